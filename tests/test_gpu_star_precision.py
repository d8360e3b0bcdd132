"""The FP64 star of the filter and of wide applies, point by point: values far below the largest
of their neighbourhood keep their digits.

Reference: the star in extended precision.  Tolerance per point, with T = sum |w v| over the star's own 37
values and u = 2^-53.  Fixed point: a value is cut by less than 2^-60 2^E (2^E: above the largest value of
the brick and its neighbours), which the weights of one sign, 10.6 in all, turn into 10.6 units, and the sum
by 2.9 units; it is used where 1.71 (5 |v_0| + sum |v_1|) >= 1.71 2^-6 2^E, a lower bound of T, so
13.5 2^-60 2^E <= 4 u T.  Elsewhere more bits, or the FP64 star: a rounding in each of 18 pairs and 19
sums, 20 u T.  Three roundings of the result come on top: 24 u T.  Y_1 of the filter adds c v, rounded
three times.  Below the normal numbers each of the 40 roundings is to a multiple of 2^-1074 instead."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

H, RADIUS, U = 0.7, 11.3, 2.0 ** -53
SPECIES = [{"z_number": 1, "z_valence": 1.0, "r_c": 0.8, "a_gauss": 0.0, "r_gauss": 1.0, "n_proj": 0, "e_s": 0.0,
            "e_p": 0.0, "r_p": 1.0, "r_cut": 3.5, "r_start": 0.7}]
WEIGHTS = [np.longdouble(2 * (-1) ** (j + 1) * math.factorial(6) ** 2)
           / (j * j * math.factorial(6 - j) * math.factorial(6 + j)) for j in range(1, 7)]


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


def box():
    m = int(math.floor(RADIUS / H + 1e-9))
    c = np.arange(-m, m + 1) * H
    xyz = np.stack(np.meshgrid(c, c, c, indexing="ij"))
    return xyz, (xyz ** 2).sum(0) <= RADIUS ** 2 + 1e-9 * H * H


def fields(xyz, kind):
    rng = np.random.default_rng(3)
    k = 24
    out = np.empty((k,) + xyz.shape[1:])
    for j in range(k):
        d = xyz - rng.uniform(-6, 6, 3)[:, None, None, None]
        r = np.sqrt((d ** 2).sum(0))
        if kind == "orbitals":       # exp(-kappa r), some times a wave, some with noise on top
            out[j] = np.exp(-[0.5, 1.0, 1.5, 2.5][j % 4] * r)
            if j % 3 == 1:
                out[j] *= np.cos(1.1 * xyz[0] + 0.4 * xyz[1])
            if j % 3 == 2:
                out[j] *= rng.standard_normal(r.shape)
        elif kind == "gaussians":
            out[j] = np.exp(-(0.3 + 0.2 * j) * r ** 2)
        else:                        # waves: few points stand out, at their nodes and at the surface
            q = rng.normal(0, 0.6, 3)
            out[j] = np.cos(np.tensordot(q, xyz, 1) + j) * np.sin(0.3 * xyz[2] + 0.1 * j)
    return out


def star(f):
    """-1/2 Lap f and sum |w f| / (2 h^2), order 12, zero outside."""
    f = f.astype(np.longdouble)
    w0 = -2 * sum(WEIGHTS)
    out, size = 3 * w0 * f, 3 * abs(w0) * abs(f)
    for ax in range(1, 4):
        n = f.shape[ax]
        for j, w in enumerate(WEIGHTS, 1):
            a = [slice(None)] * 4
            b = [slice(None)] * 4
            a[ax], b[ax] = slice(j, n), slice(0, n - j)
            for x, y in ((tuple(a), tuple(b)), (tuple(b), tuple(a))):
                out[y] += w * f[x]
                size[y] += abs(w) * abs(f[x])
    h2 = 2 * np.longdouble(H) ** 2
    return -out / h2, size / h2


@pytest.mark.parametrize("kind", ["orbitals", "gaussians", "waves"])
@pytest.mark.parametrize("call", ["apply", "filter"])
def test_star_point_by_point(kscf, kind, call):
    xyz, inside = box()
    f = np.where(inside, fields(xyz, kind), 0.0)
    # points in lexicographic order, x fastest
    P = torch.tensor(np.ascontiguousarray(f.transpose(0, 3, 2, 1)[:, inside.transpose(2, 1, 0)].T), device="cuda")
    z = np.array([1], dtype=np.int32)
    grid, ham = kscf.build_cluster(np.zeros((1, 3)), z, SPECIES, RADIUS, H, center=np.zeros(3))
    n, k = P.shape
    assert n == grid.info["n_points"] and n * k >= 1.5e5      # a narrower apply runs the FP64 star
    kscf.kscf_set_potential(ham, torch.zeros(ham.n_slots, dtype=torch.float64, device="cuda"))
    X = torch.zeros((ham.n_slots, 32), dtype=torch.float64, device="cuda")[:, :k]
    kscf.kscf_points_to_slots(ham, P, X)
    ref, size = star(f)
    tol = 24 * U * size + 40 * np.longdouble(2.0 ** -1074)
    if call == "apply":
        Y = kscf.kscf_hamiltonian_apply(ham, X, torch.full_like(X, 7.0))
    else:
        a, b, a0 = 1.0, 70.0, -2.0
        e, c = (b - a) / 2, (b + a) / 2
        scale = np.longdouble(e / (a0 - c)) / e
        Y = kscf.kscf_chebyshev_filter(ham, X, 1, a, b, a0)
        ref, tol = scale * (ref - c * f), abs(scale) * (tol + 3 * U * abs(c * f)) + 2 * U * abs(scale * (ref - c * f))
    got = kscf.kscf_slots_to_points(ham, Y, torch.empty_like(P)).cpu().numpy()
    full = np.zeros(f.shape)
    full.transpose(0, 3, 2, 1)[:, inside.transpose(2, 1, 0)] = got.T
    err = abs(np.where(inside, full - ref, 0))
    assert np.all(err <= np.where(inside, tol, 0))
