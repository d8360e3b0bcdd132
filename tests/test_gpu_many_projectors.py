"""Bricks with many projector atoms: more than the 32 whose coefficients the step kernels stage in
shared memory, and more than 65,535 (point, atom) pairs in one 8^3 brick, which 16 bits cannot number.

Reference: the generic FP64 kernel, which applies H on 16^3 bricks of the same points and reads the
64-bit entry pointers.  Tolerance: both kernels round each of the at most 37 + 4 * 200 + 5 operations
of a value of H y to half a unit u = 2^-53 of a partial sum, which stays below 50 max|y| (star) plus a few
max|y| (projections of Gaussians, E h^3 |chi|^2 <= 1); max|H y| > max|y|.  So 842 * 2 * 60 u < 1.2e-11
of max|H y|; 1e-11 asks for no more than a few of the roundings not to add up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

RADIUS, H = 7.0, 0.7
SPECIES = [{"z_number": 14, "z_valence": 0.02, "r_c": 0.8, "a_gauss": 0.0, "r_gauss": 1.0, "n_proj": 4, "e_s": 0.5,
            "e_p": -0.3, "r_p": 1.0, "r_cut": 16.0, "r_start": 1.2}]


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


def systems(kscf, n_atoms):
    """The same atoms, each within r_cut of every point, on 8^3 and on 16^3 bricks."""
    rng = np.random.default_rng(5)
    pos = rng.uniform(-3.5, 3.5, (n_atoms, 3))
    z = np.full(n_atoms, 14, dtype=np.int32)
    out = {b: kscf.build_cluster(pos, z, SPECIES, RADIUS, H, brick=b, center=np.zeros(3)) for b in (8, 16)}
    lex, _ = out[8][0].slots()
    pairs = int((lex.reshape(-1, 512) >= 0).sum(1).max()) * n_atoms
    assert (pairs > 65535) == (n_atoms == 200)
    return out


def in_slots(kscf, ham, P):
    X = torch.zeros((ham.n_slots, (P.shape[1] + 31) // 32 * 32), dtype=P.dtype, device="cuda")[:, :P.shape[1]]
    return kscf.kscf_points_to_slots(ham, P, X)


def apply_reference(kscf, system, P):
    ham = system[1]
    X = in_slots(kscf, ham, P)
    Y = kscf.kscf_hamiltonian_apply(ham, X, torch.zeros_like(X))
    return kscf.kscf_slots_to_points(ham, Y, torch.empty_like(P))


def filter_reference(kscf, system, P, degree, a, b, a0):
    """The scaled Chebyshev recurrence with the reference's H."""
    e, c = (b - a) / 2, (b + a) / 2
    s1 = e / (a0 - c)
    tau, s, x = 2 / s1, s1, P
    y = (apply_reference(kscf, system, x) - c * x) * (s1 / e)
    for _ in range(2, degree + 1):
        n = 1 / (tau - s)
        x, y = y, (apply_reference(kscf, system, y) - c * y) * (2 * n / e) - s * n * x
        s = n
    return y


@pytest.mark.parametrize("n_atoms", [40, 200])
@pytest.mark.parametrize("degree", [0, 1, 3])
def test_fp64_star_kernel(kscf, n_atoms, degree):
    both = systems(kscf, n_atoms)
    n = both[8][0].info["n_points"]
    k = 40 if degree == 0 else 5
    assert degree or n * k >= 1.5e5        # a narrower apply runs the generic kernel itself
    P = torch.tensor(np.random.default_rng(k).standard_normal((n, k)), device="cuda")
    ham = both[8][1]
    X = in_slots(kscf, ham, P)
    if degree == 0:
        Y = kscf.kscf_hamiltonian_apply(ham, X, torch.full_like(X, 7.0))
        lex, _ = both[8][0].slots()
        assert torch.all(Y[torch.tensor(lex < 0, device="cuda")] == 0)      # padding rows are zeroed
        ref = apply_reference(kscf, both[16], P)
    else:
        Y = kscf.kscf_chebyshev_filter(ham, X, degree, 1.0, 80.0, -2.0)
        ref = filter_reference(kscf, both[16], P, degree, 1.0, 80.0, -2.0)
    got = kscf.kscf_slots_to_points(ham, Y, torch.empty_like(P))
    assert (got - ref).abs().max() <= 1e-11 * ref.abs().max()


@pytest.mark.parametrize("brick", [8, 16])
@pytest.mark.parametrize("n_atoms", [40, 200])
def test_fp32_filter_kernel(kscf, n_atoms, brick):
    """FP32 against the FP64 reference: the 842 roundings of a step, u = 2^-24, bound nothing useful
    when they all add up; as a random walk they give sqrt(842) * 60 u = 1.0e-4 of max|y|, three times
    over the three steps."""
    both = systems(kscf, n_atoms)
    n, k, degree = both[8][0].info["n_points"], 20, 3
    P = torch.tensor(np.random.default_rng(k).standard_normal((n, k)), device="cuda")
    ham = both[brick][1]
    X = in_slots(kscf, ham, P.float())
    kscf.kscf_chebyshev_filter(ham, X, degree, 1.0, 80.0, -2.0)
    got = kscf.kscf_slots_to_points(ham, X, torch.empty_like(P, dtype=torch.float32)).double()
    ref = filter_reference(kscf, both[16], P, degree, 1.0, 80.0, -2.0)
    assert (got - ref).abs().max() <= 3e-4 * ref.abs().max()
