"""FP64 Gram and rotation on the tensor cores (56-bit integer digits) against exact sums.

Tolerances from the conversion alone: a value is rounded to 2^-56 of 2^E, its column's (Gram) or
row's / column's (rotation) bound, with 2^E at most twice the largest element, so a product is
off by at most 2 * 2^-56 * 2^E_a 2^E_b, the dropped digit products add less than 2^-60 of it, and
the result is rounded once more (twice with a scale): terms * 2^-54.9 * 2^(E_a + E_b) + 2^-52 |C|.
The reference adds Dekker products with math.fsum, which is exact."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

UNIT = 2.0 ** -54.9


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


def exact_dot(x, y):
    def split(a):
        t = 134217729.0 * a
        h = t - (t - a)
        return h, a - h
    p = x * y
    (xh, xl), (yh, yl) = split(x), split(y)
    return math.fsum(np.concatenate([p, ((xh * yh - p) + xh * yl + xl * yh) + xl * yl]))


def bound2(a, axis):
    """2^E with |a| < 2^E along the axis."""
    return np.ldexp(1.0, np.frexp(np.max(np.abs(a), axis=axis))[1])


def data(shape, seed, kind):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal(shape)
    if kind == "columns":      # columns of very different norms, one of zeros
        a *= 10.0 ** rng.uniform(-8, 8, (1, shape[1]))
        a[:, shape[1] // 2] = 0.0
    if kind == "constant":     # coherent digits: the largest sums an accumulator can hold
        a = np.full(shape, 1.0 - 2.0 ** -53)
    return a


@pytest.mark.parametrize("kind", ["normal", "columns", "constant"])
@pytest.mark.parametrize("rows,m,n", [(128, 1, 1), (129, 5, 7), (1000, 64, 64), (4097, 65, 129), (2500, 128, 193)])
def test_gram(kscf, rows, m, n, kind):
    A, B = data((rows, m), 1, kind), data((rows, n), 2, kind)
    At = torch.tensor(A, device="cuda")
    C = kscf.kscf_gram(At, torch.tensor(B, device="cuda"), scale=0.5).cpu().numpy()
    S = kscf.kscf_gram(At, At)
    assert torch.equal(S, S.T)
    S = S.cpu().numpy()
    ea, eb = bound2(A, 0), bound2(B, 0)
    rng = np.random.default_rng(3)
    picks = [(0, 0), (m - 1, n - 1)] + [(rng.integers(m), rng.integers(n)) for _ in range(40)]
    for i, j in picks:
        x = 0.5 * exact_dot(A[:, i], B[:, j])
        assert abs(C[i, j] - x) <= 0.5 * rows * UNIT * ea[i] * eb[j] + 2.0 ** -52 * abs(x)
        k = j % m
        x = exact_dot(A[:, i], A[:, k])
        assert abs(S[i, k] - x) <= rows * UNIT * ea[i] * ea[k] + 2.0 ** -52 * abs(x)


def test_gram_in_small_buffer(kscf):
    """Several row chunks in a buffer below the reported size, and no buffer at all."""
    rows, m = 9000, 70
    A = torch.tensor(data((rows, m), 1, "normal"), device="cuda")
    full = kscf.kscf_gram(A, A)
    need = kscf.kscf_gemm_workspace_size(0, rows, m, m, 0, 0)
    part = kscf.kscf_gram(A, A, work=torch.empty(need // 4 // 256 * 256, dtype=torch.uint8, device="cuda"))
    tiny = kscf.kscf_gram(A, A, work=torch.empty(256, dtype=torch.uint8, device="cuda"))
    assert torch.equal(full, part)          # integer sums: the same in any number of chunks
    assert (full - tiny).abs().max() <= rows * 2.0 ** -50 * A.abs().max() ** 2


@pytest.mark.parametrize("kind", ["normal", "columns", "constant"])
@pytest.mark.parametrize("rows,kin,kout", [(9000, 24, 24), (3000, 300, 300), (129, 257, 260), (777, 130, 65),
                                           (20000, 31, 64)])
def test_rotate(kscf, rows, kin, kout, kind):
    A, Q = data((rows, kin), 1, kind), data((kin, kout), 2, "normal")
    if kind == "columns":
        Q /= np.where(bound2(A, 0) > 0, bound2(A, 0), 1.0)[:, None]
    O = kscf.kscf_rotate(torch.tensor(A, device="cuda"), torch.tensor(Q, device="cuda")).cpu().numpy()
    ec = bound2(A, 0)
    er, eq = bound2(A / np.where(ec > 0, ec, 1.0), 1), bound2(Q * ec[:, None], 0)
    rng = np.random.default_rng(3)
    for r, j in [(0, 0), (rows - 1, kout - 1)] + [(rng.integers(rows), rng.integers(kout)) for _ in range(200)]:
        x = exact_dot(A[r], Q[:, j])
        assert abs(O[r, j] - x) <= kin * UNIT * er[r] * eq[j] + 2.0 ** -52 * abs(x)


@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf, 1e200])
def test_values_outside_the_digits(kscf, bad):
    """NaN, Inf and extreme magnitudes go through the FP64 kernels: the results of torch."""
    rows, k = 6000, 40
    A = torch.tensor(data((rows, k), 1, "normal"), device="cuda")
    Q = torch.tensor(data((k, k), 2, "normal"), device="cuda")
    A[77, 3] = bad
    for got, ref in ((kscf.kscf_gram(A, A), A.T @ A), (kscf.kscf_rotate(A, Q), A @ Q)):
        assert torch.equal(torch.isnan(got), torch.isnan(ref))
        fine = torch.isfinite(ref)
        assert torch.equal(fine, torch.isfinite(got))
        assert torch.allclose(got[fine], ref[fine], rtol=1e-9, atol=1e-9)
        inf = torch.isinf(ref)
        assert torch.equal(got[inf], ref[inf])
    kscf.kscf_check_status()
