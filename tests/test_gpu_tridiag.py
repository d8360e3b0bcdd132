"""Eigensolver at the sizes where the tridiagonalisation's paths change, against the residual and
orthogonality of the eigenpairs.  n = 2 .. 9: a cluster with CTAs that own no row or one; 159 .. 161:
the last cluster and the first grid; 305, 609: around one more row per CTA; 1023 .. 1026: more
elements than the registers hold; 1800, 2000: rows in shared and in global memory; 7100: the row
work vectors in global memory.

Bar: |A Z - Z w| and |Z^T Z - I| are O(n u) max|A| for a backward-stable solver; with a constant of
16 that is 16 n 2^-53, and 64 u below n = 4 (|A| <= 1 here, so its norm is at most n)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 7, 8, 9, 33, 64, 159, 160, 161, 305, 609, 1023, 1024, 1025, 1026, 1800, 2000, 7100])
def test_eigenpairs(kscf, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    B = torch.rand((n, n), dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    A = (B + B.T) / 2
    Zt = A.clone()
    w = kscf.kscf_sym_eig(Zt)          # row j: eigenvector j
    tol = 16 * max(n, 4) * 2.0 ** -53
    assert bool((w[1:] >= w[:-1]).all())
    assert float((Zt @ A - w[:, None] * Zt).abs().max()) <= tol
    assert float((Zt @ Zt.T - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max()) <= tol
    if n <= 609:                       # sums in a fixed order: the same bits again
        Z2 = A.clone()
        w2 = kscf.kscf_sym_eig(Z2)
        assert torch.equal(w, w2) and torch.equal(Zt, Z2)
