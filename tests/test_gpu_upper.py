"""Cholesky-QR in tensor mode where the rotation leaves out the zero blocks below the diagonal of
R^-1 (column tiles of 256): the edges of a tile, several tiles and a ragged last one.

Bars as for the other tensor-mode tests: FP32 products of unit-norm columns leave |Q^T Q - I| at a
few 1e-7 (bar 2e-6), and the span differs from X's by its FP32 rounding times cond(X) ~ 3 (1e-4)."""
import numpy as np
import pytest

from helpers import from_slots, small_cluster, subspace_gap, to_slots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("k", [255, 256, 257, 288, 513, 600])
def test_upper_rotation(species, k):
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf
    from workloads import random_block_lex
    pos, z = small_cluster()
    g, H = kscf.build_cluster(pos, z, species, 9.0, 0.7)
    lex, n = g.slots()[0], g.info["n_points"]
    X = random_block_lex(k, n, k)
    X[:, 1:] += 0.3 * X[:, :-1]        # R^-1 dense above the diagonal
    Xf = torch.tensor(to_slots(X, lex), dtype=torch.float32, device="cuda")
    kscf.kscf_orthonormalize(H, Xf, mode=kscf.KSCF_GEMM_TENSOR)
    gf = from_slots(Xf.double().cpu().numpy(), lex, n)
    h3 = 0.7 ** 3
    assert np.max(np.abs(h3 * gf.T @ gf - np.eye(k))) < 2e-6
    assert subspace_gap(gf, X, h3) < 1e-4
