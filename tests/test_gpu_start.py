"""Start of the SCF on the device: the random subspace by pairs of entries (even and odd widths,
rows that start at an odd entry, one column) and the atomic density whose negligible terms are
left out (two molecules 16 bohr apart), against the oracle.

Bars: a normal value is at most 8.6 and the oracle's angle 2 pi u is rounded (2 pi 2^-53), its and
the device's functions to a few 2^-53: 8.6 * 12 * 2^-53 < 2e-14.  A density term's exponent (at
most ~100) is rounded to 4 * 2^-53 of itself: 100 * 4 * 2^-53 + the sum's rounding < 1e-13."""
import numpy as np
import pytest

from helpers import from_slots

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


@pytest.mark.parametrize("k,ld", [(1, 1), (2, 2), (3, 5), (7, 7), (8, 8), (33, 40)])
def test_random_subspace(kscf, k, ld):
    from workloads import random_block_lex
    g = kscf.kscf_build_grid((0.0, 0.0, 0.0), 4.1, 0.7, 8)
    H = kscf.kscf_build_hamiltonian(g, np.zeros((0, 3)), np.zeros(0, np.int32), [])
    lex, n = g.slots()[0], g.info["n_points"]
    for dtype, tol in ((torch.float64, 2e-14), (torch.float32, 6e-7)):
        X = torch.full((g.info["n_slots"], ld), 77.0, dtype=dtype, device="cuda")
        kscf.kscf_random_subspace(H, X[:, :k], seed=9, k=k)
        Xh = X.double().cpu().numpy()
        assert np.all(Xh[:, k:] == 77.0) and np.all(Xh[lex < 0][:, :k] == 0)
        assert np.max(np.abs(from_slots(Xh[:, :k].copy(), lex, n) - random_block_lex(9, n, k))) <= tol


def test_atomic_density(kscf, species):
    from oracle.grid import sphere_grid
    from oracle.scf import atomic_density
    dd = 1.48 / 0.529177210903 / np.sqrt(3.0)
    one = np.array([[0.0, 0.0, 0.0], [dd, dd, dd], [dd, -dd, -dd], [-dd, dd, -dd], [-dd, -dd, dd]])
    pos = np.concatenate([one - [8.0, 0, 0], one + [8.0, 0, 0]])
    z = np.array([14, 1, 1, 1, 1] * 2, dtype=np.int32)
    g, H = kscf.build_cluster(pos, z, species, 13.0, 0.7, center=np.zeros(3))
    S = kscf.Scf(H, pos, z, species, kscf.scf_params(12, 6))
    S.start(seed=1)
    rho = from_slots(S.get(kscf.KSCF_FIELD_RHO).cpu().numpy(), g.slots()[0], g.info["n_points"])
    S.free()
    ref = atomic_density(sphere_grid(np.zeros(3), 13.0, 0.7).points(), pos, z, species)
    assert np.all(np.abs(rho - ref) <= 1e-13 * ref)
