"""Hartree solve of the SCF (one cooperative CG kernel, star in fixed point) at the sizes where
its point-per-thread variants change, on 8^3 and 16^3 bricks.

The solution V is put back through the FP64 Hamiltonian of the same grid with a zero potential
and no projectors (2 H V = -Lap_h V at points whose star lies inside the sphere), a kernel that
shares nothing with the CG.  Tolerance on |2 H V - 4 pi rho|_2 / |b|_2: 1e-12 from the stop,
plus the rounding of the FP64 star, ~43 * 2^-53 |V| per point over ~3e5 points (4e-13 of
|b|_2) and the drift of the CG's recurred residual of a few 1e-13; 5e-12 in all."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

H = 0.7
SPECIES = [{"z_number": 1, "z_valence": 1.0, "r_c": 0.8, "a_gauss": 0.0, "r_gauss": 1.0, "n_proj": 0, "e_s": 0.0,
            "e_p": 0.0, "r_p": 1.0, "r_cut": 3.5, "r_start": 0.7}]


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


# radius in grid steps: 1, 2, 3 and 4 points per thread, and the variant for larger grids
@pytest.mark.parametrize("steps", [7.3, 24.0, 30.0, 36.0, 41.0, 45.0])
@pytest.mark.parametrize("brick", [8, 16])
def test_hartree_residual(kscf, steps, brick):
    radius = steps * H
    pos = np.array([[0.3, 0.1, -0.2], [1.2, -0.4, 0.6]])
    z = np.array([1, 1], dtype=np.int32)
    grid, ham = kscf.build_cluster(pos, z, SPECIES, radius, H, brick=brick, center=np.zeros(3))
    lex, ijk = grid.slots()
    xyz = torch.tensor(ijk, dtype=torch.float64, device="cuda") * H
    live = torch.tensor(lex >= 0, device="cuda")
    rho = sum(torch.exp(-((xyz - torch.tensor(c, device="cuda")).square().sum(1)) / s ** 2) * q
              for c, s, q in [((0.2, 0.3, -0.1), 1.5, 0.05), ((-2.0, 1.0, 0.5), 2.5, 0.02), ((1.0, 1.0, 1.0), 1.0, -0.03)])
    rho = torch.where(live, rho, torch.zeros_like(rho))
    scf = kscf.Scf(ham, pos, z, SPECIES, kscf.scf_params(2, 4))
    vh, it = scf.hartree(rho)
    assert it > 0
    kscf.kscf_set_potential(ham, torch.zeros_like(rho))
    V = vh[:, None].contiguous()
    HV = kscf.kscf_hamiltonian_apply(ham, V, torch.zeros_like(V))[:, 0]
    inside = live & (xyz.square().sum(1).sqrt() < (steps - 6.01) * H)   # the whole star is in the sphere
    res = (2.0 * HV - 4.0 * math.pi * rho)[inside]
    assert inside.sum() > 0
    b = (2.0 * HV)[live]     # = A V, the right-hand side with the sphere's boundary terms
    assert res.norm() <= 5e-12 * b.norm()
