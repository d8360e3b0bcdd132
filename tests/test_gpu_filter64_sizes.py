"""FP64 filter on both sides of the lines between the star in fixed point (one, two or three parts of the
block) and the FP64 star, and narrow blocks of a grid that is wide enough for the former.

Reference: 16^3 bricks of the same points, which always run the FP64 star.  Tolerance: both stars round
each of their ~45 operations of magnitude <= 50 max|y| to 2^-53 of it at most; over the m = 4 steps
of a filter that damps, below 1e-12 of the column's maximum."""
import numpy as np
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


# 17,557 points: lines at 3.04 (one part), 25.8 (two) and 48.6 (three) columns; 97,569 points: 0.5
@pytest.mark.parametrize("radius,widths", [(11.3, [3, 4, 25, 26, 32, 49, 64]), (20.0, [1, 2, 3, 5])])
def test_both_routes(kscf, radius, widths):
    from workloads import pseudo_params, workload
    pos, z = workload("si35h36").atoms()
    systems = {b: kscf.build_cluster(pos, z, pseudo_params(), radius, 0.7, brick=b) for b in (8, 16)}
    n = systems[8][0].info["n_points"]
    for k in widths:
        P = torch.tensor(np.random.default_rng(k).standard_normal((n, k)), device="cuda")
        out = []
        for grid, ham in systems.values():
            X = torch.zeros((ham.n_slots, (k + 31) // 32 * 32), dtype=torch.float64, device="cuda")[:, :k]
            kscf.kscf_points_to_slots(ham, P, X)
            _, hi = kscf.kscf_spectral_bounds(ham)
            kscf.kscf_chebyshev_filter(ham, X, 4, 1.0, hi, -2.0)
            lex, _ = grid.slots()
            assert torch.all(X[torch.tensor(lex < 0, device="cuda")] == 0)
            out.append(kscf.kscf_slots_to_points(ham, X, torch.empty_like(P)))
        assert torch.all((out[0] - out[1]).abs().amax(0) <= 1e-12 * out[1].abs().amax(0))
