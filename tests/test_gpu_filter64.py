"""FP64 filter and apply in fixed point on 8^3 bricks: ragged widths (chunks of four columns, column
sub-blocks), columns of very different magnitudes, zeros, and values the fixed point cannot hold.

Reference: the generic FP64 star (16^3 bricks of the same points run it).  Tolerance per column:
the fixed point rounds to 2^-57 of the column's largest value within two bricks, the FP64 star to
2^-53 after each of its ~45 operations of magnitude <= 50 max|y|; both together stay below
1e-13 max|H y| (the tolerance of the apply tests) and, amplified over the m <= 6 steps of a filter
that damps, below 1e-12 of the column's maximum."""
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


@pytest.fixture(scope="module")
def systems(kscf):
    from workloads import pseudo_params, workload
    pos, z = workload("si35h36").atoms()
    return {b: kscf.build_cluster(pos, z, pseudo_params(), 11.3, 0.7, brick=b) for b in (8, 16)}


def block(n, k, kind):
    rng = np.random.default_rng(k)
    P = rng.standard_normal((n, k))
    if kind == "columns":
        P *= 10.0 ** rng.uniform(-120, 120, k)
        P[:, k // 2] = 0.0
    if kind == "tails":        # decays by 1e-60 across the sphere
        P *= np.exp(-np.linspace(0, 138, n))[:, None]
    return torch.tensor(P, device="cuda")


def run(kscf, system, P, degree, width):
    grid, ham = system
    n, k = P.shape
    X = torch.zeros((ham.n_slots, (k + 31) // 32 * 32), dtype=torch.float64, device="cuda")[:, :k]
    kscf.kscf_points_to_slots(ham, P, X)
    if degree == 0:
        X = kscf.kscf_hamiltonian_apply(ham, X, torch.full_like(X, 7.0))
    else:
        _, hi = kscf.kscf_spectral_bounds(ham)
        kscf.kscf_chebyshev_filter(ham, X, degree, 1.0, hi, -2.0, block=width)
    return kscf.kscf_slots_to_points(ham, X, torch.empty_like(P))


@pytest.mark.parametrize("kind", ["normal", "columns", "tails"])
@pytest.mark.parametrize("degree,k,width", [(0, 29, 0), (0, 64, 0), (1, 1, 0), (2, 3, 0), (6, 33, 0), (5, 101, 32), (3, 64, 0)])
def test_against_fp64_star(kscf, systems, kind, degree, k, width):
    P = block(systems[8][0].info["n_points"], k, kind)
    got, ref = run(kscf, systems[8], P, degree, width), run(kscf, systems[16], P, degree, width)
    top = ref.abs().amax(0)
    err = (got - ref).abs().amax(0)
    assert torch.all(err <= (1e-13 if degree == 0 else 1e-12) * top)
    assert torch.all(err[top == 0] == 0)


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e-290])
def test_values_outside_the_fixed_point(kscf, systems, bad):
    """A NaN or Inf spreads exactly as in the FP64 star; a column of tiny values keeps its digits."""
    P = block(systems[8][0].info["n_points"], 20, "normal")
    if np.isfinite(bad):
        P[:, 4] *= bad
    else:
        P[1234, 4] = bad
    got, ref = run(kscf, systems[8], P, 2, 0), run(kscf, systems[16], P, 2, 0)
    assert torch.equal(torch.isfinite(got), torch.isfinite(ref))
    assert torch.equal(torch.isnan(got), torch.isnan(ref))
    fine = torch.isfinite(ref)
    top = torch.where(fine, ref.abs(), 0.0).amax(0)
    assert torch.all(torch.where(fine, (got - ref).abs(), 0.0).amax(0) <= 1e-12 * top)


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-13), (torch.float32, 2e-5)])
def test_projections_of_wide_blocks(kscf, systems, dtype, tol):
    """The projections' kernel for many columns gives the columns what the one for few gives them
    (the same sums in another order; the apply tests' tolerances)."""
    grid, ham = systems[8]
    k = 35 * 220 if dtype == torch.float32 else 35 * 110     # above the wide variant's CTA count
    P = block(grid.info["n_points"], 40, "normal").to(dtype)
    few = torch.zeros((ham.n_slots, 64), dtype=dtype, device="cuda")[:, :40]
    kscf.kscf_points_to_slots(ham, P, few)
    many = torch.zeros((ham.n_slots, (k + 31) // 32 * 32), dtype=dtype, device="cuda")[:, :k]
    many[:, k - 40:] = few
    a = kscf.kscf_hamiltonian_apply(ham, few, torch.empty_like(few))
    b = kscf.kscf_hamiltonian_apply(ham, many, torch.empty_like(many))[:, k - 40:]
    assert (a - b).abs().max() <= tol * a.abs().max()
