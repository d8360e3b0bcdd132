"""FP64 rotation in row panels (a panel's digits fit 1 GiB): the columns' units come from all rows,
so that a panel boundary changes nothing.

Tolerance as for one panel: kin products of values rounded to 2^-56 of their row's and column's bound
2^E (at most twice the largest element), one rounding of the result and kin roundings of the FP64 reference:
2 kin 2^-54.9 max|a| max|q| 4 + kin 2^-53 sum|a q|, below kin 2^-51 * 4 max|a| max|q| with the row's and
column's maxima."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

KIN, KOUT = 850, 40
PANEL = (1 << 30) // (14 * 128 * 864) * 128      # rows whose digits (864 = 27 * 32 columns) fit


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


def operands(rows):
    gen = torch.Generator(device="cuda").manual_seed(rows)
    A = torch.randn((rows, KIN), generator=gen, dtype=torch.float64, device="cuda")
    A[-1] *= 1e6                                     # the columns' largest elements are in the last panel
    Q = torch.randn((KIN, KOUT), generator=gen, dtype=torch.float64, device="cuda")
    return A, Q


def bound(A, Q):
    """Per element: the rows are held relative to the columns' maxima."""
    c = A.abs().amax(0)
    row = (A.abs() / c).amax(1)
    return KIN * 2.0 ** -49 * row[:, None] * (Q.abs() * c[:, None]).amax(0)[None, :]


@pytest.mark.parametrize("rows", [PANEL - 1, PANEL, PANEL + 1, 2 * PANEL + 77])
def test_panels(kscf, rows):
    A, Q = operands(rows)
    assert kscf.kscf_gemm_workspace_size(1, rows, KIN, KOUT, kscf.KSCF_F64, kscf.KSCF_GEMM_NATIVE) < 1100 << 20
    err = (kscf.kscf_rotate(A, Q) - A @ Q).abs()
    assert torch.all(err <= bound(A, Q))


def test_nan_in_the_last_panel(kscf):
    """The whole product then takes the FP64 kernel."""
    A, Q = operands(PANEL + 500)
    A[-3, 5] = float("nan")
    got = kscf.kscf_rotate(A, Q)
    assert torch.equal(torch.isnan(got).any(1).nonzero()[:, 0].cpu(), torch.tensor([A.shape[0] - 3]))
    fine = ~torch.isnan(got)
    ref = torch.nan_to_num(A) @ Q
    assert torch.all(((got - ref).abs() <= KIN * 2.0 ** -50 * (A.nan_to_num().abs() @ Q.abs()))[fine])

