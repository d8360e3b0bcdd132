"""Work buffers of the FP64 products stay bounded as the rows grow (no GPU)."""
import pytest


@pytest.fixture(scope="module")
def kscf():
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf as mod
    return mod


@pytest.mark.parametrize("k", [24, 850, 4600])
def test_rotation_buffer_does_not_grow_with_the_rows(kscf, k):
    """Q itself, seven 2-byte digits of Q and of one row panel of 1 GiB, rounded up to tiles."""
    sizes = [kscf.kscf_gemm_workspace_size(1, rows, k, k, kscf.KSCF_F64, kscf.KSCF_GEMM_NATIVE)
             for rows in (50_000, 234_489, 1_400_000)]
    assert sizes == sorted(sizes)
    assert sizes[-1] <= (8 * k * k + 14 * (k + 128) * (k + 32)) + (1040 << 20)
