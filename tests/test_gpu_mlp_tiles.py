"""MLP forward and gradient at the sizes where the tile of a block changes (64 or 112 points, one
or several per block), against the oracle with the bars of the other gradient test: 5e-5 for
the output (FP32 products of 128 terms of size ~1) and 1e-4 of the largest gradient entry."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n", [1, 63, 64, 65, 9728, 9729, 17024, 17025])
def test_tiles(n):
    from oracle import learned as L
    from paper_2303_00790_gb300.build import build
    build()
    from paper_2303_00790_gb300 import kscf
    rng = np.random.default_rng(n)
    p = L.unpack(0.1 * rng.standard_normal(L.N_PARAMS).astype(np.float32).astype(np.float64))
    x = rng.standard_normal((n, 32)).astype(np.float32).astype(np.float64)
    t = rng.standard_normal(n).astype(np.float32).astype(np.float64)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    P, D, T = dev(L.pack(p)), dev(x), dev(t)
    mu, sd = torch.zeros(32, device="cuda"), torch.ones(32, device="cuda")
    y = kscf.kscf_mlp_forward(P, mu, sd, D).cpu().numpy()
    assert np.max(np.abs(y - L.forward(p, x)[0])) < 5e-5
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    g = kscf.kscf_mlp_loss_grad(P, mu, sd, D, T, loss=loss).cpu().numpy()
    ref, gr = L.loss_and_grad(p, x, t)
    gr = L.pack(gr)
    assert abs(loss.item() - ref) < 1e-5 * ref
    assert np.max(np.abs(g - gr)) < 1e-4 * np.max(np.abs(gr)) + 1e-7
