"""The network kernels' tiles of 128 samples: forward pass and gradient
against the fp64 oracle network at counts around a tile, and one training
step (samples gathered in a shuffled order) against Adam on that gradient."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1001_3411_gb300 as hopgpu
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hop():
    hopgpu.build_library()
    h = hopgpu.Hop(0)
    yield h
    h.close()


def _case(m, seed):
    rng = np.random.default_rng(seed)
    p = rng.normal(0, 0.25, hopgpu.MLP_NPARAM).astype(np.float32)
    x = np.log1p(rng.poisson(4.0, (m, 27))).astype(np.float32)
    t = rng.normal(0, 1.0, m).astype(np.float32)
    return p, x, t


# fp32 products and sums of at most 64 terms per unit, summed over the
# samples: an output is within 64 roundings (64 * 2^-24 = 4e-6) of the sum of
# its terms' magnitudes, of which the largest output is at least a few percent
@pytest.mark.parametrize("m", [1, 2, 127, 128, 129, 255, 4097, 40001])
def test_forward_and_gradient_around_a_tile(hop, m):
    p, x, t = _case(m, m)
    hop.hop_mlp_load(p, 0.0)
    pb = omlp.bf16_round(p)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = hop.hop_mlp_forward(xd).cpu().numpy()
    y_o = omlp.forward(pb, x.astype(np.float64))
    assert np.max(np.abs(y - y_o)) <= 2e-5 * np.abs(y_o).max() + 1e-5
    loss, g = hop.hop_mlp_grad(xd, td)
    loss_o, g_o = omlp.loss_and_grad(pb, x.astype(np.float64), t.astype(np.float64))
    assert loss == pytest.approx(loss_o, rel=1e-4)
    assert np.linalg.norm(g.cpu().numpy() - g_o) <= 1e-4 * np.linalg.norm(g_o)


@pytest.mark.parametrize("m", [100, 300])
def test_one_training_step(hop, m):
    """One batch holding every sample: whatever the order, Adam's first step
    moves each weight by lr * sign(gradient) where the gradient is not tiny."""
    p, x, t = _case(m, 7 + m)
    hop.hop_mlp_load(p, 0.0)
    _, g_o = omlp.loss_and_grad(omlp.bf16_round(p), x.astype(np.float64), t.astype(np.float64))
    hop.hop_mlp_train(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), epochs=1, batch=m, lr=1e-3, seed=3)
    step = hop.hop_mlp_get() - p
    big = np.abs(g_o) > 1e-3 * np.abs(g_o).max()
    assert big.sum() > 1000
    np.testing.assert_allclose(step[big], -1e-3 * np.sign(g_o[big]), rtol=1e-3, atol=2e-7)
