"""GPU parity: the rank predictor's gradient at the edges of its 32-sample tiles and of its grid (one tile per
CTA, then several), against FP64 automatic differentiation."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 31, 32, 33, 2048, 2080, 16384, 40001])
def test_gradient_at_tile_edges(batch):
    import paper_1707_05141_gb300 as bs
    bs.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(batch)
    h, f = 64, bs.SKETCH_FEATURES
    x = torch.randn(batch, f, generator=g, device="cuda")
    target = torch.rand(batch, generator=g, device="cuda") * 4
    params = torch.randn(bs.MLP_PARAMS, generator=g, device="cuda") * 0.2
    grad, loss = torch.full_like(params, 7.0), torch.full((1,), 7.0, device="cuda")
    bs.bsvd_mlp_grad(x, target, params, grad, loss)
    p = params.double().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(p, [h * f, h, h * h, h, h, 1])
    y = torch.relu(torch.relu(x.double() @ w1.view(h, f).T + b1) @ w2.view(h, h).T + b2) @ w3 + b3
    ref = ((y - target.double()) ** 2).sum() / (2 * batch)
    ref.backward()
    # every entry is a sum of `batch` products with |sum| well below the sum of magnitudes: FP32 sums in
    # chains of at most 32 * ceil(tiles / CTAs) + the CTAs' additions stay within a few hundred u of the largest
    assert (grad.double() - p.grad).abs().max() <= 2e-5 * p.grad.abs().max()
    assert abs(loss.item() - ref.item()) <= 2e-5 * ref.item()
