"""GPU parity: the rank predictor's gradient with a sample of a NaN or infinite feature, or a NaN parameter: units whose
derivative is 0 take nothing from it, so that the rest of the batch keeps its gradient."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(x, target, p, f, h):
    """The gradient in 64 bits, element by element: a product with a derivative of 0 is 0."""
    w1, b1, w2, b2, w3, b3 = np.split(p, np.cumsum([h * f, h, h * h, h, h]))
    w1, w2 = w1.reshape(h, f), w2.reshape(h, h)

    def prod(d, y):   # sum over the samples of d y where d != 0
        return np.stack([np.where(d[:, i:i + 1] != 0, d[:, i:i + 1] * y, 0).sum(0) for i in range(d.shape[1])])

    with np.errstate(all="ignore"):
        z1 = (w1[None] * x[:, None]).sum(2) + b1
        h1 = np.where(z1 > 0, z1, 0)
        z2 = (w2[None] * h1[:, None]).sum(2) + b2
        h2 = np.where(z2 > 0, z2, 0)
        r = (w3 * h2).sum(1) + b3 - target
        dy = r[:, None] / len(x)
        d2 = np.where(h2 > 0, dy * w3, 0)
        d1 = np.where(d2[:, :, None] != 0, w2[None] * d2[:, :, None], 0).sum(1)
        d1 = np.where(h1 > 0, d1, 0)
        grad = np.concatenate([prod(d1, x).ravel(), d1.sum(0), prod(d2, h1).ravel(), d2.sum(0), (dy * h2).sum(0), dy.sum(0)])
    return grad, (r ** 2).sum() / (2 * len(x))


@pytest.mark.parametrize("batch", [1, 33, 64, 2049])
@pytest.mark.parametrize("what", ["nothing", "nan feature", "inf feature", "nan weight"])
def test_zero_derivatives_take_nothing(batch, what):
    import paper_1707_05141_gb300 as bs
    bs.build()
    h, f = 64, bs.SKETCH_FEATURES
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((batch, f)).astype(np.float32)
    target = rng.random(batch).astype(np.float32) * 4
    p = (rng.standard_normal(bs.MLP_PARAMS) * 0.2).astype(np.float32)
    if what == "nan feature":
        x[batch // 2, 3] = np.nan
    elif what == "inf feature":
        x[batch // 2, 3] = np.inf      # layer 2 sees infinities of both signs: NaN before its ReLU, 0 behind it
    elif what == "nan weight":
        p[h * f + h + 5 * h + 7] = np.nan
    grad, loss = torch.full((bs.MLP_PARAMS,), 7.0, device="cuda"), torch.full((1,), 7.0, device="cuda")
    bs.bsvd_mlp_grad(torch.from_numpy(x).cuda(), torch.from_numpy(target).cuda(), torch.from_numpy(p).cuda(), grad, loss)
    ref, ref_loss = _reference(x.astype(np.float64), target.astype(np.float64), p.astype(np.float64), f, h)
    assert np.isfinite(ref).all() and np.isfinite(ref_loss)
    # the bound of the gradient test over tiles: sums of `batch` FP32 products against the largest entry
    assert np.abs(grad.cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()
    assert abs(loss.item() - ref_loss) <= 2e-5 * ref_loss
