"""Parameter gradients of the closure network over sample counts around the sizes of the backward
kernel's work split: a warp's 32 samples, a block's 4 warps, and more batches than resident warps
(a warp then sums several batches in registers), against float64 autograd."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _net(p, x):
    import torch

    h = torch.nn.functional.gelu(x @ p[:224].reshape(32, 7).t() + p[224:256])
    h = torch.nn.functional.gelu(h @ p[256:1280].reshape(32, 32).t() + p[1280:1312])
    return h @ p[1312:1344] + p[1344]


@pytest.mark.parametrize("n,offset,stride", [(1, 0, 1), (31, 2, 3), (32, 0, 1), (33, 1, 2), (129, 0, 1),
                                             (40001, 0, 1), (70000, 1, 2)])
def test_loss_gradient_matches_float64(n, offset, stride):
    import torch

    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(n)
    p = np.concatenate([rng.normal(0, 1 / np.sqrt(7), 256), rng.normal(0, 1 / np.sqrt(32), 1056),
                        rng.normal(0, 0.1, 33)]).astype(np.float32)
    m = offset + (n - 1) * stride + 1
    x = rng.normal(0, 1, (m, 7)).astype(np.float32)
    smag = rng.uniform(0.5, 1.5, m).astype(np.float32)
    target = (rng.uniform(0, 0.02, m) * smag).astype(np.float32)
    weight = smag * smag
    pd, xd, td, sd, wd = (torch.from_numpy(a).cuda() for a in (p, x, target, smag, weight))
    g = torch.full((1345,), 7.0, device="cuda")  # overwritten
    loss = lbm.lbm_closure_loss_grad(pd, xd, td, sd, wd, n, offset, stride, 0.1, g)
    pe = pd.double().requires_grad_(True)
    sel = slice(offset, None, stride)
    xe, te, se, we = (a[sel].double() for a in (xd, td, sd, wd))
    nu = torch.nn.functional.softplus(_net(pe, xe)) * 0.01 / np.log(2) * se
    ref = (we * (nu - te) ** 2).sum() / we.sum()
    ref.backward()
    # the sum of |per-sample contributions| bounds what rounding to float32 can do (4e-6 of it, the
    # bound of the gradient tests): sum_s |dL/dy_s| |dy_s/dp|, estimated per parameter group by the
    # largest derivative over samples of unit inputs
    r = (2 * we * (nu - te) * se / we.sum()).abs().sum().item() * 0.01 / np.log(2)
    err = (g.double() - pe.grad).abs().max().item()
    scale = max(1.0, float(xd.abs().max())) * 2.0  # |dy/dp| <= max |x| or |h| times bounded weights
    assert err <= 4e-6 * r * scale, (err, r * scale)
    assert abs(loss - ref.item()) <= 1e-5 * ref.item()
