"""The L1 loss (2 or 8 pixels per thread by the call's pixels) against float64, at
the edges of its rounds and of the rule."""
import numpy as np
import pytest
import torch

from oracle import render as R
from tests._util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(1, 1)], [(511, 1)], [(512, 1)], [(171, 3)], [(1024, 2048)], [(1025, 2048)],
                                   [(37, 53), (1, 513), (1024, 2000)], [(1024, 2048), (3, 5)]])
def test_loss_sizes(sizes):
    """Gradients are signs times an exactly rounded scale; the loss is a sum of at
    most 2.1M terms in trees and chains of at most 300 (1e-5 as in the loss test)."""
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context
    rng = np.random.default_rng(sum(h * w for h, w in sizes))
    ctx = Context(0)
    cu = lambda a: torch.as_tensor(a, device="cuda")
    views = []
    for h, w in sizes:
        td = rng.uniform(0.5, 4, (h, w)).astype(np.float32)
        td[rng.uniform(size=(h, w)) < 0.1] = 0.0
        td[0, 0] = 1.0
        views.append((rng.uniform(0, 1, (3, h, w)).astype(np.float32), rng.uniform(0.5, 4, (h, w)).astype(np.float32),
                      rng.uniform(0, 1, (3, h, w)).astype(np.float32), td))
    cams = [abi.make_camera(1, 1, 0, 0, w, h) for h, w in sizes]
    gc, gd = [torch.empty(v[0].shape, device="cuda") for v in views], [torch.empty(v[1].shape, device="cuda") for v in views]
    loss = torch.zeros(1, device="cuda")
    img = [[cu(v[k]) for v in views] for k in range(4)]
    abi.gs_loss_l1_batched(ctx.handle, cams, *img, 0.8, 0.2, loss, gc, gd)
    total = 0.0
    for k, v in enumerate(views):
        L, rc, rd = R.loss_image_grads(*v)
        total += float(L)
        np.testing.assert_allclose(gc[k].cpu().numpy(), rc.numpy(), rtol=1e-6, atol=0)
        np.testing.assert_allclose(gd[k].cpu().numpy(), rd.numpy(), rtol=1e-6, atol=0)
    assert abs(float(loss) - total) <= 1e-5 * total
    if len(sizes) == 1:  # the entry point without allocations takes the same sums
        one, g1, g2 = torch.zeros(1, device="cuda"), torch.empty_like(gc[0]), torch.empty_like(gd[0])
        abi.gs_loss_l1_noalloc(cams[0], img[0][0], img[1][0], img[2][0], img[3][0], 0.8, 0.2, one, g1, g2)
        assert float(one) == float(loss) and torch.equal(g1, gc[0]) and torch.equal(g2, gd[0])
    ctx.close()
