"""The training kernel at the edges of its split: batches below, at and just
past a block's rows, past the size where the partial gradients fit the
caller's scratch, and past one tile per block, against the oracle's FP64
backward (tolerance of the existing gradient test: 1e-4 of each layer's
largest gradient)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 8, 9, 48, 49, 65, 1217, 8193, 9729])
def test_gradients_at_batch_edges(nb):
    import torch

    import paper_1308_6482_gb300 as lub
    from paper_1308_6482_gb300 import build
    from paper_1308_6482_gb300.mlp import init_params, unpack
    build.build()
    rng = np.random.default_rng(100 + nb)
    x = rng.standard_normal((nb, 12)).astype(np.float32)
    t = rng.uniform(-3, 3, (nb, 4)).astype(np.float32)
    wt = rng.uniform(0, 1, (nb, 4)).astype(np.float32) if nb % 2 else None
    params = init_params(seed=4)
    params[128 * 12:128 * 13] = rng.standard_normal(128) * 0.1
    ctx = lub.Context()
    dp = torch.as_tensor(params).cuda()
    grads = torch.full_like(dp, 7.0)
    work = torch.empty(nb * lub._lib.LUB_MLP_WORK_PER_SAMPLE, device="cuda")
    guard = 1024
    rows = torch.full((nb + guard,), -3.0, device="cuda")
    lub.lub_mlp_forward_backward(ctx.h, dp, torch.as_tensor(x).cuda(), torch.as_tensor(t).cuda(),
                                 None if wt is None else torch.as_tensor(wt).cuda(), nb, grads, work, rows)
    torch.cuda.synchronize()
    assert bool((rows[nb:] == -3.0).all())
    w = {k: v.astype(np.float64) for k, v in unpack(params).items()}
    loss, g, _ = oracle.mlp_loss_grad(x.astype(np.float64), t.astype(np.float64), w,
                                      wgt=None if wt is None else wt.astype(np.float64))
    assert float(rows[:nb].double().mean().item()) == pytest.approx(loss, rel=1e-5)
    got = unpack(grads.cpu().numpy())
    for k in g:
        assert np.abs(got[k] - g[k]).max() <= 1e-4 * np.abs(g[k]).max(), k
