"""The weight gradients' sums over queries against 64 bits: no component along
the gradient, as a sum of roundings to nearest has none."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [16, 32, 64])
def test_weight_gradients_are_not_shortened(gctx, oracle, H):
    import torch
    from paper_2305_02678_gb300 import binding as B
    along = []
    for seed in range(4):
        rng = W.rng_streams(230 + seed, 4)
        size, L, n = 256, 9, 6000
        pyr = W.make_pyramid(rng[0], size, size, L, dtype=np.float32)
        model = W.make_model(rng[1], (14, H, H, 3), None)
        q = W.uniform_queries(rng[2], n, 6.0)
        dl = rng[3].normal(1, 1, (n, 3)).astype(np.float32)  # sums that do not cancel
        ref = oracle.grad(oracle.Model(size, size, L, pyr, None, model["decoder"], out_cosine=True), q,
                          dl.astype(np.float64), with_pyramid=False)["decoder"]
        mat = gctx.material(size, size, L, pyr, None, model["decoder"], precision=0, trainable=True)
        gp = torch.zeros(mat.info.n_params, device="cuda")
        B.nam_backward(gctx.h, mat.h, to_device(q), n, torch.from_numpy(dl).cuda(), gp, None,
                       torch.cuda.current_stream(), B.NAM_OUT_COSINE)
        e = gp.cpu().numpy().astype(np.float64) - ref
        for a, b in ((0, 14 * H), (15 * H, 15 * H + H * H)):  # W1, W2
            along.append(np.dot(e[a:b], ref[a:b]) / np.dot(ref[a:b], ref[a:b]))
        mat.destroy()
    # half an ulp at most, of sums that each take about a hundred roundings of
    # either sign
    assert abs(np.mean(along)) <= 2.0 ** -24
    gctx.check()
