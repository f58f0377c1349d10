"""The encoder's kernels over their paddings of the inputs (4, 8, 12, 16),
warp tiles (32 rows) and many tiles per warp: rows come out bitwise the same
in any batch, and a batch's gradient is the sum of its parts' and the
oracle's."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


def _setup(ctx, K, n):
    import torch
    rng = W.rng_streams(170 + K, 6)
    pyr = W.make_pyramid(rng[0], 64, 64, 7, dtype=np.float32)
    model = W.make_model(rng[1], (14, 16, 16, 3), None)
    enc = W.make_mlp(rng[2], (K, 32, 32, 8))
    mat = ctx.material(64, 64, 7, pyr, None, model["decoder"], precision=0, trainable=True, encoder=enc)
    q = W.uniform_queries(rng[3], n, 6.0)
    attrs = rng[4].uniform(0, 1, (n, K)).astype(np.float32)
    dl = rng[5].normal(0, 1, (n, 3)).astype(np.float32)
    dirs = {k: v for k, v in to_device(q).items() if k not in ("u", "v", "lod", "xi")}
    return mat, pyr, model, enc, q, attrs, dl, dirs, torch.from_numpy(attrs).cuda(), torch.from_numpy(dl).cuda()


def _gradient(ctx, mat, K, dirs, attrs, dl, pieces):
    import torch
    from paper_2305_02678_gb300 import binding as B
    total = torch.zeros(B.encoder_param_count(K), device="cuda", dtype=torch.float64)
    for a, b in pieces:
        gp = torch.zeros(mat.info.n_params, device="cuda")
        ge = torch.zeros(B.encoder_param_count(K), device="cuda")
        B.nam_backward_encoded(ctx.h, mat.h, {k: t[a:b].contiguous() for k, t in dirs.items()}, attrs[a:b].contiguous(),
                               b - a, dl[a:b].contiguous(), gp, ge, torch.cuda.current_stream(), B.NAM_OUT_COSINE)
        total += ge
    return total


@pytest.mark.parametrize("K,n", [(1, 31), (4, 33), (5, 128), (8, 129), (9, 64), (12, 1000), (13, 257), (16, 4099)])
def test_matches_oracle(gctx, oracle, K, n):
    import torch
    from paper_2305_02678_gb300 import binding as B
    mat, pyr, model, enc, q, attrs, dl, dirs, da, dd = _setup(gctx, K, n)
    z = torch.empty((n, 8), device="cuda")
    B.nam_encode(gctx.h, mat.h, da, n, z, torch.cuda.current_stream())
    k64 = attrs.astype(np.float64)
    z64 = oracle.encoder_forward(enc, k64)
    mag = oracle.encoder_forward([(np.abs(Wl), np.abs(bl)) for Wl, bl in enc], k64)
    # sums of up to 1 + 32 terms in FP32 over three layers, against their terms' magnitude
    assert (np.abs(z.cpu().numpy() - z64) / mag).max() <= 100 * 2.0 ** -24
    om = oracle.Model(64, 64, 7, pyr, None, model["decoder"], out_cosine=True)
    g = oracle.grad(om, dict(q, z=z64), dl.astype(np.float64), with_pyramid=False, with_z=True)
    ref = oracle.flat_encoder(oracle.encoder_grad(enc, k64, g["z"]))
    got = _gradient(gctx, mat, K, dirs, da, dd, [(0, n)]).cpu().numpy()
    err = np.abs(got - ref) / (np.abs(ref) + 1e-2 * np.abs(ref).max())
    assert err.max() <= 1e-4
    mat.destroy()
    gctx.check()


@pytest.mark.parametrize("K", [4, 7, 16])
def test_many_tiles_per_warp(gctx, K):
    import torch
    from paper_2305_02678_gb300 import binding as B
    n = 170001
    mat, *_, dirs, da, dd = _setup(gctx, K, n)
    z = torch.empty((n, 8), device="cuda")
    B.nam_encode(gctx.h, mat.h, da, n, z, torch.cuda.current_stream())
    part = torch.empty((n, 8), device="cuda")
    for a in range(0, n, 20011):
        b = min(n, a + 20011)
        B.nam_encode(gctx.h, mat.h, da[a:b].contiguous(), b - a, part[a:b], torch.cuda.current_stream())
    assert torch.equal(z, part)
    whole = _gradient(gctx, mat, K, dirs, da, dd, [(0, n)])
    parts = _gradient(gctx, mat, K, dirs, da, dd, [(a, min(n, a + 9001)) for a in range(0, n, 9001)])
    # FP32 sums of 170,000 terms in two orders, cancelling to about sqrt(n) of them
    assert float((whole - parts).norm()) <= 5e-5 * float(parts.norm())
    mat.destroy()
    gctx.check()
