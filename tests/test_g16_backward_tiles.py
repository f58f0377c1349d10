"""Reverse mode over many tiles per CTA, at the edges of its tiles and with
waits that run out: the gradient of a batch is the sum of its parts'."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


def _setup(ctx, seed, H, frame, filt, albedo, n, levels=8):
    import torch
    rng = W.rng_streams(seed, 4)
    size = 1 << (levels - 1)
    pyr = W.make_pyramid(rng[0], size, size, levels, dtype=np.float32)
    model = W.make_model(rng[1], (14, H, H, 6 if albedo else 3), (8, 16, 6) if frame else None)
    mat = ctx.material(size, size, levels, pyr, model["frame"], model["decoder"], precision=0, filter=filt,
                       trainable=True)
    dq = to_device(W.uniform_queries(rng[2], n, float(levels - 1)))
    dl = torch.from_numpy(rng[3].normal(0, 1, (n, 6 if albedo else 3)).astype(np.float32)).cuda()
    return mat, dq, dl


def _gradient(ctx, mat, dq, dl, pieces):
    """dL/dparams and dL/dpyramid summed in FP64 over the given (start, end)."""
    import torch
    from paper_2305_02678_gb300 import binding as B
    tp = torch.zeros(mat.info.n_params, device="cuda", dtype=torch.float64)
    tz = torch.zeros(mat.info.texels * 8, device="cuda", dtype=torch.float64)
    for a, b in pieces:
        gp = torch.zeros(mat.info.n_params, device="cuda")
        gz = torch.zeros(mat.info.texels * 8, device="cuda")
        B.nam_backward(ctx.h, mat.h, {k: t[a:b].contiguous() for k, t in dq.items()}, b - a, dl[a:b].contiguous(), gp,
                       gz, torch.cuda.current_stream(), B.NAM_OUT_COSINE)
        tp += gp
        tz += gz
    return tp, tz


# A sum over 64 queries on the tensor cores takes 24 steps that each cut off
# less than 2^-23 of it, and FP32 sums of the tiles add a few times 2^-24 of
# their partial sums, which cancellation makes up to about eight times the
# result: 2e-5 of a gradient's norm.
TOL = 2e-5


def _same(g, r):
    for a, b in zip(g, r):
        assert float((a - b).norm()) <= TOL * float(b.norm())


@pytest.mark.parametrize("H,frame,filt,albedo", [
    (64, True, 0, False), (64, True, 1, True), (64, False, 0, False), (32, True, 1, False), (32, False, 0, True),
    (16, True, 0, True), (16, False, 1, False),
])
def test_many_tiles_per_cta(gctx, H, frame, filt, albedo):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    step = sms * 128
    n = 5 * step + 77
    mat, dq, dl = _setup(gctx, 161, H, frame, filt, albedo, n)
    whole = _gradient(gctx, mat, dq, dl, [(0, n)])
    _same(whole, _gradient(gctx, mat, dq, dl, [(a, min(n, a + step)) for a in range(0, n, step)]))
    _same(whole, _gradient(gctx, mat, dq, dl, [(a, min(n, a + 9001)) for a in range(0, n, 9001)]))
    mat.destroy()
    gctx.check()


@pytest.mark.parametrize("levels", [1, 3, 5])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 129, 193])
def test_tile_edges_on_small_pyramids(gctx, n, levels):
    """Textures that lie wholly or in part in the coarse levels' shared sums."""
    mat, dq, dl = _setup(gctx, 162 + n, 64, True, 0, False, n, levels)
    whole = _gradient(gctx, mat, dq, dl, [(0, n)])
    _same(whole, _gradient(gctx, mat, dq, dl, [(k, k + 1) for k in range(n)]))
    mat.destroy()
    gctx.check()


def test_short_wait_limit_reports_timeout():
    """A 1 ns limit makes waits give up; the kernel drains its MMAs, frees its
    TMEM and reports, and the next context's gradient is right."""
    import torch
    from paper_2305_02678_gb300 import Context
    from paper_2305_02678_gb300 import binding as B
    n = 100000
    with Context(0, wait_timeout_ns=1) as short:
        mat, dq, dl = _setup(short, 163, 64, True, 0, False, n)
        for _ in range(3):
            _gradient(short, mat, dq, dl, [(0, n)])
        with pytest.raises(B.NamError) as e:
            short.check()
        assert e.value.status == B.NAM_ERR_TIMEOUT
        short.check()  # the error word was cleared (no launch since)
        mat.destroy()
    with Context(0) as ok:
        mat, dq, dl = _setup(ok, 163, 64, True, 0, False, n)
        _same(_gradient(ok, mat, dq, dl, [(0, n)]), _gradient(ok, mat, dq, dl, [(0, 40001), (40001, n)]))
        ok.check()
        mat.destroy()
