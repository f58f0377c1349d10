"""Launches of many tiles per CTA: the operand buffers between the fetch and
the chain warpgroups are used over and over, and every query must come out
bitwise as in launches of one tile per CTA (where no buffer is used twice)."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


def _pieces(mat, dq, n, size):
    import torch
    return torch.cat([mat.eval({k: t[a:a + size] for k, t in dq.items()}) for a in range(0, n, size)])


@pytest.mark.parametrize("precision,H,NH,frame,filt,latent", [
    (1, 64, 2, (8, 16, 6), 0, np.float16),
    (1, 64, 3, (8, 12), 1, np.float16),
    (2, 64, 2, (8, 16, 6), 0, np.float16),
    (1, 32, 2, (8, 12), 0, np.float16),
    (1, 16, 2, None, 1, np.float32),
    (1, 16, 2, (8, 16, 6), 0, np.float16),
    (1, 64, 2, (8, 16, 6), 0, np.float32),
    (2, 64, 3, (8, 12), 0, np.float32),
    (0, 64, 2, (8, 16, 6), 0, np.float16),
    (0, 64, 3, (8, 12), 1, np.float32),
    (0, 32, 2, None, 0, np.float32),
    (0, 16, 2, (8, 12), 0, np.float16),
])
def test_many_tiles_per_cta(gctx, precision, H, NH, frame, filt, latent):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = W.rng_streams(141, 3)
    pyr = W.make_pyramid(rng[0], 128, 128, 8, dtype=latent)
    nin = 20 if frame == (8, 12) else 14
    model = W.make_model(rng[1], (nin,) + (H,) * NH + (3,), frame)
    kw = {"act_scale": np.full(NH + 1, 0.004, np.float32)} if precision == 2 else {}
    mat = gctx.material(128, 128, 8, pyr, model["frame"], model["decoder"], precision=precision, filter=filt, **kw)
    n = sms * 128 * 33 + 77
    dq = to_device(W.uniform_queries(rng[2], n, 7.0))
    whole = mat.eval(dq)
    assert torch.equal(whole, _pieces(mat, dq, n, sms * 128))
    mat.destroy()
    gctx.check()


def test_many_chunks_per_cta_mixed_materials(gctx):
    """Materials of very different sizes, so that chains of one CTA hold, give
    up and reload weight slots while their operands arrive."""
    import torch
    from paper_2305_02678_gb300 import binding as B
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = W.rng_streams(142, 30)
    mats = []
    for k in range(12):
        model = W.make_model(rng[k], (14, 64, 64, 3), (8, 16, 6))
        mats.append(gctx.material(64, 64, 7, W.make_pyramid(rng[12 + k], 64, 64, 7, dtype=np.float16), model["frame"],
                                  model["decoder"]))
    n = sms * 128 * 9 + 5
    dq = to_device(W.uniform_queries(rng[24], n, 6.0))
    ids = np.minimum(rng[25].geometric(0.35, n) - 1, 11).astype(np.int32)
    out = torch.empty((n, 3), device="cuda")
    B.nam_eval_binned(gctx.h, [m.h for m in mats], dq, torch.from_numpy(ids).cuda(), n, out,
                      torch.cuda.current_stream())
    for k, m in enumerate(mats):
        idx = torch.from_numpy(np.nonzero(ids == k)[0]).cuda()
        sub = {f: t[idx].contiguous() for f, t in dq.items()}
        assert torch.equal(out[idx], _pieces(m, sub, idx.numel(), sms * 128)), k
        m.destroy()
    gctx.check()


@pytest.mark.parametrize("latent", [np.float16, np.float32])
def test_sampler_many_tiles_per_cta(gctx, latent):
    import torch
    from paper_2305_02678_gb300 import binding as B
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = W.rng_streams(143, 5)
    model = W.make_model(rng[0], (14, 16, 16, 3), None)
    mat = gctx.material(128, 128, 8, W.make_pyramid(rng[1], 128, 128, 8, dtype=latent), None, model["decoder"],
                        sampler=W.make_mlp(rng[2], (11, 32, 32, 32, 9)))
    n, size = sms * 128 * 20 + 33, sms * 128
    dq = to_device(W.uniform_queries(rng[3], n, 7.0))
    u = torch.from_numpy(rng[4].random((n, 3), dtype=np.float32)).cuda()

    def sample(a, b):
        wo, pdf = torch.empty((b - a, 3), device="cuda"), torch.empty(b - a, device="cuda")
        B.nam_sample(gctx.h, mat.h, {k: t[a:b] for k, t in dq.items()}, b - a, u[a:b], wo, pdf,
                     torch.cuda.current_stream())
        return wo, pdf

    wo, pdf = sample(0, n)
    parts = [sample(a, min(a + size, n)) for a in range(0, n, size)]
    assert torch.equal(wo, torch.cat([p[0] for p in parts]))
    assert torch.equal(pdf, torch.cat([p[1] for p in parts]))
    mat.destroy()
    gctx.check()


@pytest.mark.parametrize("nmat,n", [(3, 2048), (700, 2049), (4096, 300007)])
@pytest.mark.parametrize("coherent", [False, True])
def test_binning_segments_and_bad_ids(gctx, nmat, n, coherent):
    """Material counts up to the limit, partly filled segments, runs of one
    material, and ids outside the range at both ends of int32."""
    import torch
    from paper_2305_02678_gb300 import binding as B
    from paper_2305_02678_gb300 import NamError
    rng = W.rng_streams(144, 6)
    two = [gctx.material(32, 32, 6, W.make_pyramid(rng[k], 32, 32, 6, dtype=np.float16), None,
                         W.make_model(rng[2 + k], (14, 16, 16, 3), None)["decoder"]) for k in range(2)]
    handles = [two[k % 2].h for k in range(nmat)]
    dq = to_device(W.uniform_queries(rng[4], n, 5.0))
    ids = rng[5].integers(0, nmat, n).astype(np.int32)
    if coherent:
        ids = np.repeat(ids, 200)[:n].copy()
    bad = rng[5].integers(0, n, 9)
    ids[bad] = np.resize(np.array([-1, nmat, -2 ** 31, 2 ** 31 - 1], np.int64), 9).astype(np.int32)
    ref = torch.stack([m.eval(dq) for m in two])
    ok = (ids >= 0) & (ids < nmat)
    want = torch.full((n, 3), -7.0, device="cuda")
    idx = torch.from_numpy(np.nonzero(ok)[0]).cuda()
    want[idx] = ref[torch.from_numpy(ids[ok] % 2).long().cuda(), idx]
    for call in (B.nam_eval_binned, B.nam_eval_select):
        out = torch.full((n, 3), -7.0, device="cuda")
        call(gctx.h, handles, dq, torch.from_numpy(ids).cuda(), n, out, torch.cuda.current_stream())
        assert torch.equal(out, want)
        with pytest.raises(NamError):
            gctx.check()
    for m in two:
        m.destroy()
    gctx.check()
