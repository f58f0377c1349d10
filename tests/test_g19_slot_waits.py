"""The weight slots of launches that mix materials: waits for a slot end at the
context's limit, and a slot is not reloaded while a warpgroup still reads it."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


def _materials(ctx, rng, count):
    return [ctx.material(64, 64, 7, W.make_pyramid(rng[k], 64, 64, 7, dtype=np.float16), m["frame"], m["decoder"])
            for k in range(count)
            for m in [W.make_model(rng[count + k], (14, 64, 64, 3), (8, 16, 6))]]


@pytest.mark.parametrize("entry", ["nam_eval_binned", "nam_eval_select"])
def test_short_wait_limit_reports_timeout(entry):
    """Every chain of a CTA wants another material, more of them than there are
    slots, and no wait may last: the launches end with an error status, and a
    context with the default limit then evaluates the same queries."""
    import torch
    from paper_2305_02678_gb300 import Context
    from paper_2305_02678_gb300 import binding as B
    call = getattr(B, entry)
    rng = W.rng_streams(191, 18)
    n = 200000
    dq = to_device(W.uniform_queries(rng[16], n, 6.0))
    ids = torch.from_numpy(rng[17].integers(0, 8, n).astype(np.int32)).cuda()
    out = torch.empty((n, 3), device="cuda")
    with Context(0, wait_timeout_ns=1) as short:
        mats = _materials(short, rng, 8)
        for _ in range(3):
            call(short.h, [m.h for m in mats], dq, ids, n, out, torch.cuda.current_stream())
        with pytest.raises(B.NamError) as e:
            short.check()
        assert e.value.status == B.NAM_ERR_TIMEOUT
        short.check()  # the error word was cleared (no launch since)
    with Context(0) as ok:
        mats = _materials(ok, rng, 8)
        call(ok.h, [m.h for m in mats], dq, ids, n, out, torch.cuda.current_stream())
        ok.check()
        for k, m in enumerate(mats):
            idx = torch.nonzero(ids == k)[:, 0]
            assert torch.equal(out[idx], m.eval({f: t[idx].contiguous() for f, t in dq.items()})), k


@pytest.mark.parametrize("tiles", [1, 5, 6, 9])
def test_last_tiles_of_a_cta_keep_their_weights(gctx, tiles):
    """CTAs whose chains finish on a few tiles each, of more materials than
    slots: a chain that is done gives its slot to one that still needs it."""
    import torch
    from paper_2305_02678_gb300 import binding as B
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = W.rng_streams(192, 14)
    mats = _materials(gctx, rng, 6)
    n = sms * tiles * 128
    dq = to_device(W.uniform_queries(rng[12], n, 6.0))
    ids = rng[13].integers(0, 6, sms * tiles)
    ref = torch.stack([m.eval(dq) for m in mats])
    want = ref[torch.from_numpy(np.repeat(ids, 128)).cuda(), torch.arange(n, device="cuda")]
    items = [(128 * k, 128, int(i)) for k, i in enumerate(ids)]  # in tile order: neighbours differ
    for _ in range(20):
        out = torch.empty((n, 3), device="cuda")
        B.nam_eval_multi(gctx.h, [m.h for m in mats], dq, items, out, torch.cuda.current_stream())
        assert torch.equal(out, want)
    for m in mats:
        m.destroy()
    gctx.check()
