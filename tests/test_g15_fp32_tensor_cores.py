"""FP32 evaluation on the tensor cores (split operands; materials whose weights
are fixed) against the per-thread FP32 kernel (the same material made
trainable): every shape both run, inputs of large and small magnitude, and
inputs that are not finite."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


def _pair(gctx, rng, H, frame, filt=0, address=0, scale=1.0, tex=(64, 64, 7), out=3):
    pyr = (W.make_pyramid(rng[0], *tex, dtype=np.float32) * scale).astype(np.float32)
    m = W.make_model(rng[1], (14, H, H, out), frame)
    mk = lambda t: gctx.material(*tex, pyr, m["frame"], m["decoder"], precision=0, filter=filt, address=address,
                                 trainable=t)
    return mk(False), mk(True)


# Both kernels sum at most 65 products per output and layer; the split leaves
# out less than 2^-23 of a product and each of the MMA's at most 25 additions
# loses at most 2^-23 of the largest partial sum.  Three layers of that, with
# the partial sums of these Glorot-initialised decoders within a factor of
# eight of the result's RMS: 3 * 8 * 27 * 2^-23 = 8e-5 of the RMS at worst.
TOL = 8e-5


@pytest.mark.parametrize("H", [16, 32, 64])
@pytest.mark.parametrize("frame", [None, (8, 16, 6)])
@pytest.mark.parametrize("n,filt,address,scale,out", [(1, 0, 0, 1.0, 3), (129, 1, 1, 1.0, 6), (30011, 0, 0, 1.0, 3),
                                                      (4000, 0, 1, 2.0 ** 40, 3), (4000, 1, 0, 2.0 ** -40, 3)])
def test_matches_per_thread_kernel(gctx, H, frame, n, filt, address, scale, out):
    rng = W.rng_streams(151, 3)
    tc, simt = _pair(gctx, rng, H, frame, filt, address, scale, out=out)
    q = W.uniform_queries(rng[2], n, 6.0)
    dq = to_device(q)
    a, b = (np.concatenate([t.cpu().numpy() for t in (m.eval_albedo(dq) if out == 6 else (m.eval(dq),))], 1)
            for m in (tc, simt))
    assert np.isfinite(a).all()
    # rows of a nearly degenerate frame amplify both kernels' rounding alike:
    # the frame itself is computed by the same operations in both
    rms = np.sqrt(np.mean(b.astype(np.float64) ** 2))
    assert np.abs(a.astype(np.float64) - b).max() <= TOL * rms
    for m in (tc, simt):
        m.destroy()
    gctx.check()


@pytest.mark.parametrize("frame", [None, (8, 16, 6)])
def test_non_finite_inputs(gctx, frame):
    rng = W.rng_streams(152, 3)
    tc, simt = _pair(gctx, rng, 64, frame)
    n = 600
    q = W.uniform_queries(rng[2], n, 6.0)
    for k, (f, v) in enumerate([("wix", np.nan), ("woz", np.inf), ("wiy", -np.inf), ("u", np.nan), ("v", np.inf),
                                ("lod", np.nan), ("wox", 3e38)]):
        q[f][k::40] = v
    dq = to_device(q)
    a, b = tc.eval(dq).cpu().numpy().astype(np.float64), simt.eval(dq).cpu().numpy().astype(np.float64)
    assert np.array_equal(np.isnan(a), np.isnan(b))
    fin = np.isfinite(b)
    assert np.array_equal(a[~fin & ~np.isnan(b)], b[~fin & ~np.isnan(b)])
    clean = np.ones(n, bool)
    clean[[i for k in range(7) for i in range(k, n, 40)]] = False
    rms = np.sqrt(np.mean(b[clean] ** 2))
    big = np.maximum(np.abs(b), rms)
    with np.errstate(invalid="ignore"):
        assert (np.abs(a - b)[fin] <= TOL * big[fin]).all()
    for m in (tc, simt):
        m.destroy()
    gctx.check()
