"""FP32 evaluation of fixed weights at the ends of FP32's range, against the
per-thread kernel (the same material made trainable)."""
import numpy as np
import pytest

import workloads as W
from conftest import to_device

pytestmark = pytest.mark.gpu


def _pair(ctx, rng, H, out=3, scale=(1.0, 1.0, 1.0), frame=None):
    """Decoder weights scaled per layer, those behind the first layer made
    positive (so that infinite units do not cancel)."""
    pyr = W.make_pyramid(rng[0], 64, 64, 7, dtype=np.float32)
    m = W.make_model(rng[1], (14, H, H, out), frame)
    dec = [(Wl * np.float32(s), bl * np.float32(s)) for (Wl, bl), s in zip(m["decoder"], scale)]
    dec[1:] = [(np.abs(Wl), bl) for Wl, bl in dec[1:]]
    return [ctx.material(64, 64, 7, pyr, m["frame"], dec, precision=0, trainable=t) for t in (False, True)]


def _eval(mats, dq, out):
    return [np.concatenate([t.cpu().numpy() for t in (m.eval_albedo(dq) if out == 6 else (m.eval(dq),))], 1)
            .astype(np.float64) for m in mats]


# Scales of the layers: the first overflows for the queries with directions of
# 1e12; for nearly all; the second and the output layer for those of 1e12
@pytest.mark.parametrize("H,out", [(16, 3), (32, 6), (64, 3)])
@pytest.mark.parametrize("scale", [(1e28, 1.0, 1e-28), (1e38, 1.0, 1e-30), (1e6, 1e22, 1.0), (1.0, 1.0, 1e28)])
def test_overflow_of_a_layer(gctx, H, out, scale):
    rng = W.rng_streams(211, 3)
    mats = _pair(gctx, rng, H, out, scale)
    n = 700
    q = W.uniform_queries(rng[2], n, 6.0)
    for k, f in enumerate(("wix", "wiy", "wiz", "wox", "woy", "woz")):
        q[f][k::35] *= 1e12
    a, b = _eval(mats, to_device(q), out)
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
    f = np.isfinite(b)
    assert np.array_equal(a[~f & ~np.isnan(b)], b[~f & ~np.isnan(b)])
    # sums of positive and negative terms in different orders in the first layer,
    # of positive ones behind it: up to 65 roundings of 2^-24 a layer, against the row's scale
    row = np.abs(np.where(f, b, 0.0)).max(1, keepdims=True) * np.ones_like(b)
    with np.errstate(invalid="ignore"):
        assert (np.abs(a - b)[f] <= 3 * 65 * 2.0 ** -24 * 8 * row[f]).all()
    for m in mats:
        m.destroy()
    gctx.check()


@pytest.mark.parametrize("H,out,frame", [(16, 3, None), (32, 6, (8, 16, 6)), (64, 3, (8, 16, 6)), (64, 6, None)])
def test_rows_out_of_range_are_the_per_thread_kernels(gctx, H, out, frame):
    """Bit for bit, whether the results are finite (directions of up to 1e25 with
    weights of 1e-3 and less) or not."""
    rng = W.rng_streams(212, 3)
    pyr = W.make_pyramid(rng[0], 64, 64, 7, dtype=np.float32)
    m = W.make_model(rng[1], (14, H, H, out), frame)
    dec = [(Wl * np.float32(1e-3), bl) for Wl, bl in m["decoder"]]
    mats = [gctx.material(64, 64, 7, pyr, m["frame"], dec, precision=0, trainable=t) for t in (False, True)]
    n = 1400
    q = W.uniform_queries(rng[2], n, 6.0)
    rows = np.arange(0, n, 7)
    for f in ("wix", "wiy", "wiz", "wox", "woy", "woz"):
        q[f][rows] *= 1e25
    q["wix"][rows[::5]] = np.inf
    q["woy"][rows[1::5]] = np.nan
    dq = to_device(q)
    a, b = ([t.cpu().numpy() for t in (m.eval_albedo(dq) if out == 6 else (m.eval(dq),))] for m in mats)
    for x, y in zip(a, b):
        assert np.isfinite(y[rows[2::5]]).all()
        assert np.array_equal(x[rows].view(np.int32), y[rows].view(np.int32))
    for m in mats:
        m.destroy()
    gctx.check()


def test_budget_without_room_for_the_split_weights():
    """A budget that just holds the pyramid and the masters still takes the
    material, which then runs the per-thread kernel."""
    from paper_2305_02678_gb300 import Context, NamError
    rng = W.rng_streams(213, 3)
    pyr = W.make_pyramid(rng[0], 32, 32, 6, dtype=np.float32)
    m = W.make_model(rng[1], (14, 64, 64, 3), (8, 16, 6))
    dq = to_device(W.uniform_queries(rng[2], 500, 5.0))
    with Context(0) as ctx:
        t = ctx.material(32, 32, 6, pyr, m["frame"], m["decoder"], precision=0, trainable=True)
        want = t.eval(dq).cpu().numpy()
        need = pyr.nbytes + 4 * t.info.n_params
        assert ctx.material(32, 32, 6, pyr, m["frame"], m["decoder"], precision=0).info.resident_bytes > need
    with Context(0, hbm_budget_bytes=need) as ctx:
        f = ctx.material(32, 32, 6, pyr, m["frame"], m["decoder"], precision=0)
        assert f.info.resident_bytes == need == ctx.stats().resident_bytes
        assert np.array_equal(f.eval(dq).cpu().numpy(), want)
        f.destroy()
        assert ctx.stats().resident_bytes == 0
    with Context(0, hbm_budget_bytes=need - 1) as ctx, pytest.raises(NamError):
        ctx.material(32, 32, 6, pyr, m["frame"], m["decoder"], precision=0)


def _family(kind, rng, dec):
    """Weights other than Glorot's uniform ones."""
    f = {"glorot": lambda w: w, "positive": np.abs,
         "heavy": lambda w: (w / np.abs(w).max()) ** 3 * np.abs(w).max() * 2}[kind]
    return [(np.ascontiguousarray(f(w), np.float32), b) for w, b in dec]


@pytest.mark.parametrize("H", [16, 32, 64])
@pytest.mark.parametrize("kind", ["glorot", "positive", "heavy"])
def test_error_against_64_bits_is_the_per_thread_kernels(gctx, oracle, H, kind):
    rng = W.rng_streams(214, 4)
    pyr = W.make_pyramid(rng[0], 128, 128, 8, dtype=np.float32)
    dec = _family(kind, rng[3], W.make_model(rng[1], (14, H, H, 3), None)["decoder"])
    q = W.uniform_queries(rng[2], 30000, 7.0)
    ref = oracle.eval(oracle.Model(128, 128, 8, pyr, None, dec), q)
    dq = to_device(q)
    err = []
    for t in (False, True):
        mat = gctx.material(128, 128, 8, pyr, None, dec, precision=0, trainable=t)
        err.append(np.linalg.norm(mat.eval(dq).cpu().numpy().astype(np.float64) - ref))
        mat.destroy()
    assert err[0] <= 1.1 * err[1]  # (a tenth for the chance of one batch's roundings)


def test_error_of_three_hidden_layers(gctx, oracle):
    """No per-thread form to compare with: four layers of sums whose roundings,
    2^-24 each, add up like random ones, are well within 2^-21 of the result."""
    rng = W.rng_streams(215, 3)
    pyr = W.make_pyramid(rng[0], 128, 128, 8, dtype=np.float32)
    dec = W.make_model(rng[1], (14, 64, 64, 64, 3), None)["decoder"]
    q = W.uniform_queries(rng[2], 30000, 7.0)
    ref = oracle.eval(oracle.Model(128, 128, 8, pyr, None, dec), q)
    mat = gctx.material(128, 128, 8, pyr, None, dec, precision=0)
    err = np.linalg.norm(mat.eval(to_device(q)).cpu().numpy().astype(np.float64) - ref)
    assert err <= 2.0 ** -21 * np.linalg.norm(ref)
    mat.destroy()
