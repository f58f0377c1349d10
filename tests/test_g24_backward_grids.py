"""Reverse mode where its grid changes: a tile per CTA up to the SM count, then a
tile per group of a CTA, then several; and the pyramid levels whose sums a CTA
keeps in shared memory, which depend on its share of the queries."""
import pytest

from test_g16_backward_tiles import _gradient, _same, _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,frame,albedo,levels", [(16, True, False, 8), (32, False, True, 7), (64, True, False, 9)])
@pytest.mark.parametrize("tiles", [1, 2])
@pytest.mark.parametrize("extra", [0, 1, 64, 333])
def test_around_the_sm_count(gctx, H, frame, albedo, levels, tiles, extra):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = tiles * sms * 64 + extra
    mat, dq, dl = _setup(gctx, 241, H, frame, 0, albedo, n, levels)
    whole = _gradient(gctx, mat, dq, dl, [(0, n)])
    _same(whole, _gradient(gctx, mat, dq, dl, [(a, min(n, a + 3333)) for a in range(0, n, 3333)]))
    mat.destroy()
    gctx.check()
