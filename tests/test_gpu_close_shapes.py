"""rs3_close_argmax at the edges of its tiles: one to four 128-column strips and
images wider than a tile, rows that do not fill the last tile, every radius,
streams with more objects than a cluster has CTAs, and arrays that start on no
16-byte (4-byte) boundary, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2608_22526_gb300 import rs3, synth
from tests._harness import to_dev, to_host

pytestmark = pytest.mark.gpu


def _off(t, skew):
    """The tensor's values in storage that starts `skew` elements later."""
    buf = torch.empty(t.numel() + skew, dtype=t.dtype, device=t.device)
    buf[skew:] = t.reshape(-1)
    return buf[skew:].view(t.shape)


def _check(objs, h, w, R, s, seed, skew=0, punch=None):
    rng = np.random.default_rng(seed)
    L = synth.decoder_logits(rng, sum(objs), h, w)
    if punch is not None:                # one pixel in twenty of every object
        L[rng.random(L.shape) < 0.05] = punch
    U, G = sum(objs), len(objs)
    gs = np.concatenate([[0], np.cumsum(objs)]).astype(np.int32)
    mk = lambda *shape: _off(torch.full(shape, 77, dtype=torch.uint8, device="cuda"), skew)
    pal, clo, grd = mk(G, h, w), mk(U, h, w), mk(U, h // s, w // s)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    rs3.rs3_close_argmax(_off(to_dev(L), skew), to_dev(gs), G, U, h, w, R, s, pal, clo, grd, st)
    pal, clo, grd = to_host(pal), to_host(clo), to_host(grd)
    assert int(st.item()) == 0
    for g in range(G):
        c_ref, p_ref = orc.close_argmax(L[gs[g]:gs[g + 1]], R)
        assert np.array_equal(pal[g], p_ref), f"palette of stream {g}"
        assert np.array_equal(clo[gs[g]:gs[g + 1]], c_ref), f"closed masks of stream {g}"
        for o in range(objs[g]):
            assert np.array_equal(grd[gs[g] + o], orc.downsample(c_ref[o], s))


@pytest.mark.parametrize("w", [32, 128, 160, 256, 288, 384, 416, 512, 544, 1056])
def test_widths(w):
    _check([3, 1], 45, w, 4, 1, 300 + w)


@pytest.mark.parametrize("R", range(9))
def test_radii(R):
    _check([2, 4], 50, 640, R, 2, 400 + R)


@pytest.mark.parametrize("objs,h,w,s", [([11, 0, 3], 52, 96, 4), ([1] * 40, 100, 256, 4), ([3] * 30, 96, 384, 6),
                                        ([20], 23, 64, 1), ([9, 9], 384, 512, 32), ([2, 2], 48, 288, 3)])
def test_streams_and_rows(objs, h, w, s):
    _check(objs, h, w, 4, s, 500 + h)


@pytest.mark.parametrize("skew", [1, 2, 3, 4])
def test_unaligned_arrays(skew):
    _check([2, 1], 40, 160, 4, 4, 600 + skew, skew=skew)
    _check([2, 1], 40, 160, 3, 4, 600 + skew, skew=skew)


@pytest.mark.parametrize("skew", [0, 1])
@pytest.mark.parametrize("objs,punch", [([1, 1], -np.inf), ([3, 2], -np.inf), ([8], -np.inf), ([11, 2], -np.inf), ([1] * 30, -np.inf),
                                        ([1, 1], np.nan), ([1] * 30, np.nan)])
def test_closed_pixels_of_any_logit_have_a_label(objs, punch, skew):
    """Suppressed pixels (-inf, or NaN where one object is alone) that the closure
    fills belong to the object, as every closed pixel that no other object takes
    does."""
    _check(objs, 64, 160, 4, 4, 700 + len(objs), skew=skew, punch=punch)


@pytest.mark.parametrize("objs,h,w,R,skew", [([8], 256, 256, 4, 0), ([8], 256, 256, 2, 0), ([8], 256, 256, 4, 1), ([5], 300, 640, 4, 0),
                                             ([16], 130, 512, 7, 0), ([3], 40, 96, 4, 0)])
def test_one_stream_of_several_objects(objs, h, w, R, skew):
    """The sizes whose tiles are shared by clusters: as many as are resident at
    once, with one, two or more objects for each of their CTAs."""
    _check(objs, h, w, R, 4 if h % 4 == 0 else 2, 800 + h, skew=skew)
