"""Seeds and write keep-sets at the edges of their kernels: bands with no rows,
rows that end inside a bit word, dilations beyond a word and beyond the grid,
the largest grid, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2608_22526_gb300 import rs3, synth
from tests._harness import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U,h,w,s", [(1, 5, 16, 1), (3, 8, 32, 8), (2, 37, 48, 1), (60, 96, 160, 16), (1, 2048, 1536, 16), (2, 16, 8192, 16)])
def test_seeds(U, h, w, s):
    rng = np.random.default_rng(h * 7 + w)
    M = synth.pixel_masks(rng, U, h, w)
    M[U - 1] = 0
    if U > 1:
        M[U - 1, h // 2, w - 1] = 1                      # one pixel
        M[0, 0, 0] = 3
    track = torch.full((U, 6), -5, dtype=torch.int32, device="cuda")
    grd = torch.full((U, h // s, w // s), 77, dtype=torch.uint8, device="cuda")
    box = torch.full((U, h // s, w // s), 77, dtype=torch.uint8, device="cuda")
    rs3.rs3_seed_from_masks(to_dev(M), U, h, w, s, track, grd, box)
    alone = torch.full((U, 6), -5, dtype=torch.int32, device="cuda")
    rs3.rs3_seed_from_masks(to_dev(M), U, h, w, s, alone, None, None)
    t, g, b = to_host(track), to_host(grd), to_host(box)
    assert np.array_equal(t, to_host(alone))
    for u in range(U):
        ref = orc.seed_track(M[u], s)
        assert list(t[u]) == list(ref), u
        assert np.array_equal(g[u], orc.downsample(M[u], s))
        want = np.zeros((h // s, w // s), np.uint8)
        if ref[4]:
            want[ref[0]:ref[2] + 1, ref[1]:ref[3] + 1] = 1
        assert np.array_equal(b[u], want)


@pytest.mark.parametrize("U,h,w,s", [(3, 1040, 1056, 16), (20, 1024, 896, 32), (1, 40000, 32, 8), (1, 8, 200000, 8), (2, 1030, 2064, 2),
                                     (200, 256, 256, 16), (400, 128, 128, 8), (7, 96, 208, 1), (50, 144, 144, 3)])
def test_seeds_of_large_and_of_many_masks(U, h, w, s):
    """Masks past 1 MB, or 16 MB in all, are spread in bands over all SMs; many
    small ones get a CTA or two each."""
    test_seeds(U, h, w, s)


def _dilated(S, m, n, r):
    """Cells within Chebyshev distance r of a set one, by window counts (the
    oracle visits every window's cells: too slow for large radii)."""
    c = np.zeros((m + 1, n + 1), np.int64)
    c[1:, 1:] = np.cumsum(np.cumsum(S.reshape(m, n) != 0, 0), 1)
    y, x = np.arange(m), np.arange(n)
    ya, yb = np.maximum(y - r, 0), np.minimum(y + r, m - 1) + 1
    xa, xb = np.maximum(x - r, 0), np.minimum(x + r, n - 1) + 1
    return (c[yb][:, xb] - c[ya][:, xb] - c[yb][:, xa] + c[ya][:, xa] > 0).astype(np.uint8).reshape(-1)


@pytest.mark.parametrize("m,n", [(1, 1), (40, 1), (17, 31), (33, 64), (20, 65), (3, 200), (128, 128), (16384, 1), (1, 16384)])
@pytest.mark.parametrize("D_w", [0, 5, 31, 32, 70, 20000])
@pytest.mark.parametrize("union", [0, 1])
def test_write_keepsets(m, n, D_w, union):
    rng = np.random.default_rng([m, n, D_w])
    ug = np.array([0, 7, 0, -2, 7, 7], np.int32)           # any id groups units
    U, mn = len(ug), m * n
    S = np.zeros((U, mn), np.uint8)
    for u in range(U - 1):
        S[u, rng.integers(0, mn, size=1 + mn // 50)] = 1 + u
    for fall in (0, 1):
        p = rs3.default_params(D_w=D_w, union_mode=union, fall_through=fall)
        kw = torch.full((U, mn), 77, dtype=torch.uint8, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        rs3.rs3_write_keepset(to_dev(S), to_dev(ug), U, m, n, p, kw, st)
        ref = np.empty((U, mn), np.uint8)
        for u in range(U):
            seed = np.any(S[ug == ug[u]] != 0, axis=0) if union else S[u] != 0
            frac = seed.mean()
            ref[u] = 1 if fall and (frac > 0.95 or frac < 0.05) else _dilated(seed, m, n, D_w)
        assert np.array_equal(to_host(kw), ref), fall
        if D_w <= 5 and mn <= 4096:
            assert np.array_equal(ref, orc.write_keepset(S, ug, m, n, D_w, fall_through=fall, union_mode=union))


@pytest.mark.parametrize("U,G,m,n", [(600, 3, 30, 33), (40, 1, 64, 64), (9, 2, 2100, 7), (17, 1, 5, 300)])
def test_write_keepsets_of_large_groups(U, G, m, n):
    """More units than the CTA lists at a time, more than eight of a group, rows
    shorter and longer than a word."""
    rng = np.random.default_rng([U, m, n])
    ug = rng.integers(0, G, U).astype(np.int32)
    S = np.zeros((U, m * n), np.uint8)
    S[np.arange(U)[::2], rng.integers(0, m * n, size=U)[::2]] = 255
    p = rs3.default_params(D_w=3, union_mode=1, fall_through=0)
    kw = torch.full((U, m * n), 77, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    rs3.rs3_write_keepset(to_dev(S), to_dev(ug), U, m, n, p, kw, st)
    ref = [_dilated(np.any(S[ug == g] != 0, axis=0), m, n, 3) for g in range(G)]
    assert np.array_equal(to_host(kw), np.stack([ref[g] for g in ug]))
