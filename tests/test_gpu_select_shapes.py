"""The selection at the edges of its kernel: rows that end inside a bit word,
radii beyond a word, grids of one column and the largest grid, units from one
(eight CTAs each) to hundreds (one CTA), narrow and wide channels, keys that
crowd into one histogram bin, groups whose units are interleaved or invalid,
bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2608_22526_gb300 import rs3, synth
from tests._harness import to_dev, to_host

pytestmark = pytest.mark.gpu


def _masks(rng, U, m, n, density):
    M = np.zeros((U, m, n), np.uint8)
    for u in range(U):
        kind = u % 4
        if kind == 0:                                   # a rectangle, perhaps at the border
            y, x = rng.integers(0, m), rng.integers(0, n)
            M[u, y:y + 1 + m // 3, x:x + 1 + n // 3] = 255
        elif kind == 1:
            M[u] = rng.random((m, n)) < density
        elif kind == 2:
            M[u, rng.integers(0, m), rng.integers(0, n)] = 1
    return M.reshape(U, m * n)                          # every fourth unit's mask is empty


def _run(m, n, C, dtype, ug, G, union, rho=0.3, r_s=4, c=14, seed=0, outlier=False, rounds=2, density=0.02, bbox=0, both=False):
    rng = np.random.default_rng([seed, m, n, C])
    U, mn = len(ug), m * n
    ug = np.asarray(ug, np.int32)
    k = rs3.rs3_kmax(rho, mn)
    p = rs3.default_params(rho=rho, r_s=r_s, c=c, union_mode=int(union), bbox_mode=bbox)
    track = np.zeros((U, 6), np.int32)
    track_d = torch.zeros((U, 6), dtype=torch.int32, device="cuda")
    idx = torch.full((U, max(k, 1)), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((U,), -7, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.full((rs3.rs3_select_workspace_bytes(G, U, m, n),), 255, dtype=torch.uint8, device="cuda")
    track_n, idx_n, cnt_n = track_d.clone(), idx.clone(), cnt.clone()
    for t in range(rounds):
        M = _masks(rng, U, m, n, density)
        if t:
            M = np.roll(M, 1, axis=0)                   # other units lose their object (Eq. 4)
        z = rng.standard_normal((G, mn, C), dtype=np.float32)
        if outlier:                                     # one key stretches the range: the rest share a bin
            z[:, rng.integers(0, mn)] *= 1e8
            z[:, rng.integers(0, mn)] = 0
        z = synth.f32_to_bf16_bits(z) if dtype == "bf16" else z
        rs3.rs3_select_queries(to_dev(z), dtype, G, m, n, C, to_dev(M), to_dev(ug), U, track_d, p, idx, cnt, ws, st)
        sel = orc.select(z, dtype, M, ug, track, m, n, rho, r_s, c, int(union), bbox_mode=bbox)
        c_d, i_d = to_host(cnt), to_host(idx)
        assert np.array_equal(c_d, sel.count), (t, c_d, sel.count)
        for u in range(U):
            assert np.array_equal(i_d[u, :c_d[u]], sel.keep(u)), (t, u)
        assert np.array_equal(to_host(track_d), track), t
        if both:                                        # the one launch of calls without a workspace
            rs3.rs3_select_queries_noalloc(to_dev(z), dtype, G, m, n, C, to_dev(M), to_dev(ug), U, track_n, p, idx_n, cnt_n, st)
            assert torch.equal(cnt, cnt_n) and torch.equal(idx, idx_n) and torch.equal(track_d, track_n), t
    assert int(st.item()) == 0


@pytest.mark.parametrize("m,n", [(40, 1), (300, 31), (37, 33), (64, 64), (50, 65), (20, 97), (128, 128), (1, 500), (5, 1100), (16384, 1)])
@pytest.mark.parametrize("union", [False, True])
def test_grids(m, n, union):
    _run(m, n, 64, "bf16", [0, 1, 0, 1, 0, 0], 2, union)


@pytest.mark.parametrize("r_s,c", [(0, 0), (31, 2), (32, 40), (75, 14)])
def test_radii(r_s, c):
    _run(48, 130, 32, "f32", [0, 0, 1, 1], 2, False, r_s=r_s, c=c, rounds=3, density=0.001)


@pytest.mark.parametrize("C,dtype", [(8, "bf16"), (40, "f32"), (128, "bf16"), (256, "f32"), (264, "bf16"), (768, "bf16"), (4096, "f32")])
def test_channels(C, dtype):
    _run(40, 36, C, dtype, [0, 1, 1, 0, 1], 2, False, rho=0.1, density=0.2)


@pytest.mark.parametrize("U,G,union", [(1, 1, False), (43, 5, False), (45, 45, True), (130, 9, False), (400, 3, True), (333, 20, False)])
def test_cluster_sizes(U, G, union):
    rng = np.random.default_rng(U)
    _run(24, 28, 64, "bf16", rng.integers(0, G, U), G, union, seed=U)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rho", [0.02, 0.3, 0.9])
def test_crowded_bin(dtype, rho):
    _run(64, 64, 64, dtype, [0, 0, 0, 0], 1, True, rho=rho, outlier=True, density=0.4, r_s=9)


def test_seed_box_prior():
    _run(33, 47, 64, "bf16", [0, 0, 1], 2, False, bbox=1)


@pytest.mark.parametrize("union", [False, True])
def test_units_without_a_grid_are_skipped(union, C=64, more=0):
    """A group id out of range latches RS3_EINVAL, its unit keeps its tracker and
    selects nothing, the others are selected as usual."""
    m, n, G = 30, 40, 2
    rng = np.random.default_rng(3)
    ug = np.array([0, 5, 1, -1, 0] + [0] * more, np.int32)
    U, mn = len(ug), m * n
    M = _masks(rng, U, m, n, 0.05)
    M[:, 7:200] = 1
    z = synth.f32_to_bf16_bits(rng.standard_normal((G, mn, C), dtype=np.float32))
    k = rs3.rs3_kmax(0.3, mn)
    track_d = torch.full((U, 6), 3, dtype=torch.int32, device="cuda")
    idx = torch.zeros((U, k), dtype=torch.int32, device="cuda")
    cnt = torch.full((U,), -7, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(rs3.rs3_select_workspace_bytes(G, U, m, n), dtype=torch.uint8, device="cuda")
    p = rs3.default_params(rho=0.3, union_mode=int(union))
    rs3.rs3_select_queries(to_dev(z), "bf16", G, m, n, C, to_dev(M), to_dev(ug), U, track_d, p, idx, cnt, ws, st)
    good = np.flatnonzero((ug >= 0) & (ug < G))
    track = np.full((len(good), 6), 3, np.int32)
    sel = orc.select(z, "bf16", M[good], ug[good], track, m, n, 0.3, 4, 14, int(union))
    c_d, i_d, t_d = to_host(cnt), to_host(idx), to_host(track_d)
    assert int(st.item()) == rs3.RS3_EINVAL
    assert c_d[1] == 0 and c_d[3] == 0 and np.all(t_d[[1, 3]] == 3)
    for i, u in enumerate(good):
        assert c_d[u] == sel.count[i] and np.array_equal(i_d[u, :c_d[u]], sel.keep(i))
        assert np.array_equal(t_d[u], track[i])


@pytest.mark.parametrize("m,n,C,dtype,ug,G,union,rho", [
    (64, 64, 2048, "bf16", [0], 1, False, 0.1), (64, 64, 1024, "f32", [0, 1], 2, False, 0.3), (50, 65, 4096, "bf16", [0, 1, 0], 2, False, 0.02),
    (128, 128, 1024, "bf16", [0], 1, True, 0.3), (64, 64, 256, "bf16", [0] * 70, 1, False, 0.2), (37, 33, 64, "bf16", [0, 1] * 9, 2, True, 0.3),
    (24, 28, 264, "f32", [0] * 75, 1, True, 1.0), (40, 1, 64, "bf16", [0] * 9, 1, True, 0.3), (1, 500, 8, "bf16", [0] * 12, 1, True, 0.0),
    (300, 31, 40, "f32", [0] * 10, 1, True, 0.05), (16384, 1, 64, "bf16", [0] * 9, 1, True, 0.3), (2, 2, 64, "bf16", [0] * 9, 1, True, 0.5),
    (1, 3, 64, "bf16", [0] * 9, 1, True, 0.5)])
def test_three_launches(m, n, C, dtype, ug, G, union, rho):
    """Calls of wide rows, of many objects on one grid and of large unions go
    through the workspace in three launches; the one launch of a call without a
    workspace selects the same."""
    _run(m, n, C, dtype, ug, G, union, rho=rho, density=0.3, both=True, bbox=len(ug) == 18)
    if len(ug) > 1:
        _run(m, n, C, dtype, ug, G, not union, rho=rho, density=0.3, both=True)


@pytest.mark.parametrize("union", [False, True])
def test_units_without_a_grid_in_three_launches(union):
    test_units_without_a_grid_are_skipped(union, C=4096, more=10)
