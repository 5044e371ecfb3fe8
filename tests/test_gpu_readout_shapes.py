"""The readout at the edges of its tiles: kept counts and bank lengths around
the query and key tiles of each kernel (CUDA cores: 32 keys, 64 or 128 rows;
tensor cores: 64 or 128 keys, 128 rows or pairs of that), every head width,
ring pieces and pointer rows that leave partial tiles, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2608_22526_gb300 import rs3, synth
from tests._harness import F32_REL, bf16_ulp, to_dev, to_host, widen

pytestmark = pytest.mark.gpu


def _draw(rng, dtype, shape, scale=1.0):
    x = rng.standard_normal(shape, dtype=np.float32) * np.float32(scale)
    return synth.f32_to_bf16_bits(x) if dtype == "bf16" else x


def _check(dtype, got, exact, vmax, rope, what):
    """bf16: half a step of the result for its one rounding, plus 2^-9 of the
    greatest value for the probabilities' rounding (sum p |v| / l <= max |v|) and
    as much again for the sums; with RoPE the rotated queries are rounded too,
    which moves a score of the size drawn here by about 2^-9, and p by as much.
    fp32: the relative bound of the other parity tests."""
    err = np.abs(widen(got, dtype) - exact)
    if not err.size:
        return
    if dtype == "bf16":
        excess = float(np.max(err - 0.5 * bf16_ulp(exact)))
        assert excess <= (2.0 if rope else 1.0) * 2.0 ** -8 * vmax, f"{what}: {excess} beyond one rounding"
    else:
        assert float(err.max()) <= F32_REL * max(float(np.abs(exact).max()), 1e-30), f"{what}: {err.max()}"


def _case(dtype, H, d, counts, rows, n_ptr=0, rope=False, sharp=1.0, ramp=0.0, seed=0, ws_bytes=None, tile=None, cap=0):
    """One group, a unit per (count, rows) pair: `rows` bank rows in two ring
    frames, then n_ptr pointer rows.  ramp > 0 makes later keys score higher,
    so that a row's softmax reference has to move.  cap: rows of the bank's ring, of
    which two frames are used."""
    rng = np.random.default_rng([seed, d, len(counts)])
    U, m, n = len(counts), 24, 25
    mn, D = m * n, H * d
    k_max = max(counts)
    bank = rs3.Bank(U, H, d, dtype, mn, 0, 2, max(cap, 2 * mn), 2, n_ptr)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    q = _draw(rng, dtype, (1, mn, D), sharp)
    K, V = [[] for _ in range(U)], [[] for _ in range(U)]
    for f in range(2):
        k, v = _draw(rng, dtype, (U, mn, D)), _draw(rng, dtype, (U, mn, D))
        if ramp:
            x = widen(k, dtype) + ramp * (f * mn + np.arange(mn))[None, :, None] * widen(q, dtype)[:, :1] / mn
            k = synth.f32_to_bf16_bits(x.astype(np.float32)) if dtype == "bf16" else x.astype(np.float32)
        mask = np.zeros((U, mn), np.uint8)
        for u in range(U):
            r = rows[u] // 2 + (rows[u] % 2 if f == 0 else 0)
            mask[u, np.sort(rng.permutation(mn)[:r])] = 1
            K[u].append(k[u][mask[u] == 1])
            V[u].append(v[u][mask[u] == 1])
        rs3.rs3_bank_commit(bank, to_dev(k), to_dev(v), to_dev(mask), 0, st)
    if n_ptr:
        kp, vp = _draw(rng, dtype, (U, n_ptr, D)), _draw(rng, dtype, (U, n_ptr, D))
        rs3.rs3_bank_set_pointers(bank, to_dev(kp), to_dev(vp), st)
        for u in range(U):
            K[u].append(kp[u])
            V[u].append(vp[u])
    idx = np.zeros((U, k_max), np.int32)
    for u, c in enumerate(counts):
        idx[u, :c] = np.sort(rng.permutation(mn)[:c])
    res = _draw(rng, dtype, (U, mn, D))
    tab = rng.uniform(0, 6.28, (mn, d // 2)) if rope else None
    table = np.ascontiguousarray(np.stack([np.cos(tab), np.sin(tab)], -1).astype(np.float32)) if rope else None
    ws_bytes = rs3.rs3_readout_workspace_bytes(U, H, d, k_max, dtype) if ws_bytes is None else ws_bytes
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    ug = torch.zeros(U, dtype=torch.int32, device="cuda")
    cnt = torch.tensor(counts, dtype=torch.int32, device="cuda")
    out = to_dev(res)
    attn = torch.empty_like(out)
    dev = to_dev(q), to_dev(idx), None if table is None else to_dev(table)

    def call(r, o):
        rs3.rs3_memory_readout(dev[0], dtype, 1, mn, H, d, ug, dev[1], cnt, k_max, bank, dev[2], r, o, 0.0, ws, st)

    call(None, attn)
    call(out, out)
    attn, out = to_host(attn), to_host(out)
    if tile is not None:                                 # query rows of an item: the kernel that the plan chose
        assert ws.view(torch.int32)[4].item() == tile
    for u, c in enumerate(counts):
        cells = idx[u, :c]
        vmax, A = 1.0, np.zeros((c, D))
        if c and rows[u] + n_ptr:
            Ku, Vu = np.concatenate(K[u]), np.concatenate(V[u])
            vmax = float(np.abs(widen(Vu, dtype)).max())
            A = orc.readout(q[0], dtype, H, d, cells, Ku, Vu, dtype, rope=table)
        what = f"unit {u}: {c} queries, {rows[u]} rows"
        _check(dtype, attn[u][cells], A, vmax, rope, what)
        _check(dtype, out[u][cells], widen(res[u][cells], dtype) + A, vmax, rope, what)
        other = np.setdiff1d(np.arange(mn), cells)
        assert np.all(widen(attn[u][other], dtype) == 0.0)
        assert np.array_equal(out[u][other], res[u][other])
    assert int(st.item()) == 0


COUNTS = [1, 31, 33, 64, 65, 127, 128, 129, 255, 257, 513, 0]
ROWS = [1, 2, 63, 64, 65, 31, 129, 255, 257, 513, 1100, 300]


@pytest.mark.parametrize("dtype,H,d", [("f32", 1, 16), ("f32", 3, 32), ("f32", 2, 64), ("f32", 1, 128), ("f32", 1, 256),
                                       ("bf16", 4, 16), ("bf16", 2, 32), ("bf16", 2, 64), ("bf16", 1, 128), ("bf16", 1, 256)])
@pytest.mark.parametrize("rope,n_ptr", [(False, 0), (True, 7)])
def test_tile_edges(dtype, H, d, rope, n_ptr):
    _case(dtype, H, d, COUNTS, ROWS, n_ptr=n_ptr, rope=rope)


@pytest.mark.parametrize("dtype,H,d", [("bf16", 2, 64), ("bf16", 1, 128), ("f32", 1, 64)])
@pytest.mark.parametrize("part", range(4))
def test_tile_edges_of_few_units(dtype, H, d, part):
    """Too few query tiles for two per CTA."""
    _case(dtype, H, d, COUNTS[part::4], ROWS[part::4], n_ptr=3, rope=part % 2 == 1)


@pytest.mark.parametrize("dtype,H,d", [("f32", 2, 64), ("f32", 1, 256), ("bf16", 2, 64), ("bf16", 1, 128), ("bf16", 1, 256)])
def test_one_group_cut_over_every_slice(dtype, H, d):
    """One unit with few queries: its keys are spread over all CTAs and merged."""
    _case(dtype, H, d, [37], [1200])


@pytest.mark.parametrize("dtype,H,d", [("f32", 1, 64), ("f32", 1, 128), ("bf16", 1, 64), ("bf16", 1, 128), ("bf16", 1, 256)])
def test_rising_scores_move_the_reference(dtype, H, d):
    """Scores that grow along the bank by far more than 2^8 between tiles: the
    running reference moves and what is accumulated is rescaled."""
    _case(dtype, H, d, [200, 3, 129, 64], [1200, 900, 700, 1000], ramp=3.0)
    _case(dtype, H, d, [256, 3, 129, 64, 250, 255, 1, 128, 500, 512] * 2, [1200, 900, 700, 1000, 130, 1100, 600, 257, 384, 128] * 2, ramp=3.0)


@pytest.mark.parametrize("d", [64, 128, 256])
def test_partial_query_tiles_of_whole_items(d):
    """More groups than CTAs, so that most items hold a whole group and write their
    rows directly: warps in which only some rows have a query, a warp with none
    beside them, over every chunk of columns of the epilogue."""
    counts = [1, 31, 33, 100, 127, 129, 160, 5, 97, 140, 180, 65] * 15
    rows = [70, 129, 64, 200, 33, 140, 65, 257, 10, 128, 130, 90] * 15
    _case("bf16", 1, d, counts, rows, rope=True, seed=3, tile=128)


def _one_tile_bytes(U, H, d, k_max):
    """Workspace of 256 rows of partial results per SM: header, a range set per
    unit, item ranges, items, merge entries, (O, m, l) per row."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    up = lambda x: (x + 255) // 256 * 256
    groups = U * H * max(1, -(-k_max // 128))
    return (up(128) + up(8 * n_sm) + up(96 * U) + up(32 * (groups + n_sm)) + up(32 * min(groups, n_sm)) +
            up(256 * n_sm * d * 4) + up(256 * n_sm * 8))


@pytest.mark.parametrize("dtype,H,d", [("bf16", 4, 64), ("bf16", 4, 128), ("f32", 2, 64)])
def test_smaller_calls_in_a_workspace_sized_for_the_largest(dtype, H, d):
    """Keep-sets of two query tiles in a workspace sized for three (which the
    one-tile kernel serves, with half the partial rows), and every path in a
    workspace that only the smaller one fits; less than that is refused."""
    U, counts = 8, [200, 256, 3, 129, 255, 64, 130, 250]
    rows = [300, 150, 700, 64, 900, 129, 40, 500]
    _case(dtype, H, d, counts, rows, ws_bytes=rs3.rs3_readout_workspace_bytes(U, H, d, 384, dtype))
    cap = 70000 if dtype == "bf16" and d == 64 else 0     # of the size that the plan would choose for
    least = _one_tile_bytes(U, H, d, 256)
    assert least < rs3.rs3_readout_workspace_bytes(U, H, d, 256, dtype)
    _case(dtype, H, d, counts, rows, rope=True, n_ptr=5, ws_bytes=least, cap=cap)
    with pytest.raises(rs3.RS3Error) as e:
        _case(dtype, H, d, counts, rows, ws_bytes=least - 256)
    assert e.value.code == rs3.RS3_ECAPACITY


PAIRS = [512, 511, 500, 1, 385, 130, 512, 0, 400, 490, 257, 512] * 4
PAIR_ROWS = [1100, 1200, 1025, 1000, 1151, 900, 1200, 1100, 1153, 1199, 1024, 1100] * 4


@pytest.mark.parametrize("H,d", [(4, 64), (4, 128), (8, 64)])
@pytest.mark.parametrize("rope,ramp", [(True, 0.0), (False, 3.0)])
def test_two_query_tiles(H, d, rope, ramp):
    """Enough score tiles for the plan to take two query tiles per CTA: pairs that
    are full, half empty and empty, partial keys in every piece of the bank."""
    _case("bf16", H, d, PAIRS, PAIR_ROWS, n_ptr=3, rope=rope, ramp=ramp, seed=5, tile=256, cap=12000 * d // 64)


@pytest.mark.parametrize("H,d", [(4, 64), (2, 128)])
def test_small_keep_sets_take_one_query_tile(H, d):
    """Few kept queries: one tile per CTA, as the plan finds for the large bank and
    the call's sizes say for the small one."""
    counts, rows = [512, 40, 129, 1, 100, 60] + [33] * 18, [200] * 24
    _case("bf16", H, d, counts, rows, rope=True, seed=6, tile=128, cap=80000 // H)
    _case("bf16", H, d, counts, rows, rope=True, seed=6, tile=128)


def test_two_query_tiles_of_one_unit():
    """One unit, whose pairs get whole slices each, and a unit count past the plan's threads."""
    _case("bf16", 40, 64, [512], [1200], seed=7, tile=256, cap=30000)
    _case("bf16", 1, 64, [512, 250, 70] * 100, [1100, 900, 300] * 100, seed=8, tile=256, cap=5000)
