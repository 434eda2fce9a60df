"""GPU parity of block-causal paged GQA verify attention (spec_verify_attention) with
the oracle, through the C ABI: within 1e-2 max-abs on outputs (bf16 inputs, fp32
accumulation, bf16 outputs) and 1e-3 on the log-sum-exp."""

import numpy as np
import pytest
import torch

from paper_2609_04010_gb300 import binding
from paper_2609_04010_gb300 import workloads as W

from helpers import attn_tensors, compare_attention, gpu_attention, sample_rows

pytestmark = pytest.mark.gpu

# the CUDA-core kernel, the row-tile tensor-core kernel (AUTO's choice) and the
# keys-on-lanes tensor-core kernel (where it applies; elsewhere the row-tile one)
PATHS = [binding.ATTN_CUDA_CORES, binding.ATTN_TENSOR_CORES, binding.ATTN_TENSOR_CORES_KEYS_ON_LANES]

SMALL = [
    dict(batch=2, gamma=4, num_q_heads=8, num_kv_heads=8, head_dim=64, page_size=16, ctx=(0, 300)),
    dict(batch=3, gamma=8, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=16,
         ctx=(1, 700)),
    dict(batch=2, gamma=16, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=32,
         ctx=(100, 500)),
    dict(batch=2, gamma=32, num_q_heads=64, num_kv_heads=8, head_dim=128, page_size=64,
         ctx=(200, 333)),
    dict(batch=4, gamma=1, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=16,
         ctx=(0, 1000)),
    dict(batch=1, gamma=3, num_q_heads=6, num_kv_heads=2, head_dim=64, page_size=64, ctx=0),
    dict(batch=2, gamma=64, num_q_heads=8, num_kv_heads=4, head_dim=64, page_size=16,
         ctx=(0, 150)),
    # 512 rows per kv head: two row tiles of two M tiles each
    dict(batch=2, gamma=32, num_q_heads=128, num_kv_heads=8, head_dim=128, page_size=16,
         ctx=(10, 300)),
    # a group that does not divide 128, with two M tiles
    dict(batch=2, gamma=64, num_q_heads=6, num_kv_heads=2, head_dim=128, page_size=32,
         ctx=(5, 200)),
    # keys-on-lanes shapes: group 1 with 64-token pages, 48 rows (not a multiple of 32),
    # group 2 with 64 rows, and contexts shorter than one 128-key tile
    dict(batch=3, gamma=4, num_q_heads=8, num_kv_heads=8, head_dim=128, page_size=64,
         ctx=(0, 700)),
    dict(batch=2, gamma=12, num_q_heads=16, num_kv_heads=4, head_dim=128, page_size=16,
         ctx=(127, 385)),
    dict(batch=5, gamma=32, num_q_heads=16, num_kv_heads=8, head_dim=128, page_size=32,
         ctx=(1, 260)),
    dict(batch=4, gamma=16, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=16,
         ctx=(0, 100)),
    # two KV heads per block with 64-token pages (32 KB page boxes), head dim 128 and 64
    dict(batch=3, gamma=16, num_q_heads=16, num_kv_heads=4, head_dim=128, page_size=64,
         ctx=(50, 900)),
    dict(batch=2, gamma=10, num_q_heads=32, num_kv_heads=8, head_dim=64, page_size=64,
         ctx=(300, 700)),
]


def oracle_attn(oracle_mod, inp, rows=None):
    return oracle_mod.verify_attention(inp.q, inp.k_cache, inp.v_cache, inp.page_table,
                                       inp.kv_len, inp.gamma, rows=rows)


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("case", range(len(SMALL)))
def test_small_shapes_full(oracle_mod, case, path):
    inp = W.make_attn_inputs(seed=case, **SMALL[case])
    g_out, g_lse = gpu_attention(inp, path)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert np.all(st == 0)
    compare_attention(g_out, g_lse, o_out, o_lse)


def random_shape(seed):
    """A seeded random attention problem: GQA group, KV heads, head dim, page size,
    block size and ragged contexts drawn over the ranges the kernels take (up to 512
    query rows per KV head), with spare pages in the pool."""
    rng = np.random.default_rng(1000 + seed)
    group = int(rng.choice([1, 2, 3, 4, 6, 8, 16]))
    hkv = int(rng.choice([1, 2, 4, 8]))
    gamma = int(rng.integers(1, max(2, min(64, 512 // group)) + 1))
    lo = int(rng.integers(0, 900))
    hi = lo + int(rng.integers(0, 700))
    return dict(batch=int(rng.integers(1, 5)), gamma=gamma, num_q_heads=group * hkv,
                num_kv_heads=hkv, head_dim=int(rng.choice([64, 128])),
                page_size=int(rng.choice([16, 32, 64])), ctx=(lo, hi),
                extra_pages=int(rng.integers(0, 8)))


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("seed", range(20))
def test_random_shapes(oracle_mod, seed, path):
    shape = random_shape(seed)
    inp = W.make_attn_inputs(seed=seed, **shape)
    g_out, g_lse = gpu_attention(inp, path)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert np.all(st == 0)
    compare_attention(g_out, g_lse, o_out, o_lse)


@pytest.mark.parametrize("name", ["tiny", "llama8b", "serve64", "long70b"])
def test_named_workloads_sampled(oracle_mod, name):
    """Full-size workloads, in the launch configuration the benchmark times (automatic
    kernel choice), on sampled (sequence, position, head) rows."""
    inp = W.workload(name).attn_inputs(seed=0)
    g_out, g_lse = gpu_attention(inp, binding.ATTN_AUTO)
    rows = sample_rows(inp, 48)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp, rows)
    assert np.all(st == 0)
    err, lerr = compare_attention(g_out, g_lse, o_out, o_lse, rows)
    print(f"{name}: max abs err {err:.2e}, lse err {lerr:.2e}")


@pytest.mark.parametrize("name", ["llama8b", "serve64"])
def test_named_workload_every_row(oracle_mod, name):
    """Full-size workloads in the benchmark's launch configuration, every (sequence,
    block position, head) row element-wise against the oracle (2,048 rows at llama8b,
    32,768 at serve64)."""
    inp = W.workload(name).attn_inputs(seed=0)
    g_out, g_lse = gpu_attention(inp, binding.ATTN_AUTO)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert np.all(st == 0)
    err, lerr = compare_attention(g_out, g_lse, o_out, o_lse)
    print(f"{name} every row: max abs err {err:.2e}, lse err {lerr:.2e}")


@pytest.mark.parametrize("path", PATHS)
def test_page_order_invariance_bitwise(path):
    inp = W.make_attn_inputs(3, 8, 32, 8, 128, 16, (50, 400), permute_pages=False, seed=11)
    base, base_lse = gpu_attention(inp, path)
    perm = np.random.default_rng(2).permutation(inp.num_pages)
    inv = np.argsort(perm)
    inp.k_cache = inp.k_cache[perm]
    inp.v_cache = inp.v_cache[perm]
    inp.page_table = np.where(inp.page_table >= 0, inv[np.maximum(inp.page_table, 0)],
                              -1).astype(np.int32)
    out, lse = gpu_attention(inp, path)
    np.testing.assert_array_equal(out, base)
    np.testing.assert_array_equal(lse, base_lse)


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("path", PATHS)
def test_bad_pages_and_lengths(oracle_mod, path, head_dim):
    inp = W.make_attn_inputs(4, 4, 8, 2, head_dim, 16, (20, 300), seed=12)
    inp.page_table[1, 2] = inp.num_pages + 5
    inp.kv_len[2] = 2  # shorter than the block
    t = attn_tensors(inp)
    out = torch.empty_like(t[0])
    lse = torch.empty(t[0].shape[:3], dtype=torch.float32, device="cuda")
    a = binding.attn_args(*t, out, lse, path=path)
    ws = binding.new_workspace(binding.workspace_size(attn=a))
    binding.verify_attention_args(a, ws)
    code, flags = binding.read_device_status(ws)
    assert code == 5 and flags == (binding.FLAG_BAD_PAGE | binding.FLAG_BAD_KV_LEN)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert list(st) == [0, 1, 1, 0]
    compare_attention(out.float().cpu().numpy(), lse.cpu().numpy(), o_out, o_lse)


@pytest.mark.parametrize("path", PATHS)
def test_garbage_in_unused_slots_is_ignored(oracle_mod, path):
    inp = W.make_attn_inputs(2, 5, 16, 4, 128, 16, (30, 41), seed=13)
    for b in range(2):
        L = int(inp.kv_len[b])
        last = inp.page_table[b, (L - 1) // 16]
        inp.k_cache[last, :, L % 16:] = 0x7FC0  # NaN in the unused tail of the last page
        inp.v_cache[last, :, L % 16:] = 0x7FC0
    g_out, g_lse = gpu_attention(inp, path)
    o_out, o_lse, _ = oracle_attn(oracle_mod, inp)
    compare_attention(g_out, g_lse, o_out, o_lse)


def test_deterministic_repeat():
    inp = W.make_attn_inputs(2, 8, 32, 8, 128, 16, (500, 2000), seed=14)
    t = attn_tensors(inp)
    out1, lse1 = binding.verify_attention(*t)
    out2, lse2 = binding.verify_attention(*t)
    assert torch.equal(out1, out2) and torch.equal(lse1, lse2)


# The small-group kernel (automatic choice): 1 to 64 query rows per KV head (edges of its
# 16-row tiles), 2, 4 and 8 KV heads per block, every page size, contexts that end inside
# a 16-key step, units whole in a block, split over a few blocks and over many.
# (The cases of 48, 49 and 64 rows are the row-tile kernel's: the small-group one takes up to
# 32, whose edges are in test_rows_at_the_kernels_edges.)
GROUPS = [
    dict(batch=1, gamma=1, num_q_heads=2, num_kv_heads=2, head_dim=128, page_size=16, ctx=0),
    dict(batch=24, gamma=1, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=16, ctx=(0, 900)),
    dict(batch=1, gamma=1, num_q_heads=8, num_kv_heads=8, head_dim=64, page_size=32, ctx=6000),
    dict(batch=20, gamma=3, num_q_heads=40, num_kv_heads=8, head_dim=128, page_size=32, ctx=(5, 700)),
    dict(batch=3, gamma=4, num_q_heads=16, num_kv_heads=4, head_dim=128, page_size=64, ctx=(100, 2000)),
    dict(batch=40, gamma=16, num_q_heads=8, num_kv_heads=8, head_dim=128, page_size=16, ctx=(1, 300)),
    dict(batch=5, gamma=17, num_q_heads=6, num_kv_heads=6, head_dim=128, page_size=16, ctx=(60, 700)),
    dict(batch=40, gamma=8, num_q_heads=16, num_kv_heads=4, head_dim=128, page_size=64, ctx=(1, 500)),
    dict(batch=7, gamma=11, num_q_heads=12, num_kv_heads=4, head_dim=128, page_size=16, ctx=(0, 333)),
    dict(batch=2, gamma=48, num_q_heads=2, num_kv_heads=2, head_dim=128, page_size=32, ctx=(0, 1500)),
    dict(batch=30, gamma=49, num_q_heads=4, num_kv_heads=4, head_dim=64, page_size=16, ctx=(0, 400)),
    dict(batch=9, gamma=64, num_q_heads=8, num_kv_heads=8, head_dim=64, page_size=64, ctx=(3, 900)),
    dict(batch=50, gamma=2, num_q_heads=32, num_kv_heads=8, head_dim=64, page_size=16, ctx=(0, 500)),
    dict(batch=300, gamma=2, num_q_heads=4, num_kv_heads=2, head_dim=128, page_size=16, ctx=(0, 90)),
]


@pytest.mark.parametrize("case", range(len(GROUPS)))
def test_small_groups(oracle_mod, case):
    inp = W.make_attn_inputs(seed=200 + case, **GROUPS[case])
    g_out, g_lse = gpu_attention(inp, binding.ATTN_AUTO)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert np.all(st == 0)
    compare_attention(g_out, g_lse, o_out, o_lse)


# The row-tile kernel's ranges: short units kept whole (one and two M tiles, head pairs, more
# units than blocks), and whole blocks for each of fewer units.
RANGES = [
    dict(batch=8, gamma=32, num_q_heads=40, num_kv_heads=8, head_dim=64, page_size=16, ctx=(200, 440)),
    dict(batch=25, gamma=16, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=16, ctx=(0, 300)),
    dict(batch=90, gamma=10, num_q_heads=10, num_kv_heads=2, head_dim=128, page_size=32, ctx=(1, 200)),
    dict(batch=5, gamma=32, num_q_heads=20, num_kv_heads=4, head_dim=128, page_size=16, ctx=1000),
]


@pytest.mark.parametrize("case", range(len(RANGES)))
def test_row_tile_ranges(oracle_mod, case):
    inp = W.make_attn_inputs(seed=260 + case, **RANGES[case])
    g_out, g_lse = gpu_attention(inp, binding.ATTN_AUTO)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert np.all(st == 0)
    compare_attention(g_out, g_lse, o_out, o_lse)


@pytest.mark.parametrize("case", [0, 2, 3, 6, 9])
def test_small_groups_tree_mask(oracle_mod, case):
    inp = W.make_attn_inputs(seed=230 + case, **GROUPS[case])
    B, N = inp.batch, inp.gamma
    rng = np.random.default_rng(case)
    masks = np.zeros((B, N), np.uint64)
    for b in range(B):
        for j in range(N):
            up = masks[b, int(rng.integers(0, j))] if j else np.uint64(0)
            masks[b, j] = up | np.uint64(1 << j)
    out, lse = binding.verify_attention(*attn_tensors(inp), tree_mask=torch.from_numpy(masks.view(np.int64)).cuda())
    o_out, o_lse, st = oracle_mod.verify_attention(inp.q, inp.k_cache, inp.v_cache, inp.page_table,
                                                   inp.kv_len, N, tree_mask=masks)
    assert np.all(st == 0)
    compare_attention(out.float().cpu().numpy(), lse.cpu().numpy(), o_out, o_lse)


@pytest.mark.parametrize("gamma,head_dim,page", [(1, 128, 16), (8, 128, 32), (4, 64, 64), (16, 128, 16)])
def test_small_groups_bad_inputs_and_garbage(oracle_mod, gamma, head_dim, page):
    inp = W.make_attn_inputs(5, gamma, 16, 4, head_dim, page, (150, 400), seed=240 + gamma)
    inp.page_table[1, 2] = inp.num_pages + 5
    inp.page_table[4, int(inp.kv_len[4] - 1) // page] = -3
    inp.kv_len[2] = inp.page_table.shape[1] * page + 1  # longer than its pages
    for b in (0, 3):  # NaN in the unused tail of the last page
        L = int(inp.kv_len[b])
        last = inp.page_table[b, (L - 1) // page]
        if L % page:
            inp.k_cache[last, :, L % page:] = 0x7FC0
            inp.v_cache[last, :, L % page:] = 0x7FC0
    t = attn_tensors(inp)
    out = torch.empty_like(t[0])
    lse = torch.empty(t[0].shape[:3], dtype=torch.float32, device="cuda")
    a = binding.attn_args(*t, out, lse)
    ws = binding.new_workspace(binding.workspace_size(attn=a))
    for _ in range(2):  # the workspace serves the next call
        out.fill_(1.0)
        binding.verify_attention_args(a, ws)
        code, flags = binding.read_device_status(ws)
        assert code == 5 and flags == (binding.FLAG_BAD_PAGE | binding.FLAG_BAD_KV_LEN)
        o_out, o_lse, st = oracle_attn(oracle_mod, inp)
        assert list(st) == [0, 1, 1, 0, 1]
        compare_attention(out.float().cpu().numpy(), lse.cpu().numpy(), o_out, o_lse)


def check_whole_and_split(inp, tree_mask=None):
    """A call whose page table is as wide as its contexts (short units whole in a block) against
    the same call with a wide table (the general path: split by tiles and merged). Both take
    each tile's probabilities against its own maximum, so they differ by fp32 rounding, which
    may move a bf16 output to its neighbour (2^-7 of it), and in tiles 2^8 below a row's
    maximum by their probabilities' rounding (2^-8 of a weight of 2^-8, on either side)."""
    t = list(attn_tensors(inp))
    out, lse = binding.verify_attention(*t, tree_mask=tree_mask)
    pt = t[3]
    t[3] = torch.full((pt.shape[0], 64), -1, dtype=pt.dtype, device=pt.device)
    t[3][:, :pt.shape[1]] = pt
    w_out, w_lse = binding.verify_attention(*t, tree_mask=tree_mask)
    a, b = out.double(), w_out.double()
    most = t[2].double().abs().max()
    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 2.0 ** -15 * most).all())
    assert bool(((lse - w_lse).abs() <= 1e-5 + 2.0 ** -20 * w_lse.abs()).all())


# Short units of the row-tile kernel (whole in a block whatever their number, up to three
# 64-key tiles of the page table): one and two M tiles, head pairs, odd Hkv, a key on each
# side of a tile's edge, and the first table that splits.
@pytest.mark.parametrize("keys", [34, 64, 65, 128, 129, 192, 193])
@pytest.mark.parametrize("batch,gamma,hq,hkv,dim", [(1, 33, 8, 8, 128), (2, 16, 8, 2, 128), (1, 33, 12, 3, 64),
                                                    (3, 32, 8, 1, 128), (1, 32, 64, 2, 64), (2, 4, 3, 1, 128)])
@pytest.mark.parametrize("tree", [False, True])
def test_row_tile_short_units(batch, gamma, hq, hkv, dim, keys, tree):
    inp = W.make_attn_inputs(batch, gamma, hq, hkv, dim, 16, keys - gamma, True, seed=keys + hq)
    for b in range(1, batch):  # shorter ones in the same table
        inp.kv_len[b] = max(gamma, keys - 41 * b)
    masks = None
    if tree:
        rng = np.random.default_rng(keys)
        masks = np.zeros((batch, gamma), np.uint64)
        for b in range(batch):
            for j in range(gamma):
                up = masks[b, int(rng.integers(0, j))] if j else np.uint64(0)
                masks[b, j] = up | np.uint64(1 << j)
        masks = torch.from_numpy(masks.view(np.int64)).cuda()
    check_whole_and_split(inp, masks)


@pytest.mark.parametrize("gains", [(1.0, 12.0, 1.0), (12.0, 1.0, 1.0), (1.0, 1.0, 12.0), (12.0, 1.0, 12.0),
                                   (0.01, 8.0, 0.5)])
@pytest.mark.parametrize("gamma,hq,hkv", [(33, 8, 2), (32, 16, 2), (16, 8, 2)])
def test_row_tile_short_units_falling_and_rising_maxima(gamma, hq, hkv, gains):
    # three tiles of keys whose scores' scales differ by up to 16: each tile's probabilities are
    # taken against its own maximum, more than 2^8 above or below the others'
    inp = W.make_attn_inputs(2, gamma, hq, hkv, 128, 64, 192 - gamma, True, seed=77)
    k = inp.k_cache
    for b in range(2):
        for t in range(3):
            page = inp.page_table[b, t]
            x = (k[page].astype(np.uint32) << 16).view(np.float32) * np.float32(gains[t])
            k[page] = (torch.from_numpy(x).to(torch.bfloat16).view(torch.int16).numpy()).view(np.uint16)
    check_whole_and_split(inp)


@pytest.mark.parametrize("gamma,hq,hkv,dim", [(1, 8, 2, 128), (4, 8, 2, 128), (8, 8, 2, 128), (4, 16, 4, 128),
                                              (8, 16, 4, 128), (8, 16, 8, 64), (2, 12, 6, 64)])
@pytest.mark.parametrize("keys,seed", [(120, 1), (128, 2), (113, 3), (33, 4)])
def test_small_groups_short_units_falling_and_rising_maxima(oracle_mod, gamma, hq, hkv, dim, keys, seed):
    # units of at most eight stages (one, two and four key groups) whose pages' scores differ in
    # scale by up to 240, so that the stages' maxima rise and fall by far more than 2^2. P and
    # the output are bf16 (2^-8 relative each): an element is off by at most 2^-7 of
    # sum_k p_k |v_k| (the oracle's output with V's magnitudes), and 5% of it for the fp32 terms.
    inp = W.make_attn_inputs(3, gamma, hq, hkv, dim, 16, keys - gamma, True, seed=seed)
    gains = np.random.default_rng(seed).choice([0.05, 0.5, 1.0, 4.0, 12.0], inp.num_pages).astype(np.float32)
    x = (inp.k_cache.astype(np.uint32) << 16).view(np.float32) * gains[:, None, None, None]
    inp.k_cache[:] = torch.from_numpy(x).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    inp.kv_len[1] = max(gamma, keys - 37)
    out, lse = gpu_attention(inp, binding.ATTN_AUTO)
    args = (inp.page_table, inp.kv_len, gamma)
    o_out, o_lse, st = oracle_mod.verify_attention(inp.q, inp.k_cache, inp.v_cache, *args)
    o_abs, _, _ = oracle_mod.verify_attention(inp.q, inp.k_cache, inp.v_cache & np.uint16(0x7FFF), *args)
    assert np.all(st == 0)
    assert np.all(np.abs(out - o_out) <= 1.05 * 2.0 ** -7 * o_abs + 1e-6)
    np.testing.assert_allclose(lse, o_lse, rtol=0, atol=1e-3)


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 31, 32, 33, 34])  # up to 32: the small-group kernel
@pytest.mark.parametrize("hkv,dim,page", [(4, 128, 16), (2, 128, 64), (8, 64, 32), (6, 64, 16)])
def test_rows_at_the_kernels_edges(oracle_mod, rows, hkv, dim, page):
    inp = W.make_attn_inputs(3, rows, hkv, hkv, dim, page, (100, 900), True, seed=300 + rows)
    g_out, g_lse = gpu_attention(inp, binding.ATTN_AUTO)
    o_out, o_lse, st = oracle_attn(oracle_mod, inp)
    assert np.all(st == 0)
    compare_attention(g_out, g_lse, o_out, o_lse)
