"""GPU parity of the original-GQA decode path (mla_gqa_append,
mla_gqa_decode_attn; Sec. 3.1 Eqs. 1-4) against the fp64 oracle on the same
seeded inputs, at every workload's shape.

Bars: appended values bit-exact and keys within one bf16 rounding of the
exact rotation (as for the MLA append); attention outputs within
max|d| <= 2e-2 max|ref| and mean relative error <= 5e-3 (the softmax weights
are rounded to bf16 before they multiply the bf16 values, as in the MLA path).
"""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_27269_gb300 import abi
from paper_2607_27269_gb300 import workloads as wl
from tests.helpers import bf16_to_f64, bits, rel_errors

pytestmark = pytest.mark.gpu

MAX_TOL, MEAN_TOL = 2e-2, 5e-3


def assert_close(got, ref, what):
    mx, mean = rel_errors(got, ref)
    assert mx <= MAX_TOL and mean <= MEAN_TOL, f"{what}: max {mx:.3e} mean {mean:.3e}"


def devices(gw, splits=0):
    s = gw.shape
    dims = abi.GqaDims(gw.num_heads, gw.num_kv_groups, gw.d, gw.sm_scale, s.rope_style, s.rope_base)
    bt = None if gw.block_table is None else gw.block_table.cuda()
    cache = abi.Cache(gw.v_cache.cuda(), gw.k_cache.cuda(), gw.capacity, bt, s.page_size if s.paged else 0,
                      gw.num_pages)
    step = abi.GqaStep(dims, cache, gw.kv_len.numel(), gw.q.shape[1], int(gw.kv_len.max()), splits)
    return dims, cache, step


def oracle_run(gw):
    s = gw.shape
    dims = orc.GqaDims(gw.num_heads, gw.num_kv_groups, gw.d, gw.d, gw.sm_scale, s.rope_style, s.rope_base)
    bt = None if gw.block_table is None else gw.block_table.numpy().astype(np.int32).copy()
    cache = orc.Cache(c_kv=bits(gw.v_cache), k_rope=bits(gw.k_cache), c_tok_stride=gw.d, r_tok_stride=gw.d,
                      c_blk_stride=gw.k_cache.shape[1] * gw.d, r_blk_stride=gw.k_cache.shape[1] * gw.d,
                      capacity=gw.capacity, block_table=bt, page_size=s.page_size if s.paged else 0,
                      num_pages=gw.num_pages)
    orc.gqa_append(dims, cache, bits(gw.k_new), bits(gw.v_new), gw.start_pos.numpy())
    res = orc.gqa_decode(dims, cache, bits(gw.q), gw.kv_len.numpy())
    return cache, res


def run(gw, splits=0):
    dims, cache, step = devices(gw, splits)
    abi.gqa_append(dims, cache, gw.k_new.cuda(), gw.v_new.cuda(), gw.start_pos.cuda())
    o = step(gw.q.cuda(), gw.kv_len.cuda())
    code = abi.check_status()
    assert code == abi.MLA_OK, abi.status_name(code)
    return cache, step


@pytest.mark.parametrize("name", wl.ORDER)
def test_gqa_decode_matches_oracle(name):
    w = wl.small(name, seed=61)
    gw = wl.gqa(w, seed=61)
    cache, step = run(gw)
    ocache, ref = oracle_run(gw)
    # the append: values bit-exact, keys within one rounding, nothing else touched
    assert np.array_equal(bits(cache.c_kv.cpu()), ocache.c_kv)
    got_k = bits(cache.k_rope.cpu()).astype(np.int32)
    d = np.abs(got_k - ocache.k_rope.astype(np.int32))
    assert d.max() <= 1 and (d > 0).mean() < 0.01
    assert_close(step.o.cpu().numpy(), ref["o"], "o")
    assert_close(step.lse.cpu().numpy(), ref["lse"], "lse")


@pytest.mark.parametrize("splits", [1, 3, 7])
def test_gqa_split_counts_and_paged(splits):
    """Several units per CTA and ragged tails in both layouts; the paged and
    contiguous runs of the same logical cache agree bit for bit."""
    shape = wl.SHAPES["llama1b_paged_b128_h32_r512_t128_8192"]
    wp = wl.make(shape, seed=62, batch=4, kv_range=(70, 650))
    gp = wl.gqa(wp, seed=62)
    cache_p, step_p = run(gp, splits)
    ocache, ref = oracle_run(gp)
    G = gp.num_kv_groups
    assert_close(step_p.o.cpu().numpy(), ref["o"], "o")
    # the same logical cache laid out contiguously
    cap = int(gp.kv_len.max())
    B, d = 4, gp.d
    kc = torch.zeros(B * G, cap, d, dtype=torch.bfloat16)
    vc = torch.zeros(B * G, cap, d, dtype=torch.bfloat16)
    for u in range(B * G):
        for t in range(int(gp.kv_len[u // G]) - shape.q_len):     # the rows before this step's append
            pg = int(gp.block_table[u, t // 64])
            kc[u, t], vc[u, t] = gp.k_cache[pg, t % 64], gp.v_cache[pg, t % 64]
    gc = dataclasses.replace(gp, shape=dataclasses.replace(shape, paged=False), k_cache=kc, v_cache=vc,
                             block_table=None, num_pages=0, capacity=cap)
    _, step_c = run(gc, splits)
    assert torch.equal(step_p.o.cpu(), step_c.o.cpu())


@pytest.mark.parametrize("hpg,q_len,d,paged,style", [
    (1, 1, 64, False, 0), (3, 1, 128, True, 1), (8, 1, 128, False, 0), (3, 3, 64, True, 0), (5, 5, 64, False, 1),
    (6, 4, 128, True, 0), (5, 5, 128, False, 0), (8, 4, 64, True, 1), (11, 3, 64, False, 0), (8, 6, 128, False, 1),
    (7, 8, 64, True, 0), (8, 16, 64, False, 0), (8, 16, 128, True, 0)])
def test_gqa_row_counts_and_stage_tails(hpg, q_len, d, paged, style):
    """Query rows from 1 to 128 (one to eight row groups of 8 or 16 rows, as so
    few tiles take) against units that end around every load stage and tile
    boundary; rows past a unit's end hold NaN and must not reach an output."""
    check_row_counts_and_stage_tails(hpg, q_len, d, paged, style)


@pytest.mark.parametrize("width", [8, 16, 24, 32])
@pytest.mark.parametrize("hpg,q_len,d,paged,style", [
    (3, 3, 64, True, 0), (5, 5, 64, False, 1), (6, 4, 128, True, 0), (5, 5, 128, False, 0), (8, 4, 64, True, 1),
    (8, 6, 128, False, 1), (7, 8, 64, True, 0), (8, 16, 64, False, 0), (8, 16, 128, True, 0)])
def test_gqa_row_widths(hpg, q_len, d, paged, style, width, tuning):
    """The same with warps of up to 8, 16, 24 and 32 rows (24 at most at width
    128), which batches of many tiles take."""
    tuning(GBMLA_GQA_ROWS=width)
    check_row_counts_and_stage_tails(hpg, q_len, d, paged, style)


def check_row_counts_and_stage_tails(hpg, q_len, d, paged, style):
    lens = [1, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 192, 300]
    G, B = 2, len(lens)
    shape = wl.Shape("rows", B, hpg * G, G, d, 64, d, 128, 0, q_len, 300, 300, paged=paged, rope_style=style)
    w = wl.make(shape, seed=63)
    w.kv_len = torch.tensor([max(t, q_len) for t in lens], dtype=torch.int32)
    w.start_pos = w.kv_len - q_len
    gw = wl.gqa(w, seed=63)
    for u in range(B * G):
        kv = int(gw.kv_len[u // G])
        for t in range(kv, -(-kv // 64) * 64 if paged else gw.capacity):
            at = (int(gw.block_table[u, t // 64]), t % 64) if paged else (u, t)
            gw.k_cache[at] = float("nan")
            gw.v_cache[at] = float("nan")
    _, step = run(gw)
    _, ref = oracle_run(gw)
    assert_close(step.o.cpu().numpy(), ref["o"], "o")
    assert_close(step.lse.cpu().numpy(), ref["lse"], "lse")


@pytest.mark.parametrize("heads,groups,d", [(64, 8, 64), (32, 8, 64), (40, 8, 128), (14, 2, 64)])
@pytest.mark.parametrize("splits", [0, 5])
def test_gqa_workspace_covers_smaller_calls(heads, groups, d, splits):
    """Buffers sized once for the longest chunk, batch and cache hold every
    smaller call's partials (units + S - 1 slots of q_len * H/G rows), although
    its partition count may be the larger one."""
    dims = abi.GqaDims(heads, groups, d, d ** -0.5)
    for batch, q_len, kv in [(8, 5, 2048), (8, 16, 2200), (3, 16, 900), (61, 7, 4096)]:
        if q_len * heads // groups > 128:
            continue
        o_bytes, lse_bytes, _ = abi.gqa_workspace_size(dims, batch, q_len, kv, splits)
        for b in range(1, batch + 1, 1 + batch // 8):
            for q in range(1, q_len + 1):
                for t in range(q, kv + 1, 1 + kv // 50):
                    s = abi.gqa_workspace_size(dims, b, q, t, splits)[2]
                    rows = (b * groups + s - 1) * q * (heads // groups)
                    assert rows * d * 4 <= o_bytes and rows * 4 <= lse_bytes, (b, q, t, s)


def test_gqa_shorter_chunk_in_the_longest_chunks_buffers():
    """8 heads a group, 64 units of up to 2048 tokens: four queries are one row
    group and take more partitions than five, and twice as many slots.  With
    num_splits 0 in buffers sized for five queries nothing past them is written
    and the results are those of buffers of their own."""
    B, G, d, cap = 8, 8, 64, 2048
    g = torch.Generator(device="cuda").manual_seed(64)
    k, v = (torch.randn(B * G, cap, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn(B, 4, 8 * G, d, generator=g, device="cuda").bfloat16()
    kv = torch.tensor([cap - 97 * b for b in range(B)], dtype=torch.int32, device="cuda")
    dims, cache = abi.GqaDims(8 * G, G, d, d ** -0.5), abi.Cache(v, k, cap)
    own = abi.GqaStep(dims, cache, B, 4, cap)
    want = own(q, kv).clone()
    o_bytes, lse_bytes, _ = abi.gqa_workspace_size(dims, B, 5, cap)
    step = abi.GqaStep(dims, cache, B, 4, cap)
    step.num_splits = 0
    step.o_part = torch.full((o_bytes // 4 + (1 << 22),), 7.0, device="cuda")    # sized for five queries, and a guard
    step.lse_part = torch.full((lse_bytes // 4 + (1 << 16),), 7.0, device="cuda")
    step(q, kv)
    assert abi.check_status() == abi.MLA_OK
    assert torch.equal(step.o, want) and torch.equal(step.lse, own.lse)
    assert (step.o_part[o_bytes // 4:] == 7.0).all() and (step.lse_part[lse_bytes // 4:] == 7.0).all()


@pytest.mark.parametrize("lens", [(200, 301, 150), (200, 2, 150), (301, 2, -5), (0, 0, 0)])
def test_gqa_lengths_that_cannot_be_served_are_recorded(lens):
    """A length above the stated maximum or below q_len: recorded, the unit
    left out, the other units right; nothing but such lengths too."""
    q_len, most = 3, 300
    shape = wl.Shape("lens", len(lens), 8, 2, 64, 64, 64, 128, 0, q_len, most, most)
    gw = wl.gqa(wl.make(shape, seed=65), seed=65)
    dims, cache, step = devices(gw)
    abi.gqa_append(dims, cache, gw.k_new.cuda(), gw.v_new.cuda(), gw.start_pos.cuda())
    good = torch.tensor([n if q_len <= n <= most else q_len for n in lens], dtype=torch.int32, device="cuda")
    step(gw.q.cuda(), good)
    assert abi.check_status() == abi.MLA_OK
    want = step.o.clone()
    step(gw.q.cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda"))
    assert abi.check_status() == abi.MLA_ERR_DEVICE_BOUNDS
    for b, n in enumerate(lens):
        if q_len <= n <= most:
            # another partition of the tiles: other roundings of the weights, as in the bars above
            assert_close(step.o[b].cpu().numpy(), want[b].cpu().numpy(), f"o[{b}]")


@pytest.mark.parametrize("at", [5, 40, 70, 127])
@pytest.mark.parametrize("d", [64, 128])
def test_gqa_largest_weight_of_the_first_tile_is_exact(d, at):
    """One token of 128 outweighs each other one 128.5 times, a ratio halfway
    between two bf16 values.  The exponent base is the maximum of the first
    tile, wherever in it that lies: the large weight is 1 and the small ones
    1/128.5, which bf16 holds to 1.6e-5.  (Over a base of 1 the large weight would
    be 128, and the output 2e-3 off.)  Values +1 and -1: o = (128.5 - 127) /
    (128.5 + 127), each weight's error halved."""
    k = torch.zeros(1, 128, d, dtype=torch.bfloat16)
    v = torch.full((1, 128, d), -1.0, dtype=torch.bfloat16)
    q = torch.zeros(1, 1, 1, d, dtype=torch.bfloat16)
    k[0, at, d // 2 - 1] = q[0, 0, 0, d // 2 - 1] = 1.0  # a pair that a base of 1e30 does not turn
    v[0, at] = 1.0
    dims = abi.GqaDims(1, 1, d, float(np.log(128.5)), 0, 1e30)
    step = abi.GqaStep(dims, abi.Cache(v.cuda(), k.cuda(), 128), 1, 1, 128)
    o = step(q.cuda(), torch.tensor([128], dtype=torch.int32, device="cuda"))
    assert abi.check_status() == abi.MLA_OK
    assert (o.double() - 1.5 / 255.5).abs().max().item() <= 2e-5
