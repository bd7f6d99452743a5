"""The grouped GEMM at the sizes where its tilings can go wrong: rows just past
a tile and unevenly divided, output widths past a whole block of columns and not
a multiple of eight or four, split and unsplit K, the projection's column tiles.

Both products are compared with fp64 sums of the very operands they read (W_O
of the o that W_UV wrote), so the bar is one rounding to bf16 of an fp32 sum:
half a unit in the last place plus the accumulation error of the fp32 sum, a
bound proportional to the sum of the products' magnitudes."""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest
import torch

from paper_2607_27269_gb300 import abi
from paper_2607_27269_gb300 import workloads as wl
from tests.helpers import bf16_to_f64, bits, oracle_step, rel_errors
from tests.test_gpu_project import assert_one_rounding, check_projection, run_projection

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,heads,groups,rank,d_v,hidden", [
    (1, 8, 8, 512, 64, 264),      # one row, K split four ways, a part block of eight columns
    (65, 32, 8, 512, 64, 2048),   # two tiles of 33 rows
    (129, 32, 8, 512, 64, 2056),  # two tiles of 65 rows, split over a cluster, eight columns in the last tile
    (160, 32, 8, 512, 64, 1030),  # split; rows of C at odd multiples of four bytes
    (160, 4, 2, 128, 64, 1030),   # the same rows unsplit (K of four chunks)
    (64, 4, 2, 128, 64, 1024),    # the tallest tile of 64-row products, unsplit
    (17, 4, 2, 128, 64, 1030),    # the same products, rows of C at odd multiples of four bytes
    (13, 14, 2, 256, 64, 898),    # short tiles, split, rows of C at odd multiples of four bytes
    (200, 32, 8, 512, 64, 2048),  # two tiles of 100 rows, 128 columns wide, split
    (384, 32, 8, 512, 64, 2044),  # three tiles, 64 columns wide, unsplit
    (300, 8, 4, 256, 128, 516),   # unsplit, rows of C eight-byte aligned
    (700, 16, 4, 192, 40, 1024),  # 40-wide heads, three chunks of rank
    (640, 32, 8, 512, 64, 264),   # more tiles of o_lat than SMs: 68 rows each, two CTAs an SM
    (96, 16, 4, 512, 128, 512),   # 128-wide heads, a ring of four stages under eight chunks
    (41, 80, 80, 512, 128, 512),  # one head a group, 128 columns: the last stage's rows read past the ring
    (48, 80, 80, 512, 128, 264),  # the tallest such tile
    (45, 40, 40, 512, 256, 264),  # two column tiles a group
])
def test_out_proj_tiles(rows, heads, groups, rank, d_v, hidden):
    g = torch.Generator().manual_seed(rows + hidden)
    o_lat = torch.randn(rows, 1, heads, rank, generator=g)
    w_uv = (torch.randn(groups, d_v, rank, generator=g) * rank ** -0.5).bfloat16()
    w_o = (torch.randn(hidden, heads * d_v, generator=g) * (heads * d_v) ** -0.5).bfloat16()
    o = torch.full((rows, 1, heads, d_v), 7.0, dtype=torch.bfloat16, device="cuda")
    out = torch.full((rows + 1, 1, hidden), 7.0, dtype=torch.bfloat16, device="cuda")  # one guard row
    d = abi.Dims(heads, groups, 64, 64, d_v, rank, hidden)
    abi.out_proj(d, o_lat.cuda(), w_uv.cuda(), w_o.cuda(), o, out[:rows])
    assert abi.check_status() == abi.MLA_OK
    a = bf16_to_f64(bits(o_lat.bfloat16())).reshape(rows, groups, heads // groups, rank)  # the GEMM reads o_lat as bf16
    u = bf16_to_f64(bits(w_uv))
    exact = np.einsum("tghr,gvr->tghv", a, u)
    mag = np.einsum("tghr,gvr->tghv", np.abs(a), np.abs(u))
    got = bits(o.cpu())
    shape = (rows, 1, heads, d_v)
    assert_one_rounding(got, exact.reshape(shape), mag.reshape(shape), "o")
    a, u = bf16_to_f64(got).reshape(rows, heads * d_v), bf16_to_f64(bits(w_o))
    got = bits(out.cpu())
    assert_one_rounding(got[:rows, 0], a @ u.T, np.abs(a) @ np.abs(u).T, "out")
    assert (out[rows:] == 7.0).all()


@pytest.mark.parametrize("rows", [1, 8, 17, 20, 24, 25, 32, 33, 65])
@pytest.mark.parametrize("hidden,heads", [(3072, 24), (4096, 32), (5120, 40)])
def test_gqa_out_proj_tiles(rows, hidden, heads):
    """An fp32 activation as wide as the output against a few dozen rows: rings
    of many short stages, K split and not; 17 to 32 rows leave the last stage's
    products reading past the ring."""
    g = torch.Generator().manual_seed(rows + hidden)
    width = heads * 128
    o = torch.randn(rows, 1, heads, 128, generator=g)
    w_o = (torch.randn(hidden, width, generator=g) * width ** -0.5).bfloat16()
    out = torch.full((rows + 1, 1, hidden), 7.0, dtype=torch.bfloat16, device="cuda")  # one guard row
    abi.gqa_out_proj(abi.GqaDims(heads, 8, 128, 128 ** -0.5), o.cuda(), w_o.cuda(), out[:rows])
    assert abi.check_status() == abi.MLA_OK
    a, u = bf16_to_f64(bits(o.bfloat16())).reshape(rows, width), bf16_to_f64(bits(w_o))  # the GEMM reads o as bf16
    assert_one_rounding(bits(out.cpu())[:rows, 0], a @ u.T, np.abs(a) @ np.abs(u).T, "out")
    assert (out[rows:] == 7.0).all()


@pytest.mark.parametrize("rows", [41, 48])
def test_decode_step_many_single_head_groups(rows):
    """The whole step where W_UV runs one head a group in tiles of 41 to 48 rows."""
    s = wl.Shape("groups80", rows, 80, 80, 64, 32, 128, 512, 0, 1, 70, 200)
    w = wl.make(s, seed=45)
    dw = abi.to_device(w)
    step = abi.DecodeStep(dw.dims, dw.cache, rows, 1, dw.max_kv_len)
    step(dw.q_nope, dw.q_pe, dw.kv_len, dw.w_uk, dw.w_uv, None, c_new=dw.c_new, kr_new=dw.kr_new, start_pos=dw.start_pos)
    assert abi.check_status() == abi.MLA_OK
    mx, mean = rel_errors(bf16_to_f64(bits(step.o.cpu())), oracle_step(w)["o"])
    assert mx <= 2e-2 and mean <= 5e-3, (mx, mean)  # the bars of the parity tests


@pytest.mark.parametrize("name,batch,n_new,rank,heads,with_q", [
    ("llama1b_chunk5_b32_h32_r512_t4096", 26, 5, 320, 16, True),   # 130 rows: two tiles of 65, rank past a column tile
    ("llama1b_chunk5_b32_h32_r512_t4096", 100, 5, 512, 32, True),  # 500 rows, four tiles
    ("llama1b_chunk5_b32_h32_r512_t4096", 300, 5, 512, 32, True),  # 1500 rows: several waves
    ("qwen05b_b16_h14_r256_t2048", 17, 1, 256, 14, True),          # 17 rows: short stages
    ("llama1b_chunk5_b32_h32_r512_t4096", 129, 1, 192, 32, False), # no queries
])
def test_projection_tiles(name, batch, n_new, rank, heads, with_q):
    s = dataclasses.replace(wl.SHAPES[name], rank=rank, num_heads=heads, q_len=n_new)
    w = wl.make(s, seed=44, batch=batch, kv_range=(s.q_len + 1, 60))
    p = wl.projection(w, seed=44)
    dw, qn, qp = run_projection(w, p, with_q)
    check_projection(w, p, dw, qn, qp, with_q)
