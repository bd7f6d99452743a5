"""The tensor-core attention's walk over a partition's tiles where it changes
gear: more than 32 sequences in a partition (they are scanned 32 at a time),
more than 32 tiles of one paged sequence (so are its pages), and scores that
outgrow the exponent base of their column (the base moves, O^T is rescaled).

Outputs against the fp64 oracle within the step's bar; the moving bases against
the CUDA-core kernel, which reads the same bf16 queries (at scores of some
hundreds the rounding of the queries alone would exceed the oracle's bar)."""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest

from paper_2607_27269_gb300 import abi
from paper_2607_27269_gb300 import workloads as wl
from tests.helpers import oracle_step
from tests.test_gpu_parity import assert_close, run_step

pytestmark = pytest.mark.gpu

PAGED = "llama1b_paged_b128_h32_r512_t128_8192"


@pytest.mark.parametrize("q_len", [1, 5])  # 32 and 2 x 80 query rows
@pytest.mark.parametrize("batch,kv_range,splits", [
    (70, (6, 140), 1),       # 70 sequences in one partition: three scans
    (33, (6, 140), 2),
    (2, (4200, 5500), 1),    # 33 to 43 tiles of one sequence, two pages each
    (3, (4097, 4225), 2),    # a partition that begins inside a sequence
])
def test_walk_over_many_sequences_and_pages(q_len, batch, kv_range, splits):
    s = dataclasses.replace(wl.SHAPES[PAGED], q_len=q_len)
    w = wl.make(s, seed=61, batch=batch, kv_range=kv_range)
    step = run_step(abi.to_device(w), num_splits=splits)
    seqs = sorted({0, batch // 2, min(31, batch - 1), min(32, batch - 1), batch - 1})
    ref = oracle_step(w, seqs=seqs)
    assert_close(step.o_lat.cpu().numpy()[seqs], np.asarray(ref["o_lat"])[seqs], "o_lat")
    assert_close(step.lse.cpu().numpy()[seqs], np.asarray(ref["lse"])[seqs], "lse")


@pytest.mark.parametrize("q_len", [1, 5])
@pytest.mark.parametrize("splits", [1, 3])
def test_exponent_bases_move(q_len, splits, tuning):
    s = dataclasses.replace(wl.SHAPES[PAGED], q_len=q_len)
    w = wl.make(s, seed=62, batch=3, kv_range=(900, 1200))
    for b in range(3):
        for t in range(int(w.start_pos[b])):
            # tile by tile larger and smaller scores, the largest late
            f = (1.0, 8.0, 0.25, 16.0, 2.0, 32.0, 1.0, 24.0, 4.0, 1.0)[min(t // 128, 9)]
            page, slot = int(w.block_table[b, t // s.page_size]), t % s.page_size
            w.c_kv[page, slot] *= f
            w.k_rope[page, slot] *= f
    res = {}
    for kern in ("simt", "tc"):
        tuning(GBMLA_ATTN_KERNEL=kern)
        step = run_step(abi.to_device(w), num_splits=splits)
        res[kern] = (step.o_lat.cpu().numpy().astype(np.float64), step.lse.cpu().numpy().astype(np.float64))
    assert np.ptp(res["simt"][1]) > 50  # (the scores did grow)
    assert_close(res["tc"][0], res["simt"][0], "o_lat")
    assert np.abs(res["tc"][1] - res["simt"][1]).max() < 1e-2
