"""GPU parity of mla_acceptance_stats (Sec. 3.3, Eqs. 9-10) against the fp64
oracle on the same seeded logits.

Bars: the argmaxes and the greedy decision are integers decided on the
logits themselves, so they must match exactly (lowest index on ties);
alpha_sample is an fp32 sum of ~10^5 probabilities formed with fp32
exponentials (each within a few ulp) and summed hierarchically (at most a few
hundred serial additions per thread, then trees), so its error is ~1e-5 at
most: the bar is 1e-4 absolute.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_27269_gb300 import abi
from paper_2607_27269_gb300 import workloads as wl
from tests.helpers import bf16_to_f64, bits

pytestmark = pytest.mark.gpu

ALPHA_TOL = 1e-4


def values(t: torch.Tensor) -> np.ndarray:
    return bf16_to_f64(bits(t)) if t.dtype == torch.bfloat16 else t.double().numpy()


def padded(x: torch.Tensor) -> torch.Tensor:
    """x on the GPU in rows padded to a 16-byte multiple (a view of the first vocab entries)."""
    per = 16 // x.element_size()
    stride = (x.shape[1] + per - 1) // per * per
    buf = torch.zeros(x.shape[0], stride, dtype=x.dtype, device="cuda")
    buf[:, :x.shape[1]] = x.cuda()
    return buf[:, :x.shape[1]]


def check(draft: torch.Tensor, target: torch.Tensor):
    alpha, ad, at, gr = abi.acceptance_stats(padded(draft), padded(target))
    torch.cuda.synchronize()
    ref = orc.acceptance(values(draft), values(target))
    assert np.array_equal(ad.cpu().numpy(), ref["argmax_draft"])
    assert np.array_equal(at.cpu().numpy(), ref["argmax_target"])
    assert np.array_equal(gr.cpu().numpy(), ref["greedy"])
    err = np.abs(alpha.cpu().numpy().astype(np.float64) - ref["alpha_sample"])
    assert err.max() <= ALPHA_TOL, err.max()
    return ref


@pytest.mark.parametrize("name", wl.ORDER)
def test_acceptance_matches_oracle(name):
    lg = wl.logits(name, seed=51, rows=6)
    ref = check(lg.draft, lg.target)
    assert 0.05 < ref["alpha_sample"].mean() < 0.99      # the inputs exercise the overlap, not an edge


def test_acceptance_fp32_logits_and_identical_rows():
    lg = wl.logits("qwen05b_b16_h14_r256_t2048", seed=52, rows=5)
    check(lg.draft.float(), lg.target.float())
    ref = check(lg.target, lg.target)
    assert np.all(ref["greedy"] == 1)


def test_acceptance_ties_ragged_and_tiny_vocabularies():
    g = torch.Generator().manual_seed(53)
    for vocab in (13, 1003, 40961):
        d = (torch.randn(4, vocab, generator=g) * 2).to(torch.bfloat16)
        t = (torch.randn(4, vocab, generator=g) * 2).to(torch.bfloat16)
        # equal maxima far apart (different slices of the cluster): the lowest index wins
        d[0, vocab - 1] = d[0, 0] = 30.0
        t[1, vocab // 2] = t[1, 1] = 30.0
        check(d, t)


def test_acceptance_row_stride_and_empty():
    g = torch.Generator().manual_seed(54)
    full = (torch.randn(3, 1008, generator=g) * 3).to(torch.bfloat16).cuda()
    full2 = (torch.randn(3, 1008, generator=g) * 3).to(torch.bfloat16).cuda()
    d, t = full[:, :1001], full2[:, :1001]          # rows 1008 apart, 1001 tokens used
    alpha, ad, at, gr = abi.acceptance_stats(d, t)
    ref = orc.acceptance(values(d.cpu()), values(t.cpu()))
    assert np.array_equal(ad.cpu().numpy(), ref["argmax_draft"])
    assert np.abs(alpha.cpu().numpy() - ref["alpha_sample"]).max() <= ALPHA_TOL
    e = torch.empty(0, 100, dtype=torch.bfloat16, device="cuda")
    abi.acceptance_stats(e, e)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_acceptance_many_rows_ties_ragged_and_strided(dtype):
    """160 rows (clusters of two or more CTAs, or one a row): ragged vocabularies (a tail past the last
    whole vector; a vocabulary shorter than one vector), equal maxima far
    apart (the lowest index wins), identical rows (greedy agreement, alpha =
    1) and rows padded to a longer stride -- every row against the oracle."""
    g = torch.Generator().manual_seed(56)
    rows = 160
    for vocab in (7, 1003, 40961):
        d = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
        t = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
        d[0, vocab - 1] = d[0, 0] = 30.0
        t[1, vocab // 2] = t[1, 1] = 30.0
        d[rows - 1, vocab - 1] = 40.0  # the maximum in the tail
        t[7] = d[7]
        ref = check(d, t)
        assert ref["greedy"][7] == 1 and abs(ref["alpha_sample"][7] - 1.0) < 1e-12
    # rows 1040 entries apart, 1001 used
    full = (torch.randn(rows, 1040, generator=g) * 3).to(dtype).cuda()
    full2 = (torch.randn(rows, 1040, generator=g) * 3).to(dtype).cuda()
    dd, tt = full[:, :1001], full2[:, :1001]
    alpha, ad, at, gr = abi.acceptance_stats(dd, tt)
    ref = orc.acceptance(values(dd.cpu()), values(tt.cpu()))
    assert np.array_equal(ad.cpu().numpy(), ref["argmax_draft"])
    assert np.array_equal(at.cpu().numpy(), ref["argmax_target"])
    assert np.abs(alpha.cpu().numpy().astype(np.float64) - ref["alpha_sample"]).max() <= ALPHA_TOL


@pytest.mark.parametrize("name", ["qwen05b_b16_h14_r256_t2048", "llama1b_paged_b128_h32_r512_t128_8192"])
def test_acceptance_full_rows_sampled(name):
    """Every row of the workload on the GPU (the size bench.py times); the
    oracle checks a sample of rows."""
    lg = wl.logits(name, seed=55)
    alpha, ad, at, gr = abi.acceptance_stats(lg.draft.cuda(), lg.target.cuda())
    rows = lg.draft.shape[0]
    pick = np.unique(np.linspace(0, rows - 1, 8).astype(int))
    ref = orc.acceptance(values(lg.draft[pick]), values(lg.target[pick]))
    assert np.array_equal(ad.cpu().numpy()[pick], ref["argmax_draft"])
    assert np.array_equal(gr.cpu().numpy()[pick], ref["greedy"])
    assert np.abs(alpha.cpu().numpy()[pick] - ref["alpha_sample"]).max() <= ALPHA_TOL


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rows,vocab", [(2, 1), (3, 8), (2, 2049), (5, 4099), (700, 515), (61, 9001), (1200, 37)])
def test_acceptance_masked_logits_and_cluster_sizes(rows, vocab, dtype):
    """Few and many rows, clusters of one, seven and eight CTAs (the sizes
    these shapes are given), slices with no vector at all, groups that end
    inside and several rows per cluster; logits masked with -inf and with the type's lowest value (whole vectors of
    them, a thread's first ones included) weigh nothing.  Error: the sums are
    trees of fp32 exponentials, as above."""
    g = torch.Generator().manual_seed(57)
    d = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
    t = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
    low = torch.finfo(dtype).min
    keep = max(1, vocab // 3)
    d[0, keep:] = float("-inf")
    t[0, :vocab - keep] = float("-inf")
    d[1, keep:] = low
    t[1, keep:] = low
    check(d, t)
    if vocab > 40:
        d[rows - 1, : vocab // 2] += 60.0  # the base is raised late, and by much
        t[rows - 1, vocab // 2:] += 60.0
        check(d, t)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("cluster", range(1, 9))
def test_acceptance_every_cluster_size(cluster, dtype, tuning):
    """Each cluster size, also those that no shape above is given: three rows
    and more a cluster (both sets of exchange slots are used again; up to 456
    clusters run at a time), slices of unequal length, a tail past the last
    whole vector, fewer vectors than CTAs, equal maxima in different slices (the
    first wins), rows whose maximum every CTA but one has not seen."""
    tuning(GBMLA_ACCEPT_CLUSTER=cluster)
    g = torch.Generator().manual_seed(58)
    rows, n = 3 * 456 + 5, 16 // torch.empty((), dtype=dtype).element_size()
    for vocab in (3 * n + 1, 8 * n, 1003, 4099):
        d = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
        t = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
        at = torch.randint(0, vocab, (rows, 2), generator=g)
        r = torch.arange(rows)
        d[r, at[:, 0]] = d[r, at[:, 1]] = 12.0
        t[r[::2], at[::2, 1]] = 12.0
        t[r[1::2], at[1::2, 0]] = 12.0
        ref = check(d, t)
        assert 0 < ref["greedy"].mean() < 1


@pytest.mark.parametrize("rows,vocab,dtype", [(512, 32000, torch.bfloat16), (560, 50257, torch.float32),
                                              (640, 128256, torch.float32)])
def test_acceptance_cluster_choice(rows, vocab, dtype, tuning):
    """The size that the launcher picks is near the fastest of the eight where
    they differ most (waves that the rows do not fill; rows past the L2's size).
    The model is within a few percent; the bar leaves room for other load on the
    GPU, and the worst sizes take two to three times the best one's time."""
    target = torch.randn(rows, (vocab + 7) // 8 * 8, device="cuda")
    draft = (target + torch.randn_like(target)).to(dtype)[:, :vocab]
    target = target.to(dtype)[:, :vocab]
    out = [torch.empty(rows, dtype=t, device="cuda") for t in (torch.float32,) + 3 * (torch.int32,)]

    def us(size):
        tuning(GBMLA_ACCEPT_CLUSTER=size)
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(20):
                abi.acceptance_stats(draft, target, *out)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 50)
        return min(times)

    picked, each = us(0), [us(size) for size in range(1, 9)]
    assert picked <= 1.25 * min(each), (picked, each)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("mask", [-1e4, -65504.0, -1e9, -1e10, -1e20, -1e30, -1e38])
@pytest.mark.parametrize("rows,vocab", [(15, 73), (11, 536), (40, 4096), (9, 50257)])
def test_acceptance_finite_masks(rows, vocab, mask, dtype):
    """Masks by a large negative number: most of a row, whole vectors and threads'
    whole shares of it, weigh nothing, as -inf does."""
    g = torch.Generator().manual_seed(59)
    d = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
    t = (torch.randn(rows, vocab, generator=g) * 2).to(dtype)
    for share in (0.3, 0.9, 0.999):
        out = torch.rand(rows, vocab, generator=g) < share
        out[:, vocab // 2] = False
        check(d.masked_fill(out, mask), t.masked_fill(out, mask))
