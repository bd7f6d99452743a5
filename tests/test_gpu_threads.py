"""Host threads that call the library at the same time, each on its own stream
and with shapes of its own: a launch must not depend on what another thread
sets for its launch of the same kernel (the shared memory a kernel may ask for
is one value per kernel, not per launch)."""
from __future__ import annotations

import threading

import pytest
import torch

from paper_2607_27269_gb300 import abi

pytestmark = pytest.mark.gpu


def _out_proj(rows, rank, heads, seed):
    """A call of W_UV and W_O (2 groups, 64 columns out) and the buffer it writes last."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape, dtype=torch.bfloat16):
        return torch.randn(*shape, generator=g, device="cuda").to(dtype)

    o_lat, w_uv, w_o = normal(rows, 1, heads, rank, dtype=torch.float32), normal(2, 64, rank), normal(64, heads * 64)
    o, out = (torch.empty(rows, 1, *n, dtype=torch.bfloat16, device="cuda") for n in ((heads, 64), (64,)))
    d = abi.Dims(heads, 2, 64, 64, 64, rank, 64)
    return lambda: abi.out_proj(d, o_lat, w_uv, w_o, o, out), out


def _project(rows, hidden, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda").bfloat16()

    cache = abi.Cache(normal(rows, 4, 128), normal(rows, 4, 64), 4)
    h, w_dkv, w_kr = normal(rows, 1, hidden), normal(128, hidden), normal(64, hidden)
    start = torch.zeros(rows, dtype=torch.int32, device="cuda")
    d = abi.Dims(8, 2, 64, 64, 64, 128, hidden)
    return lambda: abi.project_append(d, cache, h, w_dkv, w_kr, None, start), cache.c_kv[:, :1]


def _absorb(rows, rank, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda").bfloat16()

    q_nope, q_pe, w_uk = normal(rows, 1, 8, 64), normal(rows, 1, 8, 64), normal(2, 64, rank)
    kv = torch.full((rows,), 9, dtype=torch.int32, device="cuda")
    q_abs = torch.empty(rows, 1, 8, rank + 64, dtype=torch.bfloat16, device="cuda")
    d = abi.Dims(8, 2, 64, 64, 64, rank)
    return lambda: abi.absorb_q(d, q_nope, q_pe, kv, w_uk, q_abs), q_abs


def _attn(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda").bfloat16()

    d = abi.Dims(8, 2, 64, 64, 64, 128, sm_scale=128 ** -0.5)
    cache = abi.Cache(normal(2, 256, 128), normal(2, 256, 64), 256)
    kv, q_abs = torch.full((2,), 200, dtype=torch.int32, device="cuda"), normal(2, 1, 8, 192)
    o_bytes, lse_bytes, splits = abi.workspace_size(d, 2, 1, 200)
    o_part, lse_part = torch.empty(o_bytes // 4, device="cuda"), torch.empty(lse_bytes // 4, device="cuda")
    o_lat = torch.empty(2, 1, 8, 128, device="cuda")

    def call():
        abi.decode_attn(d, cache, kv, 200, q_abs, o_part, lse_part, splits)
        abi.combine(d, 2, 1, kv, 200, o_part, lse_part, o_lat, None, splits)

    return call, o_lat


def _gqa(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda").bfloat16()

    kv, q = torch.full((2,), 200, dtype=torch.int32, device="cuda"), normal(2, 1, 8, 64)
    step = abi.GqaStep(abi.GqaDims(8, 2, 64, 0.125), abi.Cache(normal(4, 256, 64), normal(4, 256, 64), 256), 2, 1, 200)
    return lambda: step(q, kv), step.o


@pytest.mark.parametrize("make", [lambda: _out_proj(5, 128, 8, 7), lambda: _project(5, 64, 8),
                                  lambda: _absorb(5, 128, 9), lambda: _attn(10), lambda: _gqa(11)],
                         ids=["out_proj", "project", "absorb", "attn", "gqa"])
def test_a_threads_first_call(make):
    """A host thread that has made no CUDA call yet has no context: the
    library's call is the first, and tensor maps cannot be encoded without one."""
    call, out = make()
    call()
    torch.cuda.synchronize()
    want = out.clone()
    out.zero_()
    torch.cuda.synchronize()
    errors = []

    def work():
        try:
            call()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert not errors, errors[0]
    assert abi.check_status() == abi.MLA_OK
    torch.cuda.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("small,large", [
    (lambda: _out_proj(1, 64, 8, 1), lambda: _out_proj(64, 512, 32, 2)),
    (lambda: _project(1, 64, 3), lambda: _project(64, 2048, 4)),
    (lambda: _absorb(1, 128, 5), lambda: _absorb(2048, 512, 6)),
], ids=["out_proj", "project", "absorb"])
def test_threads_with_different_shapes(small, large, monkeypatch):
    calls = [make() for _ in range(4) for make in (small, large)]
    streams = [torch.cuda.Stream() for _ in calls]
    raw = []  # each call's library function and arguments: a loop over them leaves the threads little time in Python

    class Recorder:
        def __getattr__(self, name):
            return lambda *args: raw.append((getattr(library, name), args)) or abi.MLA_OK

    library = abi.lib()
    with monkeypatch.context() as m:
        m.setattr(abi, "lib", Recorder)
        for (call, _), stream in zip(calls, streams):
            with torch.cuda.stream(stream):
                call()
    for fn, args in raw:
        assert fn(*args) == abi.MLA_OK
    torch.cuda.synchronize()
    want = [out.clone() for _, out in calls]
    bad = []
    start = threading.Barrier(len(calls))

    def work(fn, args):
        start.wait()
        bad.extend(code for code in (fn(*args) for _ in range(4000)) if code != abi.MLA_OK)

    threads = [threading.Thread(target=work, args=r) for r in raw]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad, (len(bad), abi.status_name(bad[0]))
    assert abi.check_status() == abi.MLA_OK
    for (_, out), ref in zip(calls, want):
        assert torch.equal(out, ref)
