"""Calls beside another kernel: what else is resident on the GPU must not change a result.

The persistent prefill kernel hands part of its work to whichever CTA is free, decode and small
prefills run as clusters, and every kernel starts while the one before it in its stream still runs;
all of this goes another way when a kernel of another stream keeps some of the SMs."""
import ctypes
import os
import shutil
import subprocess
import time

import pytest
import torch

from paper_2410_16663_b200 import inputs as synth
from tests.test_parity_gpu import check_status, fa  # noqa: F401  (fa: the fixture)

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _rand(shape, dtype, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    return torch.randn(shape, device=DEV, generator=gen).to(dtype)


class Neighbour:
    """A finite call that holds one SM per head: one query tile over `keys` keys, about 0.6 us per 128 keys."""

    def __init__(self, fa, sms, keys):
        self.fa, self.sms = fa, sms
        self.q = _rand((1, 128, sms, 128), torch.float16, 1)
        self.k, self.v = (_rand((1, keys, 1, 128), torch.float16, s) for s in (2, 3))
        self.o = torch.empty_like(self.q)

    def run(self):
        self.fa.fa_forward_ex(self.q, self.k, self.v, self.o, None, False, 0.1, variant=3)


def beside_neighbour(fa, call, outs, sms, keys=131072, overlaps=True):
    """Runs call() alone and again beside a Neighbour that outlasts it; the outputs, filled with NaN
    before each run, must be the same bit for bit."""
    near = Neighbour(fa, sms, keys)

    def clear():
        for t in outs:
            t.fill_(float("nan"))

    near.run()
    clear()
    call()
    torch.cuda.synchronize()
    alone = [t.clone() for t in outs]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    end1, end2 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clear()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        near.run()
        end1.record()
    with torch.cuda.stream(s2):
        call()
        end2.record()
    torch.cuda.synchronize()
    check_status(fa)
    if overlaps:   # else the neighbour was gone too early and nothing has been tested
        assert end2.elapsed_time(end1) > 0
    for a, b in zip(alone, outs):
        assert not torch.isnan(a).any()
        assert torch.equal(a, b), f"{int((a != b).sum())} of {a.numel()} values differ"


def _dense(B, H, Hkv, Sq, Skv, d, dtype, o_dtype=None, seed=5):
    q = _rand((B, Sq, H, d), dtype, seed)
    k, v = (_rand((B, Skv, Hkv, d), dtype, seed + i) for i in (1, 2))
    o = torch.empty(q.shape, dtype=o_dtype or dtype, device=DEV)
    return q, k, v, o, torch.empty(B, H, Sq, device=DEV)


# (16, 32, 128): three rounds of items on 148 SMs and a remainder; then six and thirteen; the head-by-head
# order with its last two rounds claimed; d = 64 and the fp32 output
@pytest.mark.parametrize("sms", [1, 16, 32])
@pytest.mark.parametrize("B,H,Hkv,Sq,Skv,d,dtype,o_dtype", [
    (16, 32, 32, 128, 128, 128, torch.float16, None),
    (8, 32, 32, 512, 512, 128, torch.float16, None),
    (4, 32, 32, 2048, 2048, 128, torch.bfloat16, None),
    (1, 4, 2, 148 * 128 + 1, 300, 128, torch.float16, None),
    (8, 32, 8, 512, 512, 64, torch.float16, None),
    (8, 32, 32, 512, 512, 128, torch.bfloat16, torch.float32),
])
def test_prefill_beside_a_kernel_that_holds_sms(fa, B, H, Hkv, Sq, Skv, d, dtype, o_dtype, sms):  # noqa: F811
    q, k, v, o, lse = _dense(B, H, Hkv, Sq, Skv, d, dtype, o_dtype)
    beside_neighbour(fa, lambda: fa.fa_forward_ex(q, k, v, o, lse, Sq == Skv, 0.1), [o, lse], sms)


@pytest.mark.parametrize("sms", [16, 32])
def test_prefill_fp8_beside_a_kernel_that_holds_sms(fa, sms):  # noqa: F811
    q, k, v, o, lse = _dense(8, 32, 32, 512, 512, 128, torch.float16)
    q8, k8, v8 = synth.fp8_operands(q, k, v, 0.125, 0.25, 0.0625)
    beside_neighbour(fa, lambda: fa.fa_forward_fp8(q8, k8, v8, o, lse, True, 0.1, 0.125, 0.25, 0.0625), [o, lse], sms)


@pytest.mark.parametrize("sms", [16, 32])
def test_other_forms_beside_a_kernel_that_holds_sms(fa, sms):  # noqa: F811
    # a packed batch (all of its list claimed)
    lens = [700, 33, 1290, 128, 512, 1] * 3
    cu = torch.tensor([0] + lens).cumsum(0).to(torch.int32).to(DEV)
    q, k, v = (_rand((sum(lens), 16, 128), torch.bfloat16, s) for s in (7, 8, 9))
    o, lse = torch.empty_like(q), torch.empty(16, sum(lens), device=DEV)
    beside_neighbour(fa, lambda: fa.fa_forward_varlen(q, k, v, o, lse, cu, cu, max(lens), max(lens), True, 0.1), [o, lse], sms)
    # a query tile shared by a cluster's CTAs, d = 256, the short d = 64 kernels
    for B, H, Hkv, Sq, Skv, d in ((1, 8, 2, 200, 4000, 128), (1, 8, 8, 700, 700, 256), (40, 12, 12, 197, 197, 64), (64, 12, 12, 100, 100, 64)):
        q, k, v, o, lse = _dense(B, H, Hkv, Sq, Skv, d, torch.float16)
        beside_neighbour(fa, lambda: fa.fa_forward(q, k, v, o, lse, True, 0.1), [o, lse], sms, overlaps=False)
    # decode: chunks merged in one cluster, and split with a merge kernel
    for B, Hkv, smax in ((1, 5, 8192), (16, 8, 9000)):
        q, o, lse = _rand((B, 1, 2 * Hkv, 128), torch.float16, 11), torch.empty(B, 1, 2 * Hkv, 128, dtype=torch.float16, device=DEV), torch.empty(B, 2 * Hkv, device=DEV)
        k, v = (_rand((B, smax, Hkv, 128), torch.float16, s) for s in (12, 13))
        sl = torch.tensor([smax - 77 * b for b in range(B)], dtype=torch.int32, device=DEV)
        ws = torch.empty(fa.fa_decode_workspace_bytes(B, 2 * Hkv, Hkv, smax, 128) + 16, dtype=torch.uint8, device=DEV)
        beside_neighbour(fa, lambda: fa.fa_decode(q, k, v, o, lse, sl, 0.1, ws), [o, lse], sms, overlaps=False)


# Calls that feed one another.  Every call starts while the one before it may still run; call i reads what call i - 1
# wrote, as its queries, its keys or its values in turn (the other two are its own), and writes over what
# that one read.  step(i, src, dst) is one call, src and dst [B, S, H, d] of 16 bits; the softmax scale grows from
# call to call, so that no two of them write the same.
def _scale(i):
    return 0.2 + 0.03 * i


def _dense_steps(fa, B, H, S, d, causal, dtype=torch.float16, o_dtype=None):
    own = [_rand((B, S, H, d), dtype, 20 + i) for i in range(3)]
    o32 = torch.empty(B, S, H, d, device=DEV) if o_dtype else None

    def step(i, src, dst):
        q, k, v = (src if i % 3 == n else own[n] for n in range(3))
        fa.fa_forward_ex(q, k, v, dst if o32 is None else o32, None, causal, _scale(i))
        if o32 is not None:
            dst.copy_(o32)

    return (B, S, H, d), dtype, step


def _fp8_steps(fa, B, H, S, causal):
    own = [_rand((B, S, H, 128), torch.float16, 30 + i).to(torch.float8_e4m3fn) for i in range(3)]
    x8 = torch.empty_like(own[0])

    def step(i, src, dst):
        x8.copy_(src)
        q, k, v = (x8 if i % 3 == n else own[n] for n in range(3))
        fa.fa_forward_fp8(q, k, v, dst, None, causal, _scale(i), 1.0, 1.0, 1.0)

    return (B, S, H, 128), torch.float16, step


def _packed_steps(fa, lens, H, d, page):
    """Prefix sums, lengths and block table are written on the device right before each call, which takes
    the sequences in another order than the one before."""
    n, total = len(lens), sum(lens)
    own = [_rand((total, H, d), torch.bfloat16, 40 + i) for i in range(3)]
    cu, sl = torch.zeros(n + 1, dtype=torch.int32, device=DEV), torch.zeros(n, dtype=torch.int32, device=DEV)
    pages = -(-max(lens) // page) if page else 0
    table = torch.zeros(n, max(1, pages), dtype=torch.int32, device=DEV)
    orders = [torch.tensor(lens[i % n:] + lens[:i % n], dtype=torch.int32).to(DEV) for i in range(n)]
    tables = [torch.randperm(n * pages).to(torch.int32).view(n, pages).to(DEV) for _ in range(n)] if page else None
    pool = torch.zeros(2, n * pages, page, H, d, dtype=torch.bfloat16, device=DEV) if page else None
    if page:
        pool.copy_(_rand(pool.shape, torch.bfloat16, 44))

    def step(i, src, dst):
        src, dst = src.view(total, H, d), dst.view(total, H, d)
        cu[1:].copy_(orders[i % n].cumsum(0))
        if not page:
            q, k, v = (src if i % 3 == m else own[m] for m in range(3))
            fa.fa_forward_varlen(q, k, v, dst, None, cu, cu, max(lens), max(lens), True, _scale(i))
        else:
            sl.copy_(orders[i % n])
            table.copy_(tables[i % n])
            if i % 3:   # as keys or values: the first rows of the pool
                pool[i % 3 - 1].view(-1, H, d)[:total].copy_(src)
            fa.fa_forward_varlen_paged(own[0] if i % 3 else src, pool[0], pool[1], table, dst, None, cu, sl, max(lens), max(lens), True, _scale(i))

    return (1, total, H, d), torch.bfloat16, step


def _decode_and_prefill_steps(fa, B, H):
    """A decode, a small prefill over its output, a decode with the prefill's output as its queries, ..."""
    q0, k, v = _rand((1, B, H, 128), torch.float16, 50), _rand((B, 900, H, 128), torch.float16, 51), _rand((B, 900, H, 128), torch.float16, 52)
    sl = torch.tensor([900 - 31 * b for b in range(B)], dtype=torch.int32, device=DEV)
    ws = torch.empty(fa.fa_decode_workspace_bytes(B, H, H, 900, 128) + 16, dtype=torch.uint8, device=DEV)

    def step(i, src, dst):
        if i % 2 == 0:
            fa.fa_decode(src.view(B, 1, H, 128), k, v, dst.view(B, 1, H, 128), None, sl, _scale(i), ws)
        else:
            fa.fa_forward(q0 if i % 4 == 1 else src, src, src, dst, None, True, _scale(i))

    return (1, B, H, 128), torch.float16, step


@pytest.mark.parametrize("form", [
    lambda fa: _dense_steps(fa, 1, 2, 512, 128, True),
    lambda fa: _dense_steps(fa, 1, 1, 5, 128, False),
    lambda fa: _dense_steps(fa, 1, 4, 2048, 128, True),            # query tiles shared by a cluster's CTAs
    lambda fa: _dense_steps(fa, 1, 3, 3000, 128, False, torch.bfloat16),
    lambda fa: _dense_steps(fa, 3, 5, 700, 128, True),
    lambda fa: _dense_steps(fa, 8, 32, 512, 128, True),            # a full grid
    lambda fa: _dense_steps(fa, 4, 16, 600, 64, True),
    lambda fa: _dense_steps(fa, 2, 6, 700, 128, True, o_dtype=torch.float32),
    lambda fa: _fp8_steps(fa, 2, 8, 700, True),
    lambda fa: _packed_steps(fa, [300, 33, 128, 517, 1], 4, 128, 0),
    lambda fa: _packed_steps(fa, [300, 33, 128, 517, 1], 4, 64, 0),
    lambda fa: _packed_steps(fa, [300, 33, 128, 517, 1], 4, 128, 128),
    lambda fa: _decode_and_prefill_steps(fa, 16, 4),
], ids=["small", "few rows", "shared tiles", "shared tiles bf16", "medium", "full grid", "d64", "fp32 output", "fp8", "packed", "packed d64",
        "paged", "decode and prefill"])
def test_calls_that_read_what_the_call_before_wrote(fa, form):  # noqa: F811
    # The calls one by one, and queued up behind a call that outlasts their enqueueing: bit for bit the same.
    near = Neighbour(fa, 4, 524288)
    ends = []
    for alone in (True, False):
        torch.manual_seed(3)
        shape, dtype, step = form(fa)
        x0 = _rand(shape, dtype, 3)
        bufs, seen = [x0.clone(), torch.full_like(x0, float("nan"))], []
        near.run()
        torch.cuda.synchronize()
        gone = torch.cuda.Event()
        if not alone:
            near.run()
            gone.record()
        for i in range(12):
            step(i, bufs[i & 1], bufs[1 - (i & 1)])
            if alone:
                seen.append(bufs[1 - (i & 1)].clone())
                torch.cuda.synchronize()
        assert alone or not gone.query()   # else the calls did not queue up and nothing has been tested
        torch.cuda.synchronize()
        check_status(fa)
        for a, b in zip(seen, seen[2:]):   # a call that read a buffer as it was before would be found out
            assert torch.isfinite(a).all() and torch.isfinite(b).all() and not torch.equal(a, b)
        ends.append(bufs)
    assert all(torch.equal(a, b) for a, b in zip(*ends))


# 120 CTAs each, fewer than the SMs, and a merge kernel: chunks of one length out of the longest sequence's, and out of the lengths
# that the device finds (one and three tokens, 8-bit keys)
@pytest.mark.parametrize("B,Hkv,smax,sq,fp8", [(3, 1, 40000, 1, False), (12, 5, 5861, 1, False), (12, 5, 5861, 3, False), (7, 8, 19641, 1, True)],
                         ids=["by the longest", "by the lengths", "by the lengths, 3 tokens", "by the lengths, 8-bit"])
def test_decodes_whose_lengths_are_written_right_before(fa, B, Hkv, smax, sq, fp8):  # noqa: F811
    # Each call's lengths are written on the device right before it, in another order than the call before had them, and its
    # queries are the output of that call: one by one, and queued up behind a call that outlasts their enqueueing, bit for bit.
    near = Neighbour(fa, 4, 524288)
    k, v = (_rand((B, smax, Hkv, 128), torch.float16, s) for s in (61, 62))
    if fp8:
        k, v = (t.to(torch.float8_e4m3fn).view(torch.uint8) for t in (k, v))
    lens = [smax, sq, 128, 129] + [max(sq, smax * (2 * b + 1) // (2 * B + 3)) for b in range(B)]
    orders = [torch.tensor((lens * 2)[i:i + B], dtype=torch.int32).to(DEV) for i in range(len(lens))]
    sl = torch.zeros(B, dtype=torch.int32, device=DEV)
    ws = torch.empty(fa.fa_decode_append_workspace_bytes(B, sq, Hkv, Hkv, smax, 128) + 16, dtype=torch.uint8, device=DEV)
    x0 = _rand((B, sq, Hkv, 128), torch.float16, 63)
    ends = []
    for alone in (True, False):
        bufs, seen = [x0.clone(), torch.full_like(x0, float("nan"))], []
        sl.zero_()
        ws.fill_(0xff)   # NaNs
        near.run()
        torch.cuda.synchronize()
        gone = torch.cuda.Event()
        if not alone:
            near.run()
            gone.record()
        for i in range(20):
            src, dst = bufs[i & 1], bufs[1 - (i & 1)]
            sl.copy_(orders[i % len(lens)])
            if fp8:
                fa.fa_decode_fp8(src, k, v, dst, None, sl, 0.3, 1.0, 1.0, ws)
            else:
                fa.fa_decode_ex(src, k, v, dst, None, sl, 0.3, ws)
            if alone:
                seen.append(dst.clone())
                torch.cuda.synchronize()
        assert alone or not gone.query()   # else the calls did not queue up and nothing has been tested
        torch.cuda.synchronize()
        check_status(fa)
        for a, b in zip(seen, seen[1:]):
            assert torch.isfinite(a).all() and torch.isfinite(b).all() and not torch.equal(a, b)
        ends.append(bufs)
    assert all(torch.equal(a, b) for a, b in zip(*ends))


@pytest.mark.parametrize("B,Hkv,smax,sq", [(3, 1, 40000, 1), (12, 5, 5861, 2), (1, 5, 8192, 1)], ids=["by the longest", "by the lengths", "cluster"])
def test_captured_decodes_take_the_lengths_of_the_replay(fa, B, Hkv, smax, sq):  # noqa: F811
    # two decodes in one graph, the second with the first one's output as its queries; each replay bit for bit what the
    # calls give with its lengths
    k, v = (_rand((B, smax, Hkv, 128), torch.float16, s) for s in (71, 72))
    q = _rand((B, sq, Hkv, 128), torch.float16, 73)
    sl = torch.full((B,), smax, dtype=torch.int32, device=DEV)
    ws = torch.empty(fa.fa_decode_append_workspace_bytes(B, sq, Hkv, Hkv, smax, 128) + 16, dtype=torch.uint8, device=DEV)
    outs = [torch.empty_like(q), torch.empty_like(q), torch.empty(B, Hkv, sq, device=DEV)]

    def calls():
        fa.fa_decode_ex(q, k, v, outs[0], None, sl, 0.1, ws)
        fa.fa_decode_ex(outs[0], k, v, outs[1], outs[2], sl, 0.3, ws)

    calls()   # (set-up before the capture)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    seen = []
    for lens in ([smax] * B, [smax // (b + 2) for b in range(B)], [1 + 128 * b for b in range(B)], [0] + [smax - 5] * (B - 1)):
        sl.copy_(torch.tensor(lens, dtype=torch.int32))
        ws.fill_(0xff)
        calls()
        want = [t.clone() for t in outs]
        for t in outs:
            t.fill_(float("nan"))
        ws.fill_(0xff)
        graph.replay()
        torch.cuda.synchronize()
        check_status(fa)
        assert all(torch.equal(a, b) for a, b in zip(want, outs)) and not torch.isnan(outs[1]).any()
        seen.append(want[1])
    assert not any(torch.equal(a, b) for a, b in zip(seen, seen[1:]))


@pytest.fixture(scope="module")
def early_release(tmp_path_factory):
    """early_release(ns, src, dst): see gpu_helpers/early_release.cu; on the current stream."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("early_release") / "early_release.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "gpu_helpers", "early_release.cu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xcompiler", "-fPIC", src,
                    "-o", out], check=True, timeout=600)
    fn = ctypes.CDLL(out).early_release
    fn.argtypes = [ctypes.c_ulonglong, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]

    def call(ns, src, dst):
        assert fn(ns, src.data_ptr(), dst.data_ptr(), src.numel() * src.element_size(), torch.cuda.current_stream().cuda_stream) == 0

    return call


WAIT_LIMIT_S = 4   # of every bounded wait in the kernels


def test_a_kernel_before_that_outlasts_every_wait_limit(fa, early_release):  # noqa: F811
    # The call starts while that kernel runs, which writes the call's values at its end, more than a wait limit later: no
    # wait of the call may count that time.  The forms of the ping-pong kernel whose grids leave room for one
    # another, each behind a kernel and on a stream of its own.
    forms = []   # (values, output and log-sum-exp, call)
    # (the second: a query tile shared by a cluster's CTAs)
    for H, Sq, Skv, d, o_dtype in ((2, 512, 512, 128, None), (2, 100, 2048, 128, None), (2, 700, 700, 64, None), (2, 512, 512, 128, torch.float32)):
        q, k, v, o, lse = _dense(1, H, H, Sq, Skv, d, torch.float16, o_dtype)
        forms.append((v, [o, lse], lambda q=q, k=k, v=v, o=o, lse=lse: fa.fa_forward_ex(q, k, v, o, lse, True, 0.1)))
    q, k, v, o, lse = _dense(1, 2, 2, 512, 512, 128, torch.float16)
    q8, k8, v8 = synth.fp8_operands(q, k, v, 0.125, 0.25, 0.0625)
    forms.append((v8, [o, lse], lambda q=q8, k=k8, v=v8, o=o, lse=lse: fa.fa_forward_fp8(q, k, v, o, lse, True, 0.1, 0.125, 0.25, 0.0625)))
    lens = [300, 33, 128]
    cu = torch.tensor([0] + lens).cumsum(0).to(torch.int32).to(DEV)
    q, k, v = (_rand((sum(lens), 2, 128), torch.bfloat16, s) for s in (7, 8, 9))
    o, lse = torch.empty_like(q), torch.empty(2, sum(lens), device=DEV)
    forms.append((v, [o, lse], lambda q=q, k=k, v=v, o=o, lse=lse: fa.fa_forward_varlen(q, k, v, o, lse, cu, cu, max(lens), max(lens), True, 0.1)))
    kp, vp, table = (t.to(DEV) for t in synth.paged_from_packed(k.cpu(), v.cpu(), lens, 128, seed=3))
    sl = torch.tensor(lens, dtype=torch.int32, device=DEV)
    o, lse = torch.empty_like(q), torch.empty(2, sum(lens), device=DEV)
    forms.append((vp, [o, lse], lambda q=q, kp=kp, vp=vp, o=o, lse=lse: fa.fa_forward_varlen_paged(q, kp, vp, table, o, lse, cu, sl, max(lens), max(lens), True, 0.1)))
    for _, _, call in forms:
        call()
    torch.cuda.synchronize()
    check_status(fa)
    alone = [[t.clone() for t in outs] for _, outs, _ in forms]
    sources, streams = [v.clone() for v, _, _ in forms], [torch.cuda.Stream() for _ in forms]
    for v, outs, _ in forms:
        v.view(torch.uint8).zero_()
        for t in outs:
            t.fill_(float("nan"))
    torch.cuda.synchronize()
    t0 = time.monotonic()
    for (v, _, call), src, stream in zip(forms, sources, streams):
        with torch.cuda.stream(stream):
            early_release(int((WAIT_LIMIT_S + 1) * 1e9), src, v)
            call()
    torch.cuda.synchronize()
    assert WAIT_LIMIT_S + 0.5 < time.monotonic() - t0 < 4 * WAIT_LIMIT_S
    check_status(fa)
    for i, ((_, outs, _), want) in enumerate(zip(forms, alone)):
        for a, b in zip(want, outs):
            assert torch.equal(a, b), f"form {i}: {int((a != b).sum())} of {a.numel()} values differ"


def test_a_thread_that_gives_up_a_wait_lets_what_is_on_its_way_arrive(fa):  # noqa: F811
    # copies that the CTA's threads have issued may be on their way into its shared memory; the thread
    # whose time is up (0.05 ms here) stays for another millisecond before it and the CTA can leave
    gave_up = torch.zeros(1, dtype=torch.int32, device=DEV)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    t0.record()
    fa.fa_selftest_wait(50, gave_up)
    t1.record()
    torch.cuda.synchronize()
    assert int(gave_up.item()) == 64 and fa.fa_device_status()[:2] == (fa.FA_ERR_TIMEOUT, 990)
    assert 1.0 <= t0.elapsed_time(t1) <= 500.0
