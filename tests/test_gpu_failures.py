"""Failure reporting of the library on the GPU, exercised without faulting it.

The scoring kernel waits on mbarriers (copies landed, accumulators ready, stages free).  Every such wait is
bounded; when one runs out the thread block stops issuing work, drains what it has in flight, frees its
tensor memory and ends, and the host reads DKV_ERR_TIMEOUT from dkv_last_status.  The test makes a wait run
out the harmless way: the copy of one key tile is simply never issued (dkv_debug_withhold_tile), with the
wait limit set to about a millisecond.  Nothing traps, no address is invalid, the context stays usable.
"""
import contextlib
import ctypes

import numpy as np
import pytest
import torch

from oracle import dynamickv as O
from paper_2412_14838_b200 import binding as B
from paper_2412_14838_b200 import build, synth
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()


def _dev(bits):
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).cuda()


@pytest.mark.parametrize("sweep", [1, 2])
def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable(sweep):
    w = synth.WORKLOADS["tiny"]
    t = synth.layer_inputs(w, 0, want_v=False)
    q, k = _dev(t["q"]), _dev(t["k"])
    ref = O.window_scores(synth.bf16_bits_to_f64(t["q"]), synth.bf16_bits_to_f64(t["k"]), w.ws, w.pool)["score"]
    ctx = B.dkv_create(B.config_of(w))
    try:
        out = torch.zeros((w.Bt, w.Hkv, w.P), dtype=torch.float32, device="cuda")
        B.dkv_set_wait_limit(ctx, 2_000_000)              # about a millisecond of SM clock
        B.dkv_debug_withhold_tile(ctx, sweep, 0)           # block 0 never gets its first key tile of that sweep
        B.dkv_score(ctx, 0, q, k, out)                     # enqueues; the kernels end by themselves
        torch.cuda.synchronize()
        code, status = B.dkv_last_status(ctx)
        assert code == B.DKV_ERR_TIMEOUT, f"expected a timeout report, got {code} {status}"
        assert 101 <= status[0] <= 107 and status[2] == 0, status
        assert "timed out" in B.strerror(code)
        code, status = B.dkv_last_status(ctx)              # reported once
        assert code == B.DKV_OK and status[0] == 0
        # the same context, hook off: a normal call gives the right scores
        B.dkv_debug_withhold_tile(ctx, 0, -1)
        B.dkv_set_wait_limit(ctx, 4_000_000_000)
        B.dkv_score(ctx, 0, q, k, out)
        torch.cuda.synchronize()
        code, status = B.dkv_last_status(ctx)
        assert code == B.DKV_OK and status[0] == 0
        U.assert_scores_close(out.cpu().numpy(), ref, "after a reported timeout")
    finally:
        B.dkv_destroy(ctx)


# A pipe with one tile and pipes with five, in which the copy after the withheld tile waits for its slot; with a limit of a millisecond,
# and with the shortest one, which any wait may exceed.
@pytest.mark.parametrize("use,sweep", [("pass", 1), ("pass", 2), ("lse", 2)])
@pytest.mark.parametrize("S,tile,limit", [(300, 0, 2_000_000), (6200, 0, 2_000_000), (6200, 3, 2_000_000), (6200, 3, 1000)])
def test_a_wait_that_runs_out_in_a_pass_is_reported_and_the_context_stays_usable(use, sweep, S, tile, limit):
    L, Hkv, G, D, ws = 4, 8, 2, 64, 16
    g = torch.Generator(device="cuda").manual_seed(S)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k, v = new(1, G * Hkv, ws, D), new(1, Hkv, S, D), new(1, Hkv, S, D)
    kb, vb = ([torch.zeros((1, Hkv, 64 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    hidden = torch.arange(S, device="cuda") > (S - ws + torch.arange(ws, device="cuda")).repeat(G)[:, None]
    logits = [(a.double().view(1, Hkv, G * ws, D) @ b.double().transpose(-1, -2) / D ** 0.5).masked_fill(hidden, -torch.inf) for a, b in zip(q, k)]
    lse = [t.logsumexp(-1).view(1, Hkv * G, ws).float().contiguous() for t in logits]
    want = [t.softmax(-1)[..., :S - ws].sum(2).cpu() for t in logits]
    ctx = B.dkv_create(B.make_config(L, G * Hkv, Hkv, D, 1, S, ws, 1, 32, 64, 2))
    run = (lambda: B.dkv_run_prefill_pass_lse(ctx, q, k, v, lse, kb, vb)) if use == "lse" else (lambda: B.dkv_run_prefill_pass(ctx, q, k, v, kb, vb))
    try:
        for _ in range(3):
            B.dkv_set_wait_limit(ctx, limit)
            B.dkv_debug_withhold_tile(ctx, sweep, tile)
            run()
            code, status = B.dkv_last_status(ctx)
            assert code == B.DKV_ERR_TIMEOUT and 101 <= status[0] <= 107, f"{code} {status}"
            assert limit == 1000 or status[2] == 0
            assert B.dkv_last_status(ctx)[0] == B.DKV_OK
            B.dkv_debug_withhold_tile(ctx, 0, -1)
            B.dkv_set_wait_limit(ctx, 4_000_000_000)
            run()
            assert B.dkv_last_status(ctx)[0] == B.DKV_OK
            for l in range(L):
                got = torch.zeros((1, Hkv, S - ws))
                B.dkv_memcpy_to_host(ctx, got, B.dkv_layer_views(ctx, l)[0], got.numel() * 4)
                assert ((got - want[l]).abs() <= 5e-5 * want[l]).all()
    finally:
        B.dkv_destroy(ctx)


@pytest.mark.parametrize("use", ["pass", "lse"])
def test_the_limit_is_for_a_tile_and_not_for_a_head(use):
    """Two heads of 65536 keys to a pipe, some 700 us, of 2 us a tile: a limit of 80 us is far from any wait for a tile."""
    L, Hkv, D, S, ws = 8, 74, 64, 65536, 16
    q, k = ([torch.randn((1, Hkv, n, D), device="cuda").to(torch.bfloat16) for _ in range(1)] * L for n in (ws, S))
    kb, vb = ([torch.zeros((1, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    lse = [torch.zeros((1, Hkv, ws), device="cuda")] * L
    ctx = B.dkv_create(B.make_config(L, Hkv, Hkv, D, 1, S, ws, 5, 4, 8, 2))
    try:
        B.dkv_set_wait_limit(ctx, 150_000)
        for _ in range(2):
            if use == "lse":
                B.dkv_run_prefill_pass_lse(ctx, q, k, k, lse, kb, vb)
            else:
                B.dkv_run_prefill_pass(ctx, q, k, k, kb, vb)
            code, status = B.dkv_last_status(ctx)
            assert code == B.DKV_OK, status
    finally:
        B.dkv_destroy(ctx)


def test_the_limit_does_not_count_the_wait_for_the_launch_before():
    """The key sums of a pass start on the SMs whose row sums have ended.  One head whose logits are far above its first key keeps
    two blocks for some 250 us longer (its row sums are computed again): the others wait, and their limit of 80 us or so stands for
    what they wait for themselves."""
    L, Hkv, D, S, ws = 32, 8, 64, 32768, 16
    g = torch.Generator(device="cuda").manual_seed(3)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k = new(1, Hkv, ws, D), new(1, Hkv, S, D)
    q[5][:, 3, :, 0], k[5][:, 3, :, 0], k[5][:, 3, 70::999, 0] = 16.0, 0.0, 100.0
    kb, vb = ([torch.zeros((1, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    ctx = B.dkv_create(B.make_config(L, Hkv, Hkv, D, 1, S, ws, 5, 4, 8, 2))
    scores = []
    try:
        for limit in (4_000_000_000, 150_000, 150_000):
            B.dkv_set_wait_limit(ctx, limit)
            B.dkv_run_prefill_pass(ctx, q, k, k, kb, vb)
            code, status = B.dkv_last_status(ctx)
            assert code == B.DKV_OK, f"limit {limit}: {status}"
            got = torch.zeros((L, Hkv, S - ws))
            for l in range(L):
                B.dkv_memcpy_to_host(ctx, got[l], B.dkv_layer_views(ctx, l)[0], got[l].numel() * 4)
            scores.append(got)
        assert all(torch.equal(x, scores[0]) for x in scores)
    finally:
        B.dkv_destroy(ctx)


def test_wait_limit_and_hook_arguments_are_checked():
    ctx = B.dkv_create(B.config_of(synth.WORKLOADS["tiny"]))
    try:
        with pytest.raises(B.DkvError) as e:
            B.dkv_set_wait_limit(ctx, 10)
        assert e.value.code == B.DKV_ERR_INVALID_ARG
        with pytest.raises(B.DkvError) as e:
            B.dkv_debug_withhold_tile(ctx, 3, 0)
        assert e.value.code == B.DKV_ERR_INVALID_ARG
    finally:
        B.dkv_destroy(ctx)


def test_two_live_contexts_with_different_layer_budgets():
    """The select kernel's shared-memory attribute belongs to the kernel, not to a context: a second context with
    a small per-layer maximum must not break the first one's launches."""
    big = synth.Workload("bigbl", 71, L=1, Hq=2, Hkv=1, D=64, Bt=1, S=12000, ws=8, pool=3, N=4096, Bl=8192, m=1,
                         recipe="iid")
    small = synth.Workload("smallbl", 72, L=1, Hq=2, Hkv=1, D=64, Bt=1, S=600, ws=8, pool=3, N=16, Bl=32, m=1,
                           recipe="iid")
    a = B.dkv_create(B.config_of(big))
    b = B.dkv_create(B.config_of(small))                   # created second, needs far less shared memory
    try:
        for ctx, w in ((a, big), (b, small), (a, big)):
            sc = synth.pooled_like_scores((w.Bt, w.Hkv, w.P), w.pool, seed=w.cid, tie_fraction=0.2)
            B.dkv_set_scores(ctx, 0, torch.from_numpy(sc).cuda())
            idx = torch.zeros((w.Bt, w.Hkv, w.Blc), dtype=torch.int32, device="cuda")
            B.dkv_select_topk(ctx, 0, idx)
            torch.cuda.synchronize()
            want = O.select_topk(sc[0, 0].astype(np.float64), w.Bl)["idx"]
            assert (idx.cpu().numpy()[0, 0] == want).all()
    finally:
        B.dkv_destroy(a)
        B.dkv_destroy(b)


@contextlib.contextmanager
def stream_that_refuses_work():
    """A stream whose capture was invalidated: the runtime refuses every launch and copy on it, on the host, until the
    capture is ended."""
    rt = ctypes.CDLL("libcudart.so.12")
    rt.cudaStreamEndCapture.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    stream = torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(handle, 2) == 0
    assert rt.cudaStreamSynchronize(handle) != 0               # not allowed in a capture
    try:
        yield stream
    finally:
        graph = ctypes.c_void_p()
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0 and not graph.value
        rt.cudaGetLastError()


class _Pass:
    """One prompt of the smallest workload on the device."""

    def __init__(self):
        self.w = w = synth.WORKLOADS["tiny"]
        bits = [synth.layer_inputs(w, l) for l in range(w.L)]
        self.q, self.k, self.v = ([_dev(t[n]) for t in bits] for n in ("q", "k", "v"))
        shape = (w.Bt, w.Hkv, w.Blc + w.ws, w.D)
        self.kb, self.vb = ([torch.zeros(shape, dtype=torch.int16, device="cuda") for _ in range(w.L)] for _ in range(2))
        shape = (w.Bt, w.Hq, 1, w.D)
        self.dq = [torch.randn(shape, device="cuda").to(torch.bfloat16) for _ in range(w.L)]
        self.out = [torch.zeros(shape, device="cuda") for _ in range(w.L)]
        self.lse = [torch.zeros((w.Bt, w.Hq, w.ws), device="cuda") for _ in range(w.L)]

    def run(self, ctx, use, stream=None):
        if use == "lse":
            B.dkv_run_prefill_pass_lse(ctx, self.q, self.k, self.v, self.lse, self.kb, self.vb, stream)
        else:
            B.dkv_run_prefill_pass(ctx, self.q, self.k, self.v, self.kb, self.vb, stream)

    def decode(self, ctx):
        B.dkv_decode_attend(ctx, 0, self.w.L, 1, self.dq, self.kb, self.vb, self.out)
        torch.cuda.synchronize()
        return torch.stack(self.out).clone()


@pytest.mark.parametrize("use", ["pass", "lse"])
def test_a_pass_that_fails_midway_leaves_no_layer_of_the_pass_before(use):
    p = _Pass()
    ctx = B.dkv_create(B.config_of(p.w))
    try:
        p.run(ctx, use)
        want = p.decode(ctx)
        with stream_that_refuses_work() as stream:
            with pytest.raises(B.DkvError) as e:
                p.run(ctx, use, stream)
            assert e.value.code == B.DKV_ERR_CUDA and B.dkv_last_cuda_error(ctx) != 0
        for call in (lambda: p.decode(ctx), lambda: B.dkv_rebudget(ctx, p.w.L), lambda: B.dkv_select_topk(ctx, 0),
                     lambda: B.dkv_compact_all(ctx, p.w.L, p.kb, p.vb)):
            with pytest.raises(B.DkvError) as e:
                call()
            assert e.value.code == B.DKV_ERR_STATE
        p.run(ctx, use)
        assert torch.equal(p.decode(ctx), want)
    finally:
        B.dkv_destroy(ctx)


def test_a_refused_call_is_reported_once():
    w = synth.WORKLOADS["tiny"]
    a, b = B.dkv_create(B.config_of(w)), B.dkv_create(B.config_of(w))
    d = torch.zeros(w.Bt * w.Hkv * w.S * w.D, device="cuda")
    try:
        with stream_that_refuses_work() as stream:
            launched = B.dkv_launch_count(a)
            for call in (lambda: B.dkv_select_positions(a, 0, 4, 4, stream), lambda: B.dkv_reset(a, stream),
                         lambda: B.dkv_score_static(B.config_of(w), d, d, d, stream)):
                with pytest.raises(B.DkvError) as e:
                    call()
                assert e.value.code == B.DKV_ERR_CUDA
            assert B.dkv_launch_count(a) == launched
        for ctx in (b, a):
            B.dkv_select_positions(ctx, 0, 4, 4)
    finally:
        B.dkv_destroy(a)
        B.dkv_destroy(b)


def test_a_host_buffer_pass_that_fails_midway_leaves_no_layer():
    w = synth.WORKLOADS["tiny"]
    p = _Pass()
    pin = lambda tensors: [t.cpu().pin_memory() for t in tensors]
    q, k, v, kb, vb = (pin(x) for x in (p.q, p.k, p.v, p.kb, p.vb))
    counts, again = (np.zeros((w.Bt, w.L), dtype=np.int32) for _ in range(2))
    rt = ctypes.CDLL("libcudart.so.12")
    rt.cudaStreamEndCapture.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    other, graph = ctypes.c_void_p(torch.cuda.Stream().cuda_stream), ctypes.c_void_p()
    ctx = B.dkv_create(B.config_of(w))
    try:
        B.dkv_run_prefill_pass_host(ctx, q, k, v, kb, vb, counts)
        # while another stream is captured in the strictest mode the runtime refuses some calls, the read of the counts
        # into ordinary memory among them
        assert rt.cudaStreamBeginCapture(other, 0) == 0
        try:
            with pytest.raises(B.DkvError) as e:
                B.dkv_run_prefill_pass_host(ctx, q, k, v, kb, vb, again)
            assert e.value.code == B.DKV_ERR_CUDA and B.dkv_last_cuda_error(ctx) != 0
        finally:
            rt.cudaStreamEndCapture(other, ctypes.byref(graph))
            rt.cudaGetLastError()
        for call in (lambda: B.dkv_rebudget(ctx, 1), lambda: p.decode(ctx)):
            with pytest.raises(B.DkvError) as e:
                call()
            assert e.value.code == B.DKV_ERR_STATE
        B.dkv_get_counts(ctx, again)
        assert (again == 0).all()
        B.dkv_run_prefill_pass_host(ctx, q, k, v, kb, vb, again)
        assert (again == counts).all()
    finally:
        B.dkv_destroy(ctx)


def test_a_host_buffer_pass_that_finds_too_little_memory_keeps_none_of_it():
    # two layers of keys and values in flight: 2 x 3 x 512 MB of staging
    w = synth.Workload("staging", 73, L=2, Hq=8, Hkv=8, D=128, Bt=8, S=32768, ws=8, pool=3, N=16, Bl=32, m=1, recipe="iid")
    some = torch.zeros(1 << 20, dtype=torch.uint8)            # never read: the call fails before it copies anything
    counts = np.zeros((w.Bt, w.L), dtype=np.int32)
    torch.cuda.empty_cache()
    ctx = B.dkv_create(B.config_of(w))
    free = torch.cuda.mem_get_info()[0]
    taken = torch.empty(free - (900 << 20), dtype=torch.uint8, device="cuda")
    try:
        before = torch.cuda.mem_get_info()[0]
        for _ in range(3):
            with pytest.raises(B.DkvError) as e:
                B.dkv_run_prefill_pass_host(ctx, *[[some] * w.L] * 5, counts)
            assert e.value.code == B.DKV_ERR_NOMEM
        assert torch.cuda.mem_get_info()[0] > before - (64 << 20)
    finally:
        del taken
        torch.cuda.empty_cache()
        B.dkv_destroy(ctx)
