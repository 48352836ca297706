"""The sizes at which the launches of a selection, the budget updates and the host-buffer pass change their form."""
import numpy as np
import pytest
import torch

from oracle import dynamickv as O
from paper_2412_14838_b200 import binding as B
from paper_2412_14838_b200 import build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()


# one block a head below 8192 positions or above 18 heads, four to 24575 positions or from 10 to 18 heads, else eight;
# "same": more equal scores than the list holds
@pytest.mark.parametrize("P,Hkv,Bl,kind", [(8191, 2, 100, "ties"), (8192, 1, 1, "ties"), (8193, 18, 333, "ties"), (8200, 19, 64, "ties"),
                                           (24575, 3, 700, "ties"), (24576, 9, 64, "ties"), (24577, 10, 64, "ties"), (24609, 2, 4096, "ties"),
                                           (9001, 2, 500, "same"), (30011, 1, 500, "same")])
def test_select_of_one_layer(P, Hkv, Bl, kind):
    w = synth.Workload("sel", 41, L=1, Hq=Hkv, Hkv=Hkv, D=64, Bt=1, S=P + 8, ws=8, pool=7, N=Bl, Bl=Bl, m=1, recipe="iid")
    sc = synth.pooled_like_scores((1, Hkv, P), 7, seed=P, tie_fraction=0.2)
    if kind == "same":
        sc[...] = 0.25
        sc[:, :, P - 100:P - 90] = 0.5
    h = B.dkv_create(B.config_of(w))
    try:
        B.dkv_set_scores(h, 0, torch.from_numpy(sc).cuda())
        idx = torch.empty((1, Hkv, w.Blc), dtype=torch.int32, device="cuda")
        rank = torch.empty_like(idx)
        B.dkv_select_topk(h, 0, idx, rank)
        idx, rank = idx.cpu().numpy(), rank.cpu().numpy()
    finally:
        B.dkv_destroy(h)
    for head in range(Hkv):
        ref = O.select_topk(sc[0, head].astype(np.float64), Bl)
        assert (idx[0, head] == ref["idx"]).all() and (rank[0, head] == ref["rank"]).all(), f"head {head}"


@pytest.mark.parametrize("L,m", [(7, 1), (8, 1), (9, 1), (17, 2)])       # the updates of a pass run up to eight at a time
def test_updates_of_a_pass_and_pageable_results(L, m):
    w = synth.Workload("upd", 42, L=L, Hq=4, Hkv=2, D=64, Bt=2, S=333, ws=9, pool=3, N=20, Bl=60, m=m, recipe="sink")
    bits = [{n: np.ascontiguousarray(a).view(np.int16) for n, a in synth.layer_inputs(w, l).items()} for l in range(L)]
    q, k, v = ([torch.from_numpy(t[n]).cuda() for t in bits] for n in "qkv")
    shape = (w.Bt, w.Hkv, w.Blc + w.ws, w.D)
    kb, vb = ([torch.zeros(shape, dtype=torch.int16, device="cuda") for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.config_of(w))
    try:
        B.dkv_run_prefill_pass(h, q, k, v, kb, vb)
        torch.cuda.synchronize()
        counts = np.zeros((w.Bt, L), dtype=np.int32)
        B.dkv_get_counts(h, counts)
        hist = []
        for l in range(L):
            sc = np.empty((w.Bt, w.Hkv, w.P), dtype=np.float32)
            B.dkv_memcpy_to_host(h, sc, B.dkv_layer_views(h, l)[0], sc.nbytes)
            hist.append(sc)
        for b in range(w.Bt):
            ref = np.full(L, w.Blc, dtype=np.int64)
            for l in [n for n in range(1, L + 1) if n % m == 0 or n == L]:
                ref = np.asarray(O.rebudget([hist[i][b].astype(np.float64) for i in range(l)], ref, w.N, w.Bl, L)["counts"])
            assert counts[b].tolist() == ref.tolist()
        out = [[np.zeros(shape, dtype=np.int16) for _ in range(L)] for _ in range(2)]        # not page-locked
        again = np.zeros_like(counts)
        B.dkv_run_prefill_pass_host(h, *([torch.from_numpy(t[n]) for t in bits] for n in "qkv"), out[0], out[1], again)
        # the calls a layer, an update every m layers: the same launches a layer, so the same scores, counts and rows to the bit
        B.dkv_reset(h)
        for l in range(L):
            B.dkv_score(h, l, q[l], k[l])
            B.dkv_select_topk(h, l)
            B.dkv_compact(h, l, k[l], v[l], kb[l], vb[l])
            if (l + 1) % m == 0 or l + 1 == L:
                B.dkv_rebudget(h, l + 1)
                B.dkv_compact_all(h, l + 1, kb[:l + 1], vb[:l + 1])
        B.dkv_get_counts(h, counts)
        assert (again == counts).all()
        for l in range(L):
            for b in range(w.Bt):
                n = int(counts[b, l]) + w.ws
                for got, want in ((out[0], kb), (out[1], vb)):
                    assert (got[l][b, :, :n] == want[l][b, :, :n].cpu().numpy()).all(), f"layer {l}"
                    assert (got[l][b, :, n:] == 0).all()                     # the rest of the caller's buffers is left alone
    finally:
        B.dkv_destroy(h)


# one block a head where positions + 16 rows are below 20480 or heads are more than 74, else four, or eight from 24576
# positions with up to 37 heads
@pytest.mark.parametrize("P,L,Hkv,Bl", [(19583, 2, 3, 56), (19584, 2, 3, 56), (6177, 2, 2, 1001), (19951, 74, 1, 33), (19953, 25, 3, 33), (24575, 2, 2, 700),
                                        (24577, 37, 1, 40), (24576, 19, 2, 40), (24601, 2, 1, 5000)])
def test_select_and_gather_of_a_pass(P, L, Hkv, Bl):
    w = synth.Workload("sg", 43, L=L, Hq=Hkv, Hkv=Hkv, D=64, Bt=1, S=P + 7, ws=7, pool=3, N=max(1, Bl // 2), Bl=Bl, m=4, recipe="iid")
    g = torch.Generator(device="cuda").manual_seed(P)
    rand = lambda heads, rows: [torch.randn((1, heads, rows, w.D), generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(L)]
    q, k, v = rand(w.Hq, w.ws), rand(Hkv, w.S), rand(Hkv, w.S)
    k[0][:, 0, :P] = 0                                       # a head of equal scores
    kb, vb = ([torch.zeros((1, Hkv, w.Blc + w.ws, w.D), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.config_of(w))
    try:
        B.dkv_run_prefill_pass(h, q, k, v, kb, vb)
        torch.cuda.synchronize()
        counts = np.zeros((1, L), dtype=np.int32)
        B.dkv_get_counts(h, counts)
        for l in range(L):
            n, sc = int(counts[0, l]), np.empty((Hkv, P), dtype=np.float32)
            scores, idx = B.dkv_layer_views(h, l)
            B.dkv_memcpy_to_host(h, sc, scores, sc.nbytes)
            kept = B.read_device_i32(h, idx, (Hkv, w.Blc))[:, :n]
            want = np.argsort(-sc, axis=1, kind="stable")[:, :n]
            assert (kept == want).all(), f"layer {l}"
            rows = torch.from_numpy(np.concatenate([want, np.tile(np.arange(P, w.S), (Hkv, 1))], axis=1)).cuda()
            for src, buf in ((k, kb), (v, vb)):
                assert torch.equal(buf[l][0, :, :n + w.ws], torch.gather(src[l][0], 1, rows[:, :, None].expand(-1, -1, w.D)))
    finally:
        B.dkv_destroy(h)


# steps over many heads whose rows make fewer 16-row blocks than the launch has warps, about as many, and more
@pytest.mark.parametrize("L,Bt,Hkv,G,D,N,nq", [(11, 2, 4, 1, 128, 73, 1), (16, 1, 4, 7, 128, 56, 1), (20, 1, 2, 2, 64, 4, 3), (19, 1, 2, 4, 128, 300, 4),
                                               (12, 2, 4, 3, 64, 190, 1), (32, 1, 8, 4, 64, 64, 1)])
def test_decoding_step_over_short_heads(L, Bt, Hkv, G, D, N, nq):
    w = synth.Workload("dec", 44, L=L, Hq=G * Hkv, Hkv=Hkv, D=D, Bt=Bt, S=1205, ws=8, pool=3, N=N, Bl=2 * N, m=3, recipe="iid")
    g = torch.Generator(device="cuda").manual_seed(N)
    rand = lambda *shape: [torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(L)]
    q, k, v = (rand(Bt, heads, rows, D) for heads, rows in ((w.Hq, w.ws), (Hkv, w.S), (Hkv, w.S)))
    q = [x * (0.3 + l / L) for l, x in enumerate(q)]
    kb, vb = ([torch.zeros((Bt, Hkv, w.Blc + w.ws, D), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.config_of(w))
    try:
        B.dkv_run_prefill_pass(h, q, k, v, kb, vb)
        counts = np.zeros((Bt, L), dtype=np.int32)
        B.dkv_get_counts(h, counts)
        for _ in range(2):                                   # the second call finds what the first has left
            dq, out = rand(Bt, w.Hq, nq, D), [torch.zeros((Bt, w.Hq, nq, D), device="cuda") for _ in range(L)]
            B.dkv_decode_attend(h, 0, L, nq, dq, kb, vb, out)
            torch.cuda.synchronize()
            for l in range(L):
                for b in range(Bt):
                    n = int(counts[b, l]) + w.ws
                    kk, vv = (x[l][b, :, :n].double().repeat_interleave(G, dim=0) for x in (kb, vb))
                    want = (dq[l][b].double() @ kk.transpose(1, 2) / D ** 0.5).softmax(-1) @ vv
                    assert (out[l][b] - want).abs().max() <= 1e-5 * want.abs().max(), f"layer {l}, sample {b}"
    finally:
        B.dkv_destroy(h)


# Heads of one key tile, or of one in sweep 2 and few in sweep 1: the two MMA issuers of score_tc.cuh take tiles in turn, so that either
# has none of many heads.  Calls for one layer, all builds; scores are the same in every call.
@pytest.mark.parametrize("G,ws,D", [(1, 16, 64), (2, 32, 64), (3, 32, 128), (4, 32, 128), (7, 32, 128), (8, 32, 64)])
@pytest.mark.parametrize("S,Bt,lse", [(100, 64, False), (100, 64, True), (130, 32, False), (300, 3, False)])
def test_heads_of_one_tile(G, ws, D, S, Bt, lse):
    Hkv, pool, P = 8, 5, S - ws
    g = torch.Generator(device="cuda").manual_seed(S)
    q, k = (torch.randn(n, generator=g, device="cuda").to(torch.bfloat16) for n in ((Bt, G * Hkv, ws, D), (Bt, Hkv, S, D)))
    t = q.double().view(Bt, Hkv, G * ws, D) @ k.double().transpose(-1, -2) / D ** 0.5
    last = P + torch.arange(ws, device="cuda").repeat(G)
    t.masked_fill_(torch.arange(S, device="cuda") > last[:, None], -torch.inf)
    want = torch.nn.functional.max_pool1d(t.softmax(-1)[..., :P].sum(2), pool, 1, pool // 2)
    given = t.logsumexp(-1).view(Bt, Hkv * G, ws).float().contiguous()
    h = B.dkv_create(B.make_config(1, G * Hkv, Hkv, D, Bt, S, ws, pool, 4, 8, 1))
    try:
        first = None
        for _ in range(20):
            got = torch.zeros((Bt, Hkv, P), device="cuda")
            if lse:
                B.dkv_score_lse(h, 0, q, k, given, got)
            else:
                B.dkv_score(h, 0, q, k, got)
            first = got if first is None else first
            assert torch.equal(got, first)
        assert ((first - want).abs() <= 5e-5 * want).all()       # |t| < 128 in 32 bits: 2^-18 ln 2, and the sums
        assert B.dkv_last_status(h)[0] == B.DKV_OK
    finally:
        B.dkv_destroy(h)


def test_a_pass_over_heads_of_one_tile():
    L, Hkv, G, D, Bt, S, ws, pool = 32, 8, 4, 128, 8, 100, 32, 5
    g = torch.Generator(device="cuda").manual_seed(1)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k = new(Bt, G * Hkv, ws, D), new(Bt, Hkv, S, D)
    kb, vb = ([torch.zeros((Bt, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.make_config(L, G * Hkv, Hkv, D, Bt, S, ws, pool, 4, 8, 4))
    try:
        for _ in range(20):
            B.dkv_run_prefill_pass(h, q, k, k, kb, vb)
        last = S - ws + torch.arange(ws, device="cuda").repeat(G)
        for l in range(L):
            t = q[l].double().view(Bt, Hkv, G * ws, D) @ k[l].double().transpose(-1, -2) / D ** 0.5
            t.masked_fill_(torch.arange(S, device="cuda") > last[:, None], -torch.inf)
            want = torch.nn.functional.max_pool1d(t.softmax(-1)[..., :S - ws].sum(2), pool, 1, pool // 2).cpu()
            got = torch.zeros((Bt, Hkv, S - ws))
            B.dkv_memcpy_to_host(h, got, B.dkv_layer_views(h, l)[0], got.numel() * 4)
            assert ((got - want).abs() <= 5e-5 * want).all(), f"layer {l}"
        assert B.dkv_last_status(h)[0] == B.DKV_OK
    finally:
        B.dkv_destroy(h)
