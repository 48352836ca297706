"""Decode attention where its kernels can go wrong: row counts around the 16-row blocks, query counts around the 8 and
16 a warp holds, few heads (a cluster per head) and many (equal slices of all rows), against torch in double precision."""
import numpy as np
import pytest
import torch

from paper_2412_14838_b200 import binding as B
from paper_2412_14838_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()


@pytest.mark.parametrize("L,Hkv,G,nq,D,Bt,ws,keep", [
    (1, 1, 1, 1, 64, 1, 1, [0]),                          # a single row
    (2, 2, 4, 1, 128, 1, 7, [8, 9]),                      # 15 and 16 rows
    (3, 2, 4, 2, 128, 2, 8, [9, 300, 1017]),              # 17 rows; one full round of a cluster and a row more
    (2, 4, 3, 3, 64, 1, 5, [123, 4000]),                  # 9 queries a head group: the 16-query build
    (1, 2, 1, 17, 128, 1, 4, [77]),                       # 17: two rounds of queries
    (2, 1, 8, 8, 64, 1, 32, [500, 31]),                   # 64, the most
    (12, 8, 4, 1, 128, 1, 16, [0, 1, 2, 900, 0, 17, 333, 0, 0, 2048, 5, 64]),   # slices over lengths that differ
    (9, 8, 4, 4, 128, 3, 8, [0, 1500, 8, 0, 40, 23, 900, 0, 7]),
    (5, 12, 2, 1, 64, 4, 3, [13, 14, 400, 0, 2]),
    (70, 2, 3, 1, 64, 1, 2, [i * 7 % 90 for i in range(70)]),                   # more layers than one launch takes
])
def test_decode_attention(L, Hkv, G, nq, D, Bt, ws, keep):
    S, Bl = max(keep) + ws + 10, max(max(keep), 1)
    g = torch.Generator(device="cuda").manual_seed(L * 100 + nq)
    ctx = B.dkv_create(B.make_config(L, Hkv * G, Hkv, D, Bt, S, ws, 1, 1, Bl, 1))
    try:
        rows = Bl + ws
        new = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
        kb, vb = ([torch.full((Bt, Hkv, rows, D), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
        q = [new(Bt, Hkv * G, nq, D) for _ in range(L)]
        out = [torch.zeros((Bt, Hkv * G, nq, D), device="cuda") for _ in range(L)]
        for l in range(L):
            B.dkv_select_positions(ctx, l, 0, keep[l])
            B.dkv_compact(ctx, l, new(Bt, Hkv, S, D), new(Bt, Hkv, S, D), kb[l], vb[l])
        for _ in range(2):                                # the second call finds the first one's scratch
            B.dkv_decode_attend(ctx, 0, L, nq, q, kb, vb, out)
        torch.cuda.synchronize()
        for l in range(L):
            n = keep[l] + ws
            k, v = (x[l][:, :, :n].double().repeat_interleave(G, dim=1) for x in (kb, vb))
            want = torch.softmax(q[l].double() @ k.transpose(-1, -2) / np.sqrt(D), dim=-1) @ v
            err = (out[l].double() - want).abs().max() / want.abs().max()
            assert err < 3e-6, f"layer {l}: {err:.2e}"
        first = [o.clone() for o in out]
        for l in range(L):                                # one layer a call: the same results to rounding
            B.dkv_decode_attend(ctx, l, 1, nq, q[l:l + 1], kb[l:l + 1], vb[l:l + 1], out[l:l + 1])
        torch.cuda.synchronize()
        assert all((a - b).abs().max() <= 3e-6 * b.abs().max() for a, b in zip(out, first))
    finally:
        B.dkv_destroy(ctx)


def test_first_step_on_a_stream_that_does_not_wait_for_the_default_one():
    L, Hkv, G, D, S, ws = 10, 8, 4, 128, 700, 8              # heads enough for the slices, which count arrivals
    g = torch.Generator(device="cuda").manual_seed(7)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k, v, dq = new(1, Hkv * G, ws, D), new(1, Hkv, S, D), new(1, Hkv, S, D), new(1, Hkv * G, 1, D)
    kb, vb = ([torch.zeros((1, Hkv, 300 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    out, again = ([torch.zeros((1, Hkv * G, 1, D), device="cuda") for _ in range(L)] for _ in range(2))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = B.dkv_create(B.make_config(L, Hkv * G, Hkv, D, 1, S, ws, 3, 100, 300, 2))
    try:
        torch.cuda._sleep(200_000_000)                       # the default stream is busy for a tenth of a second
        B.dkv_run_prefill_pass(ctx, q, k, v, kb, vb, side)
        B.dkv_decode_attend(ctx, 0, L, 1, dq, kb, vb, out, side)
        side.synchronize()
        first = [o.clone() for o in out]
        torch.cuda.synchronize()
        B.dkv_run_prefill_pass(ctx, q, k, v, kb, vb)
        B.dkv_decode_attend(ctx, 0, L, 1, dq, kb, vb, again)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) and a.abs().max() > 0 for a, b in zip(first, again))
    finally:
        B.dkv_destroy(ctx)
