"""Kernels that begin before the one before them has ended: calls queued one behind the other, each on data that the call before
it has just replaced, give what the same calls give with the GPU idle in between."""
import pytest
import torch

from paper_2412_14838_b200 import binding as B
from paper_2412_14838_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()


@pytest.mark.parametrize("Hkv,G,D,keep,ws", [(8, 4, 128, 500, 8), (2, 3, 64, 1, 2), (1, 8, 128, 1030, 1)])
def test_decoding_behind_the_gather_of_its_rows(Hkv, G, D, keep, ws):
    n, S = 6, keep + ws + 50
    g = torch.Generator(device="cuda").manual_seed(keep)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(n)]
    k, v, q = new(1, Hkv, S, D), new(1, Hkv, S, D), new(1, Hkv * G, 1, D)
    kb, vb = (torch.zeros((1, Hkv, keep + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(2))
    queued, alone = ([torch.zeros((1, Hkv * G, 1, D), device="cuda") for _ in range(n)] for _ in range(2))
    ctx = B.dkv_create(B.make_config(1, Hkv * G, Hkv, D, 1, S, ws, 1, 1, keep, 1))
    try:
        for out, wait in ((queued, False), (alone, True)):
            torch.cuda.synchronize()
            for i in range(n):
                B.dkv_select_positions(ctx, 0, 0, keep)
                B.dkv_compact(ctx, 0, k[i], v[i], kb, vb)
                if wait:
                    torch.cuda.synchronize()
                B.dkv_decode_attend(ctx, 0, 1, 1, [q[i]], [kb], [vb], [out[i]])
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) and a.abs().max() > 0 for a, b in zip(queued, alone))
    finally:
        B.dkv_destroy(ctx)


# heads enough for a block each; few long ones, which clusters share; ten updates in two batches; budgets that reach 0
@pytest.mark.parametrize("L,Hkv,D,S,N,Bl,m", [(6, 8, 64, 1500, 40, 100, 2), (2, 2, 64, 25000, 64, 200, 2), (10, 2, 64, 700, 9, 40, 1),
                                              (3, 1, 128, 200, 1, 1, 2)])
def test_passes_queued_over_different_prompts(L, Hkv, D, S, N, Bl, m):
    n, ws = 4, 8
    g = torch.Generator(device="cuda").manual_seed(S)
    new = lambda scale, *s: [[(scale * (1 + l) * torch.randn(s, generator=g, device="cuda")).to(torch.bfloat16) for l in range(L)] for _ in range(n)]
    q, k, v = new(0.5, 1, 2 * Hkv, ws, D), new(0.7, 1, Hkv, S, D), new(1.0, 1, Hkv, S, D)
    buffers = lambda: [[torch.zeros((1, Hkv, Bl + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(n)]
    one, two = (buffers(), buffers()), (buffers(), buffers())
    ctx = B.dkv_create(B.make_config(L, 2 * Hkv, Hkv, D, 1, S, ws, 3, N, Bl, m))
    try:
        for (kb, vb), wait in ((one, False), (two, True)):
            torch.cuda.synchronize()
            for i in range(n):
                B.dkv_run_prefill_pass(ctx, q[i], k[i], v[i], kb[i], vb[i])
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert not torch.equal(one[0][0][0], one[0][1][0])
        for a, b in zip(one, two):
            assert all(torch.equal(a[i][l], b[i][l]) for i in range(n) for l in range(L))
        assert B.dkv_last_status(ctx)[0] == B.DKV_OK
    finally:
        B.dkv_destroy(ctx)
