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
