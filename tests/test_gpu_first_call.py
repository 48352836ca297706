"""First calls in a process of their own: what a kernel needs before its first launch is set by the context, or the call,
whose shape reaches it, and not by an earlier caller."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys, torch
from paper_2412_14838_b200 import binding as B
B.load()
use, *shapes = eval(sys.argv[1])
for Hq, Hkv, D, ws in shapes:                               # ws * Hq / Hkv window rows
    L, S = 3, 900
    g = torch.Generator(device="cuda").manual_seed(ws)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k, v = new(1, Hq, ws, D), new(1, Hkv, S, D), new(1, Hkv, S, D)
    kb, vb = ([torch.zeros((1, Hkv, 64 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    one = torch.zeros((1, Hkv, S - ws), device="cuda")
    cfg = B.make_config(L, Hq, Hkv, D, 1, S, ws, 1, 32, 64, 2)
    logits = q[0].double() @ k[0].double().repeat_interleave(Hq // Hkv, dim=1).transpose(-1, -2) / D ** 0.5
    logits.masked_fill_(torch.arange(S, device="cuda") > (S - ws + torch.arange(ws, device="cuda"))[:, None], float("-inf"))
    want = logits.softmax(-1)[..., :S - ws].sum(2).view(1, Hkv, -1, S - ws).sum(2)
    close = lambda x: ((x - want).abs().max() <= 1e-4 * want.max()).item()
    if use == "static":
        B.dkv_score_static(cfg, q[0], k[0], one)
        assert close(one), "static"
    elif use == "lse":
        ctx = B.dkv_create(cfg)
        lse = [logits.logsumexp(-1).float().contiguous()] * L
        B.dkv_run_prefill_pass_lse(ctx, q, k, v, lse, kb, vb)
        B.dkv_memcpy_to_host(ctx, host := torch.zeros(one.shape), B.dkv_layer_views(ctx, 0)[0], host.numel() * 4)
        assert close(host.cuda()), "pass with log-denominators"
        assert B.dkv_last_status(ctx)[0] == B.DKV_OK
        B.dkv_destroy(ctx)
    else:
        ctx = B.dkv_create(cfg)
        B.dkv_score(ctx, 0, q[0], k[0], one)
        assert close(one), "one layer"
        B.dkv_run_prefill_pass(ctx, q, k, v, kb, vb)
        B.dkv_memcpy_to_host(ctx, host := torch.zeros(one.shape), B.dkv_layer_views(ctx, 0)[0], host.numel() * 4)
        assert close(host.cuda()), "pass"
        B.dkv_destroy(ctx)
print("ok")
"""

SHAPES = [(4, 2, 64, 16), (8, 2, 128, 16), (6, 2, 128, 32), (8, 2, 128, 32), (8, 2, 64, 32), (14, 2, 128, 32)]   # 32 .. 224 window rows


@pytest.mark.parametrize("case", [(u, s) for u in ("pass", "lse") for s in SHAPES] + [("static", *SHAPES)], ids=str)
def test_first_call_of_a_process(case):
    res = subprocess.run([sys.executable, "-c", CHILD, repr(case)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stderr[-2000:]
