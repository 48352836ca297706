"""Scoring at the window-row counts where the kernel changes its build (32, 64 and 128 rows per KV head) and around them."""
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


@pytest.mark.parametrize("G,ws,D,S", [(1, 1, 64, 130), (1, 31, 128, 1000), (4, 8, 64, 2055), (3, 11, 128, 700), (7, 9, 64, 1555),
                                      (2, 32, 128, 4097), (5, 13, 128, 900), (4, 32, 64, 1300), (3, 43, 128, 777)])
def test_scores_match_oracle(G, ws, D, S):
    w = synth.Workload("rows", 95, L=1, Hq=2 * G, Hkv=2, D=D, Bt=2, S=S, ws=ws, pool=3, N=4, Bl=8, m=1, recipe="sink")
    t = synth.layer_inputs(w, 0, want_v=False)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()
    h = B.dkv_create(B.config_of(w))
    try:
        out = torch.zeros((w.Bt, w.Hkv, w.P), dtype=torch.float32, device="cuda")
        B.dkv_score(h, 0, dev(t["q"]), dev(t["k"]), out)
        torch.cuda.synchronize()
        ref = O.window_scores(synth.bf16_bits_to_f64(t["q"]), synth.bf16_bits_to_f64(t["k"]), w.ws, w.pool)["score"]
        U.assert_scores_close(out.cpu().numpy(), ref, f"{w.M} window rows")
    finally:
        B.dkv_destroy(h)
