"""Scoring of whole passes at the sizes where the sweeps change: window rows around their 16-row steps and the second plane, keys
around a tile, heads that lie in one pipe's range and in many, logits that a row's reference cannot hold."""
import numpy as np
import pytest
import torch

from oracle import dynamickv as O
from paper_2412_14838_b200 import binding as B
from paper_2412_14838_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    B.load()


def _scores(q, k, ws, pool):
    """Eq. 1-2 in 64 bits: q [Bt, Hq, ws, D], k [Bt, Hkv, S, D] -> [Bt, Hkv, S - ws]."""
    (Bt, Hkv, S, D), G = k.shape, q.shape[1] // k.shape[1]
    t = q.double().view(Bt, Hkv, G * ws, D) @ k.double().transpose(-1, -2) / D ** 0.5
    last = S - ws + torch.arange(ws, device="cuda").repeat(G)
    t.masked_fill_(torch.arange(S, device="cuda") > last[:, None], -torch.inf)
    return torch.nn.functional.max_pool1d(t.softmax(-1)[..., :S - ws].sum(2), pool, 1, pool // 2), t.logsumexp(-1).view(Bt, Hkv * G, ws)


def _passes(L, Hkv, G, D, Bt, S, ws, pool, change=None, most=5e-5, sweeps=False):
    """Both kinds of pass; a score is a sum of 2^(t - lse): with |t| < 128 in 32 bits each is off by 2^-18 ln 2 at most, and the
    instruction for 2^x and the sums add a few 2^-22.  sweeps: the pass has to be scored by row sums, key sums and pooling."""
    g = torch.Generator(device="cuda").manual_seed(S)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k, v = new(Bt, G * Hkv, ws, D), new(Bt, Hkv, S, D), new(Bt, Hkv, S, D)
    if change:
        change(q, k)
    P, rows = S - ws, min(8, S - ws) + ws
    kb, vb = ([torch.zeros((Bt, Hkv, rows, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    want, lse = zip(*(_scores(q[l], k[l], ws, pool) for l in range(L)))
    lse = [x.float().contiguous() for x in lse]
    h = B.dkv_create(B.make_config(L, G * Hkv, Hkv, D, Bt, S, ws, pool, 4, 8, 2))
    try:
        if sweeps:
            B.dkv_profile(h, True)
            B.dkv_run_prefill_pass(h, q, k, v, kb, vb)
            scoring = B.dkv_profile_read(h)
            B.dkv_profile(h, False)
            assert (scoring["score_stats"][1], scoring["score_emit"][1]) == (-(-L // 32), 2 * -(-L // 32))
        for run in (lambda: B.dkv_run_prefill_pass(h, q, k, v, kb, vb), lambda: B.dkv_run_prefill_pass_lse(h, q, k, v, lse, kb, vb)):
            run()
            for l in range(L):
                got = torch.zeros((Bt, Hkv, P))
                B.dkv_memcpy_to_host(h, got, B.dkv_layer_views(h, l)[0], got.numel() * 4)
                off = (got.cuda().double() - want[l]).abs() / want[l].clamp_min(1e-25)
                assert off.max() <= most, f"layer {l}: {off.max():.1e}"
            assert B.dkv_last_status(h)[0] == B.DKV_OK
    finally:
        B.dkv_destroy(h)


# (window rows G * ws: 1, 32, 33, 64, 65, 96, 97, 128, 130, 192, 256)
@pytest.mark.parametrize("G,ws,D", [(1, 1, 64), (1, 32, 128), (3, 11, 64), (2, 32, 64), (5, 13, 128), (3, 32, 128), (1, 97, 64), (4, 32, 64),
                                    (5, 26, 64), (6, 32, 128), (8, 32, 64)])
def test_window_rows(G, ws, D):
    _passes(2, 2, G, D, 1, 900, ws, 5)


# the last tile full, with one key, with the prefix ending at its start; fewer tiles than pipes; heads in many pipes and many in one
@pytest.mark.parametrize("L,Hkv,Bt,S,pool", [(1, 1, 1, 9, 1), (1, 1, 1, 128, 3), (1, 2, 1, 129, 7), (3, 1, 1, 136, 255), (2, 3, 2, 2049, 7),
                                             (2, 1, 1, 20011, 3), (33, 6, 3, 257, 9), (2, 2, 1, 2056, 5)])
def test_lengths(L, Hkv, Bt, S, pool):
    _passes(L, Hkv, 2, 64, Bt, S, 8, pool)


def test_a_call_of_128_rows_over_many_tiles():
    _passes(32, 8, 4, 128, 2, 8200, 32, 7)


def test_logits_that_are_far_above_the_first_key_of_a_segment():
    def far(q, k):                                           # up to 200 above it: 2^288 times its exponential
        q[0][:, :, :, 0], k[0][..., 0], k[0][:, 0, 700:705, 0] = 16.0, 0.0, 100.0
    _passes(2, 2, 2, 64, 1, 2000, 8, 5, far, most=2e-4)      # |t| < 512: 2^-16 ln 2 and more


# Such logits in some heads only, first and last ones of a pipe's range among them: two planes, four accumulator stages and two, heads
# in many pipes, many heads in one, several hundred (head, plane) pairs.
@pytest.mark.parametrize("L,Hkv,G,D,Bt,S,ws", [(2, 2, 7, 128, 1, 2000, 32), (3, 2, 4, 64, 1, 20011, 32), (33, 6, 2, 64, 3, 257, 8),
                                               (33, 3, 5, 64, 2, 200, 26), (1, 1, 1, 64, 1, 128, 3), (4, 8, 3, 128, 1, 6200, 27)])
@pytest.mark.parametrize("every", [1, 5])
def test_heads_with_logits_beyond_their_references(L, Hkv, G, D, Bt, S, ws, every):
    def far(q, k):
        n = 0
        for x, y in zip(q, k):
            x[..., 0] = 16.0
            for b in range(Bt):
                for h in range(Hkv):
                    y[b, h, :, 0] = 0.0
                    if n % every == 0:
                        y[b, h, S // 3::37, 0] = 100.0
                        y[b, h, S // 2::53, 0] = -100.0
                    n += 1
    _passes(L, Hkv, G, D, Bt, S, ws, 5, far, most=2e-4)


@pytest.mark.parametrize("bad", [1, 64])
def test_a_head_with_such_logits_costs_a_few_sweeps_of_its_own(bad):
    L, Hkv, S, ws, D = 8, 8, 32768, 32, 128
    g = torch.Generator(device="cuda").manual_seed(1)
    new = lambda *s: [torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for _ in range(L)]
    q, k = new(1, 3 * Hkv, ws, D), new(1, Hkv, S, D)
    kb, vb = ([torch.zeros((1, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.make_config(L, 3 * Hkv, Hkv, D, 1, S, ws, 5, 4, 8, 2))

    def time():
        best = 1e9
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            B.dkv_run_prefill_pass(h, q, k, k, kb, vb)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    try:
        time()
        clean = time()
        for i in range(bad):
            k[i // Hkv][0, i % Hkv, 100, 0] = torch.nan
        assert time() <= 4 * clean                           # two more sweeps for the row sums, which are less than half of a pass
        assert B.dkv_last_status(h)[0] == B.DKV_OK
    finally:
        B.dkv_destroy(h)


# One key of every 128 a little less than 88.7 nats (128 bits) above the others: the sums of the segments are finite, and would
# not be together.  |t| < 256: 2^-17 ln 2 a factor.
@pytest.mark.parametrize("nats", [82.0, 83.5, 84.0, 87.0, 88.5, 89.0, 95.0])
@pytest.mark.parametrize("L,Hkv,S", [(1, 1, 32768), (1, 3, 4999), (40, 8, 520)])    # a head in 256 segments, in 40, in one or two
def test_sums_of_segments_that_no_float_can_hold_together(L, Hkv, S, nats):
    def far(q, k):
        for x, y in zip(q, k):
            x[..., 0], y[..., 0], y[:, 0, 5::128, 0] = 16.0, 0.0, nats / 2
    _passes(L, Hkv, 1, 64, 1, S, 8, 5, far, most=1e-4)


# A sum of nearly 2^128 relative to its own reference, and another part whose reference is 126.6 bits above that one, so that the
# factor between them is below the smallest normal float; in another quarter of the tile, and in another segment.
@pytest.mark.parametrize("at", [32, 3 * 128])
def test_a_large_sum_beside_a_large_reference(at):
    def far(q, k):
        q[0][...], k[0][...] = 0.0, 0.0
        q[0][..., :2] = 16.0
        k[0][:, :, 5, 0], k[0][:, :, at, 0], k[0][:, :, at, 1] = 44.25, 43.5, 0.375      # 88.5 and 87.75 nats
    _passes(1, 1, 1, 64, 1, 2056, 8, 1, far, most=1e-4)


def test_a_head_with_a_key_that_is_no_number_spoils_no_other():
    g = torch.Generator(device="cuda").manual_seed(1)
    new = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    q, k = new(1, 6, 8, 64), new(1, 3, 700, 64)
    k[0, 1, 300, 5] = torch.nan
    kb = torch.zeros((1, 3, 16, 64), device="cuda", dtype=torch.bfloat16)
    h = B.dkv_create(B.make_config(1, 6, 3, 64, 1, 700, 8, 3, 4, 8, 2))
    try:
        B.dkv_run_prefill_pass(h, [q], [k], [k], [kb], [kb.clone()])
        got = torch.zeros((1, 3, 692))
        B.dkv_memcpy_to_host(h, got, B.dkv_layer_views(h, 0)[0], got.numel() * 4)
        want = _scores(q, k, 8, 3)[0].cpu()
        assert got[0, 1].isnan().all()
        assert ((got[0, ::2] - want[0, ::2]).abs() <= 5e-5 * want[0, ::2]).all()
    finally:
        B.dkv_destroy(h)


# the builds are 16 window rows apart: 16, 17, 48, 49, 80, 81, 112, 113 rows, two planes of 72 and of 112, and of 88 with 16 empty ones
@pytest.mark.parametrize("G,ws,D", [(1, 16, 64), (1, 17, 128), (3, 16, 128), (7, 7, 64), (5, 16, 64), (3, 27, 128), (7, 16, 128), (1, 113, 64),
                                    (5, 28, 128), (7, 32, 64), (7, 24, 128)])
def test_window_rows_around_sixteens(G, ws, D):
    _passes(2, 2, G, D, 1, 900, ws, 5)


def test_a_context_of_many_heads_takes_no_statistics_for_groups_of_layers():
    L, Bt, Hkv, S, ws, D = 32, 32, 8, 264, 8, 64
    P = S - ws
    cfg = B.make_config(L, Hkv, Hkv, D, Bt, S, ws, 3, 4, 8, 2)
    B.dkv_destroy(B.dkv_create(cfg))                         # loads the kernels
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    h = B.dkv_create(cfg)
    try:
        # scores and candidates (4 and 8 bytes a position), unpooled scores and histograms; the rest is below 16 MB
        known = L * Bt * (Hkv * P * 4 + max(Hkv * P * 8, Hkv * 384 * 4) + 2048 * 4)
        assert free - torch.cuda.mem_get_info()[0] <= known + (24 << 20)
        g = torch.Generator(device="cuda").manual_seed(7)
        for l in range(5):                                   # three sets of statistics in turn
            q, k = (torch.randn((Bt, Hkv, n, D), generator=g, device="cuda").to(torch.bfloat16) for n in (ws, S))
            got = torch.zeros((Bt, Hkv, P), device="cuda")
            B.dkv_score(h, l, q, k, got)
            want = _scores(q, k, ws, 3)[0]
            assert ((got - want).abs() <= 5e-5 * want).all()
    finally:
        B.dkv_destroy(h)


# As many segments in a pipe as a prompt of one tile a head can have: 40000 samples of 8 heads, far logits in all.
def test_a_thousand_segments_of_one_tile():
    def far(q, k):
        q[0][..., 0], k[0][..., 0], k[0][:, :, 3, 0] = 16.0, 0.0, 100.0
    _passes(1, 8, 1, 64, 40000, 16, 1, 1, far, most=2e-4)


# Heads of 2048 tiles, each on one pipe or two.  What a pipe adds one key after the other is 256 tiles: 1024 additions of a thread,
# each off by 2^-25 of the sum in the mean, is 1e-6 of it and less for the 64 such sums of a row; logits of |t| < 64 are off by 2^-19
# and 2^-20 in the mean.  (Added to the end of the head, 8192 of them, the largest mean error of a head was 5.4e-6.)
@pytest.mark.parametrize("far", [False, True])
def test_the_error_of_a_row_sum_does_not_grow_with_the_prompt(far):
    Bt, Hkv, S, ws, D = 37, 4, 262144, 8, 64
    P = S - ws
    g = torch.Generator(device="cuda").manual_seed(1)
    q = (3 * torch.randn((Bt, Hkv, ws, D), generator=g, device="cuda")).to(torch.bfloat16)
    k = torch.empty((Bt, Hkv, S, D), device="cuda", dtype=torch.bfloat16)
    for x in k:
        x.normal_(generator=g)
    if far:                                                  # in a later part of some heads, and only there
        q[3:5, ..., 0], k[3:5, ..., 0], k[3:5, :, 150000, 0] = 16.0, 0.0, 60.0
    kb = torch.zeros((Bt, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16)
    h = B.dkv_create(B.make_config(1, Hkv, Hkv, D, Bt, S, ws, 1, 4, 8, 2))
    try:
        B.dkv_run_prefill_pass(h, [q], [k], [k], [kb], [kb.clone()])
        got = torch.zeros((Bt, Hkv, P))
        B.dkv_memcpy_to_host(h, got, B.dkv_layer_views(h, 0)[0], got.numel() * 4)
        for b in range(Bt):
            want = _scores(q[b:b + 1], k[b:b + 1], ws, 1)[0][0]
            off = (got[b].cuda().double() - want) / want.clamp_min(1e-25)
            if far and 3 <= b < 5:                           # |t| < 256
                assert off.abs().max() <= 1e-4
            else:
                assert off.mean(-1).abs().max() <= 2.5e-6, f"sample {b}: {off.mean(-1).abs().max():.1e}"
    finally:
        B.dkv_destroy(h)


def _masked(q, k):                                           # keys that no query sees: logits of minus infinity, first ones of heads too
    for x, y in zip(q, k):
        x[..., 0] = x[..., 0].abs() + 1
        y[:, 0, :300, 0], y[..., 5::7, 0] = -torch.inf, -torch.inf


# two planes of 80 rows and 64, and of 112; and one
@pytest.mark.parametrize("G,ws,D", [(9, 16, 64), (7, 32, 128), (4, 32, 64), (1, 16, 64)])
def test_keys_at_minus_infinity_count_for_nothing(G, ws, D):
    _passes(20, 2, G, D, 1, 1000, ws, 1, _masked, sweeps=True)


def test_parts_of_a_long_head_at_minus_infinity():
    """Heads of 1024 tiles, about one to a pipe, whose first two parts of 256 tiles hold no key that counts."""
    L, Hkv, S, ws, D = 32, 8, 131072, 16, 64
    P, masked = S - ws, 66000
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k = (torch.randn((1, Hkv, n, D), generator=g, device="cuda").to(torch.bfloat16) for n in (ws, S))
    q[..., 0], k[:, :, :masked, 0] = q[..., 0].abs() + 1, -torch.inf
    kb, vb = ([torch.zeros((1, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.make_config(L, Hkv, Hkv, D, 1, S, ws, 1, 4, 8, 32))
    try:
        B.dkv_run_prefill_pass(h, [q] * L, [k] * L, [k] * L, kb, vb)
        want = _scores(q, k, ws, 1)[0]
        got = torch.zeros((1, Hkv, P))
        for l in range(L):
            B.dkv_memcpy_to_host(h, got, B.dkv_layer_views(h, l)[0], got.numel() * 4)
            assert (got[..., :masked] == 0).all()
            assert ((got.cuda() - want).abs() <= 5e-5 * want).all()
        assert B.dkv_last_status(h)[0] == B.DKV_OK
    finally:
        B.dkv_destroy(h)


def test_digit_counters_beyond_31_bits():
    """32 layers of 32768 samples have 2^31 counters, which every pass has to clear: counts of a pass after others."""
    L, Bt, S, ws, D, N, Bl = 32, 32768, 12, 1, 64, 4, 8
    P = S - ws
    g = torch.Generator(device="cuda").manual_seed(1)
    new = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    k, q = new(Bt, 1, S, D), [new(Bt, 1, ws, D) for _ in range(L)]
    lse = [torch.full((Bt, 1, ws), 3.0, device="cuda")] * L
    kb, vb = ([torch.zeros((Bt, 1, Bl + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
    h = B.dkv_create(B.make_config(L, 1, 1, D, Bt, S, ws, 1, N, Bl, L))
    try:
        for run in (lambda q: B.dkv_run_prefill_pass_lse(h, q, [k] * L, [k] * L, lse, kb, vb), lambda q: B.dkv_run_prefill_pass(h, q, [k] * L, [k] * L, kb, vb)):
            run(q[::-1])
            run(q)
            assert B.dkv_last_status(h)[0] == B.DKV_OK
            counts = torch.zeros((Bt, L), dtype=torch.int32)
            B.dkv_get_counts(h, counts)
            scores = torch.zeros((L, Bt, 1, P))
            for l in range(L):
                B.dkv_memcpy_to_host(h, scores[l], B.dkv_layer_views(h, l)[0], scores[l].numel() * 4)
            for b in (0, 1, Bt // 2 - 1, Bt // 2, Bt - 1):
                want = O.rebudget([x.numpy() for x in scores[:, b]], [Bl] * L, N, Bl, L)["counts"]
                assert np.array_equal(counts[b], want), f"sample {b}"
    finally:
        B.dkv_destroy(h)


# Passes of 128 rows of 128 dims that are scored by groups of layers, the last group smaller (25, 25, 25, 22 layers; 26, 26, 26, 23;
# 17, 16), with fewer tiles than SMs.  The fourth group's statistics go where the first one's were.
@pytest.mark.parametrize("L,S", [(97, 500), (101, 500), (101, 896), (33, 896)])
def test_last_group_with_fewer_tiles_than_the_one_before(L, S):
    _passes(L, 1, 4, 128, 1, S, 32, 5)


# enough tiles (two an SM) for passes of two planes: 129 to 256 rows, planes that share rows and planes that do not, all of one size
# of the builds and of the largest; without and with logits whose sums have to be computed again, in either plane
@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("G,ws,D", [(1, 129, 64), (5, 26, 64), (5, 28, 128), (9, 16, 64), (7, 24, 128), (6, 32, 64), (7, 32, 128), (3, 75, 64),
                                    (8, 32, 128), (8, 32, 64)])
def test_two_planes(G, ws, D, far):
    def change(q, k):
        for n, (x, y) in enumerate(zip(q, k)):
            x[..., 0], y[..., 0] = 0.0, 0.0
            if n % 3 == 0:                                   # in this layer for the last query head, which is in the second plane
                x[:, -1, :, 0], y[:, -1, 500::61, 0] = 16.0, 100.0
            elif n % 3 == 1:                                 # for the first query head of a key head
                x[:, ::G, :, 0], y[:, 0, 500::61, 0] = 16.0, 100.0
    _passes(20, 2, G, D, 1, 1000, ws, 5, change if far else None, most=2e-4 if far else 5e-5, sweeps=True)


# At the line where score_tc.cuh takes passes of more than 207 rows over heads of two tiles, one of them without a scored position
# (samples: fewest that it takes, one less; a row less; one position more).
@pytest.mark.parametrize("G,ws,D,Bt,S,sweeps", [(8, 26, 128, 7, 150, False), (8, 26, 128, 6, 150, True), (9, 23, 128, 7, 147, True), (8, 32, 128, 7, 156, False),
                                                (8, 32, 128, 7, 157, True), (8, 32, 64, 14, 130, False), (8, 32, 64, 13, 130, True)])
def test_many_short_heads_of_many_rows(G, ws, D, Bt, S, sweeps):
    L, Hkv, pool = 16, 8, 5                                   # 256 tiles a sample
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert sms == 148, "the samples are for 148 SMs"
    _passes(L, Hkv, G, D, Bt, S, ws, pool, sweeps=sweeps)
    if not sweeps:
        q, k = (torch.randn((Bt, n, m, D), device="cuda").to(torch.bfloat16) for n, m in ((G * Hkv, ws), (Hkv, S)))
        kb, vb = ([torch.zeros((Bt, Hkv, 8 + ws, D), device="cuda", dtype=torch.bfloat16) for _ in range(L)] for _ in range(2))
        h = B.dkv_create(B.make_config(L, G * Hkv, Hkv, D, Bt, S, ws, pool, 4, 8, 2))
        try:
            before = B.dkv_launch_count(h)
            B.dkv_run_prefill_pass(h, [q] * L, [k] * L, [k] * L, kb, vb)
            assert B.dkv_launch_count(h) - before == 2 + 3 + 1       # sweep 1, sweep 2, the updates, selection
        finally:
            B.dkv_destroy(h)
