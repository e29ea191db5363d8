"""What the tensor-core GEMM is cut into (host code, no GPU): the plan's
tile width, splits, exchange, accumulators, TMEM and shared memory over sizes
drawn from the whole range."""
import ctypes as C
import random

import pytest

STORE, SILU, ADD, GEGLU = 0, 1, 2, 3
NONE, L2, BF16, FP32 = 0, 1, 2, 3   # how splits exchange their partials
SMS, SM_SMEM, TMEM = 152, 228 * 1024, 512


def load_plan():
    from paper_2609_34170_gb300 import build, load
    build.build()
    fn = load().ravel_debug_gemm_plan
    fn.restype = None
    fn.argtypes = [C.c_int] * 7 + [C.c_size_t, C.c_int, C.c_void_p, C.c_void_p]
    clusters = (C.c_int * 4)(76, 36, 15, 7)
    out = (C.c_int * 7)()

    def call(m, n, k, epi, out_bf16, xbf16, aligned=1, ws=24 << 20):
        fn(m, n, k, epi, out_bf16, xbf16, aligned, ws, SMS, clusters, out)
        return dict(zip(("pair", "bn", "splits", "exchange", "accs", "cols", "smem"), out))

    return call


@pytest.fixture(scope="module")
def plan():
    return load_plan()


def _draws(n, seed):
    rng = random.Random(seed)
    for _ in range(n):
        m = int(4225 ** rng.random())
        k = 8 * rng.randint(1, 512) if rng.random() < 0.5 else rng.choice([64, 128, 256, 512, 1024, 2048, 4096])
        nn = rng.choice([32, 100, 1024, 1536, 2560, 8192, rng.randint(16, 4096)])
        epi = rng.choice([STORE, STORE, SILU, ADD, GEGLU])
        yield (m, (nn + 127) // 128 * 128 if epi == GEGLU else nn, k, epi,
               1 if epi == GEGLU else 0 if epi == ADD else rng.randint(0, 1), rng.randint(0, 1), rng.random() < 0.8)


def test_waiting_launches_share_an_sm_only_if_tmem_holds_both(plan):
    """CTAs that wait for others of their cluster may meet another stream's on
    an SM, each holding TMEM that the other's peers need: whatever fits the
    SM's shared memory together must fit its TMEM."""
    splits, pairs = set(), set()
    for m, n, k, epi, bf, xb, al in _draws(20000, 1):
        p = plan(m, n, k, epi, bf, xb, int(al))
        assert 0 < p["smem"] <= 227 * 1024 and 32 <= p["cols"] <= TMEM, (m, n, k, p)
        if p["splits"] > 1:
            splits.add((p["smem"] + 1024, p["cols"]))   # 1 KB of each CTA is the system's
        elif p["pair"]:
            pairs.add((p["smem"] + 1024, p["cols"]))
    for smem, cols in splits:   # at most its share of TMEM: any set of them fits
        assert cols * SM_SMEM <= TMEM * smem, (smem, cols)
    for smem, cols in pairs:
        for s2, c2 in splits:
            assert smem + s2 > SM_SMEM or cols + c2 <= TMEM, (smem, cols, s2, c2)


def test_shares_in_bf16_only_where_splits_are_many(plan):
    """A share rounded to bf16 loses up to 2^-8 of its size: only a step's launch does
    that, and only where 64- or 128-token tiles split into slices of at most 32
    tokens on the SMs that there are."""
    def check(m, n, k, epi, bf, xb, al):
        p = plan(m, n, k, epi, bf, xb, al)
        many = 2 if m <= 64 else 4
        if not xb or (n + 127) // 128 * ((m + 127) // 128) * many > SMS or (k + 63) // 64 < many:
            assert p["exchange"] != BF16, (m, n, k, epi, p)
        assert (p["exchange"] == NONE) == (p["splits"] == 1), p
        return p

    for d in _draws(20000, 2):
        check(*d[:6], int(d[6]))
    for m in range(1, 1200):   # the projections of the two experts, all token counts
        for n, k, epi, bf in ((2560, 1024, STORE, 1), (1024, 2048, ADD, 0), (1024, 4096, ADD, 0), (8192, 1024, GEGLU, 1),
                              (1536, 1024, STORE, 1), (1024, 1024, ADD, 0)):
            p = check(m, n, k, epi, bf, 1, 1)
            if m == 50:   # one robot: the exchange that the step was tuned with
                assert p["exchange"] == (BF16 if p["splits"] > 1 else NONE)


def test_fp32_results_sum_one_k_tile_per_accumulator(plan):
    """The tensor cores truncate, so a sum's error grows with its length: where
    the result stays fp32, each k-tile has an accumulator of its own as far as
    TMEM holds them (two tiles' worth where a CTA has several); past 32 k-tiles
    four share them where outputs are aligned."""
    for m, n, k, epi, bf, _, al in _draws(20000, 3):
        for xb in (0, 1):
            p = plan(m, n, k, epi, bf, xb, int(al))
            per_item = -(-((k + 63) // 64) // p["splits"])
            items = -(-((n + 127) // 128 * -(-m // p["bn"])) // SMS) if p["splits"] == 1 else 1
            width = 32
            while width < p["bn"]:
                width *= 2
            fit = max(1, TMEM // width // (2 if items > 1 else 1))
            halves = 2 if (n + 127) // 128 * ((m + 127) // 128) * 2 <= SMS else 1
            if bf or p["pair"] or p["exchange"] == BF16:
                assert p["accs"] == 1, (m, n, k, p)
            else:
                assert p["accs"] == min(per_item, fit, halves if xb else 4 if per_item > 32 and al else fit), (m, n, k, xb, p)
    for m, n, k in ((1, 32, 128), (16, 128, 128), (50, 1024, 1024), (128, 1024, 1024), (240, 512, 560), (256, 100, 4096)):
        p = plan(m, n, k, STORE, 0, 0)
        assert -(-((k + 63) // 64) // (p["splits"] * p["accs"])) == 1, (m, n, k, p)
    # a step's O and down without splits: two halves, as the widest split of 128 tokens summed
    assert plan(800, 1024, 2048, ADD, 0, 1)["accs"] == plan(800, 1024, 4096, ADD, 0, 1)["accs"] == 2


def test_slices_through_l2_go_out_in_few_chunks(plan):
    """An unaligned split's slice costs a round trip per chunk of 16, 8 or 4
    tokens: the plans of shapes that had been slower than with wider slices."""
    for m, n, k in ((200, 2049, 6216), (426, 749, 3088), (316, 1245, 2872), (167, 1715, 2632)):
        p = plan(m, n, k, ADD, 0, 0, 0)
        slice_ = p["bn"] // p["splits"]
        assert p["exchange"] in (NONE, L2) and (p["splits"] == 1 or slice_ % 16 == 0), (m, n, k, p)


def test_fp32_rows_only_where_they_were_measured_faster():
    """Each side of the line between the fp32 row and tile kernels, at sizes
    whose times its comment gives."""
    from paper_2609_34170_gb300 import build, load
    build.build()
    rows = load().ravel_debug_rows_gemm
    for m, n, k in ((1, 75776, 4096), (24, 75776, 1024), (64, 2560, 1024), (192, 2560, 1024), (256, 1024, 4096),
                    (96, 4096, 4096), (192, 2048, 256)):
        assert rows(m, n, k, STORE) == rows(m, n, k, GEGLU) == 1, (m, n, k)
    for m, n, k in ((25, 75776, 1024), (128, 4096, 4096), (192, 4096, 4096), (128, 8192, 1024), (200, 8192, 1024),
                    (257, 33, 516), (8, 100, 250)):
        assert rows(m, n, k, STORE) == rows(m, n, k, GEGLU) == 0, (m, n, k)
    for m, n, k in ((100, 8192, 1024), (192, 3000, 1024), (250, 2048, 256)):   # GeGLU saves a launch
        assert (rows(m, n, k, STORE), rows(m, n, k, GEGLU)) == (0, 1), (m, n, k)
