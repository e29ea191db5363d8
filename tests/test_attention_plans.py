"""What the tensor-core attention is cut into (host code, no GPU)."""
import ctypes as C
import random

import pytest

SMS = 152


@pytest.fixture(scope="module")
def plan():
    from paper_2609_34170_gb300 import build, load
    build.build()
    fn = load().ravel_debug_attention_plan
    fn.restype = None
    fn.argtypes = [C.c_int] * 7 + [C.c_size_t, C.c_int, C.c_void_p, C.c_void_p]
    clusters, out = (C.c_int * 4)(76, 36, 15, 7), (C.c_int * 5)()

    def call(B, H, F, Hq, Hkv, hd, P):
        fn(B, H, F, Hq, Hkv, hd, P, 32 << 20, SMS, clusters, out)
        return dict(zip(("tiles", "TQ", "splits", "bf16", "smem"), out))

    return call


def _most_splits(B, H, F, Hq, Hkv, hd, P):
    """Splits of two 64-key pieces each on the SMs that 128-row tiles leave idle
    (64-row tiles where eight of each fit half the SMs)."""
    G, hdp = Hq // Hkv, -(-hd // 16) * 16
    pieces = -(-P // 64) - (-(H + F) // 64)
    tiles = -(-H // max(1, 128 // G))
    rows, small = -(-H // tiles), -(-H // max(1, 64 // G))
    if tiles * B * Hkv * 2 <= SMS and max(1, 64 // G) < rows and small * B * Hkv * 16 <= SMS and pieces >= 3:
        tiles = small
    ctas, s = tiles * B * Hkv, 1
    if ctas * 2 > SMS:
        return 1
    while (s * 2 <= min((pieces + 1) // 2, SMS // ctas, 16) and hdp // (s * 2) % 4 == 0
           and s * 2 * ctas * 128 * (hdp + 2) * 4 <= 32 << 20):
        s *= 2
    return s


def test_partials_in_bf16_only_where_splits_are_many(plan):
    rng = random.Random(1)
    shapes = [(b, h, 32, 16, 4, 64, p) for b in range(1, 14) for h in (8, 30, 50) for p in (64, 128, 512, 2048)]
    for _ in range(20000):
        hkv = rng.choice([1, 1, 2, 4, 8])
        shapes.append((int(65 ** rng.random()), rng.randint(1, 60), rng.randint(0, 40), hkv * rng.choice([1, 2, 4, 8]), hkv,
                       8 * rng.randint(1, 32), int(2049 ** rng.random())))
    for s in shapes:
        p, most = plan(*s), _most_splits(*s)
        hdp = -(-s[5] // 16) * 16
        assert most > 1 or p["splits"] == 1, (s, p)
        assert not p["bf16"] or (hdp // most % 8 == 0 and hdp // p["splits"] % 8 == 0), (s, p, most)
        assert p["tiles"] * p["TQ"] >= s[1] and p["TQ"] * (s[3] // s[4]) <= 128, (s, p)
        # nothing that waits for a peer with TMEM taken fits beside it (30 KB is the least that a split GEMM takes)
        assert 200 * 1024 < p["smem"] <= 227 * 1024, (s, p)
    # one robot's two experts, and a group of robots, keep their bf16 merge
    assert plan(1, 50, 16, 8, 1, 256, 816)["bf16"] and plan(8, 30, 32, 16, 4, 64, 512)["bf16"]
    assert plan(16, 16, 16, 8, 1, 256, 2048)["bf16"]
