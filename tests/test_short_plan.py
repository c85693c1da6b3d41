"""Launch geometry of the kernels for short vectors (host logic only)."""
import pytest

from paper_2309_13307_b200 import binding


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


VECTORS = [*range(1, 70), 100, 128, 129, 255, 256, 257, 400, 1000, 1024, 1025, 2000, 2048, 2049, 3000, 4095, 4096, 4097]


@pytest.mark.parametrize("sm_count", [1, 2, 5, 8, 9, 20, 132, 148])
def test_a_reconstruction_has_a_thread_per_block_and_range(sm_count):
    """... and the CTAs cover the vector: the sums over the ranges read a place per thread."""
    seen = 0
    for m in VECTORS:
        for q in sorted({1, 2, 3, 7, 33, 100, 1000, 49_152 // m, 49_152 // m - 1, 30_000 // m, 9000 // m}):
            for d in (4 * q - 3, 4 * q):
                p = binding.core_debug_short_plan(m, d, sm_count=sm_count) if d > 0 else {"ctas": 0}
                if p["ctas"] == 0:
                    continue
                seen += 1
                assert p["alone_per"] * p["slices"] <= p["alone_threads"] <= 512, (m, d)
                assert p["alone_ctas"] * p["alone_per"] >= (d + 3) // 4 > (p["alone_ctas"] - 1) * p["alone_per"]
    assert seen > 500


@pytest.mark.parametrize("sm_count", [20, 148])
def test_no_lane_adds_up_a_long_chain(sm_count):
    """A message's rounding error grows with the square root of the longest chain of additions: at most 24 blocks per lane (16 where the lanes, a
    power of two, use all threads), fewer than the 32 steps in a tile of the kernel for longer rows."""
    seen = 0
    for m in VECTORS:
        for q in range(1, 49_152 // m + 1, max(1, 49_152 // m // 40)):
            p = binding.core_debug_short_plan(m, 4 * q, sm_count=sm_count)
            if p["ctas"]:
                seen += 1
                assert p["per"] <= 24 * p["lanes"], (m, q)
                assert p["lanes"] * m <= 512 or p["lanes"] == 1
    assert seen > 500
