"""Launch geometry of the kernels for short vectors (host logic only)."""
import pytest

from paper_2309_13307_b200 import binding


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


# machines, d, m, dtype, offset (elements beyond 16 bytes), padding of the rows, CTAs of the one launch (0: separate kernels)
ROUTES = [
    (1, 1, 1, "f32", 0, 0, 1), (1, 3, 4096, "bf16", 1, 0, 1), (1, 2, 4097, "f32", 0, 0, 0), (1, 100, 7, "f32", 1, 0, 1), (1, 250, 7, "bf16", 0, 0, 2),
    (1, 300, 7, "f32", 0, 1, 4), (1, 36, 300, "f32", 3, 0, 8), (1, 700, 9, "bf16", 3, 0, 8), (1, 999, 48, "f32", 1, 0, 8),
    # most counters for one machine, most blocks of a CTA, and beyond
    (1, 12_288, 16, "f32", 0, 0, 8), (1, 12_289, 16, "bf16", 0, 0, 0), (1, 12_285, 16, "bf16", 5, 0, 8), (1, 81_920, 1, "f32", 0, 0, 8), (1, 81_921, 1, "f32", 0, 0, 0),
    (1, 81_917, 2, "f32", 2, 0, 8), (1, 81_921, 2, "bf16", 0, 0, 0), (1, 33_001, 5, "f32", 0, 0, 8), (1, 65_534, 3, "bf16", 0, 0, 8),
    # shared memory
    (1, 128, 1489, "f32", 0, 0, 0), (1, 120, 1400, "f32", 1, 0, 8), (1, 17, 4096, "bf16", 0, 0, 0), (1, 4, 4096, "f32", 0, 0, 1),
    # several machines: every number of them, clusters of every size
    (2, 129, 30, "f32", 0, 0, 2), (2, 7000, 2, "bf16", 1, 3, 8), (2, 1000, 1, "f32", 0, 0, 1), (3, 260, 9, "f32", 1, 2, 4), (3, 999, 20, "bf16", 0, 0, 8),
    (3, 16_384, 6, "f32", 0, 0, 8), (4, 130, 16, "bf16", 0, 2, 2), (4, 4096, 16, "f32", 0, 0, 8), (4, 520, 12, "f32", 3, 0, 8),
    (5, 129, 12, "bf16", 1, 0, 2), (5, 1001, 7, "f32", 2, 1, 8), (6, 257, 9, "f32", 0, 0, 4), (6, 2003, 9, "bf16", 3, 0, 8), (7, 140, 7, "f32", 1, 0, 1),
    (7, 1203, 11, "bf16", 0, 0, 8), (8, 64, 8, "bf16", 0, 0, 1), (8, 700, 3, "f32", 1, 0, 4), (8, 1500, 20, "bf16", 0, 0, 8),
    # most counters for two to four machines, and for more
    (2, 12_288, 8, "bf16", 0, 0, 8), (2, 12_289, 8, "bf16", 0, 0, 0), (4, 12_288, 8, "f32", 0, 0, 8), (4, 12_289, 8, "f32", 0, 0, 0),
    (8, 4096, 8, "f32", 0, 0, 8), (8, 4097, 8, "f32", 0, 0, 0), (5, 4093, 8, "f32", 1, 0, 8), (9, 300, 7, "f32", 0, 0, 0),
    # few columns for many vectors; large tiles, many blocks of all machines, many sums
    (4, 54, 256, "f32", 0, 0, 0), (3, 219, 200, "f32", 1, 0, 0), (2, 555, 40, "bf16", 0, 0, 0), (5, 141, 100, "bf16", 0, 0, 0), (2, 44_234, 1, "bf16", 1, 0, 0),
    (8, 32_111, 1, "bf16", 0, 0, 0), (8, 16_054, 2, "f32", 0, 0, 0), (4, 2599, 37, "bf16", 0, 0, 0), (4, 400, 34, "f32", 0, 0, 0), (2, 18, 2000, "f32", 1, 0, 0),
]
# rows added up, d, m, CTAs
ROW_ROUTES = [(2, 5, 3, 1), (148, 300, 5, 2), (164, 3500, 8, 8), (165, 3500, 8, 0), (8, 16_000, 8, 8), (9, 16_000, 8, 0), (26, 18_174, 2, 0), (148, 2561, 65, 0),
              (80, 2500, 64, 8), (2, 12_289, 16, 0), (500, 54, 16, 1), (2000, 54, 16, 0)]


@pytest.mark.parametrize("n,d,m,dtype,offset,pad,ctas", ROUTES)
def test_routes_of_rounds(n, d, m, dtype, offset, pad, ctas):
    assert binding.core_debug_short_plan(m, d, machines=n)["ctas"] == ctas


@pytest.mark.parametrize("rows,d,m,ctas", ROW_ROUTES)
def test_routes_of_sums_of_rows(rows, d, m, ctas):
    assert binding.core_debug_short_plan(m, d, rows=rows)["ctas"] == ctas


def test_what_a_round_takes_its_reconstruction_takes_too():
    """A round gives the bits of its parts, so wherever it is one launch the reconstruction alone is the kernel with the same sums."""
    for n in range(1, 9):
        for m in VECTORS:
            for d in (1, 60, 333, 1000, 4096, 16_384, 44_234, 81_920, 98_304):
                p = binding.core_debug_short_plan(m, d, machines=n)
                assert p["ctas"] == 0 or p["alone_ctas"] > 0, (n, m, d)


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
