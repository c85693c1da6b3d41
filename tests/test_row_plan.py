"""Launch geometry of the kernel that projects one row or the sum of several (host logic only): every plan fits a CTA's shared
memory and covers all vectors and coordinates, and the workspace has room for its partial sums."""
import pytest

from paper_2309_13307_b200 import binding


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


def check_plan(p, m, d):
    assert p["smem"] <= 227 * 1024
    assert p["smem"] >= 64 * p["tile_q"] and p["smem"] >= 16 * p["tj"] * p["tq"]     # two tiles; the final reduction
    assert 1 <= p["tj"] * p["tq"] <= p["compute"] and p["tile_q"] % p["tq"] == 0
    assert p["grid_y"] * p["tj"] * 4 >= m
    assert p["tiles"] * 4 * p["tile_q"] >= d > (p["tiles"] - 1) * 4 * p["tile_q"]
    assert 1 <= p["grid_x"] <= min(p["tiles"], p["columns"])


LENGTHS = sorted({int(1e9 ** (i / 150)) for i in range(1, 151)} | {1_130_000, 2_324_170, 25_557_032, 124_439_808, 1_000_000_000})


@pytest.mark.parametrize("sm_count", [148, 132, 1])
def test_every_plan_fits(sm_count):
    turns = 0
    for m in [*range(1, 131), 170, 191, 256, 400, 511, 512, 513, 1000, 1024, 1030, 2048, 3073, 4096, 4200, 8192, 100_000]:
        for d in LENGTHS:
            for rows, misaligned in ((1, 0), (1, 4), (2, 0), (5, 4)):
                p = binding.core_debug_row_plan(m, d, rows=rows, misaligned=misaligned, sm_count=sm_count)
                check_plan(p, m, d)
                turns += p["turn"]
    assert turns > 1000


@pytest.mark.parametrize("rows", [55, 56, 148, 2368])
@pytest.mark.parametrize("dtype", [binding.CORE_F32, binding.CORE_BF16])
def test_many_rows_have_room_for_their_ranges(rows, dtype):
    """From twice as many rows as warps on, the first tile is added up from ranges of the rows, at most a segment of 64 blocks
    per warp, beside the first tile."""
    for m in (1, 16, 64, 165, 459, 700, 1024, 4096, 20_000):
        for d in LENGTHS[::3]:
            for ldg in ((d + 7) // 8 * 8, d + 1):
                p = binding.core_debug_row_plan(m, d, rows=rows, ldg=ldg, dtype=dtype)
                check_plan(p, m, d)
                warps, table = (28, 65_536 + 12_288) if p["turn"] else (10, 0)
                assert p["smem"] >= table + 32 * p["tile_q"] + warps * 64 * 16


@pytest.mark.parametrize("dtype,size", [(binding.CORE_F32, 4), (binding.CORE_BF16, 2)])
def test_a_single_row_has_one_plan_wherever_it_starts(dtype, size):
    """Plan and kernel decide the order of the sums: for one row they follow from its length and the number of vectors alone."""
    for m in [*range(1, 40), 64, 100, 1024]:
        for d in (4097, 262_144, 2_097_152, 2_097_155, 25_557_032):
            plans = [binding.core_debug_row_plan(m, d, ldg=d + pad, dtype=dtype, misaligned=off)
                     for pad in (0, 1, 2, 8) for off in range(0, 16, size)]
            assert all(p == plans[0] for p in plans), (m, d)


def test_short_rows_of_many_vectors_keep_the_polynomials():
    """More than 512 vectors take the table of angles from 3 * 2^24 Gaussians on, fewer from 2^24."""
    for m, least in ((512, 1 << 24), (513, 3 << 24), (768, 3 << 24), (1024, 3 << 24), (4096, 3 << 24), (16_384, 3 << 24)):
        for rows in (1, 2):
            assert not binding.core_debug_row_plan(m, least // m - 1, rows=rows)["turn"]
            assert binding.core_debug_row_plan(m, (least // m + 3) // 4 * 4, rows=rows)["turn"]


@pytest.mark.parametrize("dtype,size", [(binding.CORE_F32, 4), (binding.CORE_BF16, 2)])
def test_many_rows_with_the_table_have_short_tiles(dtype, size):
    """Beyond half a byte to stage per vector: 32 steps per tile and generating thread, and room for the columns there too."""
    for m in (100, 200, 357, 1000):
        for d in (262_144, 1_000_000, 4_000_000, 20_000_000):
            for rows in (m // (2 * size), m // (2 * size) + 1, m // 3 - 1):
                plan = binding.core_debug_row_plan(m, d, rows=rows, dtype=dtype)
                if plan["turn"]:
                    heavy = 2 * size * rows > m
                    assert plan["tile_q"] <= (32 if heavy else 128) * plan["tq"], (m, d, rows)
                    assert plan["grid_x"] <= plan["columns"] and plan["tiles"] * plan["tile_q"] * 4 >= d
