"""The least-squares pass rounds its copies out to 16 bytes; nothing beyond the data matrices may be touched by that, however
short the rows are and however many CTAs they are cut over (host arithmetic only: the kernel's own index functions)."""
import pytest

from paper_2309_13307_b200 import binding


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 7, 54])
def test_short_rows_stay_inside_for_every_number_of_rows(d):
    for rows in range(1, 1500):
        for misaligned in (0, 4, 8, 12):
            units, before, behind = binding.core_debug_ls_reads(1, rows, d, False, misaligned)
            assert units == min(rows, 148) and (before, behind) == (0, 0), (rows, misaligned)


@pytest.mark.parametrize("n,rows,d", [(3, 7, 1), (50, 3, 1), (7, 33, 2), (147, 1, 3), (64, 16, 65), (2, 999, 257), (9, 120, 784),
                                      (3, 151, 2049), (3, 60, 5500), (5, 7, 12001), (2, 75, 16384)])
def test_rows_of_several_machines_stay_inside(n, rows, d):
    for apart in (False, True):
        for sm_count in (148, 132, 3):
            for misaligned in (0, 4, 8, 12):
                units, before, behind = binding.core_debug_ls_reads(n, rows, d, apart, misaligned, sm_count)
                assert units > 0 and (before, behind) == (0, 0), (apart, sm_count, misaligned)


def test_long_rows_of_one_cta_have_room_for_two_slots():
    """Every length up to 16384 takes the single pass (no unit would mean two passes over A)."""
    for d in [*range(8193, 16384, 61), 13824, 13825, *range(14050, 14090), 14336, 16384]:
        for apart in (False, True):
            assert binding.core_debug_ls_reads(3, 60, d, apart, 4)[0] > 0, d
