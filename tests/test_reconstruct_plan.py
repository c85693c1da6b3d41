"""Which reconstruction kernel a shape takes (host logic only)."""
import pytest

from paper_2309_13307_b200 import binding


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


@pytest.mark.parametrize("sm_count", [148, 132])
def test_long_vectors_never_take_the_kernel_for_short_ones(sm_count):
    """Eight steps of 512 blocks per SM and more: the one for short vectors has a CTA for every 256 blocks, with start-up, table and
    message each."""
    long = 8 * sm_count * 512 * 4
    for d in (long, long + 1, 3_000_000, 4_000_000, 16_000_000, 100_000_000, 1_000_000_000):
        for m in (*range(1, 65), 100, 512, 513, 2048, 2049, 8192, 8193, 100_000):
            kernel, joins = binding.core_debug_reconstruct_plan(d, m, sm_count)
            assert kernel == ("wide" if m <= 3 or m > 8192 else kernel) and kernel != "short", (d, m)
            assert not joins, "thousands of CTAs would each form the whole message"


def test_messages_are_joined_only_by_the_kernel_that_can():
    seen = set()
    for m in (1, 2, 3, 4, 6, 8, 16, 64, 256, 512, 513, 1024, 8192, 8193):
        for d in (1, 100, 4096, 20_000, 94_719, 94_721, 300_000, 1_000_000, 2_400_000, 3_000_000, 30_000_000):
            kernel, joins = binding.core_debug_reconstruct_plan(d, m)
            assert kernel == "short" or not joins
            seen.add((kernel, joins))
    assert seen == {("short", False), ("short", True), ("wide", False), ("turn", False)}
