"""How a host round is cut into slabs (host arithmetic only): every coordinate once, starts where the kernels accept them, and
output slabs that leave no wave of the reconstruction's CTAs half empty."""
import pytest

from paper_2309_13307_b200 import binding

GROUP = 2048                    # coordinates of a CTA's step in the reconstruction for long vectors


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2309_13307_b200 import build
    build.build()


@pytest.mark.parametrize("d", [1, 3, 4096, 4097, 100_000, 262_145, 1_000_003, 2_424_832, 4_000_000, 8_183_808, 25_557_032, 124_439_808,
                               1_000_000_000])
@pytest.mark.parametrize("n,dtype", [(1, binding.CORE_F32), (2, binding.CORE_F32), (16, binding.CORE_BF16), (64, binding.CORE_F32)])
def test_slabs_cover_the_vector(d, n, dtype):
    for output, most in ((False, (64 << 20) // (n * (2 if dtype == binding.CORE_BF16 else 4))), (True, (16 << 20) // 4)):
        for sm_count in (148, 132, 1):
            slabs = binding.core_debug_host_slabs(d, n, dtype, output, sm_count)
            assert sum(slabs) == d and min(slabs) > 0 and max(slabs) <= max(most, 4096)
            starts = [sum(slabs[:i]) for i in range(len(slabs))]
            assert all(s % GROUP == 0 for s in starts), "launch_reconstruct takes starts on whole steps of a CTA"


@pytest.mark.parametrize("d", [30_000_000, 124_439_808, 1_000_000_000])
@pytest.mark.parametrize("sm_count", [148, 132])
def test_long_output_slabs_are_whole_waves(d, sm_count):
    wave = 3 * sm_count * GROUP
    slabs = binding.core_debug_host_slabs(d, output=True, sm_count=sm_count)
    long = [s for s in slabs if s >= 8 * sm_count * GROUP]           # those the kernel for long vectors takes
    assert all(s % wave == 0 for s in long)
    assert sum(long) >= 0.7 * d and len(slabs) <= 16 + d // (4 * wave)
