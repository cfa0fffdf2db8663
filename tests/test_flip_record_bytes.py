"""The flip record of a round too large for the record of levels takes at most
8 GiB, whatever the row length (rows are padded to whole 32-bit words, so
that short and ragged ones take more than a bit a sample): the memory that a
job is said to need is bounded by it.  Host arithmetic, no GPU."""
import pytest

import paper_0812_2964_gb300 as mc

GIB = 2 ** 30


def _words(L, p, S):
    return p * (-(-S * L * ((L + 31) // 32) // 32) * 32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    mc.build()


# (the last sizes are below the limit, which they keep)
@pytest.mark.parametrize("L,p,S", [(4, 4096, 1_000_000), (8, 4096, 200_000), (12, 4096, 110_000), (36, 4096, 12_000),
                                   (100, 2048, 3_300), (32, 16384, 4_096), (128, 1024, 4_096), (8, 4096, 65_536)])
def test_record_is_at_most_8_gib(L, p, S):
    assert 2 ** 33 < p * S * L * L <= 2 ** 36
    record = 4 * _words(L, p, S)
    held = mc.mc_job_device_bytes(L, p, S)
    rest = mc.mc_job_device_bytes(L, p, 1) + 4 * GIB      # the job, and its checkpoints' limit
    assert held <= rest + 8 * GIB
    assert (held >= record) == (record <= 8 * GIB)
