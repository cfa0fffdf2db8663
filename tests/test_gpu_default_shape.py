"""Where a job's chains go one a warp by default: on both sides of the lines
up to which that is the faster form for young weights too (on the 152 SMs they
were measured on)."""
import pytest

import paper_0812_2964_gb300 as mc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,per_scheduler", [(8, 6), (12, 5), (16, 7), (20, 6), (24, 8), (28, 7), (32, 8), (40, 16),
                                             (48, 8), (64, 10), (96, 10), (100, 16), (128, 8)])
def test_line_between_the_forms(L, per_scheduler):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for p, one in ((4 * sms * per_scheduler, True), (4 * sms * per_scheduler + 1, False)):
        g = mc.Job(L, p, 1, 1)
        info = g.info()
        g.close()
        assert ((info["placement"], info["chains_per_warp"]) == (1, 1)) == one, (L, p, info)
