"""The diagnostics beside the passes."""
import pytest

import paper_2310_19855_gb300 as gi
from _gpu_time import us
from _gpu_util import require_gpu

pytestmark = pytest.mark.gpu

import torch  # noqa: E402


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def test_the_accumulation_alone_is_no_slower_than_the_update_it_is_part_of():
    n, log2 = 1_000_000, 20
    rec = torch.rand((13, n), device="cuda") * 6.0 - 3.0
    rec[9] = 1.0
    view = gi.make_view(0, 640, 360, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    slots = torch.empty(n, dtype=torch.int32, device="cuda")
    h = gi.gi_cache_create(log2, first_touch=gi.GI_FIRST_TOUCH_LIST)
    try:
        hits = gi.hits_from_planes(rec, n)
        gi.gi_cache_update(h, hits, view, slots)
        scratch = torch.zeros((8 << log2,), dtype=torch.int32, device="cuda")
        first = torch.zeros(1, dtype=torch.int32, device="cuda")
        alone = us(lambda: gi.gi_diag_update_atomics(slots, n, log2, scratch, first, gi.GI_FIRST_TOUCH_LIST))
        assert alone <= us(lambda: gi.gi_cache_update(h, hits, view, slots))
    finally:
        gi.gi_cache_destroy(h)
