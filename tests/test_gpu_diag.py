"""The diagnostics beside the passes."""
import pytest

import paper_2310_19855_gb300 as gi
from _gpu_time import us
from _gpu_util import dev, require_gpu
from test_gpu_shared_cells import gather

pytestmark = pytest.mark.gpu

import torch  # noqa: E402


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def test_the_accumulation_alone_takes_no_longer_than_the_update_it_is_part_of():
    # a million records in 32 cells, where the additions are nearly all of the update
    n, log2 = 1_000_000, 20
    rec = dev(gather(n, 32, 3))
    view = gi.make_view(0, 640, 360, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    slots = torch.empty(n, dtype=torch.int32, device="cuda")
    h = gi.gi_cache_create(log2, first_touch=gi.GI_FIRST_TOUCH_LIST)
    try:
        hits = gi.hits_from_planes(rec, n)
        gi.gi_cache_update(h, hits, view, slots)
        scratch = torch.zeros((8 << log2,), dtype=torch.int32, device="cuda")
        first = torch.zeros(1, dtype=torch.int32, device="cuda")
        alone = us(lambda: gi.gi_diag_update_atomics(slots, n, log2, scratch, first, gi.GI_FIRST_TOUCH_LIST))
        update = us(lambda: gi.gi_cache_update(h, hits, view, slots))
        assert alone < 1.25 * update, (alone, update)
    finally:
        gi.gi_cache_destroy(h)
