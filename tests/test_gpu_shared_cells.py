"""Records of a warp that share cells: the tile cache and GI_MERGE_WARP merge them where a warp holds at
most half as many cells as hits.  Merged or not, every form must give the same cells, sums and counts,
and many records in few cells must not cost a multiple of the same records spread out."""
import numpy as np
import pytest

import paper_2310_19855_gb300 as gi
import workload as wl
from _gpu_time import update_us
from _gpu_util import dev, require_gpu, u32

pytestmark = pytest.mark.gpu

import torch  # noqa: E402


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _view():
    return gi.make_view(0, 640, 360, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)


def gather(n, cells, seed):
    """n records at `cells` places (record i at place i mod cells), misses among them."""
    rec = wl.records_random(n, seed, extent=20.0)
    at = np.arange(n) % cells
    rec[0:6] = rec[0:6, at]
    rec[10:13] = rec[10:13, at]
    rec[9] = np.where(np.isfinite(rec[9]), np.float32(1.0), rec[9])
    return rec


def _cells(kw, rec):
    n = rec.shape[1]
    h = gi.gi_cache_create(**kw)
    try:
        r, s = dev(rec), torch.empty(n, dtype=torch.int32, device="cuda")
        gi.gi_cache_update(h, gi.hits_from_planes(r, n), _view(), s)
        torch.cuda.synchronize()
        st = gi.gi_cache_stats(h)
        ids = u32(s)
        hit = np.isfinite(rec[9])
        assert np.all(ids[~hit] == gi.GI_SLOT_MISS) and np.all(ids[hit] < gi.GI_SLOT_FAR)
        ex = gi.gi_cache_export(h)
        assert st["dropped"] == 0 and int(ex["count"].sum()) == int(hit.sum())
        return {k: ex[k] for k in ("identity", "sum", "count")}, st["clamped"]
    finally:
        gi.gi_cache_destroy(h)


FORMS = [dict(log2_slots=14, merge=1), dict(log2_slots=14, merge=1, first_touch=1), dict(log2_slots=21, merge=1),
         dict(log2_slots=14, tiles=True)]


@pytest.mark.parametrize("kw", FORMS, ids=["bitmap", "list", "large", "tiles"])
@pytest.mark.parametrize("cells", [1, 2, 8, 15, 16, 17, 31, 700])
def test_shared_cells_get_the_sums_of_their_records(kw, cells):
    # 9,999 records (a ragged last warp): by place in turn, and shuffled, with one clamped radiance
    rec = gather(9_999, cells, 31)
    rec[6, 5] = np.float32(1e9)
    plain = dict(kw, merge=0)
    want = _cells(plain, rec)
    mixed = rec[:, np.random.default_rng(1).permutation(rec.shape[1])]
    for got in (_cells(kw, rec), _cells(kw, np.ascontiguousarray(mixed))):
        for k in want[0]:
            assert np.array_equal(want[0][k], got[0][k]), k
        assert want[1] == got[1]


def test_one_tile_cell_costs_no_multiple_of_many():
    # a million additions to one address, one after the other, take a millisecond; merged by warps 54 us,
    # in a thousand cells 41
    n = 1_000_000
    assert update_us(dict(log2_slots=16, tiles=True), gather(n, 1, 3)) < 6 * update_us(
        dict(log2_slots=16, tiles=True), gather(n, 1_009, 3))
