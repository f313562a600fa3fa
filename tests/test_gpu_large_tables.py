"""Tables of 2^21 slots and more in the bitmap form, whose resolve walks shares of rank words."""
import numpy as np
import pytest

import paper_2310_19855_gb300 as gi
import workload as wl
from _gpu_time import update_us
from _gpu_util import dev, require_gpu
from test_gpu_dense import _same
from test_gpu_shared_cells import gather

pytestmark = pytest.mark.gpu

import torch  # noqa: E402


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _view(frame):
    return gi.make_view(frame, 640, 360, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)


def _update(h, rec, frame, slots=None):
    n = rec.shape[1]
    s = torch.empty(n, dtype=torch.int32, device="cuda") if slots is None else slots
    gi.gi_cache_update(h, gi.hits_from_planes(rec, n), _view(frame), s)
    return s


def _pair(log2, **kw):
    return [gi.gi_cache_create(log2, first_touch=ft, cell_size=0.05, **kw)
            for ft in (gi.GI_FIRST_TOUCH_AUTO, gi.GI_FIRST_TOUCH_LIST)]


@pytest.mark.parametrize("f16", [0, 1])
def test_shares_with_more_touched_slots_than_a_block_lists(f16):
    # 2.4 million cells in 2^22 slots: more than 2048 in every block's share of the rank words
    caches = _pair(22, resolved_format=f16)
    try:
        rec = [dev(wl.records_random(1_300_000, k, extent=40.0)) for k in (1, 2)]
        for frame in range(2):
            for h in caches:
                for r in rec:
                    _update(h, r, frame)
            torch.cuda.synchronize()
            assert gi.gi_cache_stats(caches[0])["touched"] > 2048 * 1024
            if frame:
                _same(*caches)
            for h in caches:
                gi.gi_cache_resolve(h, frame)
            torch.cuda.synchronize()
        _same(*caches)
    finally:
        for h in caches:
            gi.gi_cache_destroy(h)


@pytest.mark.parametrize("log2", [24, 25])
def test_several_shares_per_block_answer_like_the_list_form(log2):
    n = 400_000
    caches = _pair(log2, evict_frames=3)
    try:
        recs = [wl.records_random(n, k, extent=8.0) for k in range(4)]
        for frame in range(6):
            for h in caches:
                for k in (0, 1 + frame % 3):  # some cells in every frame, others in every third
                    _update(h, dev(recs[k]), frame)
                gi.gi_cache_resolve(h, frame)
            torch.cuda.synchronize()
            stats = [gi.gi_cache_stats(h) for h in caches]
            assert all(stats[0][k] == stats[1][k] for k in ("occupied", "live", "touched", "dropped"))
            for k in range(4):
                out = [torch.empty((n, 4), device="cuda") for _ in caches]
                for h, o in zip(caches, out):
                    gi.gi_cache_query(h, o, n, points=gi.hits_from_planes(dev(recs[k]), n), view=_view(frame))
                assert torch.equal(*out)
    finally:
        for h in caches:
            gi.gi_cache_destroy(h)


def test_few_records_in_a_large_table_cost_no_multiple():
    # 65,536 records: 14 us over 2^20 slots, 22 us over 2^24; a counter addition per 512 slots took 37 us there
    rec = wl.records_random(65_536, 5, extent=3.0)
    assert update_us(dict(log2_slots=24), rec) < 2.2 * update_us(dict(log2_slots=20), rec)


def test_few_cells_of_a_large_table_do_not_share_a_line():
    # eight cells, a million records: with their accumulators in one 256-byte run 526 us, now 92 (over 2^20 slots 110)
    rec = gather(1_000_000, 8, 3)
    assert update_us(dict(log2_slots=22), rec) < 2.5 * update_us(dict(log2_slots=20), rec)


def test_a_captured_resolve_ages():
    # cells of set B, touched before the replays only, must lose their side-by-side accumulators
    a, b = dev(wl.records_random(20_011, 1, extent=3.0)), dev(wl.records_random(50_021, 2, extent=9.0))
    h = gi.gi_cache_create(21, cell_size=0.05, evict_frames=1 << 20)
    try:
        st = torch.cuda.Stream()
        s = torch.empty(20_011, dtype=torch.int32, device="cuda")
        n = a.shape[1]
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            _update(h, a, 0)
            gi.gi_cache_resolve(h, 0)
            torch.cuda.synchronize()
            only_a = gi.gi_diag_dense_cells(h)
            assert 0 < only_a <= n
            _update(h, b, 0)
            gi.gi_cache_resolve(h, 0)
        torch.cuda.synchronize()
        assert gi.gi_diag_dense_cells(h) > 2 * only_a
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st, capture_error_mode="relaxed"):
            gi.gi_cache_update(h, gi.hits_from_planes(a, n), _view(0), s, stream=st)
            gi.gi_cache_resolve(h, 0, stream=st)
        for _ in range(16):
            graph.replay()
        torch.cuda.synchronize()
        assert gi.gi_diag_dense_cells(h) == only_a
        got = gi.gi_cache_export(h)
        assert np.all(got["count"] == 0)
    finally:
        gi.gi_cache_destroy(h)
