"""Tables of 2^21 slots and more in the bitmap form, whose resolve walks shares of rank words."""
import numpy as np
import pytest

import paper_2310_19855_gb300 as gi
import workload as wl
from _gpu_time import update_us
from _gpu_util import dev, require_gpu
from paper_2310_19855_gb300.pipeline import BatchPipeline, Pipeline, view_of
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


@pytest.mark.parametrize("use_graph", [False, True])
def test_batched_large_and_small_tables_equal_single_views_past_the_aging(use_graph):
    # 20 frames: side-by-side accumulators added to, resolved, aged and ranked again in the batched kernels
    sizes, log2 = ((160, 96), (96, 64), (200, 120)), (21, 16, 21)
    data = []
    for cfg, seed in wl.batched_views(3, sizes=sizes):
        scene = wl.make_scene(cfg, seed)
        data.append([wl.make_frame(cfg, f, scene, seed_base=seed) for f in range(3)])
    gb = [[dev(fr.gbuffer) for fr in v] for v in data]
    rec = [[dev(fr.records) for fr in v] for v in data]
    bp = BatchPipeline([(w, h, n) for (w, h), n in zip(sizes, log2)], 64)
    singles = [Pipeline(w, h, 64, n) for (w, h), n in zip(sizes, log2)]
    try:
        for k in range(20):
            f = 0 if k < 17 else k % 3  # 17 frames of the same cells, then others
            views = [view_of(v[f].camera, k) for v in data]
            bp.frame([g[f] for g in gb], [r[f] for r in rec], views, use_graph=use_graph)
            for v, sp in enumerate(singles):
                sp.frame(gb[v][f], rec[v][f], views[v])
            if k in (0, 1, 9, 16, 19):
                torch.cuda.synchronize()
                for v, sp in enumerate(singles):
                    st = bp.views[v]
                    ea, eb = gi.gi_cache_export(st["cache"]), gi.gi_cache_export(sp.cache)
                    for name in ("identity", "sum", "count", "stamp", "value"):
                        assert np.array_equal(ea[name], eb[name]), (k, v, name)
                    assert gi.gi_diag_dense_cells(st["cache"]) == gi.gi_diag_dense_cells(sp.cache)
                    assert torch.equal(st["probes"].sh, sp.probes.sh) and torch.equal(st["irr"], sp.irr)
        assert gi.gi_diag_dense_cells(singles[0].cache) > 0 and gi.gi_diag_dense_cells(singles[1].cache) == 0
    finally:
        bp.close()
        for sp in singles:
            sp.close()


@pytest.mark.parametrize("f16", [0, 1])
def test_cold_marks_of_a_large_table_equal_a_small_one(f16):
    # the answered records are the hits on cells resolved without history: fresh cells, cells seen again,
    # evicted ones, and across a compaction of either table
    n = 20_000
    lo, hi = (-9.0,) * 3, (9.0,) * 3
    SI = wl.surrogate_inputs
    cfg = gi.make_nrc_config(lo, hi, log2_table=14, resolutions=SI.SMALL_RESOLUTIONS, batch=1024, train_steps=1,
                             lr=1e-30, trust=1e30, query_lod=4, max_records=n, max_queries=n)
    nrc = gi.gi_nrc_create(cfg)
    caches = [gi.gi_cache_create(log2, cell_size=0.05, evict_frames=2, rebuild_load=0.25, resolved_format=f16)
              for log2 in (21, 20)]
    try:
        gi.gi_nrc_set_params(nrc, *SI.params(3, 14))
        near = [dev(wl.records_random(n, k, extent=2.0)) for k in range(4)]
        fill = [dev(wl.records_random(300_000, 50 + k, extent=40.0)) for k in range(2)]
        cold = []
        for frame, k in enumerate((0, 1, 0, 2, 2, 0, 1, 3, 3, 0)):
            picked = []
            for h in caches:
                if frame in (3, 5):
                    _update(h, fill[frame == 5], frame)
                s = _update(h, near[k], frame)
                gi.gi_cache_resolve(h, frame)
                torch.cuda.synchronize()
                if frame == 0:
                    gi.gi_nrc_train_frame(nrc, h, gi.hits_from_planes(near[k], n), s, 0)  # trusted from now on
                gi.gi_nrc_query_frame(nrc, h, gi.hits_from_planes(near[k], n), s, _view(frame))
                m = gi.gi_nrc_answers(nrc)
                r = torch.empty(max(m, 1), dtype=torch.int32, device="cuda")
                rad = torch.empty((max(m, 1), 4), device="cuda")
                gi.gi_nrc_answers(nrc, r, rad, m)
                picked.append(torch.sort(r[:m])[0])
            assert torch.equal(*picked), (frame, [p.numel() for p in picked])
            cold.append(picked[0].numel())
        assert cold[0] > 0.9 * n and cold[2] < 0.1 * n and 0 < cold[1] and cold[4] < 0.1 * n  # seen, seen again
        assert cold[5] > 0.5 * n  # evicted
        assert all(gi.gi_cache_stats(h)["rebuilds"] >= 1 for h in caches)
    finally:
        for h in caches:
            gi.gi_cache_destroy(h)
        gi.gi_nrc_destroy(nrc)
