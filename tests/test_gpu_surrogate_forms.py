"""The surrogate's kernels come in forms picked by the number of samples (levels per group of the far-hit
encoding, CTAs per tile of the inference); every form computes a sample's answer with the same operations,
so all must agree bit for bit."""
import numpy as np
import pytest

import paper_2310_19855_gb300 as gi
import workload as wl
from _gpu_util import dev, require_gpu, u32

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

SI = wl.surrogate_inputs


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _network(n, aabb=SI.CORNELL_AABB):
    cfg = gi.make_nrc_config(*aabb, log2_table=14, resolutions=SI.SMALL_RESOLUTIONS, batch=4096, train_steps=1,
                             lr=1e-30, trust=1e30, query_lod=0, max_records=n, max_queries=n)
    nrc = gi.gi_nrc_create(cfg)
    gi.gi_nrc_set_params(nrc, *SI.params(3, 14))
    return nrc


def _infer(nrc, P, N, n):
    out = torch.empty((n, 4), device="cuda")
    gi.gi_nrc_infer(nrc, gi.make_points(P, N, n), out)
    return out


@pytest.mark.parametrize("n", [1, 127, 128, 129, 5000, 80_001])
def test_inference_of_any_count_equals_tile_by_tile(n):
    nrc = _network(128)
    try:
        pos, nrm = SI.points(5, n)
        P, N = dev(pos), dev(nrm)
        whole = _infer(nrc, P, N, n)
        for a in sorted({0, (n // 2) // 128 * 128, (n - 1) // 128 * 128}):
            m = min(128, n - a)
            part = _infer(nrc, P[:, a:a + m].contiguous(), N[:, a:a + m].contiguous(), m)
            assert torch.equal(whole[a:a + m], part), a
    finally:
        gi.gi_nrc_destroy(nrc)


@pytest.mark.parametrize("n", [33, 9_999, 30_011, 70_001, 140_003, 260_001])
def test_answers_of_a_view_equal_the_inference_of_their_points(n):
    # from below two samples a warp up to groups of 16 levels
    rec = wl.records_random(n, 11, extent=0.9, cam=(0.0, 1.0, 0.0))
    view = gi.make_view(0, 640, 360, (0, 1, 3), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    R = dev(rec)
    hits = gi.hits_from_planes(R, n)
    cache = gi.gi_cache_create(18)
    nrc = _network(n)
    try:
        slots = torch.empty(n, dtype=torch.int32, device="cuda")
        gi.gi_cache_update(cache, hits, view, slots)
        gi.gi_cache_resolve(cache, 0)
        gi.gi_nrc_train_frame(nrc, cache, hits, slots, 0)  # a step too small to move a parameter: trusted
        gi.gi_nrc_query_frame(nrc, cache, hits, slots, view)
        m = gi.gi_nrc_answers(nrc)
        assert m == int(np.isfinite(rec[9]).sum())  # every hit is cold or of LOD >= 0
        records = torch.empty(m, dtype=torch.int32, device="cuda")
        rad = torch.empty((m, 4), device="cuda")
        gi.gi_nrc_answers(nrc, records, rad, m)
        at = torch.from_numpy(u32(records).astype(np.int64)).cuda()
        assert torch.equal(torch.sort(at)[0], torch.nonzero(torch.isfinite(R[9]))[:, 0])
        P, N = R[0:3, at].contiguous(), R[3:6, at].contiguous()
        assert torch.equal(rad, _infer(nrc, P, N, m))
    finally:
        gi.gi_nrc_destroy(nrc)
        gi.gi_cache_destroy(cache)


def test_answers_in_groups_of_16_levels_equal_the_inference_of_their_points():
    # 741,000 answers: their groups of 16 levels are four items a warp, no longer run than shorter groups'
    test_answers_of_a_view_equal_the_inference_of_their_points(780_003)


@pytest.mark.parametrize("log2", [13, 16])
def test_adam_steps_the_listed_entries_of_either_chunk(log2):
    # 64 entries a warp for small tables, 256 for others; a first step moves a touched entry by lr g / (|g| + eps)
    # (float32: half an ulp of |p| < 1, and 2^-20 of the step), the others not at all
    lr, eps, T = 1e-2, 1e-15, 1 << log2
    rng = np.random.default_rng(7)
    table, w1, w2, w3 = SI.params(3, log2)
    grad = np.zeros(table.shape, np.float32)
    hit = rng.random((16, T)) < 0.1
    hit[3] = True
    hit[5], hit[6] = False, np.arange(T) % 64 == 63
    grad[hit] = rng.normal(size=(int(hit.sum()), 2)).astype(np.float32)
    cfg = gi.make_nrc_config(*SI.CORNELL_AABB, log2_table=log2, resolutions=SI.SMALL_RESOLUTIONS, lr=lr, adam_eps=eps,
                             max_records=128, max_queries=128)
    nrc = gi.gi_nrc_create(cfg)
    try:
        gi.gi_nrc_set_params(nrc, table, w1, w2, w3)
        gi.gi_nrc_set_gradients(nrc, grad, np.zeros_like(w1), np.zeros_like(w2), np.zeros_like(w3))
        gi.gi_nrc_adam(nrc)
        got = gi.gi_nrc_get_params(nrc, log2)[0]
        g = grad.astype(np.float64)
        want = table - lr * g / (np.abs(g) + eps)
        assert np.array_equal(got[~hit], table[~hit])
        assert np.abs(got - want).max() < 2.0 ** -24 * np.abs(want).max() + 2.0 ** -20 * lr
        assert not np.any(gi.gi_nrc_get_gradients(nrc, log2)[0])
    finally:
        gi.gi_nrc_destroy(nrc)
