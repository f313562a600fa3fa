"""Probe passes at the edges of their range."""
import numpy as np
import pytest

import paper_2310_19855_gb300 as gi
from _gpu_time import us
from _gpu_util import require_gpu
from paper_2310_19855_gb300.pipeline import ProbeBuffers

pytestmark = pytest.mark.gpu

import torch  # noqa: E402


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def test_the_last_tile_of_the_largest_image_searches_above_level_0():
    # the empty mask word (all ones) equals the pixel of tile (8191, 8191), which a 65,535-pixel image has
    n = 65_535
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 165 << 30:
        pytest.skip("needs 165 GB of device memory")
    view = gi.make_view(0, n, n, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    pb = ProbeBuffers(n, n)
    lay = pb.layout
    assert (lay.tiles_x, lay.tiles_y) == (8192, 8192)
    pb.mask.fill_(-1)
    pb.nrm.zero_()
    pb.sh.zero_()
    x = y = 65_523  # a probe in tile (8190, 8190), found from (8191, 8191) at level 1
    word = int(np.array((y << 16) | x, np.uint32).view(np.int32))
    pb.mask[8190 * 8192 + 8190] = word
    pb.mask[lay.mip_offset[1] + 4095 * lay.mip_w[1] + 4095] = word
    p = 8190 * 8192 + 8190
    pb.pos[p] = torch.tensor((0.0, 0.0, -2.0, 2.0), device="cuda")
    pb.nrm[p] = torch.tensor((0.0, 0.0, 1.0, 1.0), device="cuda")
    pb.sh[p, 0:3] = 1.0
    gbuf = torch.empty((n, n, 4), device="cuda")
    gbuf[..., 3] = -1.0
    gbuf[-3:, -3:] = torch.tensor((0.0, 0.0, 1.0, 2.0), device="cuda")
    out = torch.empty((n, n, 4), device="cuda")
    gi.gi_probes_interpolate(gi.make_gbuffer(gbuf, n, n), view, pb.struct, out)
    torch.cuda.synchronize()
    flag = out[-4:, -4:, 3].cpu().numpy()
    del gbuf, out, pb
    torch.cuda.empty_cache()
    assert np.all(np.isin(flag[1:, 1:], (gi.GI_INTERP_OK, gi.GI_INTERP_RELAXED))), flag
    assert flag[0, 0] == gi.GI_INTERP_SKY


def test_filter_of_a_view_without_probes_only_copies():
    # 10 us for a 1080p view of sky, 28 us with probes; searching for the absent probes' neighbours took 22 us
    w, h = 1920, 1080
    view = gi.make_view(0, w, h, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    took = []
    for dist in (float("inf"), 2.0):
        gbuf = torch.tensor((0.0, 0.0, 1.0, dist), device="cuda").repeat(h, w, 1)
        pb = ProbeBuffers(w, h)
        gi.gi_probes_spawn(gi.make_gbuffer(gbuf, w, h), view, pb.struct)
        a = torch.rand((pb.layout.num_probes, 64, 4), device="cuda")
        b = torch.empty_like(a)
        took.append(us(lambda: gi.gi_probes_filter(pb.struct, view, a, b, 0)))
        if dist > 2.0:
            assert torch.equal(a, b)
    assert took[0] < 0.6 * took[1], took


def test_more_rays_per_probe_cost_in_proportion():
    # 641 x 359 pixels: 6.1 us with 64 rays per probe, 10.9 us with 128; 18.3 us where the gathers did not fly together
    w, h = 641, 359
    view = gi.make_view(0, w, h, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    gbuf = torch.tensor((0.0, 0.0, 1.0, 2.0), device="cuda").repeat(h, w, 1)
    pb = ProbeBuffers(w, h)
    gi.gi_probes_spawn(gi.make_gbuffer(gbuf, w, h), view, pb.struct)
    n = pb.layout.num_probes * 128
    rec = torch.rand((13, n), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda") * 6.0 - 3.0
    rec[9] = 1.0
    slots = torch.empty(n, dtype=torch.int32, device="cuda")
    c = gi.gi_cache_create(20)
    try:
        gi.gi_cache_update(c, gi.hits_from_planes(rec, n), view, slots)
        gi.gi_cache_resolve(c, 0)
        t = [us(lambda: gi.gi_probes_integrate(c, pb.struct, slots, rpp), k=20) for rpp in (64, 128)]
        assert t[1] < 2.3 * t[0], t
    finally:
        gi.gi_cache_destroy(c)
