"""A pass may be scheduled while the one before it still runs; it must still see everything that pass
wrote.  Frames enqueued back to back equal frames with a synchronisation after each pass, bit for bit,
and a captured frame equals an enqueued one."""
import numpy as np
import pytest

import paper_2310_19855_gb300 as gi
import paper_2310_19855_gb300.pipeline as pl
import workload as wl
from _gpu_util import dev, require_gpu

pytestmark = pytest.mark.gpu

import torch  # noqa: E402

CFG = dict(wl.CONFIGS[2], width=152, height=88, n_boxes=256, room=(24.0, 8.0, 24.0), frames=8)
SEED = wl.scene.SEED_BASE + 9100


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _frames(upscale):
    scene = wl.make_scene(CFG, SEED)
    out = []
    for f in range(4):
        fr = wl.make_frame(CFG, f, scene, seed_base=SEED, upscale=upscale, motion=True)
        out.append((fr, dev(fr.gbuffer), dev(fr.records), dev(fr.motion), pl.view_of(fr.camera, f)))
    return out


def _waits(monkeypatch):
    for name in [n for n in vars(pl) if n.startswith(("gi_cache_", "gi_probes_")) and callable(getattr(pl, n))]:
        def call(*a, _f=getattr(pl, name), **k):
            r = _f(*a, **k)
            torch.cuda.synchronize()
            return r
        monkeypatch.setattr(pl, name, call)


@pytest.mark.parametrize("log2,kw", [(16, {}), (22, {}), (16, dict(merge=1)), (14, dict(tiles=True))])
def test_passes_enqueued_together_equal_passes_one_at_a_time(monkeypatch, log2, kw):
    frames = _frames(2)
    got = []
    for wait in (False, True):
        if wait:
            _waits(monkeypatch)
        p = pl.TemporalPipeline(CFG["width"], CFG["height"], frames[0][0].rays_per_probe, log2, upscale=2,
                                filtered=True, **kw)
        try:
            torch.cuda.synchronize()
            for _, g, r, m, v in frames:
                p.frame(g, r, m, v)
            torch.cuda.synchronize()
            ex = gi.gi_cache_export(p.cache)
            got.append((p.irr.cpu().numpy(), p.atlas.cpu().numpy(), np.sort(ex["identity"]),
                        ex["value"][np.argsort(ex["identity"], kind="stable")]))
        finally:
            p.close()
    for a, b in zip(*got):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))


@pytest.mark.parametrize("log2", [16, 22])
def test_captured_frame_equals_enqueued(log2):
    frames = _frames(1)
    got = []
    for captured in (False, True):
        p = pl.Pipeline(CFG["width"], CFG["height"], frames[0][0].rays_per_probe, log2)
        try:
            _, g, r, _, v = frames[0]
            s = torch.cuda.Stream()
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                p.frame(g, r, v, stream=s)
            torch.cuda.synchronize()
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
                    p.frame(g, r, v, stream=s)
                for _ in range(3):
                    graph.replay()
            else:
                with torch.cuda.stream(s):
                    for _ in range(3):
                        p.frame(g, r, v, stream=s)
            torch.cuda.synchronize()
            got.append(p.irr.cpu().numpy())
        finally:
            p.close()
    assert np.array_equal(got[0].view(np.uint8), got[1].view(np.uint8))
