"""Event-timed calls for the tests that compare what two inputs cost (never absolute times)."""
import torch

import paper_2310_19855_gb300 as gi
from _gpu_util import dev


def us(fn, k=10, reps=5):
    """Shortest mean time of k calls, in microseconds."""
    for _ in range(3):
        fn()
    best = float("inf")
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(k):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / k * 1e3)
    return best


def update_us(kw, rec):
    """An update with these records and a resolve, on a cache created with kw."""
    n = rec.shape[1]
    h = gi.gi_cache_create(**kw)
    view = gi.make_view(0, 640, 360, (0, 0, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), 1.0)
    try:
        hits = gi.hits_from_planes(dev(rec), n)
        s = torch.empty(n, dtype=torch.int32, device="cuda")
        frame = iter(range(1 << 20))

        def call():
            gi.gi_cache_update(h, hits, view, s)
            gi.gi_cache_resolve(h, next(frame))
        return us(call)
    finally:
        gi.gi_cache_destroy(h)
