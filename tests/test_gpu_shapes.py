"""Launch shapes of the search, every pair, with and without module hits, and the size from which the
search with module hits takes other blocks and no early starts: the same bits each time."""
import numpy as np
import pytest

from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu

LARGE_FROM = 7 << 14   # of k_build_mod.cu


@pytest.fixture(scope="module", params=["cylinders", "modules"])
def event(request):
    B.build()
    mkgb.load_library()
    g = S.geometry_phase2_modular_disks() if request.param == "modules" else S.geometry_phase2()
    ev = S.simulate_event(g, 400, 17, 0, pt_sampler=S.sample_pt_phase2, eta_max=2.5, noise_total=1000)
    b = S.concat_events([ev], g.n_layers)
    ctx = pipeline.make_context(g, S.default_params())
    ctx.load_hits(1, b.hit_off, b.hit_xyz, b.hit_cov, hit_module=b.hit_mod if request.param == "modules" else None)
    return request.param, g, b, ctx


def _search(g, ctx, seeds):
    ctx.seed(np.ascontiguousarray(seeds))
    return ctx.build(mkgb.alloc_tracks(seeds.shape[0], g.max_plan, ovl=True))


def test_every_pair_of_shapes(event):
    kind, g, b, ctx = event
    ref = _search(g, ctx, b.seed_hits)
    assert (ref["ovl"] >= 0).any() == (kind == "modules")
    for f in range(6):
        for s in range(3):
            ctx.set_launch(f, s)
            got = _search(g, ctx, b.seed_hits)
            for k in ref:
                assert np.array_equal(got[k], ref[k]), (f, s, k)
    best = ctx.autotune(1)
    assert best[0] < (3 if kind == "modules" else 6)
    ctx.set_launch(1, 0)


@pytest.mark.parametrize("n", [LARGE_FROM - 1, LARGE_FROM, LARGE_FROM + 33])
def test_large_batches(event, n):
    kind, g, b, ctx = event
    ref = _search(g, ctx, b.seed_hits)
    rows = np.random.default_rng(n).integers(0, b.seed_hits.shape[0], n)
    got = _search(g, ctx, b.seed_hits[rows])
    for k in ref:
        assert np.array_equal(got[k], ref[k][rows]), k
