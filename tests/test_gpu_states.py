"""A call that fails part-way leaves nothing behind that a later call would run on: after a rejected
batch of hits there are no hits and no seeds, and the search refuses (MKGB_ESTATE) until both are
loaded again."""
import dataclasses

import numpy as np
import pytest

from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    B.build()
    return mkgb.load_library()


def _refuses(call, code):
    with pytest.raises(mkgb.MkgbError, match=code):
        call()


def _event(geom, tracks=200):
    kw = {} if geom.modules is None else dict(pt_sampler=S.sample_pt_phase2, eta_max=2.5, noise_total=500)
    kw = kw or dict(eta_max=1.0, noise_per_layer=50)
    return S.concat_events([S.simulate_event(geom, tracks, 7, 0, **kw)], geom.n_layers)


def test_rejected_modules_leave_no_hits_and_no_seeds(lib):
    g = S.geometry_phase2_modular_disks()
    b = _event(g)
    ctx = pipeline.make_context(g, S.default_params())
    out = lambda: mkgb.alloc_tracks(b.seed_hits.shape[0], g.max_plan, ovl=True)
    load = lambda mod: ctx.load_hits(b.n_events, b.hit_off, b.hit_xyz, b.hit_cov, hit_module=mod)
    load(None)   # on the layers' own surfaces
    ctx.seed(b.seed_hits)
    plain = ctx.build(out())
    wrong = np.where(b.hit_mod >= 0, -1, 0).astype(np.int32)
    _refuses(lambda: load(wrong), "MKGB_EINVAL")
    _refuses(lambda: ctx.build(out()), "MKGB_ESTATE")
    _refuses(lambda: ctx.autotune(1), "MKGB_ESTATE")
    _refuses(lambda: ctx.seed(b.seed_hits), "MKGB_ESTATE")
    load(b.hit_mod)
    _refuses(lambda: ctx.build(out()), "MKGB_ESTATE")   # hits, but the seeds are of the batch before
    ctx.seed(b.seed_hits)
    assert (ctx.build(out())["ovl"] >= 0).any()
    load(None)
    ctx.seed(b.seed_hits)
    again = ctx.build(out())
    for k in plain:
        np.testing.assert_array_equal(again[k], plain[k], err_msg=k)


def test_rejected_host_batch_leaves_no_hits_and_no_seeds(lib):
    """run_host sizes its buffers before it finds that the batch has too many bins."""
    g = S.geometry_barrel()
    g = dataclasses.replace(g, n_eta=np.full_like(g.n_eta, 4096), n_phi=np.full_like(g.n_phi, 1024))
    b = _event(g)
    ctx = pipeline.make_context(g, S.default_params())
    n, w = b.seed_hits.shape[0], g.max_plan
    ctx.load_hits(b.n_events, b.hit_off, b.hit_xyz, b.hit_cov)
    ctx.seed(b.seed_hits)
    before = ctx.build(mkgb.alloc_tracks(n, w))
    events = 2 ** 31 // (4096 * 1024 * g.n_layers) + 1
    f32 = lambda *s: np.zeros(s, np.float32)
    i32 = lambda *s: np.zeros(s, np.int32)
    _refuses(lambda: ctx.run_host(events, np.zeros(events * g.n_layers + 1, np.int64), f32(0, 3), f32(0, 6), i32(0, 3),
                                  mkgb.alloc_tracks(0, w), i32(0, w), i32(0, w), f32(0, 6), f32(0, 21), f32(0, 6),
                                  f32(0, 21), f32(0), i32(0)), "MKGB_EINVAL")
    _refuses(lambda: ctx.build(mkgb.alloc_tracks(n, w)), "MKGB_ESTATE")
    _refuses(lambda: ctx.seed(b.seed_hits), "MKGB_ESTATE")
    ctx.load_hits(b.n_events, b.hit_off, b.hit_xyz, b.hit_cov)
    ctx.seed(b.seed_hits)
    again = ctx.build(mkgb.alloc_tracks(n, w))
    for k in before:
        np.testing.assert_array_equal(again[k], before[k], err_msg=k)
