"""The search's tiles of 32 seeds in its other forms, all in FP64 and backwards: batches of any number of
seeds around the tiles' edges give every seed the same bits as the whole batch (which the parity tests
compare with the oracle)."""
import numpy as np
import pytest

from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def events():
    B.build()
    mkgb.load_library()
    g = S.geometry_phase2()
    evs = [S.simulate_event(g, 500, 23, e, pt_sampler=S.sample_pt_phase2, eta_max=3.0, noise_total=2000) for e in range(2)]
    return g, S.concat_events(evs, g.n_layers)


def _context(g, batch, **params):
    ctx = pipeline.make_context(g, S.default_params(**params))
    ctx.load_hits(batch.n_events, batch.hit_off, batch.hit_xyz, batch.hit_cov)
    return ctx


def _same_rows(part, full, rows):
    for k in part:
        assert np.array_equal(part[k], full[k][rows]), k


@pytest.mark.parametrize("n", [1, 31, 33, 257])
def test_fp64_search_does_not_depend_on_the_batch(events, n):
    g, batch = events
    ctx = _context(g, batch, precision=mkgb.FP64)

    def search(seeds):
        ctx.seed(np.ascontiguousarray(seeds))
        return ctx.build(mkgb.alloc_tracks(seeds.shape[0], g.max_plan))

    full = search(batch.seed_hits)
    rows = np.random.default_rng(n).choice(batch.seed_hits.shape[0], n, replace=False)
    _same_rows(search(batch.seed_hits[rows]), full, rows)


@pytest.mark.parametrize("n", [1, 31, 33, 257])
def test_backward_search_does_not_depend_on_the_batch(events, n):
    """Tracks without their first three layers, fitted forwards and back, then searched inwards."""
    g, batch = events
    fi = pipeline.fit_inputs(batch)
    ctx = _context(g, batch)
    keep = (fi.layers >= 0).sum(1) > 5
    lay, hits = np.ascontiguousarray(fi.layers[keep, 3:]), np.ascontiguousarray(fi.hits[keep, 3:])
    m = lay.shape[0]
    out = lambda: (np.zeros((m, 6), np.float32), np.zeros((m, 21), np.float32), np.zeros(m, np.float32), np.zeros(m, np.int32))
    f, b = out(), out()
    ctx.fit(lay, hits, fi.p0[keep], fi.c0[keep], *f)
    ctx.fit_backward(lay, hits, f[0], f[1], *b)
    ok = np.nonzero(b[3] == 0)[0]
    event, first, p, c = fi.event[keep][ok], lay[ok, 0], b[0][ok], b[1][ok]

    def search(rows):
        pick = lambda a: np.ascontiguousarray(a[rows])
        return ctx.build_backward(pick(event), pick(first), pick(p), pick(c), mkgb.alloc_tracks(len(rows), g.max_plan))

    full = search(np.arange(len(ok)))
    assert (full["nfound"] > 0).mean() > 0.9
    rows = np.random.default_rng(n).choice(len(ok), n, replace=False)
    _same_rows(search(rows), full, rows)
