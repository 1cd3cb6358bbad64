"""Large batches are fitted in the order of their tracks' length and layer kinds, chunk by chunk or, with
module hits, all together: every track's results are the same bits as in a small batch, which keeps its
own order, forwards and backwards."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu

ORDER_FROM, ORDER_FROM_MOD, CHUNK = 96 * 1024, 64 * 1024, 1024   # of k_fit.cu


def _fit(g, batch, fi):
    ctx = pipeline.make_context(g, S.default_params())
    ctx.load_hits(batch.n_events, batch.hit_off, batch.hit_xyz, batch.hit_cov,
                  hit_module=None if g.modules is None else batch.hit_mod)
    n = fi.layers.shape[0]
    out = lambda: dict(p=np.zeros((n, 6), np.float32), c=np.zeros((n, 21), np.float32), x=np.zeros(n, np.float32),
                       s=np.full(n, -7, np.int32))
    f, b = out(), out()
    ctx.fit(fi.layers, fi.hits, fi.p0, fi.c0, f["p"], f["c"], f["x"], f["s"])
    ctx.fit_backward(fi.layers, fi.hits, fi.p0, fi.c0, b["p"], b["c"], b["x"], b["s"])
    return f, b


def _check(g, n, pad):
    B.build()
    mkgb.load_library()
    batch = S.concat_events([S.simulate_event(g, 700, 11, 0, pt_sampler=S.sample_pt_phase2, eta_max=3.0, noise_total=500)],
                            g.n_layers)
    fi = pipeline.fit_inputs(batch)
    lay, hits = (np.pad(a, ((0, 0), (0, pad)), constant_values=-1) for a in (fi.layers, fi.hits))
    lay[0], hits[0] = -1, -1
    lay[1, 1:] = -1
    lay[2, 2] = g.n_layers
    lay[3, 4:], hits[3, 4:] = lay[3, 3], -1   # the same layer again and again, to the row's end
    small = SimpleNamespace(layers=lay, hits=hits, p0=fi.p0, c0=fi.c0)
    rows = np.random.default_rng(n).integers(0, lay.shape[0], n)
    rows[5 * CHUNK:7 * CHUNK] = 9   # chunks of one track only
    pick = lambda a: np.ascontiguousarray(a[rows])
    large = SimpleNamespace(layers=pick(lay), hits=pick(hits), p0=pick(fi.p0), c0=pick(fi.c0))
    for a, b in zip(_fit(g, batch, small), _fit(g, batch, large)):
        for k in a:
            assert np.array_equal(a[k][rows], b[k], equal_nan=True), k


@pytest.mark.parametrize("n", [ORDER_FROM - 1, ORDER_FROM, ORDER_FROM + 1, 97 * CHUNK - 1, 97 * CHUNK + 33])
@pytest.mark.parametrize("pad", [0, 1, 40])
def test_order_changes_no_track(n, pad):
    """Lists without layers, of one layer, with a bad layer number and (pad) in rows wider than any track,
    of odd and even width."""
    _check(S.geometry_phase2(), n, pad)


@pytest.mark.parametrize("n, pad", [(ORDER_FROM_MOD - 1, 0), (ORDER_FROM_MOD, 0), (ORDER_FROM_MOD + 1, 1), (70_001, 40)])
def test_order_changes_no_track_with_modules(n, pad):
    _check(S.geometry_phase2_modular_disks(), n, pad)
