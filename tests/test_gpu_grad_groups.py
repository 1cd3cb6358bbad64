"""The reverse sweep's per-layer derivatives where a block takes several groups of 32 tracks and comes
back for more of them (batches of tens of thousands of tracks), against calls of 400 tracks (a group
per block) on the same rows, summed in FP64."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9_999, 20_011, 45_003])
def test_layer_derivatives_of_large_batches(n):
    """Every track's terms have the same bits in both, so only their order differs: FP32 sums of n terms
    per layer keep 5e-4 of the largest of their kind, the bound of the comparison with the oracle; one
    group of 32 tracks lost or counted twice moves them by 1e-3 and more."""
    B.build()
    mkgb.load_library()
    g, evs, al, xs = S.workload_aligned_fit(n_tracks=400, seed=2)
    batch = S.concat_events(evs, g.n_layers)
    fi = pipeline.fit_inputs(batch)
    ctx = pipeline.make_context(g, S.default_params())
    ctx.load_hits(batch.n_events, batch.hit_off, batch.hit_xyz, batch.hit_cov)
    L = g.n_layers
    align, xscale = (-al).astype(np.float32), xs.astype(np.float32)

    def grad(rows):
        m = len(rows)
        pick = lambda a: np.ascontiguousarray(a[rows])
        f = SimpleNamespace(layers=pick(fi.layers), hits=pick(fi.hits), p0=pick(fi.p0), c0=pick(fi.c0))
        x2, dp, da, dx, st = (np.zeros(m, np.float32), np.zeros((m, 6), np.float32), np.zeros((L, 6), np.float32),
                              np.zeros(L, np.float32), np.zeros(m, np.int32))
        ctx.fit_grad(f.layers, f.hits, f.p0, f.c0, align, xscale, x2, dp, da, dx, st)
        return da.astype(np.float64), dx.astype(np.float64), st

    rows = np.random.default_rng(n).integers(0, fi.layers.shape[0], n)
    da, dx, st = grad(rows)
    parts = [grad(rows[k:k + 400]) for k in range(0, n, 400)]
    assert np.array_equal(st, np.concatenate([p[2] for p in parts]))
    ra, rx = sum(p[0] for p in parts), sum(p[1] for p in parts)
    for c in range(6):
        assert np.abs(da[:, c] - ra[:, c]).max() <= 5e-4 * np.abs(ra[:, c]).max(), c
    assert np.abs(dx - rx).max() <= 5e-4 * np.abs(rx).max()
