"""The search's slots lie in tiles of 32 seeds and its merge takes blocks of 32 seeds: batches of any
number of seeds around those edges give every seed the same bits as the whole batch (which the
parity tests compare with the oracle), with the fewest and the most candidates per seed; and windows
with more hits than the queue and the child lists hold, against the oracle."""
import numpy as np
import pytest

import oracle
from oracle import parity as PR
from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    B.build()
    return mkgb.load_library()


@pytest.fixture(scope="module")
def events():
    g = S.geometry_phase2()
    evs = [S.simulate_event(g, 700, 5, e, pt_sampler=S.sample_pt_phase2, eta_max=3.0, noise_total=3000) for e in range(2)]
    return g, S.concat_events(evs, g.n_layers)


def _search(g, batch, params, seeds):
    ctx = pipeline.make_context(g, params)
    ctx.load_hits(batch.n_events, batch.hit_off, batch.hit_xyz, batch.hit_cov)
    ctx.seed(np.ascontiguousarray(seeds))
    return ctx.build(mkgb.alloc_tracks(seeds.shape[0], g.max_plan))


@pytest.mark.parametrize("cands", [1, 6, 8])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257])
def test_search_does_not_depend_on_the_batch(lib, events, n, cands):
    g, batch = events
    params = S.default_params(max_cands=cands)
    full = _search(g, batch, params, batch.seed_hits)
    rows = np.random.default_rng(n).choice(batch.seed_hits.shape[0], n, replace=False)
    part = _search(g, batch, params, batch.seed_hits[rows])
    for k, v in part.items():
        assert np.array_equal(v, full[k][rows]), k


@pytest.mark.parametrize("cands", [2, 8])
def test_crowded_windows_match_oracle(lib, cands):
    """30,000 noise hits per layer and wide windows: dozens of hits per window, more than eight of
    them accepted."""
    g = S.geometry_barrel()
    ev = S.simulate_event(g, 40, 9, 0, eta_max=1.0, noise_per_layer=30000)
    batch = S.concat_events([ev], g.n_layers)
    params = S.default_params(max_cands=cands, chi2_cut=1e6, deta_min=0.08, dphi_min=0.08)
    ctx = pipeline.make_context(g, params)
    ctx.load_hits(1, batch.hit_off, batch.hit_xyz, batch.hit_cov)
    ctx.seed(np.ascontiguousarray(batch.seed_hits))
    gpu = ctx.build(mkgb.alloc_tracks(batch.seed_hits.shape[0], g.max_plan))
    c = ctx.counters(0)
    assert c[1] > 12 * c[0]   # hits inside the window per searched step
    rep = PR.compare_build(gpu, PR.oracle_build(oracle.Oracle(g, params), batch))
    assert len(rep["hit_mismatch"]) == 0 and rep["param_bad"] == 0 and rep["chi2_bad"] == 0, rep
