"""The search's count of Kalman updates, where many of a search's last ones fail: they are taken off
again, as in the oracle."""
import numpy as np
import pytest

import oracle
from oracle import parity as PR
from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


def test_failed_last_updates_are_not_counted():
    """The hits of the outermost layer are moved 1 m along z and taken all the same (no chi2 to speak of
    cuts, a hit is worth more than any residual): for most tracks the update turns theta out of
    (0, pi) and fails.  2%: the margin of the parity tests' counters."""
    B.build()
    mkgb.load_library()
    g = S.geometry_barrel()
    b = S.concat_events([S.simulate_event(g, 300, 9, 0, eta_max=0.8, noise_per_layer=0)], g.n_layers)
    last = slice(int(b.hit_off[-2]), int(b.hit_off[-1]))
    b.hit_xyz = b.hit_xyz.copy()
    z = b.hit_xyz[last, 2]
    b.hit_xyz[last, 2] = -z - np.sign(z) * 100.0
    params = S.default_params(max_cands=1, chi2_cut=1e12, score_hit=1e11, score_hole=1e11, deta_min=3.0, deta_max=3.0,
                              dphi_min=0.01)
    o = PR.oracle_build(oracle.Oracle(g, params), b)["counters"]
    kept = 7 * b.seed_hits.shape[0]   # a hit on each of the seven searched layers, nearly
    assert o[2] < 0.9 * kept
    ctx = pipeline.make_context(g, params)
    ctx.load_hits(1, b.hit_off, b.hit_xyz, b.hit_cov)
    ctx.seed(b.seed_hits)
    ctx.build(mkgb.alloc_tracks(b.seed_hits.shape[0], g.max_plan))
    c = ctx.counters(0)
    for k in range(3):
        assert abs(c[k] - o[k]) <= 0.02 * o[k] + 10, (k, c, o)
