"""Duplicate removal where a row leaves the counted walk: hits on just as many tracks as that walk takes,
one fewer and one more, met before and after uncrowded hits, and rows around the least number of hits;
against the oracle, decision by decision."""
import numpy as np
import pytest

import oracle
from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu

CROWD = 24   # of k_clean.cu


@pytest.mark.parametrize("per_hit", [2, 6, 7, 8, CROWD - 1, CROWD, CROWD + 1, 3 * CROWD])
def test_crowds_match_oracle(per_hit):
    B.build()
    mkgb.load_library()
    g = S.geometry_barrel()
    ev = S.simulate_event(g, 400, 3, 0, eta_max=1.0, noise_per_layer=200)
    batch = S.concat_events([ev], g.n_layers)
    n_hits = batch.hit_xyz.shape[0]
    rng = np.random.default_rng(per_hit)
    groups, width = 40, 9
    rows = []
    for k in range(groups):   # per_hit rows with up to four hits in common, the others their own or a neighbour's
        common = rng.choice(n_hits, 4, replace=False)
        for _ in range(per_hit):
            r = rng.integers(0, n_hits, width)
            at = rng.choice(width, 4, replace=False)
            r[at] = common
            r[rng.random(width) < 0.3] = -1
            rows.append(r)
    rows = np.array(rows, np.int32)[rng.permutation(groups * per_hit)]
    score = rng.integers(0, 50, len(rows)).astype(np.float32)
    ctx = pipeline.make_context(g, S.default_params())
    ctx.load_hits(1, batch.hit_off, batch.hit_xyz, batch.hit_cov)
    for min_hits in (0, 5, 6, 7, width):
        for frac in (0.34, 0.5):
            keep = ctx.remove_duplicates(rows, score, np.zeros(len(rows), np.int32), min_hits=min_hits, frac=frac)
            ref = oracle.remove_duplicates(rows, score.astype(np.float64), n_hits, min_hits=min_hits, frac=frac)
            np.testing.assert_array_equal(keep, ref, err_msg=f"min_hits {min_hits} frac {frac}")
