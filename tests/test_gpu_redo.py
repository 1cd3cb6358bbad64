"""Long FP64 redo lists: with kappa_fp64 lowered until every update of the search is redone in FP64, the
search meets the oracle, and a seed's result does not depend on the number of seeds (how the list is
dealt out)."""
import numpy as np
import pytest

import oracle
from oracle import parity as PR
from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kappa", [1.0, 256.0])
def test_every_update_redone(kappa):
    B.build()
    mkgb.load_library()
    g = S.geometry_phase2()
    b = S.concat_events([S.simulate_event(g, 900, 13, e, pt_sampler=S.sample_pt_phase2, eta_max=3.0, noise_total=2000)
                         for e in range(2)], g.n_layers)
    params = S.default_params(kappa_fp64=kappa)
    ctx = pipeline.make_context(g, params)
    ctx.load_hits(b.n_events, b.hit_off, b.hit_xyz, b.hit_cov)

    def search(seeds):
        ctx.seed(np.ascontiguousarray(seeds))
        return ctx.build(mkgb.alloc_tracks(seeds.shape[0], g.max_plan))

    full = search(b.seed_hits)
    rep = PR.compare_build(full, PR.oracle_build(oracle.Oracle(g, params), b))
    assert len(rep["hit_mismatch"]) == 0 and rep["param_bad"] == 0 and rep["chi2_bad"] == 0, rep
    for n in (1, 33, 257):
        rows = np.random.default_rng(n).choice(b.seed_hits.shape[0], n, replace=False)
        part = search(b.seed_hits[rows])
        for k in part:
            assert np.array_equal(part[k], full[k][rows]), (n, k)
