"""The per-column cap's choice (App. B.5: the lowest energies go, ties by the larger id first) at the
column sizes where its kernel changes course -- a few entries, a block's width, the shared-memory keys'
limit and beyond -- with groups of identical ray volumes across the cut (ranked by id) and zero-action
ones; the survivors' ids must be the FP64 oracle's, all states within the parity bars, and the precision
form must keep the same ids."""
import numpy as np
import pytest

import oracle
from paper_2309_11257_gb300 import synth
from parity_util import assert_rays_match, assert_stats_match

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


@pytest.mark.parametrize("n,cap,copies", [(3, 1, 1), (130, 129, 1), (300, 100, 7), (1024, 1000, 1), (1100, 300, 40),
                                          (2600, 1700, 260), (400, 390, 400)])
@pytest.mark.parametrize("precision", [0, 1])
def test_cap_keeps_the_oracles_choice(gw, n, cap, copies, precision):
    import torch
    grid = synth.fplane_grid(nx=4, ny=4, nz=32)
    params = dict(synth.DEFAULT_PARAMS, cap_per_column=cap, saturation=0, splitting=0)
    bg = synth.perturbed(synth.uniform_background(grid), tag=75)
    r = synth.fplane_rays(grid, n, tag=76)
    rng = synth.rng(77)
    r["x"] = 75e3 + 5e3 * rng.uniform(size=n)      # all in one column, well inside it
    r["y"] = 75e3 + 5e3 * rng.uniform(size=n)
    for name in r:                                 # runs of `copies` identical volumes, ids interleaved
        r[name] = np.array(r[name])
        r[name][:] = r[name][np.arange(n) % -(-n // copies)]
    r["n"][:: max(2, n // 20)] = 0.0               # zero action: energies equal at 0
    T = gw.Tracer(grid, dict(params, precision=precision), max_rays=4 * n + 100)
    O = oracle.Model(grid, params)
    T.set_background(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in bg])
    O.set_background(*bg)
    T.add_rays(r)
    O.add_rays(r)
    T.step(60.0)
    O.step(60.0)
    g, o = T.rays(), O.rays()
    assert len(o["id"]) == cap and np.array_equal(np.sort(g["id"]), np.sort(o["id"]))
    if precision == 0:
        assert_rays_match(g, o, grid)
        assert_stats_match(T.stats(), O.stats())
