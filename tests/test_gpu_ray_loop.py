"""The ray step's loop and the launches' staging at the sizes where they change course, against the
FP64 oracle at the parity bars of the other cases: populations below a warp, just below, at and just
above one pass of the grid (two 256-thread blocks per SM of 152: 77 824 rays), whose left-over rays
are spread a warp per block; launches of more bins than the context can hold ray volumes, most of them
filtered (staged in scratch of their own instead of the free ray buffer), and of none."""
import numpy as np
import pytest

import oracle
from paper_2309_11257_gb300 import synth
from parity_util import assert_fields_match, assert_rays_match, assert_stats_match

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


@pytest.mark.parametrize("n", [1, 33, 77823, 77824, 77824 + 33])
def test_ray_loop_edges(gw, n):
    import torch
    grid = synth.fplane_grid(nx=12, ny=10, nz=32)
    params = dict(synth.DEFAULT_PARAMS, cap_per_column=0)
    bg = synth.perturbed(synth.uniform_background(grid), tag=71, rel=0.1)
    T = gw.Tracer(grid, params, max_rays=4 * n)
    O = oracle.Model(grid, params)
    T.set_background(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in bg])
    O.set_background(*bg)
    r = synth.fplane_rays(grid, n, tag=72)
    T.add_rays(r)
    O.add_rays(r)
    du = torch.zeros((grid["nz"], grid["ny"], grid["nx"]), dtype=torch.float64, device="cuda")
    dv = torch.zeros_like(du)
    for _ in range(2):
        T.step(300.0, du, dv)
        odu, odv = O.step(300.0)
    assert_rays_match(T.rays(), O.rays(), grid)
    assert_stats_match(T.stats(), O.stats())
    su, sv = O.tendency_scale()
    assert_fields_match(du.cpu().numpy(), odu, su, name="dudt")
    assert_fields_match(dv.cpu().numpy(), odv, sv, name="dvdt")


@pytest.mark.parametrize("launched", [0, 40])
@pytest.mark.parametrize("ghost", [False, True])
def test_launch_of_more_bins_than_rays(gw, launched, ghost):
    import torch
    grid = synth.sphere_grid(nx=16, ny=8, nz=20)
    params = dict(synth.DEFAULT_PARAMS)
    bg = synth.perturbed(synth.jet_background(grid, z_peak=12e3, z_width=5e3), tag=73)
    specs = synth.uniform_specs(grid, z_launch=3e3)
    specs["c"] = -300.0                   # a negative intrinsic frequency in any wind here: filtered
    keep = np.linspace(0, len(specs) - 1, launched).astype(int)
    specs["c"][keep] = 30.0
    probe = oracle.Model(grid, params)
    probe.set_background(*bg)
    probe.launch_spectral(specs)
    live = len(probe.rays()["id"])
    assert live < len(specs) - 100 and (live > 0) == (launched > 0)
    T = gw.Tracer(grid, params, max_rays=2 * live + 100)
    O = oracle.Model(grid, params)
    T.set_background(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in bg])
    O.set_background(*bg)
    assert len(specs) > T.max_rays
    for _ in range(2):
        T.launch_ghost_spectral(specs, 120.0) if ghost else T.launch_spectral(specs)
        O.launch_ghost_spectral(specs, 120.0) if ghost else O.launch_spectral(specs)
    assert_rays_match(T.rays(), O.rays(), grid)
    assert_stats_match(T.stats(), O.stats())
