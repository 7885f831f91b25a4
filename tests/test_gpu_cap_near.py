"""The per-column cap's choice where energies nearly tie: the FP64 oracle's choice among energies a relative 4e-13
apart on a grid whose latitude series is exact to FP64 (an f-plane), and 1e-10 apart on spheres so coarse that the
series of the double-float form (rows up to 9 degrees) is off by up to 1e-7, with near-inertial waves, whose
frequency is the Coriolis parameter.  Infinite energies (an action beyond FP64's range) stay, by the id among
themselves."""
import math

import numpy as np
import pytest

import oracle
from paper_2309_11257_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


def _survivors(gw, grid, params, bg, rays, dt):
    import torch
    n = len(rays["x"])
    T = gw.Tracer(grid, params, max_rays=4 * n + 100)
    O = oracle.Model(grid, params)
    T.set_background(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in bg])
    O.set_background(*bg)
    T.add_rays(rays)
    O.add_rays(rays)
    T.step(dt)
    O.step(dt)
    return np.sort(T.rays()["id"]), np.sort(O.rays()["id"])


def _set_energies(rays, energy, w, hx, hy):
    rays["n"] = energy / (w * (hx * rays["ex"] * rays["dk"]) * (hy * rays["ey"] * rays["dl"]) * (rays["ez"] * rays["dm"]))


@pytest.mark.parametrize("n,cap", [(40, 20), (300, 150), (1100, 1000)])
def test_energies_within_the_select_precision(gw, n, cap):
    grid = synth.fplane_grid(nx=4, ny=4, nz=32)
    params = dict(synth.DEFAULT_PARAMS, cap_per_column=cap, saturation=0, splitting=0, gamma_mode=0)
    rays = synth.fplane_rays(grid, n, tag=81)
    r = synth.rng(82)
    rays["x"], rays["y"] = 75e3 + 5e3 * r.uniform(size=n), 75e3 + 5e3 * r.uniform(size=n)
    kh2, m2, f2, n2 = rays["k"] ** 2 + rays["l"] ** 2, rays["m"] ** 2, 1e-8, 0.02 ** 2
    w = np.sqrt((f2 * m2 + n2 * kh2) / (kh2 + m2))
    _set_energies(rays, 1e-3 * (1.0 + 4e-13 * r.permutation(n)), w, 1.0, 1.0)
    g, o = _survivors(gw, grid, params, synth.uniform_background(grid), rays, 60.0)
    assert len(o) == cap and np.array_equal(g, o)


@pytest.mark.parametrize("ny", [2, 4])
def test_coarse_latitudes(gw, ny):
    n, cap = 200, 100
    grid = synth.sphere_grid(nx=4, ny=ny, nz=8)
    params = dict(synth.DEFAULT_PARAMS, cap_per_column=cap, saturation=0, splitting=0, gamma_mode=0)
    shape = (8, ny, 4)
    bg = (np.zeros(shape), np.zeros(shape), np.full(shape, 4e-4), np.ones(shape))
    rays = synth.sphere_rays(grid, n, tag=83, ext_scale=0.01)
    r = synth.rng(84)
    rays["x"] = 0.4 + 0.5 * r.uniform(size=n)
    rays["y"] = np.radians(r.uniform(4.0, 40.0, n))         # all in one row
    rays["z"] = r.uniform(3e3, 5e3, n)
    kh, th = 2 * math.pi / 1e6, r.uniform(0, 2 * math.pi, n)
    rays["k"], rays["l"], rays["m"] = kh * np.cos(th), kh * np.sin(th), np.full(n, -2 * math.pi / 100.0)
    rays["dk"] = rays["dl"] = np.full(n, 0.1 * kh)
    rays["dm"] = -0.1 * rays["m"]
    f2 = (2 * synth.EARTH_OMEGA * np.sin(rays["y"])) ** 2
    kh2, m2 = kh ** 2, rays["m"] ** 2
    w = np.sqrt((f2 * m2 + 4e-4 * kh2) / (kh2 + m2))
    rays["z"] = r.uniform(3e3, 5e3, n)
    rad = synth.EARTH_RADIUS + rays["z"]
    _set_energies(rays, 1e-3 * (1.0 + 1e-10 * r.permutation(n)), w, rad * np.cos(rays["y"]), rad)
    g, o = _survivors(gw, grid, params, bg, rays, 1e-3)
    assert len(o) == cap and np.array_equal(g, o)


@pytest.mark.parametrize("infinite,cap", [(30, 50), (30, 20), (100, 20)])
def test_infinite_energies(gw, infinite, cap):
    n = 100
    grid = synth.fplane_grid(nx=4, ny=4, nz=32)
    params = dict(synth.DEFAULT_PARAMS, cap_per_column=cap, saturation=0, splitting=0)
    rays = synth.fplane_rays(grid, n, tag=85)
    r = synth.rng(86)
    rays["x"], rays["y"] = 75e3 + 5e3 * r.uniform(size=n), 75e3 + 5e3 * r.uniform(size=n)
    big = r.permutation(n)[:infinite]
    rays["n"] = np.array(rays["n"])
    rays["dk"] = np.array(rays["dk"])
    rays["n"][big], rays["dk"][big] = 1e300, 1e20
    g, o = _survivors(gw, grid, params, synth.uniform_background(grid), rays, 60.0)
    assert len(o) == cap and np.array_equal(g, o)
