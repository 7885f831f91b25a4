"""Launches of far more bins than the context holds ray volumes, most of them filtered: the stream-ordered scratch
stays bounded (32 MB whatever the number of bins), and the ray volumes, their ids and the counters are those of a
context that holds one ray volume per bin, bit for bit (the launched sums to FP64 rounding); an overflow is reported."""
import ctypes as C

import numpy as np
import pytest

from paper_2309_11257_gb300 import synth

pytestmark = pytest.mark.gpu

POOL_USED_HIGH = 8     # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


def _pool_high(reset):
    """Most bytes in use in the device's default memory pool since the last reset."""
    import torch
    cu = C.CDLL("libcuda.so.1")
    pool, v = C.c_void_p(), C.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(C.byref(pool), C.c_int(torch.cuda.current_device())) == 0
    f = cu.cuMemPoolSetAttribute if reset else cu.cuMemPoolGetAttribute
    assert f(pool, C.c_int(POOL_USED_HIGH), C.byref(v)) == 0
    return v.value


def _tracer(gw, grid, bg, max_rays, precision):
    import torch
    T = gw.Tracer(grid, dict(synth.DEFAULT_PARAMS, precision=precision), max_rays=max_rays)
    T.set_background(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in bg])
    return T


def _specs(grid, launched):
    specs = np.tile(synth.uniform_specs(grid, z_launch=3e3), 12)
    specs["c"] = -300.0                   # a negative intrinsic frequency in any wind here: filtered
    keep = np.linspace(0, len(specs) - 1, launched).astype(int)
    specs["c"][keep] = 30.0
    return specs


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ghost", [False, True])
def test_scratch_is_bounded(gw, ghost, precision):
    import torch
    grid = synth.sphere_grid(nx=64, ny=32, nz=20)
    bg = synth.perturbed(synth.jet_background(grid, z_peak=12e3, z_width=5e3), tag=91)
    specs = _specs(grid, 3000)
    assert len(specs) > 2 * 2 ** 18
    out = []
    for max_rays in (len(specs) + 10000, 10000):
        T = _tracer(gw, grid, bg, max_rays, precision)
        T.synchronize()
        _pool_high(reset=True)
        for _ in range(2):
            T.launch_ghost_spectral(specs, 120.0) if ghost else T.launch_spectral(specs)
        T.synchronize()
        high = _pool_high(reset=False)
        out.append((T.rays(), T.stats()))
        assert high <= 32 << 20
    (ra, sa), (rb, sb) = out
    assert len(ra["id"]) > 0 and all(np.array_equal(ra[k], rb[k]) for k in ra)
    for k in sa:
        assert sa[k] == sb[k] if isinstance(sa[k], int) else abs(sa[k] - sb[k]) <= 1e-13 * abs(sa[k]), k


def test_background_source_beyond_the_rays(gw):
    grid = synth.sphere_grid(nx=64, ny=32, nz=20)
    bg = synth.perturbed(synth.jet_background(grid, z_peak=12e3, z_width=5e3), tag=92)
    src = synth.background_source(z_launch=2e3, c_min=0.01, c_max=40.0, n_az=32, n_c=12, lambda_h=400e3, launch_zero_flux=0)
    bins = 64 * 32 * 32 * 12
    wide = _tracer(gw, grid, bg, bins, 0)
    wide.launch_sources(src)
    n = wide.num_rays()
    assert 0 < n < bins
    T = _tracer(gw, grid, bg, n, 0)
    T.launch_sources(src)
    a, b = wide.rays(), T.rays()
    assert all(np.array_equal(a[k], b[k]) for k in a)
    assert wide.stats()["n_filtered"] == T.stats()["n_filtered"]


def test_overflow_is_reported(gw):
    grid = synth.sphere_grid(nx=64, ny=32, nz=20)
    bg = synth.perturbed(synth.jet_background(grid, z_peak=12e3, z_width=5e3), tag=93)
    specs = _specs(grid, 3000)
    T = _tracer(gw, grid, bg, 1000, 0)
    T.launch_spectral(specs)
    with pytest.raises(gw.GwamError) as e:
        T.synchronize()
    assert e.value.code == gw.GWAM_ECAPACITY


@pytest.mark.parametrize("n_az,n_c", [(1024, 1), (1, 1024), (32, 32)])
@pytest.mark.parametrize("ghost", [False, True])
def test_largest_source_tables(gw, n_az, n_c, ghost):
    """1024 bins a column, all in one direction of the source's table or in both, against the oracle."""
    import oracle
    from parity_util import assert_rays_match, assert_stats_match
    grid = synth.sphere_grid(nx=6, ny=6, nz=20)
    bg = synth.perturbed(synth.jet_background(grid, z_peak=12e3, z_width=5e3), tag=94)
    src = synth.background_source(z_launch=2e3, n_az=n_az, n_c=n_c)
    T = _tracer(gw, grid, bg, 36 * 1024, 0)
    O = oracle.Model(grid, synth.DEFAULT_PARAMS)
    O.set_background(*bg)
    T.launch_ghost(src, 120.0) if ghost else T.launch_sources(src)
    O.launch_ghost(src, 120.0) if ghost else O.launch_background(src)
    assert len(O.rays()["id"]) > 0
    assert_rays_match(T.rays(), O.rays(), grid)
    assert_stats_match(T.stats(), O.stats())
