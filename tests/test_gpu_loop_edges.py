"""The step's ray loops on grids of a few blocks, at populations around one and two passes of the grid (whole passes,
left-over rays, warps without rays; the counters that the projection clears in several parts for the next step), in
both forms: the ray volumes, ids and counts are those of the default launch shapes, bit for bit, and the drag is the
same up to the order of the FP64 additions (in the precision form up to its FP32 fields' rounding)."""
import numpy as np
import pytest

from paper_2309_11257_gb300 import synth

pytestmark = pytest.mark.gpu

THREADS, BLOCKS = 64, 3
PASS = THREADS * BLOCKS


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


@pytest.mark.parametrize("n", [1, 31, 33, PASS - 1, PASS, PASS + 1, PASS + 33, 2 * PASS - 31, 2 * PASS + 1, 7 * PASS + 5])
@pytest.mark.parametrize("precision", [0, 1])
def test_few_blocks_equal_the_default(gw, n, precision):
    import torch
    grid = synth.fplane_grid(nx=5, ny=7, nz=33)
    bg = synth.perturbed(synth.uniform_background(grid), tag=101, rel=0.1)
    rays = synth.fplane_rays(grid, n, tag=102, ext_z=1700.0)      # vertical splits in the first step
    out = []
    for cfg in (None, {k: (THREADS, BLOCKS) for k in gw.Tracer.KERNELS}):
        T = gw.Tracer(grid, dict(synth.DEFAULT_PARAMS, precision=precision, cap_per_column=40, alpha_s=1.5), max_rays=8 * n + 64)
        T.set_background(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in bg])
        if cfg:
            T.set_launch_config(cfg)
            assert T.launch_config() == cfg
        T.add_rays(rays)
        du = torch.zeros((33, 7, 5), dtype=torch.float64, device="cuda")
        dv = torch.zeros_like(du)
        for _ in range(3):
            T.step(300.0, du, dv)
        out.append((T.rays(), T.stats(), torch.stack([du, dv]).cpu().numpy()))
    (ra, sa, da), (rb, sb, db) = out
    assert all(np.array_equal(ra[k], rb[k]) for k in ra)
    for k in sa:
        assert sa[k] == sb[k] if isinstance(sa[k], int) else abs(sa[k] - sb[k]) <= 1e-13 * abs(sa[k]), k
    assert n == 1 or sa["n_split_v"] > 0
    assert np.abs(da - db).max() <= (1e-6 if precision else 1e-12) * np.abs(da).max()
