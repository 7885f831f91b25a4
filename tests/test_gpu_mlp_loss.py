"""The training loss as the FP64 sum of the squared errors (gwam_mlp_last_loss_host): a network whose
parameters are all zero has the outputs 0 exactly, so the errors are the targets.  64 of them in one row
(one thread's sum over two 32-column chunks of the epilogue), the rest zero; 64 rows x 64 outputs make the mean a
division by a power of two.  Bar: eight FP64 roundings, 8 x 2^-53 -- two per chunk, one between the chunks, the
others of the warps' and blocks' sums add zeros -- at magnitudes whose squares do not fit in FP32, too."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


@pytest.mark.parametrize("lo,hi", [(0, 0), (25, 25), (-25, -25), (-17, 20), (30, 38)])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_loss_is_the_fp64_sum_of_squares(gw, lo, hi, seed):
    import torch
    S = gw.Surrogate(n_in=8, n_out=64, n_hidden=64, n_layers=1, nlev=32, max_batch=128)
    one = np.ones
    S.set_normalization(0 * one(8), one(8), 0 * one(64), one(64), -9 * one(8), 9 * one(8))
    S.set_params([(0 * one((64, 8)), 0 * one(64)), (0 * one((64, 64)), 0 * one(64))])
    r = np.random.default_rng(seed)
    Y = np.zeros((64, 64), dtype=np.float32)
    Y[5] = (r.standard_normal(64) * 10.0 ** r.uniform(lo, hi, 64)).astype(np.float32)
    X = r.standard_normal((64, 8)).astype(np.float32)
    S.train_step(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), 64,
                 rows=torch.arange(64, dtype=torch.int32, device="cuda"), lr=0.0)
    ref = sum(Fraction(float(y)) ** 2 for y in Y[5]) / 4096
    assert abs(Fraction(S.loss()) - ref) <= ref * 8 / 2 ** 53
    assert not S.output(64).any()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_loss_of_an_infinite_or_nan_target(gw, bad):
    import torch
    S = gw.Surrogate(n_in=8, n_out=64, n_hidden=64, n_layers=1, nlev=32, max_batch=128)
    one = np.ones
    S.set_normalization(0 * one(8), one(8), 0 * one(64), one(64), -9 * one(8), 9 * one(8))
    S.set_params([(0 * one((64, 8)), 0 * one(64)), (0 * one((64, 64)), 0 * one(64))])
    Y = np.full((64, 64), 0.5, dtype=np.float32)
    Y[7, 40] = bad
    S.train_step(torch.zeros((64, 8), device="cuda"), torch.from_numpy(Y).cuda(), 64,
                 rows=torch.arange(64, dtype=torch.int32, device="cuda"), lr=0.0)
    assert np.isnan(S.loss()) if np.isnan(bad) else S.loss() == np.inf
