"""The bounded waits of the surrogate's two persistent kernels without a GPU fault (as test_gpu_gemm.py does for the
GEMM): the producers of both or of one CTA of each pair issue no copies, or all do and every wait is cut to a
microsecond, so that CTAs give up at any point.  The call reports within a fraction of a second, what was in flight
has landed (the kernels wait for it), and the next inference and training step give what they gave before, bit for
bit.  And which path an inference takes: the plan's own clusters, at the edges of its rule."""
import ctypes as C
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


def _surrogate(gw, n_in, hidden, layers, max_batch):
    S = gw.Surrogate(n_in=n_in, n_out=6, n_hidden=hidden, n_layers=layers, nlev=3, max_batch=max_batch, seed=hidden + n_in)
    one = np.ones
    S.set_normalization(0 * one(n_in), one(n_in), 0 * one(6), one(6), -9 * one(n_in), 9 * one(n_in))
    return S


def _plan(gw, S, rows):
    n = C.c_int(-1)
    return gw.lib().gwam_selftest_hidden_plan(S._h, rows, C.byref(n)), n.value


@pytest.mark.parametrize("n_in,hidden,layers", [(5, 256, 2), (368, 512, 4), (200, 256, 7)])
@pytest.mark.parametrize("tiles", [1, 2, 3])
def test_hidden_layers_give_up(gw, n_in, hidden, layers, tiles):
    import torch
    S = _surrogate(gw, n_in, hidden, layers, 40960)
    clusters = _plan(gw, S, 1)[1]
    assert clusters > 0
    ncol = min(40960, 256 * (clusters * tiles - clusters // 4) - 77)
    assert _plan(gw, S, ncol)[0] == 1
    X = torch.from_numpy(np.random.default_rng(ncol).standard_normal((ncol, n_in)).astype(np.float32)).cuda()
    mask, nfb = torch.zeros(ncol, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")

    def drag():
        o = torch.full((6, ncol), float("nan"), dtype=torch.float64, device="cuda")
        S.infer(X, o[:3], o[3:], mask, nfb)
        S.status()
        return o

    ref = drag()
    assert bool(torch.isfinite(ref).all())
    for skip, us in ((3, 2000), (1, 2000), (2, 2000), (3, 1), (1, 1), (2, 1), (0, 1), (0, 3), (0, 10), (0, 30)):
        t0 = time.perf_counter()
        rc = gw.lib().gwam_selftest_mlp_timeout(S._h, 0, ncol, skip, us)
        assert time.perf_counter() - t0 < 1.0
        assert rc == gw.GWAM_ETIMEOUT or (skip == 0 and rc == gw.GWAM_OK), (skip, us)
        assert torch.equal(drag(), ref), (skip, us)


@pytest.mark.parametrize("n_in,hidden,layers,batch", [(5, 64, 1, 64), (368, 512, 4, 4096), (200, 320, 2, 1024)])
def test_weight_gradients_give_up(gw, n_in, hidden, layers, batch):
    import torch
    S = _surrogate(gw, n_in, hidden, layers, 4096)
    r = np.random.default_rng(batch)
    X = torch.from_numpy(r.standard_normal((batch, n_in)).astype(np.float32)).cuda()
    Y = torch.from_numpy(r.standard_normal((batch, 6)).astype(np.float32)).cuda()
    rows = torch.arange(batch, dtype=torch.int32, device="cuda")

    def grads():
        S.train_step(X, Y, batch, rows=rows, lr=0.0)
        S.status()
        return [a for g in S.grads() for a in g]

    ref, par = grads(), S.params()
    for skip, us in ((1, 2000), (1, 1), (0, 1), (0, 3), (0, 10)):
        t0 = time.perf_counter()
        rc = gw.lib().gwam_selftest_mlp_timeout(S._h, 1, batch, skip, us)
        assert time.perf_counter() - t0 < 1.0
        assert rc == gw.GWAM_ETIMEOUT or (skip == 0 and rc == gw.GWAM_OK), (skip, us)
        assert all(np.array_equal(a, b) for a, b in zip(grads(), ref)), (skip, us)
    assert all(np.array_equal(a, b) for p, q in zip(S.params(), par) for a, b in zip(p, q))


def test_bad_arguments(gw):
    S = _surrogate(gw, 5, 256, 2, 40960)
    L = gw.lib()
    rows = 40960
    assert L.gwam_selftest_hidden_plan(S._h, rows, None) == 1
    for a in ((2, rows, 1, 100), (-1, rows, 1, 100), (0, 0, 1, 100), (0, rows + 1, 1, 100), (0, rows, 4, 100), (0, rows, -1, 100),
              (0, rows, 1, 0), (0, rows, 1, 2000001), (0, 100, 1, 100), (1, 100, 1, 100), (1, 128, 2, 100)):
        assert L.gwam_selftest_mlp_timeout(S._h, *a) == gw.GWAM_EINVAL, a
    assert L.gwam_selftest_mlp_timeout(None, 0, rows, 1, 100) == gw.GWAM_EINVAL
    assert L.gwam_selftest_hidden_plan(None, 1, None) == gw.GWAM_EINVAL
    assert L.gwam_selftest_hidden_plan(S._h, rows + 1, None) == gw.GWAM_EINVAL


@pytest.mark.parametrize("n_in,hidden,layers,own", [(5, 256, 2, True), (512, 512, 1, True), (513, 512, 2, False), (64, 128, 2, False),
                                                    (64, 384, 2, False), (64, 1024, 1, False)])
def test_plan_of_an_inference(gw, n_in, hidden, layers, own):
    """From three row tiles (256 rows) for five clusters on."""
    S = _surrogate(gw, n_in, hidden, layers, 40960)
    n = _plan(gw, S, 1)[1]
    assert (n > 0) == (hidden in (256, 512))
    edge = -(-3 * n // 5) if n else 20
    for rows in (1, 256 * (edge - 1), 256 * (edge - 1) + 1, 256 * edge, min(40960, 512 * edge), 40960):
        assert _plan(gw, S, rows)[0] == (1 if own and -(-rows // 256) >= edge else 0), rows
