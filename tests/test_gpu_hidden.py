"""Inference with all hidden layers in one kernel, whose layers read the rows that the warps of the same cluster
wrote a moment before: bit for bit the drag of the same network layer by layer (a surrogate of small chunks), pass
after pass, at widths that the kernel takes with one to several row tiles a cluster, and at widths and inputs that
it does not take (every layer a launch either way)."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    from paper_2309_11257_gb300 import build
    build.build()
    from paper_2309_11257_gb300 import gwam
    return gwam


def _surrogate(gw, par, n_in, hidden, layers, max_batch):
    one = np.ones
    S = gw.Surrogate(n_in=n_in, n_out=6, n_hidden=hidden, n_layers=layers, nlev=3, max_batch=max_batch)
    S.set_normalization(0 * one(n_in), one(n_in), 0 * one(6), one(6), -9 * one(n_in), 9 * one(n_in))
    S.set_params(par)
    return S


def _network(n_in, hidden, layers):
    r = np.random.default_rng(n_in + hidden)
    return [(W.astype(np.float32), (0.1 * r.standard_normal(len(b))).astype(np.float32))
            for W, b in mlp.init_params((n_in,) + (hidden,) * layers + (6,), hidden + layers)]


@pytest.mark.parametrize("n_in,hidden,layers,ncol", [(5, 256, 7, 14000), (512, 256, 3, 40001), (70, 512, 4, 9000),
                                                     (368, 512, 4, 32768), (368, 512, 7, 19999), (130, 128, 3, 20000),
                                                     (368, 384, 3, 9001), (600, 512, 2, 20000), (368, 1024, 2, 9000)])
def test_one_kernel_equals_layer_by_layer(gw, n_in, hidden, layers, ncol):
    import torch
    par = _network(n_in, hidden, layers)
    big = _surrogate(gw, par, n_in, hidden, layers, 40960)
    small = _surrogate(gw, par, n_in, hidden, layers, 1024)
    X = torch.from_numpy(np.random.default_rng(ncol).standard_normal((ncol, n_in)).astype(np.float32)).cuda()
    mask, nfb = torch.zeros(ncol, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")

    def drag(S):
        o = torch.full((6, ncol), float("nan"), dtype=torch.float64, device="cuda")
        S.infer(X, o[:3], o[3:], mask, nfb)
        return o

    ref = drag(small)
    for _ in range(5):
        assert torch.equal(drag(big), ref)
    big.status()
    small.status()
    assert int(nfb.item()) == 0 and bool(torch.isfinite(ref).all())
    rows = np.r_[0:65, ncol - 65:ncol]
    bf = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(torch.bfloat16).double().numpy()  # noqa: E731
    Yo, _ = mlp.forward([(bf(W), b.astype(np.float64)) for W, b in par], bf(X[rows].cpu().numpy()))
    got = ref[:, rows].cpu().numpy().T
    assert np.linalg.norm(got - Yo) <= 1e-2 * np.linalg.norm(Yo)      # the bar of test_gpu_mlp.py
