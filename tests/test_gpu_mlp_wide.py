"""Training steps with output layers up to the widest one accepted, at batches from one row block to many: every
tile width that the rule of gemm_pick_bn can choose has room for the epilogue's staging boxes and bias.  Outputs,
loss and gradients against the FP64 reference at the bars of test_gpu_mlp_shapes.py."""
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


def _bf16(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16).double().numpy()


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n_out", [4480, 4610, 6000, 8192])
@pytest.mark.parametrize("batch", [64, 640, 4096])
def test_training_step_with_many_outputs(gw, n_out, batch):
    import torch
    n_in, hidden = 40, 64
    S = gw.Surrogate(n_in=n_in, n_out=n_out, n_hidden=hidden, n_layers=1, nlev=n_out // 2, max_batch=4096)
    one = np.ones
    S.set_normalization(0 * one(n_in), one(n_in), 0 * one(n_out), one(n_out), -9 * one(n_in), 9 * one(n_in))
    r = np.random.default_rng(n_out + batch)
    par = [(W.astype(np.float32), (0.1 * r.standard_normal(len(b))).astype(np.float32))
           for W, b in mlp.init_params((n_in, hidden, n_out), n_out)]
    S.set_params(par)
    X, Y = r.standard_normal((batch, n_in)).astype(np.float32), r.standard_normal((batch, n_out)).astype(np.float32)
    rows = r.permutation(batch).astype(np.int32)
    S.train_step(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), batch, rows=torch.from_numpy(rows).cuda(), lr=0.0)
    p64 = [(_bf16(W), b.astype(np.float64)) for W, b in par]
    Yo, cache = mlp.forward(p64, _bf16(X[rows]))
    T = Y[rows].astype(np.float64)
    ref = mlp.backward(p64, cache, mlp.loss_grad(Yo, T))
    assert _rel(S.output(batch), Yo) <= 1e-2
    assert abs(S.loss() - mlp.loss(Yo, T)) <= 1e-2 * S.loss()
    for (gW, gb), (oW, ob) in zip(S.grads(), ref):
        assert _rel(gW, oW) <= 3e-2 and _rel(gb, ob) <= 3e-2
