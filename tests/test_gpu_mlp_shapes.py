"""Surrogate gradients, the Adam update and inference at the sizes where the kernels' tiles and splits
change -- one hidden layer of one 64-column tile, odd feature and output counts, batches of a single
and of an odd number of 64-row blocks, column counts below and just above a tile -- against the FP64
reference at the bars of test_gpu_mlp.py (BF16 rounding of the hidden activations and back-propagated
gradients: 1e-2 normwise for outputs, 3e-2 for gradients)."""
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


def _network(gw, n_in, hidden, layers, nlev, max_batch, seed):
    dims = (n_in,) + (hidden,) * layers + (2 * nlev,)
    S = gw.Surrogate(n_in=n_in, n_out=2 * nlev, n_hidden=hidden, n_layers=layers, nlev=nlev, max_batch=max_batch)
    one = np.ones
    S.set_normalization(0 * one(n_in), one(n_in), 0 * one(2 * nlev), one(2 * nlev), -9 * one(n_in), 9 * one(n_in))
    r = np.random.default_rng(seed)
    par = [(W.astype(np.float32), (0.1 * r.standard_normal(len(b))).astype(np.float32)) for W, b in mlp.init_params(dims, seed)]
    S.set_params(par)
    return S, par


@pytest.mark.parametrize("n_in,hidden,layers,nlev,batch", [(5, 64, 1, 3, 64), (70, 128, 2, 45, 320), (368, 192, 3, 90, 832),
                                                            (368, 512, 7, 90, 64), (200, 320, 2, 110, 1024)])
def test_training_step_shapes(gw, n_in, hidden, layers, nlev, batch):
    import torch
    S, par = _network(gw, n_in, hidden, layers, nlev, 1024, seed=n_in + hidden)
    r = np.random.default_rng(batch)
    X, Y = r.standard_normal((1500, n_in)).astype(np.float32), r.standard_normal((1500, 2 * nlev)).astype(np.float32)
    rows = r.choice(1500, batch, replace=False).astype(np.int32)
    Xd, Yd, rd = (torch.from_numpy(a).cuda() for a in (X, Y, rows))
    S.train_step(Xd, Yd, batch, rows=rd, lr=0.0)
    gr = S.grads()
    Yo, cache = mlp.forward([(_bf16(W), b.astype(np.float64)) for W, b in par], _bf16(X[rows]))
    ref = mlp.backward([(_bf16(W), b.astype(np.float64)) for W, b in par], cache, mlp.loss_grad(Yo, Y[rows].astype(np.float64)))
    assert _rel(S.output(batch), Yo) <= 1e-2
    assert abs(S.loss() - mlp.loss(Yo, Y[rows].astype(np.float64))) <= 1e-2 * S.loss()
    for (gW, gb), (oW, ob) in zip(gr, ref):
        assert _rel(gW, oW) <= 3e-2 and _rel(gb, ob) <= 3e-2
    # the update of the same gradients, three steps (the moments carry over)
    st, p64 = mlp.adam_init(par), [(W.astype(np.float64), b.astype(np.float64)) for W, b in par]
    for t in range(1, 4):
        S.train_step(Xd, Yd, batch, rows=rd, lr=1e-3)
        p64, st = mlp.adam_step(p64, [(W.astype(np.float64), b.astype(np.float64)) for W, b in S.grads()], st, t, 1e-3)
    for (W, b), (oW, ob) in zip(S.params(), p64):
        assert _rel(W, oW) <= 1e-5 and _rel(b, ob) <= 1e-4


@pytest.mark.parametrize("ncol", [1, 127, 129, 300, 1025])
def test_inference_column_counts(gw, ncol):
    import torch
    S, par = _network(gw, 368, 256, 2, 90, 1024, seed=4)
    X = np.random.default_rng(ncol).standard_normal((ncol, 368)).astype(np.float32)
    du = torch.zeros((90, ncol), dtype=torch.float64, device="cuda")
    dv, mask, nfb = torch.zeros_like(du), torch.zeros(ncol, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    S.infer(torch.from_numpy(X).cuda(), du, dv, mask, nfb)
    S.status()
    Yo, _ = mlp.forward([(_bf16(W), b.astype(np.float64)) for W, b in par], _bf16(X))
    got = np.concatenate([du.cpu().numpy(), dv.cpu().numpy()]).T
    assert int(nfb.item()) == 0 and _rel(got, Yo) <= 1e-2


@pytest.mark.parametrize("n_in,hidden,layers,ncol", [(5, 256, 2, 11265), (5, 512, 3, 5889), (70, 512, 2, 10001), (130, 256, 7, 20480), (512, 512, 1, 24673)])
def test_inference_many_columns(gw, n_in, hidden, layers, ncol):
    """Column counts that run all hidden layers in one kernel, with one, two and three row tiles a cluster, inputs
    of one to eight K blocks; the last case in two chunks, the second one short and layer by layer.  Right behind
    a training step the new weights are used."""
    import torch
    S, _ = _network(gw, n_in, hidden, layers, 3, 20480, seed=n_in + hidden)
    r = np.random.default_rng(ncol)
    X, Y = r.standard_normal((ncol, n_in)).astype(np.float32), r.standard_normal((ncol, 6)).astype(np.float32)
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    out = [torch.zeros((6, ncol), dtype=torch.float64, device="cuda") for _ in range(2)]
    mask, nfb = torch.zeros(ncol, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for o in out:
        if o is out[0]:
            S.train_step(Xd, Yd, 1024, lr=1e-2)
        S.infer(Xd, o[:3], o[3:], mask, nfb)
    S.status()
    assert torch.equal(out[0], out[1]) and int(nfb.item()) == 0
    Yo, _ = mlp.forward([(_bf16(W), b.astype(np.float64)) for W, b in S.params()], _bf16(X))
    assert _rel(out[0].cpu().numpy().T, Yo) <= 1e-2


@pytest.mark.parametrize("nlev,ncol", [(1, 130), (1500, 130), (4096, 130), (4096, 20000)])
def test_inference_output_widths(gw, nlev, ncol):
    """Output layers up to the widest one accepted: the epilogue's per-column parameters fit at every tile width."""
    import torch
    S, par = _network(gw, 40, 64, 1, nlev, 20480, seed=nlev)
    X = np.random.default_rng(ncol).standard_normal((ncol, 40)).astype(np.float32)
    du = torch.zeros((nlev, ncol), dtype=torch.float64, device="cuda")
    dv, mask, nfb = torch.zeros_like(du), torch.zeros(ncol, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    S.infer(torch.from_numpy(X).cuda(), du, dv, mask, nfb)
    S.status()
    rows = np.r_[0:65, ncol - 65:ncol]
    Yo, _ = mlp.forward([(_bf16(W), b.astype(np.float64)) for W, b in par], _bf16(X[rows]))
    got = np.concatenate([du[:, rows].cpu().numpy(), dv[:, rows].cpu().numpy()]).T
    assert int(nfb.item()) == 0 and _rel(got, Yo) <= 1e-2


@pytest.mark.parametrize("N", [8192, 8704, 16320])
def test_gemm_wide_with_bias(gw, N):
    """The tile width picked for few rows and many columns leaves room for the bias (bar of test_gpu_gemm.py)."""
    import ctypes as C
    import torch
    g = torch.Generator().manual_seed(N)
    A, B = torch.randn(100, 64, generator=g).to(torch.bfloat16), (torch.randn(N, 64, generator=g) / 8).to(torch.bfloat16)
    b = torch.randn(N, generator=g).float()
    Ad, Bd, bd, Cd = A.cuda(), B.cuda(), b.cuda(), torch.full((100, N), float("nan"), dtype=torch.float32, device="cuda")
    p = lambda t: C.c_void_p(t.data_ptr())
    assert gw.lib().gwam_gemm_bf16(p(Ad), p(Bd), 100, N, 64, p(bd), 0, 0, 0, p(Cd),
                                   C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    z, S = A.double() @ B.double().T + b.double(), A.double().abs() @ B.double().abs().T
    assert ((Cd.cpu().double() - z).abs() <= 2e-5 * S + 1e-6 * z.abs()).all()
