"""Infinite and NaN operands.  fp32 layers, and bf16 calls on rows the TMA unit does not take, go by the stored entries alone: such a
value reaches the outputs connected to it and no others, with the sign that arithmetic gives it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2408_11746_b200 as mst  # noqa: E402

INF, NAN = float("inf"), float("nan")


def _finite(a):
    return torch.where(a.isfinite(), a, torch.zeros_like(a))


def _product(A, W, M):
    """sum over stored (o, k) of A[t, k] W[o, k] in fp64"""
    A, W, M = A.double(), W.double(), M.bool()
    zero = torch.zeros((), dtype=torch.double, device=A.device)
    R = _finite(A) @ torch.where(M, _finite(W), zero).T
    for t in (~A.isfinite()).any(1).nonzero().flatten().tolist():
        R[t] = torch.where(M, A[t][None, :] * W, zero).sum(1)
    for o in (M & ~W.isfinite()).any(1).nonzero().flatten().tolist():
        R[:, o] = torch.where(M[o], A * W[o], zero).sum(1)
    return R


def _gradient(D, X):
    D, X = D.double(), X.double()
    G = _finite(D).T @ _finite(X)
    for o in (~D.isfinite()).any(0).nonzero().flatten().tolist():
        G[o] = (D[:, o, None] * X).sum(0)
    for i in (~X.isfinite()).any(0).nonzero().flatten().tolist():
        G[:, i] = (D * X[:, i, None]).sum(0)
    return G


def _same(got, ref, tol):
    got = got.double()
    assert torch.equal(got.isnan(), ref.isnan())
    for sign in (INF, -INF):
        assert torch.equal(got == sign, ref == sign)
    a, b = _finite(got), _finite(ref)
    assert float((a - b).norm()) <= tol * float(b.norm())


def _phi(x):
    return 0.5 * (1 + torch.erf(x / 2 ** 0.5))


def _case(O, I, T, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt, mdt = (torch.float32, mst.MST_F32) if dtype == "f32" else (torch.bfloat16, mst.MST_BF16)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda").to(dt)
    X, dY, W = n(T, I), n(T, O), n(O, I)
    M = (torch.rand(O, I, generator=g, device="cuda") < 0.3).to(torch.uint8)
    M[0, :4], M[1, :4] = 1, 0
    for A, K in ((X, I), (dY, O)):
        A[1 % T, 3] = INF
        A[T // 2, K - 1], A[T // 2, 2] = -INF, INF
        A[T - 1, K // 2] = NAN
    W[O - 1, I // 3], M[O - 1, I // 3] = INF, 1
    W[O // 2, I - 1], M[O // 2, I - 1] = NAN, 1
    W[1, 1] = INF                                # under a zero of the mask
    L = mst.Layer(0, O, I, mdt)
    L.pack(W, M)
    return X, dY, W, M, L, dt, mdt


def _products(O, I, T, dtype, tol, seed):
    X, dY, W, M, L, dt, _ = _case(O, I, T, dtype, seed)
    Y, dX = torch.zeros(T, O, dtype=dt, device="cuda"), torch.zeros(T, I, dtype=dt, device="cuda")
    L.fwd(X, Y, T)
    L.bwd_x(dY, dX, T)
    fwd, bwd = _product(X, W, M), _product(dY, W.T, M.T)
    _same(Y, fwd, tol)
    _same(dX, bwd, tol)
    # with the activation behind them
    pre, H = torch.zeros_like(Y), torch.zeros_like(Y)
    L.fwd_gelu(X, H, T, Y_pre=pre)
    _same(pre, fwd, tol)
    _same(H, fwd * _phi(fwd), tol)
    at = torch.randn(T, I, device="cuda").to(dt)
    L.bwd_x_gelu(dY, at, dX, T)
    a = at.double()
    _same(dX, bwd * (_phi(a) + a * torch.exp(-a * a / 2) / (2 * torch.pi) ** 0.5), tol)
    assert mst.mst_device_error_flags() == 0
    L.close()


@pytest.mark.parametrize("O,I,T", [(70, 90, 40), (100, 1000, 130), (1030, 300, 700), (3072, 768, 256)])
def test_fp32_products(O, I, T):
    _products(O, I, T, "f32", 1e-6, O)


@pytest.mark.parametrize("O,I,T", [(70, 90, 40), (100, 60, 3000), (1030, 300, 200)])
def test_fp32_gradients(O, I, T):
    X, dY, _, M, L, _, mdt = _case(O, I, T, "f32", O + 1)
    G, G2, dW, dW2 = torch.zeros(O, I, device="cuda"), torch.zeros(O, I, device="cuda"), torch.zeros(L.nnz, device="cuda"), torch.zeros(L.nnz, device="cuda")
    L.sddmm(dY, X, T, dW)
    L.dense_grad(dY, X, T, G)
    L.dense_grad_dw(dY, X, T, G2, dW2)
    ref = _gradient(dY, X)
    for got in (G, G2):
        _same(got, ref, 1e-6)
    for got in (dW, dW2):
        _same(got, ref[M.bool()], 1e-6)
    assert mst.mst_device_error_flags() == 0
    L.close()


@pytest.mark.parametrize("O,I,T", [
    (520, 519, 12),      # the few-token kernel on copied rows
    (519, 520, 7),       # rows of the output start anywhere
    (130, 91, 100),      # small tiles
    (515, 136, 300),
    (1100, 515, 6000),   # block pairs, rows of both results start anywhere
    (1104, 515, 6000),   # forward: copied rows, results by TMA
    (515, 1104, 6000)])  # input gradient: the same
def test_bf16_rows_that_start_anywhere(O, I, T):
    _products(O, I, T, "bf16", 1e-2, O)


def test_every_sum_not_finite():
    # a diverged run: all of it is formed again
    O, I, T = 770, 130, 600
    X, dY, W, M, L, dt, _ = _case(O, I, T, "f32", 5)
    X[:] = torch.where(torch.rand(T, I, device="cuda") < 0.2, torch.full_like(X, INF), X)
    Y, dW = torch.zeros(T, O, device="cuda"), torch.zeros(L.nnz, device="cuda")
    L.fwd(X, Y, T)
    L.sddmm(dY, X, T, dW)
    _same(Y, _product(X, W, M), 1e-6)
    _same(dW, _gradient(dY, X)[M.bool()], 1e-6)
    L.close()
