"""fc1 -> GELU -> fc2 with the activation fused behind the products, through the C ABI, against the oracle.

Each call is checked on its own inputs: the second layer's forward takes the H the library produced (its bf16 bits,
widened exactly), and the derivative is taken at the stored pre-activation bits, so no error carries across calls.
"""
import numpy as np
import pytest

import mst_inputs
import oracle
from oracle import activation as act

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    import paper_2408_11746_b200 as mst
    from gpu_util import TOL, dev, host, make_layer, rel_err, tdtype, to_dev


def _pre_activation(T, C, dtype, seed):
    y = mst_inputs.normal((T, C), 1.5, seed, 77)
    if dtype == "bf16":
        bits = mst_inputs.f32_to_bf16_bits(y)
        return mst_inputs.bf16_bits_to_f32(bits), torch.from_numpy(bits.view(np.int16)).to(dev()).view(torch.bfloat16)
    return y, torch.from_numpy(y).to(dev())


def _padded(t, ld):
    buf = torch.full((t.shape[0], ld), float("nan"), dtype=t.dtype, device=t.device)
    buf[:, : t.shape[1]] = t
    return buf


@pytest.mark.parametrize("dtype,path", [("bf16", "tensor"), ("bf16", "cuda_core"), ("f32", "cuda_core")])
@pytest.mark.parametrize("T,d,hid", [(300, 200, 520), (129, 64, 264), (1, 40, 72)])
def test_mlp_pair_small(dtype, path, T, d, hid):
    m1 = mst_inputs.uniform_mask(hid, d, mst_inputs.exact_nnz(hid, d, 0.3), 901, 1)
    m2 = mst_inputs.uniform_mask(d, hid, mst_inputs.exact_nnz(d, hid, 0.3), 901, 2)
    p1 = mst_inputs.make_layer("fc1", 1, hid, d, T, dtype, m1, 901, w_std=0.25)
    p2 = mst_inputs.make_layer("fc2", 2, d, hid, T, dtype, m2, 901, w_std=0.05)
    L1, L2 = make_layer(p1), make_layer(p2)
    for L in (L1, L2):
        L.set_path(mst.MST_PATH_TENSOR_CORE if path == "tensor" else mst.MST_PATH_CUDA_CORE)
    tol = TOL[dtype]
    X = to_dev(p1, "X")
    H = torch.empty((T, hid), dtype=tdtype(p1), device=dev())
    Ypre = torch.empty((T, hid), dtype=tdtype(p1), device=dev())
    L1.fwd_gelu(X, H, T, Y_pre=Ypre)
    H_only = torch.empty_like(H)
    L1.fwd_gelu(X, H_only, T)                       # without the pre-activation output
    torch.cuda.synchronize()
    Y1 = oracle.fwd(p1.X, p1.W, p1.mask)
    assert np.abs(Y1).max() > 2.0                    # the inputs reach both tails of the activation
    assert rel_err(host(Ypre), Y1) <= tol
    assert rel_err(host(H), act.gelu(Y1)) <= tol
    if dtype == "bf16" and path == "cuda_core":
        # without a pre-activation buffer the CUDA-core route rounds the product to bf16 before the activation
        assert rel_err(host(H_only), act.gelu(Y1)) <= tol
    else:
        assert torch.equal(H_only, H)
    # second layer on the H just produced
    Y2 = torch.empty((T, d), dtype=tdtype(p1), device=dev())
    L2.fwd(H, Y2, T)
    torch.cuda.synchronize()
    assert rel_err(host(Y2), oracle.fwd(host(H), p2.W, p2.mask)) <= tol
    # backward through fc2 and the activation in one call, derivative at given pre-activation bits
    pre_host, pre_dev = _pre_activation(T, hid, dtype, 33)
    dY = to_dev(p2, "dY")
    dPre = torch.empty((T, hid), dtype=tdtype(p1), device=dev())
    L2.bwd_x_gelu(dY, pre_dev, dPre, T)
    torch.cuda.synchronize()
    ref = oracle.bwd_x(p2.dY, p2.W, p2.mask) * act.gelu_grad(pre_host)
    assert rel_err(host(dPre), ref) <= tol
    # padded leading dimensions (the ragged store paths) give the same bits
    ld = hid + 8 if dtype == "bf16" else hid + 3
    Hp = torch.full((T, ld), float("nan"), dtype=H.dtype, device=dev())
    Yp = torch.full((T, ld), float("nan"), dtype=H.dtype, device=dev())
    mst.mst_spmm_fwd_gelu(L1.handle, X, d, T, Yp, ld, Hp, ld)
    dPp = torch.full((T, ld), float("nan"), dtype=H.dtype, device=dev())
    mst.mst_spmm_bwd_x_gelu(L2.handle, dY, d, T, _padded(pre_dev, ld), ld, dPp, ld)
    torch.cuda.synchronize()
    assert torch.equal(Hp[:, :hid], H) and torch.equal(Yp[:, :hid], Ypre) and torch.equal(dPp[:, :hid], dPre)
    assert torch.isnan(Hp[:, hid:]).all() and torch.isnan(dPp[:, hid:]).all()
    L1.close(); L2.close()
    assert mst.mst_device_error_flags() == 0


def test_mlp_pair_argument_errors():
    p = mst_inputs.uniform_layer("fc1", 1, 64, 32, 16, "bf16", 0.5, 5)
    L = make_layer(p)
    X = to_dev(p, "X")
    H = torch.empty((16, 64), dtype=torch.bfloat16, device=dev())
    with pytest.raises(mst.MstError) as e:
        mst.mst_spmm_fwd_gelu(L.handle, X, 32, 16, None, 0, H, 63)
    assert e.value.status == 2            # MST_ERR_SHAPE
    with pytest.raises(mst.MstError) as e:
        mst.mst_spmm_fwd_gelu(L.handle, X, 32, 16, H, 8, H, 64)
    assert e.value.status == 2            # MST_ERR_SHAPE
    with pytest.raises(mst.MstError) as e:
        mst.mst_spmm_bwd_x_gelu(L.handle, H, 64, 16, None, 32, X, 32)
    assert e.value.status == 1      # MST_ERR_INVALID_ARG
    mst.mst_spmm_fwd_gelu(L.handle, X, 32, 0, None, 0, H, 64)      # no tokens: nothing to do
    L.close()


def test_mlp_pair_gpt2_small_full_size():
    rng = np.random.default_rng(8)
    ps = {p.name: p for p in mst_inputs.config2()}
    p1, p2 = ps["fc1"], ps["fc2"]
    T, d, hid = p1.tokens, p1.in_features, p1.out_features
    L1, L2 = make_layer(p1), make_layer(p2)
    X = to_dev(p1, "X")
    H = torch.empty((T, hid), dtype=torch.bfloat16, device=dev())
    Ypre = torch.empty_like(H)
    L1.fwd_gelu(X, H, T, Y_pre=Ypre)
    pre_host, pre_dev = _pre_activation(T, hid, "bf16", 34)
    dPre = torch.empty_like(H)
    L2.bwd_x_gelu(to_dev(p2, "dY"), pre_dev, dPre, T)
    torch.cuda.synchronize()
    n = 3000
    t = rng.integers(0, T, n); o = rng.integers(0, hid, n)
    ti, oi = torch.from_numpy(t).to(dev()), torch.from_numpy(o).to(dev())
    y = oracle.fwd_at(p1.X, p1.W, p1.mask, t, o)
    assert rel_err(host(Ypre[ti, oi]), y) <= TOL["bf16"]
    assert rel_err(host(H[ti, oi]), act.gelu(y)) <= TOL["bf16"]
    ref = oracle.bwd_x_at(p2.dY, p2.W, p2.mask, t, o) * act.gelu_grad(pre_host[t, o])
    assert rel_err(host(dPre[ti, oi]), ref) <= TOL["bf16"]
    L1.close(); L2.close()
    assert mst.mst_device_error_flags() == 0


@pytest.mark.parametrize("T,d,hid", [(257, 64, 64), (300, 72, 136), (384, 136, 200), (513, 64, 328), (1000, 264, 776)])
def test_activation_boxes_at_tile_edges(monkeypatch, T, d, hid):
    """The 256-row kernel's activation: groups of 64 columns cut by the matrix, half-wide tiles, rows past the last box.
    Tolerance: one bf16 rounding (2^-9) of each stored value plus the operand sums' 2^-24 a term, under 2e-2 of the largest."""
    monkeypatch.setenv("MST_TC_PAIR", "1")
    m1 = mst_inputs.uniform_mask(hid, d, mst_inputs.exact_nnz(hid, d, 0.3), 902, 1)
    m2 = mst_inputs.uniform_mask(d, hid, mst_inputs.exact_nnz(d, hid, 0.3), 902, 2)
    p1 = mst_inputs.make_layer("fc1", 1, hid, d, T, "bf16", m1, 902, w_std=0.25)
    p2 = mst_inputs.make_layer("fc2", 2, d, hid, T, "bf16", m2, 902, w_std=0.05)
    L1, L2 = make_layer(p1), make_layer(p2)
    X, dY = to_dev(p1, "X"), to_dev(p2, "dY")
    H, Ypre, H_only, dPre = (torch.full((T + 1, hid), float("nan"), dtype=torch.bfloat16, device=dev()) for _ in range(4))
    L1.fwd_gelu(X, H, T, Y_pre=Ypre)
    L1.fwd_gelu(X, H_only, T)
    pre_host, pre_dev = _pre_activation(T, hid, "bf16", 35)
    L2.bwd_x_gelu(dY, pre_dev, dPre, T)
    torch.cuda.synchronize()
    Y1 = oracle.fwd(p1.X, p1.W, p1.mask)
    assert rel_err(host(Ypre[:T]), Y1) <= TOL["bf16"]
    assert rel_err(host(H[:T]), act.gelu(Y1)) <= TOL["bf16"]
    assert torch.equal(H_only[:T], H[:T])
    assert rel_err(host(dPre[:T]), oracle.bwd_x(p2.dY, p2.W, p2.mask) * act.gelu_grad(pre_host)) <= TOL["bf16"]
    for t in (H, Ypre, H_only, dPre):
        assert torch.isnan(t[T]).all()                # the row after the last is untouched
    # sums that overflow: x Phi(x) is +inf at +inf and NaN at -inf
    big = torch.zeros((T, d), dtype=torch.bfloat16, device=dev())
    row = int(np.argmax((np.abs(p1.W) * p1.mask).max(1)))
    col = int(np.argmax(np.abs(p1.W[row]) * p1.mask[row]))
    big[0, col] = 3.0e38 * float(np.sign(p1.W[row, col]))
    big[1, col] = -big[0, col]
    one = mst.Layer(3, hid, d, mst.MST_BF16)
    one.pack(to_dev(p1, "W") * 1e3, torch.from_numpy(p1.mask).to(dev()))
    one.fwd_gelu(big, H, T)
    torch.cuda.synchronize()
    assert torch.isposinf(H[0, row]) and torch.isnan(H[1, row]) and bool((H[2:T] == 0).all())
    one.close(); L1.close(); L2.close()
    assert mst.mst_device_error_flags() == 0


@pytest.mark.parametrize("pairs", ["1", "0"])
@pytest.mark.parametrize("T,O,I,pad,shift", [(300, 200, 136, 1, 0), (257, 328, 64, 2, 1), (513, 72, 72, 0, 4), (77, 33, 40, 0, 0)])
def test_pre_activation_of_any_pitch(monkeypatch, pairs, T, O, I, pad, shift):
    """Pre-activations that TMA does not take: the very values of the call whose rows it does, and the derivative in place."""
    monkeypatch.setenv("MST_TC_PAIR", pairs)
    g = torch.Generator(device="cuda").manual_seed(O + T)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()
    X, dY, W1, W2 = n(T, I), n(T, I), n(O, I), n(I, O)
    M1, M2 = ((torch.rand(s, generator=g, device="cuda") < 0.4).to(torch.uint8) for s in ((O, I), (I, O)))
    L1, L2 = mst.Layer(0, O, I, mst.MST_BF16), mst.Layer(1, I, O, mst.MST_BF16)
    L1.pack(W1, M1)
    L2.pack(W2, M2)
    even = (O + 7) // 8 * 8
    outs = []
    for ld, off in ((even, 0), (O + pad, shift)):
        whole = torch.full((T * ld + off + 8,), float("nan"), dtype=torch.bfloat16, device="cuda")
        pre = whole[off:off + T * ld].view(T, ld)
        H, dP = (torch.full((T, even), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        mst.mst_spmm_fwd_gelu(L1.handle, X, I, T, pre, ld, H, even)
        kept = pre[:, :O].clone()
        mst.mst_spmm_bwd_x_gelu(L2.handle, dY, I, T, pre, ld, dP, even)
        assert torch.equal(pre[:, :O], kept) and bool(torch.isnan(pre[:, O:]).all()) and bool(torch.isnan(whole[off + T * ld:]).all())
        mst.mst_spmm_bwd_x_gelu(L2.handle, dY, I, T, pre, ld, pre, ld)
        torch.cuda.synchronize()
        outs.append((H[:, :O].clone(), kept, dP[:, :O].clone(), pre[:, :O].clone()))
        assert bool(torch.isnan(H[:, O:]).all()) and bool(torch.isnan(dP[:, O:]).all())
    assert mst.mst_device_error_flags() == 0
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    assert torch.equal(outs[1][2], outs[1][3])
    x = X.double() @ (W1.double() * M1).T
    assert float((outs[1][0].double() - x * 0.5 * (1 + torch.erf(x / 2 ** 0.5))).norm()) <= 1e-2 * float(x.norm())
    L1.close()
    L2.close()


@pytest.mark.parametrize("pairs", ["1", "0"])
@pytest.mark.parametrize("T,hid,pitch", [(5000, 1288, 1288), (4993, 1283, 1288), (5000, 1283, 1283)])
def test_activation_of_later_tiles(monkeypatch, pairs, T, hid, pitch):
    """More tiles than run at once, so that a block goes on to a second one, whose pre-activations are on their way by then: last columns of 8,
    of 3 behind whole pieces, and rows that TMA does not take.  Every element: the sum's bf16 operands are exact and its fp32 terms lose 2^-24
    each of their magnitudes (64 terms, 2^-18 of their sum), the published erf form 2^-19 absolute and the unit's exponential and reciprocal
    less; one bf16 rounding, 2^-8 of the value."""
    monkeypatch.setenv("MST_TC_PAIR", pairs)
    I = 64
    g = torch.Generator(device="cuda").manual_seed(T + hid)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()
    X, dY, W1, W2 = n(T, I), n(T, I), n(hid, I), n(I, hid)
    M1, M2 = ((torch.rand(s, generator=g, device="cuda") < 0.3).to(torch.uint8) for s in ((hid, I), (I, hid)))
    L1, L2 = mst.Layer(0, hid, I, mst.MST_BF16), mst.Layer(1, I, hid, mst.MST_BF16)
    L1.pack(W1, M1)
    L2.pack(W2, M2)
    H, pre, at, dP = (torch.full((T, pitch), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(4))
    at[:, :hid] = n(T, hid) * 2
    mst.mst_spmm_fwd_gelu(L1.handle, X, I, T, pre, pitch, H, pitch)
    mst.mst_spmm_bwd_x_gelu(L2.handle, dY, I, T, at, pitch, dP, pitch)
    torch.cuda.synchronize()
    assert mst.mst_device_error_flags() == 0
    phi = lambda x: 0.5 * (1 + torch.erf(x / 2 ** 0.5))
    w1, w2, a = W1.double() * M1, W2.double() * M2, at[:, :hid].double()
    y, size = X.double() @ w1.T, X.double().abs() @ w1.abs().T
    d, dsize = dY.double() @ w2, dY.double().abs() @ w2.abs()
    slope = phi(a) + a * torch.exp(-a * a / 2) / (2 * torch.pi) ** 0.5
    for got, ref, magnitude in ((pre, y, size), (H, y * phi(y), size * 1.13 + y.abs()), (dP, d * slope, dsize * slope.abs() + d.abs())):
        over = (got[:, :hid].double() - ref).abs() - (ref.abs() * 2.0 ** -8 + magnitude * 2.0 ** -18)
        assert float(over.max()) <= 0, (float(over.max()), int(over.argmax()))
        assert torch.isnan(got[:, hid:]).all()
    L1.close()
    L2.close()
