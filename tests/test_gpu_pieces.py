"""fp32 layers on the tensor cores (three exact bf16 pieces per operand) and bf16 layers whose rows start anywhere or whose outputs have few tiles:
edges of the 128 x 64 / 128 x 128 tiles and of the 64-wide contraction blocks, against an fp64 product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2408_11746_b200 as mst  # noqa: E402


def _rel(got, ref):
    return float((got.double() - ref).norm() / ref.norm().clamp_min(1e-300))


def _layer_case(O, I, T, dtype, density, seed, pad=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt, mdt = (torch.float32, mst.MST_F32) if dtype == "f32" else (torch.bfloat16, mst.MST_BF16)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda").to(dt)
    X, dY, W = n(T, I + pad), n(T, O + pad), n(O, I)
    M = (torch.rand(O, I, generator=g, device="cuda") < density).to(torch.uint8)
    M[0, 0] = 1
    L = mst.Layer(0, O, I, mdt)
    L.pack(W, M)
    Y = torch.full((T, O + pad), float("nan"), dtype=dt, device="cuda")
    dX = torch.full((T, I + pad), float("nan"), dtype=dt, device="cuda")
    dW = torch.full((L.nnz,), float("nan"), device="cuda")
    G = torch.full((O, I), float("nan"), device="cuda")
    mst.mst_spmm_fwd(L.handle, X, I + pad, T, Y, O + pad)
    mst.mst_spmm_bwd_x(L.handle, dY, O + pad, T, dX, I + pad)
    mst.mst_sddmm_dw(L.handle, dY, O + pad, X, I + pad, T, dW)
    mst.mst_dense_grad(dY, O + pad, X, I + pad, T, O, I, mdt, G)
    assert mst.mst_device_error_flags() == 0
    Xr, dYr, Wr = X[:, :I].double(), dY[:, :O].double(), (W * M.to(dt)).double()
    Gr = dYr.T @ Xr
    if pad:                                     # columns beyond the matrix are not written
        assert bool(Y[:, O:].isnan().all()) and bool(dX[:, I:].isnan().all())
    out = (_rel(Y[:, :O], Xr @ Wr.T), _rel(dX[:, :I], dYr @ Wr), _rel(dW, Gr[M.bool()]), _rel(G, Gr))
    L.close()
    return out


@pytest.mark.parametrize("O,I,T", [(1, 1, 1), (64, 64, 64), (65, 63, 129), (128, 128, 128), (127, 257, 65), (300, 40, 1000),
                                   (40, 2050, 33), (2051, 130, 257)])
def test_fp32_products_are_single_precision(O, I, T):
    for err in _layer_case(O, I, T, "f32", 0.3, O + I + T):
        assert err <= 5e-7


@pytest.mark.parametrize("x,w", [(-118, 0), (0, -118), (-142, 60), (60, -142), (-60, -58), (116, -20), (-20, 116), (100, 10)])
def test_fp32_pieces_over_the_whole_range(x, w):
    # operands of size 2^x (activations, upstream gradients) and 2^w (weights; the other gradient operand), down to subnormal ones and
    # up to where sums pass 2^95; results stay in the normal range and keep single precision relative to the sum of their terms' sizes
    O, I, T = 130, 200, 140
    g = torch.Generator(device="cuda").manual_seed(x - w)
    n = lambda e, *s: (torch.randn(*s, generator=g, device="cuda", dtype=torch.double) * 2.0 ** e).float()
    X, dY, W, V = n(x, T, I), n(x, T, O), n(w, O, I), n(w, T, I)
    M = (torch.rand(O, I, generator=g, device="cuda") < 0.4).to(torch.uint8)
    L = mst.Layer(0, O, I, mst.MST_F32)
    L.pack(W, M)
    Y, dX = torch.zeros(T, O, device="cuda"), torch.zeros(T, I, device="cuda")
    dW, G = torch.zeros(L.nnz, device="cuda"), torch.zeros(O, I, device="cuda")
    L.fwd(X, Y, T)
    L.bwd_x(dY, dX, T)
    L.sddmm(dY, V, T, dW)
    L.dense_grad(dY, V, T, G)
    Wr = (W * M).double()
    Gr = dY.double().T @ V.double()
    for got, ref in ((Y, X.double() @ Wr.T), (dX, dY.double() @ Wr), (G, Gr), (dW, Gr[M.bool()])):
        assert _rel(got, ref) <= 5e-7
    L.close()


def test_fp32_extreme_magnitudes():
    # pieces of values near the top and the bottom of the normal range; sums stay finite
    O, I, T = 70, 66, 40
    X = torch.zeros(T, I, device="cuda")
    X[:, 0], X[:, 1] = 3.4028234e38, 1e-30
    W = torch.zeros(O, I, device="cuda")
    W[:, 0], W[:, 1] = 0.99999994, 1.0
    L = mst.Layer(0, O, I, mst.MST_F32)
    L.pack(W, torch.ones(O, I, dtype=torch.uint8, device="cuda"))
    Y = torch.empty(T, O, device="cuda")
    L.fwd(X, Y, T)
    ref = X.double() @ W.double().T
    assert bool(torch.isfinite(Y).all()) and float(((Y.double() - ref) / ref).abs().max()) <= 3e-7
    L.close()


@pytest.mark.parametrize("O,I,T,pad", [(65, 63, 129, 0), (255, 257, 300, 0), (64, 128, 130, 3), (513, 31, 520, 5), (1, 3, 1, 0)])
def test_bf16_rows_at_any_address(O, I, T, pad):
    y, dx, dw, g = _layer_case(O, I, T, "bf16", 0.3, O + I + T, pad)
    assert y <= 4e-3 and dx <= 4e-3 and dw <= 1e-5 and g <= 1e-5


@pytest.mark.parametrize("O,I,T", [(2304, 768, 8), (2304, 768, 9), (770, 3080, 16), (768, 3072, 17), (136, 200, 128), (1280, 1288, 40), (16, 8, 3)])
def test_bf16_products_of_few_tiles(O, I, T):
    # the latency kernel up to 16 tokens, small tiles with the contraction range split over a cluster above
    y, dx, dw, g = _layer_case(O, I, T, "bf16", 0.2, O + I + T)
    assert y <= 4e-3 and dx <= 4e-3 and dw <= 1e-5 and g <= 1e-5


@pytest.mark.parametrize("O,I,T,dtype", [(1, 1, 1, "f32"), (65, 63, 129, "f32"), (128, 33, 64, "f32"), (300, 40, 1000, "f32"), (2051, 130, 257, "f32"),
                                         (1, 3, 1, "bf16"), (129, 31, 65, "bf16"), (255, 257, 300, "bf16"), (513, 96, 1500, "bf16")])
def test_dense_gradient_of_small_tiles_with_its_entries(O, I, T, dtype):
    # the entries under the mask leave with the tile: the very values of the matrix, which are those without entries
    g = torch.Generator(device="cuda").manual_seed(O + I)
    dt, mdt = (torch.float32, mst.MST_F32) if dtype == "f32" else (torch.bfloat16, mst.MST_BF16)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda").to(dt)
    X, dY, W = n(T, I), n(T, O), n(O, I)
    M = (torch.rand(O, I, generator=g, device="cuda") < 0.3).to(torch.uint8)
    M[0, 0] = 1
    L = mst.Layer(0, O, I, mdt)
    L.pack(W, M)
    G, both = torch.full((O, I), float("nan"), device="cuda"), torch.full((O, I), float("nan"), device="cuda")
    dW = torch.full((L.nnz,), float("nan"), device="cuda")
    L.dense_grad(dY, X, T, G)
    L.dense_grad_dw(dY, X, T, both, dW)
    assert mst.mst_device_error_flags() == 0
    assert torch.equal(G, both) and torch.equal(dW, both[M.bool()])
    assert _rel(G, dY.double().T @ X.double()) <= 1e-5
    L.close()


@pytest.mark.parametrize("O,I,T,pad", [
    (96, 96, 1024, 0), (96, 96, 1025, 0),      # the most tokens the latency kernel takes, and one more
    (200, 136, 600, 0), (2304, 768, 33, 0), (5120, 1280, 17, 0), (300, 4096, 31, 0), (17, 40, 257, 0), (333, 777, 250, 3), (1280, 1288, 64, 0)])
def test_forward_of_a_few_hundred_tokens(O, I, T, pad):
    # the latency kernel or the small tiles, by their estimates
    y, dx, dw, g = _layer_case(O, I, T, "bf16", 0.2, O + I + T, pad)
    assert y <= 4e-3 and dx <= 4e-3 and dw <= 1e-5 and g <= 1e-5


@pytest.mark.parametrize("O,I,T,kernel", [
    (768, 768, 16, "small_fwd_kernel"), (768, 768, 64, "small_fwd_kernel"), (300, 4096, 31, "small_fwd_kernel"), (17, 40, 257, "small_fwd_kernel"),
    (1280, 1288, 512, "tc_split_kernel"), (3712, 114, 717, "tc_gemm_pair_kernel"), (96, 96, 1025, "tc_split_kernel"), (2048, 2048, 4000, "tc_gemm_pair_kernel")])
def test_kernel_of_a_forward_call(O, I, T, kernel):
    # sizes for which the estimates lie a factor 1.2 or more apart, or that are outside of a kernel's range
    from torch.profiler import ProfilerActivity, profile
    n = lambda *s: torch.randn(*s, device="cuda").bfloat16()
    L = mst.Layer(0, O, I, mst.MST_BF16)
    L.pack(n(O, I), (torch.rand(O, I, device="cuda") < 0.2).to(torch.uint8))
    X, Y = n(T, I), torch.empty(T, O, dtype=torch.bfloat16, device="cuda")
    L.fwd(X, Y, T)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as seen:
        L.fwd(X, Y, T)
        torch.cuda.synchronize()
    names = [e.name for e in seen.events() if "_kernel" in e.name and "prepare" not in e.name]
    assert len(names) == 1 and kernel in names[0], names
    L.close()


@pytest.mark.parametrize("O,I,T,density", [
    (5120, 1280, 8190, 0.1),     # 100 tiles on 74 pairs: 26 cut in two
    (3840, 1250, 8000, 0.3),     # 75 tiles: one cut, the others whole; ragged columns
    (1300, 1290, 9000, 0.1)])    # ragged rows and columns, nothing cut
def test_gradients_with_a_cut_last_wave(O, I, T, density):
    g = torch.Generator(device="cuda").manual_seed(O + I)
    mask = (torch.rand((O, I), device="cuda", generator=g) < density).to(torch.uint8)
    L = mst.Layer(0, O, I, mst.MST_BF16)
    L.pack(torch.ones((O, I), dtype=torch.bfloat16, device="cuda"), mask)
    dY = torch.randn((T, O), device="cuda", generator=g).bfloat16()
    X = torch.randn((T, I), device="cuda", generator=g).bfloat16()
    dW = torch.full((L.nnz,), float("nan"), device="cuda")
    G = torch.full((O, I), float("nan"), device="cuda")
    L.sddmm(dY, X, T, dW)
    L.dense_grad(dY, X, T, G)
    ref = dY.double().t() @ X.double()
    for got, want in ((dW.double(), ref[mask.bool()]), (G.double(), ref)):
        assert float((got - want).norm() / want.norm()) < 1e-5
    assert mst.mst_device_error_flags() == 0


@pytest.mark.parametrize("O,I,density,rows", [
    (64, 96, 0.02, None),        # few entries: half a word per thread
    (70, 1030, 0.27, None),      # blocks on either side of the choice, ragged rows
    (130, 200, 0.05, 3)])        # three full rows among sparse ones
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_pack_few_and_many_entries(O, I, density, rows, dtype):
    g = torch.Generator(device="cuda").manual_seed(O * I)
    mask = (torch.rand((O, I), device="cuda", generator=g) < density).to(torch.uint8)
    if rows:
        mask[5:5 + rows] = 1
    dt, mdt = (torch.float32, mst.MST_F32) if dtype == "f32" else (torch.bfloat16, mst.MST_BF16)
    W = torch.randn((O, I), device="cuda", generator=g).to(dt)
    L = mst.Layer(0, O, I, mdt)
    L.pack(W, mask)
    nnz = int(mask.sum())
    assert L.nnz == nnz
    ptr = torch.zeros(O + 1, dtype=torch.int32, device="cuda")
    col = torch.zeros(nnz, dtype=torch.int32, device="cuda")
    val = torch.zeros(nnz, dtype=dt, device="cuda")
    mst.mst_export_csr(L.handle, ptr, col, val)
    at = mask.bool().nonzero()
    assert torch.equal(col.long(), at[:, 1]) and torch.equal(val, W[mask.bool()])
    assert torch.equal(ptr[1:].long(), mask.sum(1).cumsum(0))


@pytest.mark.parametrize("T,O,I", [(1, 40, 1025), (9, 17, 2049), (16, 33, 3072), (7, 24, 2040)])   # 8, 16 and 24 warps, partial chunks
def test_few_tokens_long_rows(T, O, I):
    g = torch.Generator(device="cuda").manual_seed(T + O + I)
    W = torch.randn((O, I), device="cuda", generator=g).bfloat16()
    mask = (torch.rand((O, I), device="cuda", generator=g) < 0.2).to(torch.uint8)
    mask[0, 0] = 1
    L = mst.Layer(0, O, I, mst.MST_BF16)
    L.pack(W, mask)
    X = torch.randn((T, I), device="cuda", generator=g).bfloat16()
    Y = torch.full((T, O), float("nan"), dtype=torch.bfloat16, device="cuda")
    L.fwd(X, Y, T)
    assert _rel(Y, X.double() @ (W.double() * mask.double()).t()) < 4e-3


@pytest.mark.parametrize("O,I,T,density", [
    (96, 264, 700, 0.1),         # small tiles: a pass over the dense gradient
    (768, 1284, 4096, 0.06),     # two or more ranges: both results from the partial sums; half a word at the end of a row
    (3840, 1280, 8190, 0.1),     # one tile of the last wave cut
    (515, 770, 3000, 0.2)])      # columns that four do not divide
def test_dense_gradient_and_its_entries(O, I, T, density):
    g = torch.Generator(device="cuda").manual_seed(O * 7 + I)
    mask = (torch.rand((O, I), device="cuda", generator=g) < density).to(torch.uint8)
    L = mst.Layer(0, O, I, mst.MST_BF16)
    L.pack(torch.ones((O, I), dtype=torch.bfloat16, device="cuda"), mask)
    dY = torch.randn((T, O), device="cuda", generator=g).bfloat16()
    X = torch.randn((T, I), device="cuda", generator=g).bfloat16()
    dW = torch.full((L.nnz,), float("nan"), device="cuda")
    G = torch.full((O, I), float("nan"), device="cuda")
    L.dense_grad_dw(dY, X, T, G, dW)
    assert _rel(G, dY.double().t() @ X.double()) < 1e-5
    assert torch.equal(dW, G[mask.bool()])


@pytest.mark.parametrize("O,I,T", [(192, 200, 34), (256, 192, 130), (72, 320, 60), (40, 1032, 67), (24, 2056, 129)])   # last rows of a tile 1 to 31, clusters of 1 to 8
def test_activation_rows_of_a_partial_tile(O, I, T):
    g = torch.Generator(device="cuda").manual_seed(O + I + T)
    W = (torch.randn((O, I), device="cuda", generator=g) / I ** 0.5).bfloat16()
    mask = (torch.rand((O, I), device="cuda", generator=g) < 0.3).to(torch.uint8)
    mask[0, 0] = 1
    L, Lt = mst.Layer(0, O, I, mst.MST_BF16), mst.Layer(1, I, O, mst.MST_BF16)
    L.pack(W, mask)
    Lt.pack(W.t().contiguous(), mask.t().contiguous())
    X, pre = torch.randn((T, I), device="cuda", generator=g).bfloat16(), torch.randn((T, O), device="cuda", generator=g).bfloat16()
    H, Y, D = (torch.full((T, O), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3))
    L.fwd_gelu(X, H, T, Y_pre=Y)
    Lt.bwd_x_gelu(X, pre, D, T)
    product = X.double() @ (W.double() * mask.double()).t()
    p = pre.double().requires_grad_(True)
    torch.nn.functional.gelu(p).sum().backward()
    assert _rel(Y, product) < 4e-3 and _rel(H, torch.nn.functional.gelu(product)) < 4e-3 and _rel(D, product * p.grad) < 4e-3


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_a_call_without_memory_leaves_no_image_behind(dtype):
    # the first call of a layer with value tracking asks for more scratch than the GPU has and is refused; the next one builds the
    # image all the same
    O, I, T = 96, 65, 50
    dt, mdt = (torch.float32, mst.MST_F32) if dtype == "f32" else (torch.bfloat16, mst.MST_BF16)
    g = torch.Generator(device="cuda").manual_seed(1)
    X, W = torch.randn(T, I, generator=g, device="cuda").to(dt), torch.randn(O, I, generator=g, device="cuda").to(dt)
    M = (torch.rand(O, I, generator=g, device="cuda") < 0.3).to(torch.uint8)
    Y = torch.zeros(T, O, device="cuda", dtype=dt)
    L = mst.Layer(0, O, I, mdt)
    L.pack(W, M)
    L.track_values(True)
    with pytest.raises(mst.MstError) as e:
        L.fwd(X, Y, 1 << 36)
    assert e.value.status == 8     # MST_ERR_CUDA
    del e
    L.fwd(X, Y, T)
    assert _rel(Y, X.double() @ (W * M).double().T) <= (5e-7 if dtype == "f32" else 4e-3)
    L.close()
