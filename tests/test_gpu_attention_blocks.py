"""Strided attention where blocks take over others of their grid: grids just below, at and above what runs at once, blocks of which only
half the rows exist, halves with different numbers of far tiles.  Every element within the bounds of its data types."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    import paper_2408_11746_b200 as mst
    from test_gpu_attention_bwd import _row_bounds


def _forward_reference(qkv, B, n, H, stride):
    x = qkv.double().view(B, n, 3, H, 64).permute(2, 0, 3, 1, 4)
    back = torch.arange(n, device=qkv.device)
    back = back[:, None] - back[None, :]
    keep = (back >= 0) & ((back < stride) | (back % stride == 0))
    s = (x[0] @ x[1].mT / 8).masked_fill(~keep, float("-inf"))
    lse = torch.logsumexp(s, -1)
    return (torch.exp(s - lse[..., None]) @ x[2]).transpose(1, 2).reshape(B * n, 64 * H).bfloat16(), lse.float()


@pytest.mark.parametrize("B,n,H,stride", [
    (8, 128, 37, 64),      # 296 blocks: all of them run at once on 148 SMs
    (9, 384, 11, 128),     # 297: one starts when another is done
    (8, 256, 37, 64),      # 592: the most of which none is taken over
    (16, 256, 20, 192),    # 640
    (8, 448, 19, 64),      # an odd number of 64-row tiles: the last block has half its rows, its second half no far tiles
    (6, 704, 17, 192),     # the same, far tiles in odd and even numbers
    (6, 1152, 12, 128),    # up to sixteen far tiles, 648 blocks
    (34, 384, 19, 128),    # more than L2 holds: the batch in two parts
    (37, 384, 18, 192),    # the heads in two, as nothing divides the batch
    (98, 256, 20, 128),    # both in two
    (23, 512, 23, 256),    # one part, as the least number would be twenty-three
    (2, 1152, 6, 128),     # none to sixteen of them in blocks without successors: slots filled for the first time and again
    (1, 832, 7, 192),      # the same, odd numbers
    (1, 256, 6, 256),      # windows of the whole sequence: kernels without far tiles
    (2, 768, 5, 384),      # windows of half of it
    (3, 320, 5, 192),      # the same with half a block at the end
    (2, 64, 3, 64)])       # nothing but half a block
def test_blocks_that_take_over_others(B, n, H, stride):
    gen = torch.Generator(device="cuda").manual_seed(n + stride)
    C = 64 * H
    qkv = torch.randn(B * n, 3 * C, generator=gen, device="cuda").bfloat16()
    dO = torch.randn(B * n, C, generator=gen, device="cuda").bfloat16()
    out = torch.full((B * n + 64, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    dqkv = torch.full((B * n + 64, 3 * C), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, n), float("nan"), device="cuda")
    a, d = qkv.data_ptr(), dqkv.data_ptr()
    if n % 128 == 0:
        mst.mst_strided_attention_fwd(a, a + 2 * C, a + 4 * C, 3 * C, B, n, H, 64, stride, out, C, lse)
    else:
        o, lse = _forward_reference(qkv, B, n, H, stride)
        out[: B * n] = o
    mst.mst_strided_attention_bwd(a, a + 2 * C, a + 4 * C, 3 * C, out, C, dO, C, lse, B, n, H, 64, stride, d, d + 2 * C, d + 4 * C, 3 * C)
    torch.cuda.synchronize()
    assert mst.mst_device_error_flags() == 0
    assert torch.isnan(out[B * n:]).all() and torch.isnan(dqkv[B * n:]).all()      # nothing beyond the last row
    ref, bound = _row_bounds(qkv, dO, B, n, H, stride)
    for name, t, r, e in zip(("out", "dQ", "dK", "dV"), [out[: B * n]] + list(dqkv[: B * n].view(B * n, 3, C).unbind(1)), ref, bound):
        over = (t.double().view(B, n, H, 64).transpose(1, 2) - r).abs() - e
        # as in the test of every element: dS of the first positions cancels, 64 truncated terms of size |dOut||v|
        assert float(over.max()) <= 64 * 2.0 ** -23 * 8, (name, float(over.max()), int(over.argmax()))
