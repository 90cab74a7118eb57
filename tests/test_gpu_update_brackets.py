"""The one-launch topology update where its brackets can go wrong: equal keys everywhere, open ends, thresholds among the few
largest or smallest keys, everything grown or pruned, more layers than one launch takes, slices of one word.  Bit-exact
against the checker."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import mst_inputs  # noqa: E402
import oracle  # noqa: E402
import paper_2408_11746_b200 as mst  # noqa: E402
from gpu_util import dev, export_csr, make_layer, value_bits  # noqa: E402


def _problem(O, I, dtype, density, seed):
    m = mst_inputs.uniform_mask(O, I, mst_inputs.exact_nnz(O, I, density), seed, 1)
    return mst_inputs.make_layer("u", seed % 97, O, I, 1, dtype, m, seed)


def _check(L, p, W, M, G, zeta, target, R, step):
    n_prune, n_grow, n_rand, n_grad = oracle.mg_counts(zeta, int(M.sum()), target, M.size, R)
    Wn, Mn, *_ = oracle.mg_update(W, M, G, n_prune, n_grad, n_rand, 11, step, p.layer_id, False)
    rp, ci, vb = export_csr(L, p.dtype)
    rp_r, ci_r, v_r = oracle.to_csr(Wn, Mn)
    np.testing.assert_array_equal(rp, rp_r)
    np.testing.assert_array_equal(ci, ci_r)
    np.testing.assert_array_equal(vb, value_bits(v_r, p.dtype))
    L.validate()
    return Wn, Mn


def _gradient(kind, O, I, rng):
    if kind == "equal":
        return np.full((O, I), 0.5, np.float32)
    if kind == "two":
        return np.where(rng.random((O, I)) < 0.01, np.float32(2.0), np.float32(1.0)).astype(np.float32)
    if kind == "zero":
        return np.zeros((O, I), np.float32)
    if kind == "huge":      # most keys at the far ends of the range
        return (rng.choice([1e-38, 3e38, 1.0], (O, I), p=[0.6, 0.2, 0.2]) * rng.random((O, I))).astype(np.float32)
    return rng.standard_normal((O, I)).astype(np.float32)


@pytest.mark.parametrize("O,I,dtype,density,zeta,R,grad,weights", [
    (512, 512, "bf16", 0.3, 0.3, 0.25, "equal", "normal"), (512, 520, "f32", 0.3, 0.3, 0.25, "two", "equal"),
    (700, 333, "bf16", 0.2, 0.3, 0.25, "zero", "zero"), (512, 768, "f32", 0.1, 0.3, 0.25, "huge", "normal"),
    (1024, 768, "bf16", 0.1, 0.0005, 0.25, "normal", "normal"), (1024, 768, "bf16", 0.3, 0.3, 0.0, "normal", "equal"),
    (300, 500, "f32", 0.45, 1.0, 0.5, "normal", "normal"), (300, 500, "bf16", 0.5, 1.0, 0.25, "normal", "normal"),
    (64, 33, "bf16", 0.1, 0.5, 0.25, "normal", "normal"), (1, 5000, "f32", 0.2, 0.3, 0.25, "normal", "normal"),
    (2000, 31, "bf16", 0.2, 0.3, 0.25, "normal", "normal"), (1536, 1024, "bf16", 0.5, 0.3, 0.25, "normal", "normal")])
def test_update_with_awkward_keys(O, I, dtype, density, zeta, R, grad, weights):
    p = _problem(O, I, dtype, density, 40 + O + I)
    if weights != "normal":
        p.W[:] = 0.0 if weights == "zero" else 0.25
        if dtype == "bf16":
            p.W_bits = mst_inputs.f32_to_bf16_bits(p.W)
    rng = np.random.default_rng(O * I)
    L = make_layer(p)
    W, M = np.where(p.mask == 1, p.W, np.float32(0)).astype(np.float32), p.mask.copy()
    for step in range(2):
        G = _gradient(grad, O, I, rng)
        mst.mst_topology_update(L.handle, zeta, -1, R, 11, step, False, torch.from_numpy(G).to(dev()), want_stats=False)
        W, M = _check(L, p, W, M, G, zeta, -1, R, step)
    for target in (int(0.03 * O * I) + 1, int(0.6 * O * I)):   # sparsified, then most of it grown back
        G = _gradient(grad, O, I, rng)
        mst.mst_topology_update(L.handle, zeta, target, R, 11, target, False, torch.from_numpy(G).to(dev()), want_stats=False)
        W, M = _check(L, p, W, M, G, zeta, target, R, target)
    L.close()


def test_more_layers_than_one_launch_takes():
    shapes = [(96 + 40 * k, 64 + 33 * k, "f32" if k % 3 == 2 else "bf16", 0.1 + 0.04 * k) for k in range(11)]
    probs = [_problem(O, I, dt, d, 900 + k) for k, (O, I, dt, d) in enumerate(shapes)]
    layers = [make_layer(p) for p in probs]
    rng = np.random.default_rng(5)
    state = [(np.where(p.mask == 1, p.W, np.float32(0)).astype(np.float32), p.mask.copy()) for p in probs]
    for step in range(2):
        Gs = [rng.standard_normal(p.mask.shape).astype(np.float32) for p in probs]
        rules = [mst.RegrowRule(-1, 0.25, 11, step, 0, 0.0) for _ in probs]
        mst.mst_topology_update_many([L.handle for L in layers], [0.3] * len(probs), rules, [torch.from_numpy(g).to(dev()) for g in Gs],
                                     want_stats=False)
        state = [_check(L, p, W, M, G, 0.3, -1, 0.25, step) for L, p, (W, M), G in zip(layers, probs, state, Gs)]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("tied", [2, 100, 256, 258, 1000, 1100, 5000])
def test_threshold_among_equal_gradients(tied, dtype):
    """The threshold's bin holds as many entries as the warps rank directly (256), one or a few more, more than are compared one by one
    (1024), more than the list takes (4096): the same selection, ties by position."""
    O, I, zeta, R = 600, 768, 0.3, 0.25
    p = _problem(O, I, dtype, 0.2, 7100 + tied)
    rng = np.random.default_rng(tied)
    L = make_layer(p)
    W, M = np.where(p.mask == 1, p.W, np.float32(0)).astype(np.float32), p.mask.copy()
    for step in range(2):
        _, _, _, n_grad = oracle.mg_counts(zeta, int(M.sum()), -1, M.size, R)
        G = rng.standard_normal((O, I)).astype(np.float32)
        free = np.flatnonzero(M.reshape(-1) == 0)
        order = free[np.argsort(-np.abs(G.reshape(-1)[free]), kind="stable")]
        plateau = order[max(0, n_grad - tied // 2): n_grad + (tied + 1) // 2]
        flat = G.reshape(-1)
        flat[plateau] = np.abs(flat[order[n_grad]]) * np.where(rng.random(plateau.size) < 0.5, -1, 1)
        mst.mst_topology_update(L.handle, zeta, -1, R, 11, step, False, torch.from_numpy(G).to(dev()), want_stats=False)
        W, M = _check(L, p, W, M, G, zeta, -1, R, step)
    L.close()
    assert mst.mst_device_error_flags() == 0
