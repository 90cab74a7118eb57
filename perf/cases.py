"""Measured cases: what a training program has this library do, through its public entry points.

A case is a dict of plain values; ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the same ranges.
``prepare(case, seed)`` makes the inputs and the packed layers on the GPU, ``run(state)`` is one pass over them,
``work(case)`` the bytes and operations a pass cannot do without and ``tolerance(case)`` how far two correct
implementations may differ.

Kinds of passes:
  layers     forward, input gradient and weight gradient of masked linear layers; with ``grow`` a topology-update step:
             the dense gradient of the last micro-batch as well, then one Mixed-Growing update of every layer
  update     the Mixed-Growing update of a block's four layers alone, on gradients accumulated over earlier
             micro-batches, with the new structure handed to the optimizer
  mlp        fc1 -> GELU -> fc2 with the activation fused, forward and backward
  attention  strided sparse self-attention, forward and backward
  pack       dense weights and mask -> sparse layer, and its CSR arrays out (start of training, checkpoints)
  sample     forward only through a block's layers at a few tokens, weights unchanged from pass to pass
"""
import math

import numpy as np
import torch

import paper_2408_11746_b200 as mst

SIZE = {"bf16": 2, "fp32": 4}


# ------------------------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # one fp32 layer (GPT-2-small fc1) at a few hundred tokens: the debugging-size run, all of it in single precision
        dict(name="fp32_layer_step", kind="layers", out=3072, inp=768, tokens=256, dtype="fp32", density=0.25, skew="uniform",
             grow=True, prune=0.3, track=False),
        # a plain training pass over one GPT-2-small block, early warm-up density
        dict(name="small_block", kind="layers", width=768, tokens=8192, dtype="bf16", density=0.25, skew="uniform",
             grow=False, prune=0.0, track=True),
        # the ultra-sparse phase with rows of very different population and an update on every step
        dict(name="small_block_zipf_step", kind="layers", width=768, tokens=8192, dtype="bf16", density=0.06, skew="zipf",
             grow=True, prune=0.1, track=True),
        # GPT-2-medium block at the ultra-sparse density and a 16-sequence batch
        dict(name="medium_block", kind="layers", width=1024, tokens=16384, dtype="bf16", density=0.1, skew="uniform",
             grow=False, prune=0.0, track=True),
        # GPT-2-large block half way through the restoration phase: the largest call
        dict(name="large_block_restoring", kind="layers", width=1280, tokens=16384, dtype="bf16", density=0.5, skew="uniform",
             grow=False, prune=0.0, track=True),
        # a layer whose sizes are multiples of nothing, called without value tracking
        dict(name="ragged_layer", kind="layers", out=2051, inp=1023, tokens=1999, dtype="bf16", density=0.1, skew="uniform",
             grow=False, prune=0.0, track=False),
        # one topology update of a GPT-2-medium block (prune 0.3, random growth 0.25)
        dict(name="medium_update", kind="update", width=1024, dtype="bf16", density=0.1, skew="uniform", prune=0.3),
        # the MLP pair of GPT-2 small
        dict(name="small_mlp", kind="mlp", width=768, tokens=8192, density=0.1),
        # strided attention of GPT-2 small over 16 sequences, the paper's two strides
        dict(name="attention_256", kind="attention", batch=16, seq=1024, heads=12, stride=256),
        dict(name="attention_128", kind="attention", batch=8, seq=1024, heads=16, stride=128),
        # GPT-2-medium fc1 from dense weights and mask
        dict(name="pack_medium_fc1", kind="pack", out=4096, inp=1024, dtype="bf16", density=0.1, skew="uniform"),
        # text sampled from a sparse checkpoint, sixteen sequences side by side: the smallest calls
        dict(name="sample_small", kind="sample", width=768, tokens=16, density=0.1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _whole(rng, lo, hi):
    return max(lo, min(hi, int(round(_log(rng, lo, hi)))))


def _feature(rng, lo, hi):
    """A feature count: half of them multiples of 64, as model widths are, half anything."""
    n = _whole(rng, lo, hi)
    return max(lo, n // 64 * 64) if rng.random() < 0.5 else n


def _width(rng):
    """A model width: whole heads of 64."""
    return 64 * rng.randint(5, 20)


def draw(rng):
    kind = rng.choice(["layer", "layer", "block", "block", "block_step", "update", "mlp", "attention", "attention", "pack", "sample"])
    density = round(_log(rng, 0.02, 1.0), 3)
    sparse = round(_log(rng, 0.02, 0.25), 3)
    if kind == "layer":
        dtype = rng.choice(["fp32", "bf16"])
        return dict(kind="layers", out=_feature(rng, 96, 4096), inp=_feature(rng, 96, 2048),
                    tokens=_whole(rng, 64, 1024 if dtype == "fp32" else 4096), dtype=dtype, density=sparse,
                    skew=rng.choice(["uniform", "zipf"]), grow=rng.random() < 0.5, prune=round(rng.uniform(0.05, 0.3), 2), track=False)
    if kind == "block":
        return dict(kind="layers", width=_width(rng), tokens=_whole(rng, 1024, 16384), dtype="bf16", density=density,
                    skew="uniform", grow=False, prune=0.0, track=True)
    if kind == "block_step":
        return dict(kind="layers", width=64 * rng.randint(5, 16), tokens=_whole(rng, 1024, 16384), dtype="bf16", density=sparse,
                    skew=rng.choice(["uniform", "zipf"]), grow=True, prune=round(rng.uniform(0.05, 0.3), 2), track=True)
    if kind == "update":
        return dict(kind="update", width=_width(rng), dtype=rng.choice(["bf16", "bf16", "fp32"]), density=sparse,
                    skew=rng.choice(["uniform", "zipf"]), prune=round(rng.uniform(0.05, 0.3), 2))
    if kind == "mlp":
        return dict(kind="mlp", width=_width(rng), tokens=_whole(rng, 1024, 16384), density=sparse)
    if kind == "attention":
        return dict(kind="attention", batch=rng.randint(1, 16), seq=128 * _whole(rng, 2, 16), heads=rng.randint(6, 20),
                    stride=rng.choice([64, 128, 128, 192, 256, 256, 384, 512]))
    if kind == "pack":
        return dict(kind="pack", out=_feature(rng, 96, 5120), inp=_feature(rng, 96, 2048), dtype=rng.choice(["bf16", "bf16", "fp32"]),
                    density=density, skew=rng.choice(["uniform", "zipf"]))
    return dict(kind="sample", width=_width(rng), tokens=_whole(rng, 1, 128), density=sparse)


def _shapes(case):
    """(out_features, in_features) of the layers of a case."""
    kind = case["kind"]
    if "out" in case:
        return [(case["out"], case["inp"])]
    d = case["width"]
    if kind == "mlp":
        return [(4 * d, d), (d, 4 * d)]
    return [(3 * d, d), (d, d), (4 * d, d), (d, 4 * d)]


def _nnz(out, inp, density):
    return max(1, int(density * out * inp + 0.5))


def _attended(seq, stride):
    """Pairs of one head of one sequence: the last `stride` positions and every stride-th one before them."""
    return sum(min(i, stride - 1) + 1 + i // stride for i in range(seq))


# ------------------------------------------------------------------------------------------------------------ the inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(0x4D5354 + 7919 * seed)


def _normal(shape, std, dtype, g):
    x = torch.empty(shape, dtype=torch.float32, device="cuda").normal_(0.0, std, generator=g)
    return x if dtype == "fp32" else x.to(torch.bfloat16)


def _zipf_counts(out, inp, nnz, rng):
    """Row populations proportional to rank^-1.1 over a random row order, no row above `inp`, `nnz` in all."""
    share = np.arange(1, out + 1, dtype=np.float64) ** -1.1
    lo, hi = 0.0, nnz / share.min()
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if np.minimum(inp, mid * share).sum() < nnz else (lo, mid)
    count = np.minimum(inp, np.floor(lo * share)).astype(np.int64)
    short = nnz - int(count.sum())
    while short > 0:
        free = np.nonzero(count < inp)[0][:short]
        count[free] += 1
        short -= len(free)
    return count[rng.permutation(out)]


def _mask(out, inp, density, skew, g, seed):
    """uint8 [out, inp] with exactly _nnz(...) entries: uniform over the matrix, or uniform within rows of Zipf population."""
    nnz = _nnz(out, inp, density)
    if skew == "uniform":
        m = torch.zeros(out * inp, dtype=torch.uint8, device="cuda")
        m[torch.randperm(out * inp, generator=g, device="cuda")[:nnz]] = 1
        return m.view(out, inp)
    count = torch.from_numpy(_zipf_counts(out, inp, nnz, np.random.default_rng(seed))).cuda()
    place = torch.rand((out, inp), generator=g, device="cuda").argsort(1)
    m = torch.zeros((out, inp), dtype=torch.uint8, device="cuda")
    return m.scatter_(1, place, (torch.arange(inp, device="cuda")[None, :] < count[:, None]).to(torch.uint8))


class _Values:
    """A layer's stored values as a tensor, so that an optimizer can write them."""

    def __init__(self, address, count, dtype):
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": "<i2" if dtype == "bf16" else "<f4",
                                         "data": (address, False), "version": 3}


class _Layer:
    """One packed layer with its activations, upstream gradient and result buffers."""

    def __init__(self, index, out, inp, case, g, seed):
        self.out, self.inp, self.dtype = out, inp, case.get("dtype", "bf16")
        self.torch_dtype = torch.bfloat16 if self.dtype == "bf16" else torch.float32
        self.T = case.get("tokens", 0)
        self.nnz = _nnz(out, inp, case["density"])
        self.W = _normal((out, inp), 0.02, self.dtype, g)
        self.mask = _mask(out, inp, case["density"], case.get("skew", "uniform"), g, seed + index)
        self.layer = mst.Layer(index, out, inp, mst.MST_BF16 if self.dtype == "bf16" else mst.MST_F32)
        self.views = {}

    def packed(self, track):
        self.layer.pack(self.W, self.mask)
        self.layer.track_values(track)
        del self.W, self.mask
        return self

    def activations(self, g, backward=True):
        self.X = _normal((self.T, self.inp), 1.0, self.dtype, g)
        self.Y = torch.zeros((self.T, self.out), dtype=self.torch_dtype, device="cuda")
        if backward:
            self.dY = _normal((self.T, self.out), 0.01, self.dtype, g)
            self.dX = torch.zeros((self.T, self.inp), dtype=self.torch_dtype, device="cuda")
            self.dW = torch.zeros(self.nnz, dtype=torch.float32, device="cuda")
        return self

    def growth(self, g):
        """What an update takes and gives: the gradient accumulated over the micro-batches, the values as the optimizer has
        left them, and room for the new structure."""
        self.accumulated = _normal((self.out, self.inp), 0.4, "fp32", g)
        self.trained = _normal((self.nnz,), 0.02, self.dtype, g)
        return self.structure()

    def structure(self):
        self.row_ptr = torch.zeros(self.out + 1, dtype=torch.int32, device="cuda")
        self.col_idx = torch.zeros(self.nnz, dtype=torch.int32, device="cuda")
        self.values = torch.zeros(self.nnz, dtype=self.torch_dtype, device="cuda")
        return self

    def optimizer_writes(self):
        """The optimizer's new values go where the layer keeps its own (one of two places: an update changes sides)."""
        address, count = mst.mst_values(self.layer.handle)
        if address not in self.views:
            v = torch.as_tensor(_Values(address, count, self.dtype), device="cuda")
            self.views[address] = v.view(self.torch_dtype)
        self.views[address].copy_(self.trained)
        self.layer.values_changed()

    def export(self):
        mst.mst_export_csr(self.layer.handle, self.row_ptr, self.col_idx, self.values)
        return [self.row_ptr, self.col_idx, self.values]


class _State:
    pass


def prepare(case, seed):
    g = _generator(seed)
    s = _State()
    s.case, s.kind, s.step = case, case["kind"], 0
    if s.kind == "attention":
        B, n, H = case["batch"], case["seq"], case["heads"]
        s.C = 64 * H
        s.qkv = _normal((B * n, 3 * s.C), 1.0, "bf16", g)
        s.dOut = _normal((B * n, s.C), 1.0, "bf16", g)
        s.out = torch.zeros((B * n, s.C), dtype=torch.bfloat16, device="cuda")
        s.lse = torch.zeros((B, H, n), dtype=torch.float32, device="cuda")
        s.dqkv = torch.zeros_like(s.qkv)
        return s
    s.layers = [_Layer(i, o, n, case, g, seed) for i, (o, n) in enumerate(_shapes(case))]
    if s.kind == "pack":
        s.layers[0].structure()
        return s
    for L in s.layers:
        L.packed(True if s.kind in ("mlp", "sample", "update") else case["track"])
    if s.kind == "layers":
        for L in s.layers:
            L.activations(g)
            if case["grow"]:
                L.growth(g)
                L.G = torch.zeros((L.out, L.inp), dtype=torch.float32, device="cuda")
    elif s.kind == "update":
        for L in s.layers:
            L.growth(g)
    elif s.kind == "mlp":
        for L in s.layers:
            L.activations(g)
        s.pre = torch.zeros((case["tokens"], 4 * case["width"]), dtype=torch.bfloat16, device="cuda")
    elif s.kind == "sample":
        for L in s.layers:
            L.activations(g, backward=False)
    return s


# -------------------------------------------------------------------------------------------------------------- one pass
def _update(s):
    for L in s.layers:
        L.optimizer_writes()
    rules = [mst.RegrowRule(-1, 0.25, 1234, s.step, 0, 0.0) for _ in s.layers]
    s.step += 1
    mst.mst_topology_update_many([L.layer.handle for L in s.layers], [s.case["prune"]] * len(s.layers), rules,
                                 [L.accumulated for L in s.layers], want_stats=False)
    return [L.export() for L in s.layers]


def run(s):
    kind = s.kind
    if kind == "layers":
        grow = s.case["grow"]
        for L in s.layers:
            L.layer.values_changed()  # the optimizer has made a step since the last pass
            L.layer.fwd(L.X, L.Y, L.T)
        for L in reversed(s.layers):
            L.layer.bwd_x(L.dY, L.dX, L.T)
            if grow:
                L.layer.dense_grad_dw(L.dY, L.X, L.T, L.G, L.dW)
            else:
                L.layer.sddmm(L.dY, L.X, L.T, L.dW)
        out = [[L.Y, L.dX, L.dW] + ([L.G] if grow else []) for L in s.layers]
        return [out, _update(s)] if grow else out
    if kind == "update":
        return _update(s)
    if kind == "mlp":
        a, b = s.layers
        T = a.T
        a.layer.values_changed()
        b.layer.values_changed()
        a.layer.fwd_gelu(a.X, b.X, T, Y_pre=s.pre)
        b.layer.fwd(b.X, b.Y, T)
        b.layer.bwd_x_gelu(b.dY, s.pre, a.dY, T)
        b.layer.sddmm(b.dY, b.X, T, b.dW)
        a.layer.bwd_x(a.dY, a.dX, T)
        a.layer.sddmm(a.dY, a.X, T, a.dW)
        return [s.pre, b.X, b.Y, a.dY, a.dX, a.dW, b.dW]
    if kind == "attention":
        c, C = s.case, s.C
        q, d = s.qkv.data_ptr(), s.dqkv.data_ptr()
        mst.mst_strided_attention_fwd(q, q + 2 * C, q + 4 * C, 3 * C, c["batch"], c["seq"], c["heads"], 64, c["stride"], s.out, C, s.lse)
        mst.mst_strided_attention_bwd(q, q + 2 * C, q + 4 * C, 3 * C, s.out, C, s.dOut, C, s.lse, c["batch"], c["seq"], c["heads"], 64,
                                      c["stride"], d, d + 2 * C, d + 4 * C, 3 * C)
        return [s.out, s.lse, s.dqkv]
    if kind == "pack":
        L = s.layers[0]
        L.layer.pack(L.W, L.mask)
        return L.export()
    qkv, proj, fc1, fc2 = s.layers
    qkv.layer.fwd(qkv.X, qkv.Y, qkv.T)
    proj.layer.fwd(proj.X, proj.Y, proj.T)
    fc1.layer.fwd_gelu(fc1.X, fc2.X, fc1.T)
    fc2.layer.fwd(fc2.X, fc2.Y, fc2.T)
    return [qkv.Y, proj.Y, fc2.X, fc2.Y]


# --------------------------------------------------------------------------------------------- necessary work, tolerances
def work(case):
    kind = case["kind"]
    if kind == "attention":
        rows, C = case["batch"] * case["seq"], 64 * case["heads"]
        pairs = case["batch"] * case["heads"] * _attended(case["seq"], case["stride"])
        # q, k, v, dOut in, out and the three gradients back, one log-sum-exp a row; seven products of 64 a pair
        return {"bytes": 2.0 * rows * C * 8 + 4.0 * rows * case["heads"], "flops": 7 * 2 * 64.0 * pairs}
    e = SIZE[case.get("dtype", "bf16")]
    T, grow = case.get("tokens", 0), case.get("grow", False)
    total, flops = 0.0, 0.0
    for o, i in _shapes(case):
        nnz = _nnz(o, i, case["density"])
        stored = nnz * (e + 2) + 4 * (o + 1)
        exported = nnz * (e + 4) + 4 * (o + 1)
        update = o * i * 4 + nnz * e + stored + stored + exported  # gradient, new values, old and new structure, CSR out
        if kind == "layers":
            total += 2.0 * T * (o + i) * e + stored + 4.0 * nnz
            flops += 4.0 * T * nnz + (2.0 * T * o * i if grow else 2.0 * T * nnz)
            total += 4.0 * o * i + update if grow else 0
        elif kind == "update":
            total += update
        elif kind == "mlp":
            total += 2.0 * T * (o + i) * e + stored + 4.0 * nnz
            flops += 6.0 * T * nnz
        elif kind == "pack":
            total += o * i + nnz * e + stored + exported
        else:
            total += T * (o + i) * e + stored
            flops += 2.0 * T * nnz
    return {"bytes": total, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("pack", "update"):
        return "exact"
    if kind == "attention":
        return {"rel": 1e-2}  # softmax weights and score gradients pass through bf16
    if case.get("dtype", "bf16") == "fp32":
        return {"rel": 1e-5}
    return {"rel": 4e-3 if kind != "mlp" else 1e-2}  # bf16 results of 32-bit sums; the pair feeds rounded results on
