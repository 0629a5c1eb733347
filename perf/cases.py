"""Workloads that stand for what programs do with this library, as timed cases.

Each case is a dict of plain values; `kind` names the call path:

  map       one element-wise map over a 1-D partition
  map2d     one element-wise map over a rank-2 partition (an activation matrix
            tiled like the GEMM that produced it)
  gemm_f32  FP32 products C_i = A . B_i
  gemm_bf16 BF16 tensor-core products C_i = A . B_i
  fp8       an FP8 linear layer: the activations are scaled and quantised on
            every pass, the weights once
  grouped   a group of uneven BF16 products in one launch
  decode    batch-1 decode layers, fused or one launch per step
  mlp       forward and backward of the tile proposer's network

Launch-bound work is captured once into a graph and replayed, as such programs
do (`graph`); the rest are plain synchronous calls, the library's default.
"""
import math
import random

import torch

import paper_2606_15991_gb300 as tp

_CTX = None

# (K, N) of the linear layers that the grouped and FP8 workloads are made of
KN = [(2560, 9728), (5120, 25600), (25600, 5120), (5120, 10240)]


def _ctx():
    global _CTX
    if _CTX is None:
        torch.cuda.set_device(0)
        _CTX = tp.tp_ctx_create(0)
    return _CTX


# ----------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: one 2048-element tile, where the call itself is the cost
        {"name": "map_scale_bf16_2048", "kind": "map", "op": "scale", "dtype": "bf16", "n": 2048, "tile": 2048,
         "map": "identity", "graph": False},
        # the largest element-wise pass, streamed from HBM
        {"name": "map_axpy_f32_2p28", "kind": "map", "op": "axpy", "dtype": "f32", "n": 1 << 28, "tile": 4096,
         "map": "identity", "graph": False},
        # a gated activation over a ragged batch of tokens, tiled as the GEMM's output is
        {"name": "map_gelu_bf16_2d", "kind": "map2d", "op": "gelu_mul", "dtype": "bf16", "rows": 4001, "cols": 9728,
         "tile_r": 128, "tile_c": 256, "graph": False},
        # small FP32 products, each tile program a cluster of two K slices
        {"name": "gemm_f32_512", "kind": "gemm_f32", "M": 512, "N": 512, "K": 512, "split": 2, "products": 8,
         "graph": True},
        # an FP32 product with no aligned extent, on the default configuration
        {"name": "gemm_f32_ragged", "kind": "gemm_f32", "M": 1000, "N": 3001, "K": 777, "split": 1, "products": 1,
         "graph": False},
        # small tensor-core products of one input (the projections of a small layer)
        {"name": "gemm_bf16_1024", "kind": "gemm_bf16", "M": 1024, "N": 1024, "K": 1024, "products": 8, "graph": True},
        # the large square product
        {"name": "gemm_bf16_8192", "kind": "gemm_bf16", "M": 8192, "N": 8192, "K": 8192, "products": 1,
         "graph": False},
        # an FP8 linear layer over a prefill batch
        {"name": "fp8_linear_2000", "kind": "fp8", "dtype": "bf16", "M": 2000, "N": 10240, "K": 5120, "graph": True},
        # 64 uneven products, decode-sized to prefill-sized
        {"name": "grouped_64", "kind": "grouped", "problems": 64, "m_max": 4096, "shapes": 0},
        # decode: four fused layers, replayed for each token
        {"name": "decode_fused_4", "kind": "decode", "d": 5120, "nq": 10240, "ni": 25600, "layers": 4, "fused": True},
        # decode through the single-step entry points (a program with its own steps between them)
        {"name": "decode_steps_2", "kind": "decode", "d": 5120, "nq": 10240, "ni": 25600, "layers": 2,
         "fused": False},
        # one batch of the proposer's training: loss and every gradient
        {"name": "mlp_grad_256", "kind": "mlp", "batch": 256, "features": 5, "hidden": 64, "outputs": 72},
    ]


def _log(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["map", "map2d", "gemm_f32", "gemm_bf16", "gemm_bf16", "fp8", "grouped", "decode", "decode", "mlp"])
    op = rng.choice(["axpy", "gelu_mul", "scale", "add_accum"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "map":
        n = _log(rng, 1000, 1 << 28)
        n -= n % rng.choice([1, 8])
        return {"kind": kind, "op": op, "dtype": dtype, "n": n, "tile": rng.choice([1000, 2048, 4096, 16384]),
                "map": rng.choice(["identity", "strided", "queue"]), "graph": False}
    if kind == "map2d":
        return {"kind": kind, "op": op, "dtype": dtype, "rows": _log(rng, 16, 8192),
                "cols": _log(rng, 64, 12288, rng.choice([1, 8])),
                "tile_r": rng.choice([16, 64, 128]), "tile_c": rng.choice([64, 100, 128, 256]), "graph": False}
    if kind == "gemm_f32":
        step = rng.choice([1, 4])
        split = rng.choice([1, 1, 2])
        return {"kind": kind, "M": _log(rng, 64, 2048, step), "N": _log(rng, 64, 3072, step),
                "K": _log(rng, 32, 2048, step), "split": split, "products": 1, "graph": rng.random() < 0.5}
    if kind == "gemm_bf16":
        M, N, K = _log(rng, 1, 8192), _log(rng, 64, 8192, 8), _log(rng, 64, 8192, rng.choice([8, 64]))
        small = 2.0 * M * N * K < 2e10
        return {"kind": kind, "M": M, "N": N, "K": K, "products": 8 if small else 1, "graph": small}
    if kind == "fp8":
        k, n = rng.choice(KN)
        return {"kind": kind, "dtype": dtype, "M": _log(rng, 16, 4096), "N": n, "K": k, "graph": True}
    if kind == "grouped":
        return {"kind": kind, "problems": rng.randrange(4, 25), "m_max": rng.choice([256, 1024, 4096]),
                "shapes": rng.randrange(1, 1000)}
    if kind == "decode":
        d = _log(rng, 1000, 5120, 8)
        return {"kind": kind, "d": d, "nq": _log(rng, d, 2 * d), "ni": _log(rng, 2 * d, 5 * d, 8),
                "layers": rng.randrange(1, 4), "fused": rng.random() < 0.5}
    return {"kind": "mlp", "batch": rng.randrange(32, 513), "features": 5, "hidden": rng.choice([32, 64, 100, 128]),
            "outputs": rng.randrange(16, 128)}


def _shapes(case):
    """(M, N, K) of a group: M log-uniform on [1, m_max], (K, N) one of KN."""
    rng = random.Random(1000 + case["shapes"])
    out = []
    for _ in range(case["problems"]):
        m = max(1, min(case["m_max"], round(2.0 ** (math.log2(case["m_max"]) * rng.random()))))
        k, n = rng.choice(KN)
        out.append((m, n, k))
    return out


# ---------------------------------------------------------------------- inputs
_DT = {"f32": torch.float32, "bf16": torch.bfloat16}
_SIZE = {"f32": 4, "bf16": 2}


class _Inputs:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def normal(self, *shape, dtype=torch.float32, std=1.0):
        t = torch.randn(*shape, device="cuda", dtype=dtype, generator=self.g)
        return t if std == 1.0 else t.mul_(std)

    def uniform(self, *shape, lo=-1.0, hi=1.0):
        return torch.rand(*shape, device="cuda", generator=self.g).mul_(hi - lo).add_(lo)


def _map_inputs(case, seed):
    i = _Inputs(seed)
    shape = (case["n"],) if case["kind"] == "map" else (case["rows"], case["cols"])
    x, y = (i.normal(*shape, dtype=_DT[case["dtype"]]) for _ in range(2))
    c = i.normal(*shape, dtype=_DT[case["dtype"]]) if case["op"] == "add_accum" else None
    return x, y, c


def _gemm_inputs(case, seed):
    i = _Inputs(seed)
    M, N, K = case["M"], case["N"], case["K"]
    if case["kind"] == "gemm_f32":
        return i.uniform(M, K), [i.uniform(K, N) for _ in range(case["products"])]
    # weights are stored output-major (N x K): B is their transposed view
    return (i.normal(M, K, dtype=torch.bfloat16),
            [i.normal(N, K, dtype=torch.bfloat16) for _ in range(case["products"])])


def _fp8_inputs(case, seed):
    i = _Inputs(seed)
    return (i.normal(case["M"], case["K"], dtype=_DT[case["dtype"]]),
            i.normal(case["N"], case["K"], dtype=torch.bfloat16, std=0.02))


def _grouped_inputs(case, seed):
    i = _Inputs(seed)
    return [(i.normal(m, k, dtype=torch.bfloat16), i.normal(n, k, dtype=torch.bfloat16)) for m, n, k in _shapes(case)]


def _decode_inputs(case, seed):
    i = _Inputs(seed)
    d, nq, ni = case["d"], case["nq"], case["ni"]
    layers = [tuple(i.normal(r, k, dtype=torch.bfloat16, std=0.02) for r, k in ((nq, d), (2 * ni, d), (d, ni)))
              for _ in range(case["layers"])]
    return i.normal(d), layers


def _mlp_inputs(case, seed):
    i = _Inputs(seed)
    B, F, H, C = case["batch"], case["features"], case["hidden"], case["outputs"]
    params = []
    for rows, fan in ((H, F), (H, H), (C, H)):
        r = 1.0 / math.sqrt(fan)
        params += [i.uniform(rows, fan, lo=-r, hi=r), i.uniform(rows, lo=-r, hi=r)]
    X = i.uniform(B, F, lo=0.0, hi=14.0)     # log2 of the extents, as the proposer's features are
    X[:, 3:] = (X[:, 3:] > 7.0).float()
    T = i.uniform(B, C, lo=0.0, hi=1.0)
    V = (i.uniform(B, C, lo=0.0, hi=1.0) < 0.9).float()
    return params, X, T, V


# ----------------------------------------------------------------------- state
class _State:
    """What a program keeps between passes; `calls` launches one pass into the
    tp_exec it is given (None: a synchronous call)."""

    def __init__(self, case):
        self.case, self.ctx = case, _ctx()
        self.partitions, self.graph, self.plan, self.net = [], None, None, None
        self.outputs, self.before = {}, None

    def partition(self, t, tile, kind=None, programs=0):
        p = tp.tp_partition_create(self.ctx, t, tile)
        if kind is not None:
            tp.tp_partition_map(p, kind, programs)
        self.partitions.append(p)
        return p

    def strided(self, t, tile, programs):
        p = self.partition(t, tile)
        tp.tp_partition_map(p, tp.MAP_STRIDED, min(programs, tp.tp_partition_query(p)["num_tiles"]))
        return p

    def capture(self):
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        self.graph = tp.tp_graph_begin(self.ctx, s)
        self.calls(tp.make_exec(tp.CAPTURE, s))
        tp.tp_graph_end(self.graph)

    def __del__(self):
        try:
            if self.graph is not None:
                tp.tp_graph_destroy(self.graph)
            if self.plan is not None:
                tp.tp_grouped_plan_destroy(self.plan)
            if self.net is not None:
                tp.tp_mlp_destroy(self.net)
            for p in self.partitions:
                tp.tp_partition_destroy(p)
        except Exception:
            pass


_MAPS = {"axpy": lambda c, p, x, y, ex: tp.tp_map_axpy(c, p, 0.5, x, y, ex), "gelu_mul": tp.tp_map_gelu_mul,
         "scale": tp.tp_map_scale, "add_accum": tp.tp_map_add_accum}


def _prepare_map(s, case, seed):
    x, y, c = _map_inputs(case, seed)
    out = torch.empty_like(x) if c is None else c.clone()
    if case["kind"] == "map2d":
        p = s.partition(out, (case["tile_r"], case["tile_c"]))
    elif case["map"] == "identity":
        p = s.partition(out, (case["tile"],))
    else:
        p = s.partition(out, (case["tile"],))
        tp.tp_partition_map(p, tp.MAP_STRIDED if case["map"] == "strided" else tp.MAP_QUEUE,
                            min(tp.tp_partition_query(p)["num_tiles"], 4 * s.ctx.sm_count))
    if c is not None:
        s.before = lambda: out.copy_(c)      # the pass accumulates into fresh values
    op = _MAPS[case["op"]]
    s.calls = lambda ex: op(s.ctx, p, x, y, ex)
    s.outputs = {"out": out}


def _prepare_gemm_f32(s, case, seed):
    a, bs = _gemm_inputs(case, seed)
    cs = [torch.empty(case["M"], case["N"], device="cuda") for _ in bs]
    ps = [s.partition(c, (64, 64)) for c in cs]
    cfg = tp.gemm_config(bk=32, split_k=case["split"]) if case["split"] > 1 else None

    def calls(ex):
        for p, b in zip(ps, bs):
            tp.tp_gemm(s.ctx, p, a, b, cfg, ex)

    s.calls, s.outputs = calls, {"c": cs}


def _tile(M, N, elem):
    """Tile rows, columns and K blocks per stage: CTA pairs when they fill half
    the chip, smaller tiles below that, 64-row tiles for decode-sized M."""
    blk = 128 // elem
    if M <= 64:
        return 64, 64, 4 * blk
    if math.ceil(M / 256) * math.ceil(N / 256) >= 38:
        return 256, 256, 2 * blk
    return 128, 64, 4 * blk


def _prepare_gemm_bf16(s, case, seed):
    a, bts = _gemm_inputs(case, seed)
    bm, bn, bk = _tile(case["M"], case["N"], 2)
    cfg = tp.gemm_config(bm=bm, bn=bn, bk=bk, group_m=8)
    cs = [torch.empty(case["M"], case["N"], device="cuda", dtype=torch.bfloat16) for _ in bts]
    ps = [s.strided(c, (bm, bn), s.ctx.sm_count // 2 if bm == 256 else s.ctx.sm_count) for c in cs]

    def calls(ex):
        for p, bt in zip(ps, bts):
            tp.tp_gemm(s.ctx, p, a, bt.t(), cfg, ex)

    s.calls, s.outputs = calls, {"c": cs}


def _prepare_fp8(s, case, seed):
    x, w = _fp8_inputs(case, seed)
    M, N, K = case["M"], case["N"], case["K"]
    f8 = torch.float8_e4m3fn
    qx, qw = torch.empty(M, K, device="cuda", dtype=f8), torch.empty(N, K, device="cuda", dtype=f8)
    amax, scale = torch.zeros(2, device="cuda"), torch.zeros(2, device="cuda")
    out = torch.empty(M, N, device="cuda", dtype=torch.bfloat16)
    pq, pw = s.partition(qx, (16, K)), s.partition(qw, (16, K))
    tp.tp_amax(s.ctx, w, amax[1:2])
    tp.tp_quantize_fp8(s.ctx, pw, w, amax[1:2], scale[1:2])
    bm, bn, bk = _tile(M, N, 1)
    cfg = tp.gemm_config(bm=bm, bn=bn, bk=bk, group_m=16)
    pc = s.strided(out, (bm, bn), s.ctx.sm_count // 2 if bm == 256 else s.ctx.sm_count)

    def calls(ex):
        tp.tp_amax(s.ctx, x, amax[0:1], ex)
        tp.tp_quantize_fp8(s.ctx, pq, x, amax[0:1], scale[0:1], ex)
        tp.tp_gemm_fp8(s.ctx, pc, qx, qw.t(), scale[0:1], scale[1:2], cfg, ex)

    s.calls, s.outputs = calls, {"c": out, "codes": qx.view(torch.uint8), "amax": amax[0:1], "scale": scale[0:1]}


def _prepare_grouped(s, case, seed):
    probs = [(a, bt.t(), torch.empty(a.shape[0], bt.shape[0], device="cuda", dtype=torch.bfloat16))
             for a, bt in _grouped_inputs(case, seed)]
    s.plan = tp.tp_grouped_plan_create(s.ctx, probs)
    s.calls = lambda ex: tp.tp_grouped_gemm(s.ctx, s.plan, 0, ex)
    s.outputs = {"c": [c for _, _, c in probs]}


def _prepare_decode(s, case, seed):
    token, layers = _decode_inputs(case, seed)
    h = token.clone()
    chain = tp.DecodeChain(s.ctx, h, layers)
    s.partitions += list(chain.p.values())
    s.before = lambda: h.copy_(token)        # the token's embedding enters the residual stream
    s.calls = chain.record_fused if case["fused"] else chain.record_unfused
    names = ("h", "qkv", "a") if case["fused"] else ("h", "n", "qkv", "gu", "a", "dd")
    s.outputs = {k: getattr(chain, k) for k in names}
    s.chain = chain


def _prepare_mlp(s, case, seed):
    params, X, T, V = _mlp_inputs(case, seed)
    flat = torch.cat([p.reshape(-1) for p in params])
    s.net = tp.tp_mlp_create(s.ctx, case["features"], case["hidden"], case["outputs"], case["batch"],
                             flat.cpu().numpy())
    loss, grads = torch.zeros(1, device="cuda"), torch.empty_like(flat)
    s.calls = lambda ex: tp.tp_mlp_loss_grad(s.net, X, T, V, loss, grads, ex)
    s.outputs = {"loss": loss, "grads": grads}


_PREPARE = {"map": _prepare_map, "map2d": _prepare_map, "gemm_f32": _prepare_gemm_f32, "gemm_bf16": _prepare_gemm_bf16,
            "fp8": _prepare_fp8, "grouped": _prepare_grouped, "decode": _prepare_decode, "mlp": _prepare_mlp}


def prepare(case, seed):
    s = _State(case)
    _PREPARE[case["kind"]](s, case, seed)
    if case["kind"] == "decode" or case.get("graph"):
        s.capture()
    return s


def run(s):
    if s.before is not None:
        s.before()
    if s.graph is not None:
        tp.tp_graph_replay(s.graph, tp.make_exec())
    else:
        s.calls(None)
    return s.outputs


# ------------------------------------------------------------------------ work
def _gemm_work(M, N, K, ein, eout):
    return {"bytes": ein * (M * K + N * K) + eout * M * N, "flops": 2.0 * M * N * K}


def work(case):
    kind = case["kind"]
    if kind in ("map", "map2d"):
        n = case["n"] if kind == "map" else case["rows"] * case["cols"]
        return {"bytes": (4 if case["op"] == "add_accum" else 3) * _SIZE[case["dtype"]] * n,
                "flops": {"scale": 1, "gelu_mul": 8}.get(case["op"], 2) * n}
    if kind in ("gemm_f32", "gemm_bf16"):
        M, N, K, P = case["M"], case["N"], case["K"], case["products"]
        e = 4 if kind == "gemm_f32" else 2
        return {"bytes": e * (M * K + P * (N * K + M * N)), "flops": 2.0 * P * M * N * K}
    if kind == "fp8":
        M, N, K = case["M"], case["N"], case["K"]
        # the activations, their codes, the weights' codes, the result
        return {"bytes": _SIZE[case["dtype"]] * M * K + M * K + N * K + 2 * M * N, "flops": 2.0 * M * N * K}
    if kind == "grouped":
        each = [_gemm_work(m, n, k, 2, 2) for m, n, k in _shapes(case)]
        return {key: sum(w[key] for w in each) for key in ("bytes", "flops")}
    if kind == "decode":
        d, nq, ni = case["d"], case["nq"], case["ni"]
        weights = case["layers"] * (nq * d + 2 * ni * d + d * ni)
        return {"bytes": 2 * weights + 4 * case["layers"] * (nq + ni) + 8 * d, "flops": 2.0 * weights}
    B, F, H, C = case["batch"], case["features"], case["hidden"], case["outputs"]
    p = H * F + H + H * H + H + C * H + C
    return {"bytes": 4 * (2 * p + B * (F + 2 * C) + 1), "flops": 2.0 * B * (3 * (H * H + C * H) + 2 * H * F)}


# ------------------------------------------------------- the same in 64 bits
def _exact_map(case, seed):
    x, y, c = (None if t is None else t.double() for t in _map_inputs(case, seed))
    if case["op"] == "axpy":
        return {"out": x.mul_(0.5).add_(y)}
    if case["op"] == "scale":
        return {"out": x.mul_(y)}
    if case["op"] == "add_accum":
        return {"out": x.add_(c).add_(y)}
    u = x * x
    u.mul_(0.044715).add_(1.0).mul_(x).mul_(math.sqrt(2.0 / math.pi)).tanh_().add_(1.0)
    return {"out": u.mul_(x).mul_(0.5).mul_(y)}


def _exact_gemm(case, seed):
    a, bs = _gemm_inputs(case, seed)
    a = a.double()
    return {"c": [a @ (b.double() if case["kind"] == "gemm_f32" else b.double().t()) for b in bs]}


def _exact_fp8(case, seed):
    x, w = _fp8_inputs(case, seed)
    code, amax, scale = [], [], []
    for t in (x, w):
        m = t.float().abs().max()
        s = 448.0 / m                        # the format's scale is a 32-bit number
        code.append((t.float() * s).to(torch.float8_e4m3fn))
        amax.append(m)
        scale.append(s)
    c = code[0].double() @ code[1].double().t() / (scale[0].double() * scale[1].double())
    return {"c": c, "codes": None, "amax": amax[0].double().reshape(1), "scale": (448.0 / amax[0].double()).reshape(1)}


def _exact_grouped(case, seed):
    return {"c": [a.double() @ bt.double().t() for a, bt in _grouped_inputs(case, seed)]}


def _exact_decode(case, seed):
    h, layers = _decode_inputs(case, seed)
    h = h.double()
    ni = case["ni"]
    for wq, wgu, wd in layers:
        n = h / torch.sqrt((h * h).mean() + 1e-6)
        qkv = wq.double() @ n
        gu = wgu.double() @ n
        a = gu[:ni] * torch.sigmoid(gu[:ni]) * gu[ni:]
        dd = wd.double() @ a
        h = h + dd
    return {"h": h, "qkv": qkv, "a": a} if case["fused"] else {"h": h, "n": n, "qkv": qkv, "gu": gu, "a": a, "dd": dd}


def _exact_mlp(case, seed):
    params, X, T, V = _mlp_inputs(case, seed)
    ps = [p.double().requires_grad_(True) for p in params]
    w1, b1, w2, b2, w3, b3 = ps
    X, T, V = X.double(), T.double(), V.double()
    with torch.enable_grad():
        y = torch.relu(torch.relu(X @ w1.t() + b1) @ w2.t() + b2) @ w3.t() + b3
        loss = (V * (y - T) ** 2).sum() / V.sum().clamp(min=1.0)
        gs = torch.autograd.grad(loss, ps)
    return {"loss": loss.detach().reshape(1), "grads": torch.cat([g.reshape(-1) for g in gs])}


_EXACT = {"map": _exact_map, "map2d": _exact_map, "gemm_f32": _exact_gemm, "gemm_bf16": _exact_gemm, "fp8": _exact_fp8,
          "grouped": _exact_grouped, "decode": _exact_decode, "mlp": _exact_mlp}


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)
