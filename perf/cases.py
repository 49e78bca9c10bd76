"""Performance cases of the W4A4 bitmap-sparse SpMM: what a program that uses the library has it do.

A case is one pass through the public entry points of ``paper_2608_09291_b200.binding``:

``spmm``    ``SparseWeight.spmm``: one projection on packed INT4 activations. "int32" asks for the integer
            sums, "fp16" for the fused dequantisation. The weight is held in the default format (one mask
            bit per 2 x 1 weights, "2x1"), in the paper's 2 x 2 union format ("2x2"), or as INT2 weights
            ("w2"); rows "sorted" orders the rows of a matrix of uneven density before it is cut in strips.
``layer``   the seven projections of one decoder layer (Q, K, V, O, gate, up, down) one after the other on the
            caller's stream, into output buffers that the caller keeps.
``chain``   the same layer as chained calls, ``SparseWeight.spmm_requant``: fp16 activations in, INT4 inside,
            fp16 out; [Q;K;V] and [gate;up] are stacked, every call leaves the absmax the next one needs.
``load``    what a program pays to bring one dense pruned weight from host memory into use: encode it, upload
            it, run the first product.

The calls are eager, as a program makes them; weights, scales and activations are in hand before the pass. The
listed shapes are the LLaMA-2-7B / 13B / 70B shaped projections of this repository's configurations, its small
1024 x 1024 case, and one shape that divides into nothing.
"""
from __future__ import annotations

import math

import torch

from paper_2608_09291_b200 import binding

LARGEST = 28672 * 8192           # weights of the largest matrix (70B-shaped FFN)
LARGEST_LOAD = 11008 * 4096      # weights of the largest matrix a "load" case encodes


def listed():
    def spmm(name, M, K, s, N, out, fmt="2x1", rows="plain"):
        return {"name": name, "op": "spmm", "M": M, "K": K, "sparsity": s, "N": N, "out": out, "fmt": fmt, "rows": rows}

    return [
        # the smallest call of the repository's configurations: latency and launch cost
        spmm("single 1024 N8", 1024, 1024, 0.5, 8, "int32"),
        # 7B-shaped attention projection, a batch of 8 tokens: the benchmark's headline
        spmm("attn7b N8", 4096, 4096, 0.5, 8, "fp16"),
        # the same projection less sparse, a batch of 32
        spmm("attn7b s30 N32", 4096, 4096, 0.3, 32, "fp16"),
        # 7B-shaped FFN, uneven row density, sorted rows: single-token decode through the up projection
        spmm("ffn7b up sorted N1", 11008, 4096, 0.5, 1, "fp16", rows="sorted"),
        # ... and the long-K down projection for a batch of 32, integer sums
        spmm("ffn7b down sorted N32", 4096, 11008, 0.5, 32, "int32", rows="sorted"),
        # a whole 13B-shaped decoder layer at a batch of 16: weights stream from HBM
        {"name": "layer13b N16", "op": "layer", "hidden": 5120, "ffn": 13824, "sparsity": 0.5, "N": 16},
        # the same layer with fp16 activations travelling between the projections
        {"name": "chain13b N16", "op": "chain", "hidden": 5120, "ffn": 13824, "sparsity": 0.5, "N": 16},
        # 70B-shaped FFN up projection, a batch of 8: the bandwidth case
        spmm("ffn70b up N8", 28672, 8192, 0.6, 8, "int32"),
        # 70B-shaped FFN down projection at the largest batch the library takes
        spmm("ffn70b down N64", 8192, 28672, 0.6, 64, "fp16"),
        # INT2 weights (W2A4) at the 70B shape, a small batch
        spmm("ffn70b up w2 N16", 28672, 8192, 0.6, 16, "fp16", fmt="w2"),
        # nothing divides: odd M, odd K (byte-wise activations), the paper's union format
        spmm("ragged 2x2 N5", 5003, 3001, 0.5, 5, "fp16", fmt="2x2"),
        # model load: encode one 7B-shaped FFN matrix, then use it
        {"name": "load ffn7b", "op": "load", "M": 11008, "K": 4096, "sparsity": 0.5, "N": 8, "fmt": "2x1", "rows": "plain"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A dimension: mostly a multiple of 128 as model dimensions are, now and then any number."""
    v = _log_uniform(rng, lo, hi)
    return v if rng.random() < 0.3 else max(128, v // 128 * 128)


def draw(rng):
    """Another case of the same ranges: sizes over their logarithm, every format, output type and batch size."""
    op = rng.choices(["spmm", "layer", "chain", "load"], [14, 2, 2, 2])[0]
    s = round(rng.uniform(0.3, 0.7), 3)
    if op in ("layer", "chain"):
        hidden = max(8, _log_uniform(rng, 1024, 5120) // 64 * 64)
        ffn = max(8, int(hidden * rng.uniform(2.0, 2.7)) // 64 * 64)
        return {"op": op, "hidden": hidden, "ffn": ffn, "sparsity": s, "N": _log_uniform(rng, 1, 64)}
    most = LARGEST_LOAD if op == "load" else LARGEST
    M = _size(rng, 512, 28672)
    K = _size(rng, 512, min(28672, most // M))
    fmt = rng.choices(["2x1", "2x2", "w2"], [6, 2, 2])[0]
    case = {"op": op, "M": M, "K": K, "sparsity": s, "N": _log_uniform(rng, 1, 64),
            "fmt": fmt, "rows": rng.choice(["plain", "plain", "sorted"])}
    if case["rows"] == "sorted":
        case["sparsity"] = 0.5           # the mean of the row densities such a matrix is drawn with
    if op == "spmm":
        case["out"] = rng.choice(["fp16", "int32"])
    return case


# ---- inputs ------------------------------------------------------------------------------------
class _Draws:
    """Seeded draws on the GPU, in the distributions of paper_2608_09291_b200.workloads."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def uniform(self, lo, hi, *shape):
        return torch.rand(shape, device="cuda", generator=self.g) * (hi - lo) + lo

    def weight(self, M, K, sparsity, bits=4, row_varying=False):
        """Pruned weight in host memory (int8, as an encoder receives it): Bernoulli mask, kept values
        uniform over the nonzero values of the type."""
        out = torch.empty((M, K), dtype=torch.int8, device="cuda")
        for r in range(0, M, 4096):
            n = min(4096, M - r)
            keep = self.uniform(0.3, 0.7, n, 1) if row_varying else 1.0 - sparsity
            kept = torch.rand((n, K), device="cuda", generator=self.g) < keep
            if bits == 2:
                v = torch.randint(-2, 1, (n, K), device="cuda", generator=self.g, dtype=torch.int8)
            else:
                v = torch.randint(-8, 7, (n, K), device="cuda", generator=self.g, dtype=torch.int8)
            v += (v >= 0).to(torch.int8)                 # skip zero
            out[r:r + n] = torch.where(kept, v, torch.zeros_like(v))
        return out.cpu().numpy()

    def weight_scale(self, M, K=None):
        s = self.uniform(0.005, 0.02, M)
        if K is not None:                                # chained calls: keep the magnitude level
            s = s * (16.0 / math.sqrt(K))
        return s.to(torch.float16).cpu().numpy()

    def x(self, N, K):
        """Packed INT4 activations, uniform; the unused half of an odd row's last byte is zero."""
        x = torch.randint(0, 256, (N, (K + 1) // 2), device="cuda", generator=self.g, dtype=torch.uint8)
        if K % 2:
            x[:, -1] &= 0x0F
        return x

    def x_scale(self, N):
        return self.uniform(0.01, 0.05, N).to(torch.float16)

    def x_f16(self, N, K):
        """Hidden states: normal, a spread per token, one channel in 256 eight times larger."""
        x = torch.randn((N, K), device="cuda", generator=self.g) * self.uniform(0.2, 3.0, N, 1)
        ch = torch.randperm(K, device="cuda", generator=self.g)[: max(1, K // 256)]
        x[:, ch] *= 8.0
        return x.to(torch.float16)


def _encode_args(case):
    """(format, flags) of an encode call: the default tile, or the 2 x 2 union format."""
    flags = binding.US_ENCODE_SORT_ROWS if case["rows"] == "sorted" else 0
    if case["fmt"] == "2x1":
        return None, flags
    if case["fmt"] == "w2":
        flags |= binding.US_ENCODE_W2
    strips, K = (case["M"] + 15) // 16, case["K"]
    tile = next((t for t in (1024, 512) if strips * -(-K // t) >= 600), 256)
    return (16, tile, 2, 2), flags


def _layer_shapes(case):
    h, f = case["hidden"], case["ffn"]
    return [(h, h)] * 4 + [(f, h)] * 2 + [(h, f)]


def prepare(case, seed):
    d = _Draws(seed)
    op, N = case["op"], case["N"]
    state = {"op": op, "N": N}
    if op == "layer":
        shapes = _layer_shapes(case)
        state["weights"] = [binding.SparseWeight(d.weight(M, K, case["sparsity"]), d.weight_scale(M)) for M, K in shapes]
        xa, xb, xc, xd = d.x(N, case["hidden"]), d.x(N, case["hidden"]), d.x(N, case["hidden"]), d.x(N, case["ffn"])
        state["X"] = [xa, xa, xa, xb, xc, xc, xd]
        state["x_scale"] = [d.x_scale(N) for _ in shapes]
        state["Y"] = [torch.empty((N, M), dtype=torch.float16, device="cuda") for M, _ in shapes]
        return state
    if op == "chain":
        h, f = case["hidden"], case["ffn"]
        shapes = [(3 * h, h), (h, h), (2 * f, h), (h, f)]
        state["weights"] = [binding.SparseWeight(d.weight(M, K, case["sparsity"]), d.weight_scale(M, K)) for M, K in shapes]
        state["X"] = d.x_f16(N, h)
        state["amax"] = [binding.new_amax() for _ in range(5)]
        state["next"] = [(0, h), (0, h), (0, f), (0, h)]     # the columns each next call reads
        state["Y"] = [torch.empty((N, M), dtype=torch.float16, device="cuda") for M, _ in shapes]
        return state
    bits = 2 if case["fmt"] == "w2" else 4
    W = d.weight(case["M"], case["K"], case["sparsity"], bits, case["rows"] == "sorted")
    s_w = d.weight_scale(case["M"])
    fmt, flags = _encode_args(case)
    state["X"], state["x_scale"] = d.x(N, case["K"]), d.x_scale(N)
    if op == "load":
        state.update(W=W, w_scale=s_w, fmt=fmt, flags=flags)
        return state
    state["weight"] = binding.SparseWeight(W, s_w, fmt=fmt, flags=flags)
    if case["out"] == "int32":
        state["x_scale"] = None
    return state


def run(state):
    op, N = state["op"], state["N"]
    if op == "spmm":
        return state["weight"].spmm(state["X"], N, state["x_scale"])
    if op == "layer":
        for w, x, sx, y in zip(state["weights"], state["X"], state["x_scale"], state["Y"]):
            w.spmm(x, N, sx, out=y)
        return state["Y"]
    if op == "chain":
        src, amax = state["X"], binding.absmax_f16(state["X"], out=state["amax"][0])
        for w, y, left, cols in zip(state["weights"], state["Y"], state["amax"][1:], state["next"]):
            w.spmm_requant(src, N, amax, out=y, y_amax=left, amax_range=cols)
            src, amax = y[:, cols[0]:cols[1]], left
        return state["Y"]
    w = binding.SparseWeight(state["W"], state["w_scale"], fmt=state["fmt"], flags=state["flags"])
    y = w.spmm(state["X"], N, state["x_scale"])
    return {"y": y, "nnz": w.stats["nnz"], "active_bits": w.stats["sum_P"]}


# ---- what a pass cannot do without ---------------------------------------------------------------
def _stored(M, K, sparsity, fmt, rows):
    """Expected bytes of an encoded weight: active payload and union bitmap, no padding, no offsets."""
    if rows == "sorted":      # keep rates U(0.3, 0.7), alike within a strip: means of (1 - p)^2 and (1 - p)^4
        s2, s4 = 0.25 + 0.4 ** 2 / 12, (0.7 ** 5 - 0.3 ** 5) / (5 * 0.4)
    else:
        s2, s4 = sparsity ** 2, sparsity ** 4
    if fmt == "2x1":
        return M * K * (0.5 * (1 - s2) + 1 / 16)
    return M * K * ((0.25 if fmt == "w2" else 0.5) * (1 - s4) + 1 / 32)


def work(case):
    op, N, s = case["op"], case["N"], case["sparsity"]
    if op in ("layer", "chain"):
        h, f = case["hidden"], case["ffn"]
        shapes = _layer_shapes(case) if op == "layer" else [(3 * h, h), (h, h), (2 * f, h), (h, f)]
        read = 3 * h + f                                    # activations per token: packed INT4, or fp16 in a chain
        b = sum(_stored(M, K, s, "2x1", "plain") + 2 * N * M + 2 * M for M, K in shapes)
        b += N * read * (0.5 if op == "layer" else 2)
        return {"bytes": int(b), "flops": int(2 * N * (1 - s) * sum(M * K for M, K in shapes))}
    M, K = case["M"], case["K"]
    enc = _stored(M, K, s, case["fmt"], case["rows"])
    fp16 = case.get("out", "fp16") == "fp16"
    b = enc + N * ((K + 1) // 2) + N * M * (2 if fp16 else 4) + (2 * (M + N) if fp16 else 0)
    if op == "load":
        b += M * K + enc                                    # the dense weight read, the encoded one written
    return {"bytes": int(b), "flops": int(2 * M * K * N * (1 - s))}


def tolerance(case):
    if case["op"] == "chain":
        # an fp16 output that rounds the other way can move an INT4 code of the next call by one step
        return {"rel": 1e-2}
    if case.get("out") == "int32":
        return "exact"
    return {"rel": 1e-3, "max": 2e-3}                       # one fp16 rounding; whole numbers exactly
