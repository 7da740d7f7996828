"""The work that a user of this library has it do, as timed cases.

Every case names a path and a layer.  Paths:

  decode   one token:  y = W x over the columns the pruning test keeps          spdp_spmspv
  swiglu   the same behind a gated MLP's activation, which also makes the mask  spdp_swiglu_dp, spdp_spmspv
  host     one token whose vectors live in pinned host memory                   spdp_spmspv_host
  q4       one token on the 4-bit payload                                       spdp_pack_tiled_cbc_q4, spdp_spmspv
  batch    3 to 8 tokens in one pass                                            spdp_spmspv_batch
  prefill  many tokens, static pruning only                                     spdp_spmm
  pack     a dense pruned layer into the packed format and back                 spdp_pack_tiled_cbc, spdp_unpack

A layer is M x K fp16 with a share `sparsity` of its weights pruned by magnitude (`spread`: from column to column by
that much around it); `skip` is the share of activations below the pruning threshold, which is one number that a
program has calibrated beforehand.  Weights are N(0, 0.02^2), activations N(0, 1) or Laplace, as in the benchmark.
"""
import math
import statistics

import torch

from paper_2607_21985_b200 import spdp

_NORMAL = statistics.NormalDist()
_STD = 0.02


def _abs_normal_quantile(p):
    """The share p of |N(0, 1)| lies below this."""
    return _NORMAL.inv_cdf(0.5 + 0.5 * min(max(p, 0.0), 1.0 - 1e-9))


def listed():
    return [
        # the smallest call: nothing but latency (the size of the smoke check)
        dict(name="decode_1024x1024", path="decode", M=1024, K=1024, sparsity=0.5, skip=0.5, y="f16"),
        # one token through an attention projection of a 7B model
        dict(name="decode_4096x4096", path="decode", M=4096, K=4096, sparsity=0.5, skip=0.5, y="f16"),
        # its MLP down-projection, with the activation in front of it and nine columns in ten skipped
        dict(name="swiglu_4096x11008", path="swiglu", M=4096, K=11008, sparsity=0.7, skip=0.9, y="f16"),
        # the MLP up-projection of a 70B model: the benchmark's layer, the largest decode call
        dict(name="decode_28672x8192", path="decode", M=28672, K=8192, sparsity=0.5, spread=0.2, skip=0.4, y="f16"),
        # no multiple of any tile, very sparse, no dynamic pruning, 32-bit results
        dict(name="decode_6007x5001", path="decode", M=6007, K=5001, sparsity=0.9, skip=0.0, y="f32"),
        # one token end to end from and to the host, up-projection of a 7B model
        dict(name="host_11008x4096", path="host", M=11008, K=4096, sparsity=0.6, skip=0.5, x="laplace", y="f16"),
        # the largest layer with 4-bit weights
        dict(name="q4_28672x8192", path="q4", M=28672, K=8192, sparsity=0.5, spread=0.2, skip=0.4, y="f16"),
        # eight users' tokens at once on the largest layer
        dict(name="batch8_28672x8192", path="batch", M=28672, K=8192, tokens=8, sparsity=0.5, spread=0.2, skip=0.4, y="f16"),
        # a layer as it is loaded: into the format, and back as a check
        dict(name="pack_11008x4096", path="pack", M=11008, K=4096, sparsity=0.6),
        # a prompt of 1024 tokens on the largest layer: the most work of all
        dict(name="prefill1024_28672x8192", path="prefill", M=28672, K=8192, tokens=1024, sparsity=0.5, spread=0.2, y="f16"),
        # a short prompt on an up-projection of a 7B model
        dict(name="prefill128_11008x4096", path="prefill", M=11008, K=4096, tokens=128, sparsity=0.6, y="f16"),
        # nothing a multiple of a tile: rows, columns and tokens
        dict(name="prefill300_4001x4098", path="prefill", M=4001, K=4098, tokens=300, sparsity=0.3, y="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["decode", "decode", "decode", "swiglu", "host", "q4", "q4", "batch", "batch", "prefill", "prefill", "prefill", "pack"])
    odd = rng.random() < 0.4                       # layers of real models are multiples of 128; others are not
    step = 1 if odd else 128
    M = max(step, _log_int(rng, 512, 28672) // step * step)
    K = max(step, _log_int(rng, 512, 11008) // step * step)
    while M * K > 28672 * 8192:
        K = max(step, K // 2 // step * step)
    case = dict(path=path, M=M, K=K, sparsity=round(rng.uniform(0.3, 0.9), 2))
    if rng.random() < 0.3:
        case["spread"] = round(rng.uniform(0.05, min(0.2, 0.95 - case["sparsity"])), 2)
    if path == "pack":
        return case
    case["y"] = rng.choice(["f16", "f16", "f32"])
    if path == "prefill":
        case["tokens"] = _log_int(rng, 16, 1024)
        return case
    case["skip"] = rng.choice([0.0, 0.25, 0.4, 0.5, 0.75, 0.9]) if path != "swiglu" else rng.choice([0.5, 0.75, 0.9])
    if path == "batch":
        case["tokens"] = rng.randint(3, 8)
    if path in ("decode", "host", "q4") and rng.random() < 0.3:
        case["x"] = "laplace"
    return case


class _Layer:
    """A packed layer; gives its device memory back when it goes."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        try:
            spdp.spdp_free(self.handle)
        except Exception:
            pass


def _weights(case, gen):
    M, K = case["M"], case["K"]
    W = torch.randn(M, K, generator=gen, device="cuda", dtype=torch.float32)
    if case.get("spread"):
        s = case["sparsity"] + case["spread"] * (2.0 * torch.rand(K, generator=gen, device="cuda") - 1.0)
        cut = torch.special.ndtri(0.5 + 0.5 * s.double()).float()
    else:
        cut = torch.tensor(_abs_normal_quantile(case["sparsity"]), device="cuda")
    W[W.abs() <= cut] = 0.0
    return (W * _STD).half()


def _activations(case, gen, rows):
    shape = (rows, case["K"])
    if case.get("x") == "laplace":
        u = torch.rand(shape, generator=gen, device="cuda") - 0.5
        return (-u.sign() * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999))).half()
    return torch.randn(shape, generator=gen, device="cuda").half()


def _rule(case):
    skip = case["skip"]
    if skip <= 0.0:
        return spdp.SPDP_DP_NONE, -1.0
    return spdp.SPDP_DP_ABS_GT, -math.log(1.0 - skip) if case.get("x") == "laplace" else _abs_normal_quantile(skip)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    path, M, K = case["path"], case["M"], case["K"]
    W = _weights(case, gen)
    state = dict(path=path)
    if path == "pack":
        state.update(W=W, back=torch.empty_like(W))
        return state
    state["layer"] = _Layer(spdp.spdp_pack_tiled_cbc_q4(W) if path == "q4" else spdp.spdp_pack_tiled_cbc(W))
    del W
    ydt = torch.float32 if case["y"] == "f32" else torch.float16
    if path == "prefill":
        N, ld = case["tokens"], (K + 7) // 8 * 8            # a token's row starts on a 16-byte boundary
        X = torch.zeros(N, ld, dtype=torch.float16, device="cuda")
        X[:, :K] = _activations(case, gen, N)
        state.update(X=X[:, :K], Y=torch.empty(N, M, dtype=ydt, device="cuda"))
        return state
    if path == "swiglu":
        gate, up = _activations(case, gen, 2).unbind(0)
        size = (torch.nn.functional.silu(gate.float()) * up.float()).abs().sort().values
        state.update(gate=gate.contiguous(), up=up.contiguous(), thr=float(size[min(K - 1, int(case["skip"] * K))]),
                     x=torch.empty(K, dtype=torch.float16, device="cuda"),
                     mask=torch.empty((K + 31) // 32, dtype=torch.int32, device="cuda"),
                     y=torch.empty(M, dtype=ydt, device="cuda"))
        return state
    state["rule"], state["thr"] = _rule(case)
    if path == "batch":
        state.update(X=_activations(case, gen, case["tokens"]), Y=torch.empty(case["tokens"], M, dtype=ydt, device="cuda"))
        return state
    x = _activations(case, gen, 1)[0]
    if path == "host":
        state.update(x=x.cpu().pin_memory(), y=torch.empty(M, dtype=ydt).pin_memory())
    else:
        state.update(x=x, y=torch.empty(M, dtype=ydt, device="cuda"))
    return state


def run(state):
    path = state["path"]
    if path == "pack":
        handle = spdp.spdp_pack_tiled_cbc(state["W"])
        info = spdp.spdp_get_info(handle)
        spdp.spdp_unpack(handle, state["back"])
        spdp.spdp_free(handle)
        return dict(weights=state["back"], nnz=int(info.nnz), values_len=int(info.values_len), packed_bytes=int(info.packed_bytes))
    h = state["layer"].handle
    if path == "prefill":
        spdp.spdp_spmm(h, state["X"], state["Y"])
        return state["Y"]
    if path == "batch":
        spdp.spdp_spmspv_batch(h, state["X"], state["rule"], state["thr"], state["Y"])
        return state["Y"]
    if path == "swiglu":
        spdp.spdp_swiglu_dp(state["gate"], state["up"], state["thr"], state["x"], state["mask"])
        spdp.spdp_spmspv(h, state["x"], spdp.SPDP_DP_MASK, 0.0, state["y"], mask=state["mask"])
        return dict(x=state["x"], mask=state["mask"], y=state["y"])
    if path == "host":
        spdp.spdp_spmspv_host(h, state["x"], state["rule"], state["thr"], state["y"])
    else:
        spdp.spdp_spmspv(h, state["x"], state["rule"], state["thr"], state["y"])
    return state["y"]


def work(case):
    """Bytes of the packed column tiles that have to be fetched (bitmap, ColInfo, padded values), vectors in and out,
    multiply-adds on stored weights of kept columns."""
    path, M, K = case["path"], case["M"], case["K"]
    density = 1.0 - case["sparsity"]
    row_tiles = (M + 255) // 256
    unit, size = (32, 0.5) if path == "q4" else (8, 2.0)
    tile = 36.0 + size * (min(M, 256) * density + (unit - 1) / 2.0) + (2.0 if path == "q4" else 0.0)   # an average tile
    tokens = case.get("tokens", 1)
    kept = 1.0 - case.get("skip", 0.0)
    fetched = 1.0 - (1.0 - kept) ** tokens if path == "batch" else kept
    ybytes = M * tokens * (4 if case.get("y") == "f32" else 2)
    packed = row_tiles * K * fetched * tile + row_tiles * ((K + 15) // 16) * 4
    if path == "pack":       # the layer in, the packed form out and in again, the layer out
        return dict(bytes=4.0 * M * K + 2.0 * packed, flops=0.0)
    xbytes = 2 * K * tokens * (4 if path == "swiglu" else 1)      # swiglu: gate, up and x out and in
    return dict(bytes=packed + xbytes + ybytes, flops=2.0 * M * K * density * kept * tokens)


def tolerance(case):
    if case["path"] == "pack":
        return "exact"
    # About four times what was measured against the product in 64 bits.  16-bit results carry one rounding each
    # (2.1e-4); 32-bit results the order of 32-bit sums: 2.2e-7 on the CUDA cores, 7e-7 where the tensor cores add up a
    # few dozen steps (batch), 1.3e-5 where they add up all of K (prefill).  The swiglu path returns its activations and
    # mask too: one 16-bit step of an activation at the threshold turns one bit of the mask.
    if case["path"] == "swiglu":
        return dict(rel=8e-4, max=0.01, differ=0.005)
    if case["y"] == "f32":
        return dict(prefill=dict(rel=5e-5, max=2e-4), batch=dict(rel=3e-6, max=2e-5)).get(case["path"], dict(rel=1e-6, max=4e-6))
    return dict(rel=8e-4, max=0.004)
