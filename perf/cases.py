"""The workloads whose speed matters to a user of this library, one pass each.

A case is a dict of plain values:

* ``kind``: ``spmm`` (one ``rosko_spmm`` on a packed weight), ``batch`` (one
  ``rosko_spmm_batched`` over uneven layers) or ``prune`` (a pruning step of
  training: pack the new weight and its transpose, run both products);
* ``M, K, N``: C (M x N) = A (M x K) . B (K x N);
* ``s``: the share of zeros of A; ``pattern``: where its nonzeros are;
* ``form``: ``f32``, ``bf16`` (FP32 result), ``i8`` (INT32 result) or
  ``i8f`` (INT8 codes, dequantised FP32 result);
* ``relu``: B is a post-ReLU activation (half of it zero) or N(0, 1);
* ``residual``: C += A.B into a residual instead of C = A.B.
"""
import math

import torch

from paper_2307_03930_gb300 import inputs as gen
from paper_2307_03930_gb300 import rosko

FORMS = {"f32": rosko.F32, "bf16": rosko.BF16, "i8": rosko.I8, "i8f": rosko.I8}


def _case(name, M, K, N, s, form, kind="spmm", pattern="magnitude", relu=False, residual=False,
          count=1, shapes=0):
    c = {"kind": kind, "M": M, "K": K, "N": N, "s": s, "form": form, "pattern": pattern,
         "relu": relu, "residual": residual}
    if kind == "batch":
        c.update(count=count, shapes=shapes)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a layer so small that only launches and host work count
        _case("tiny_f32_s90", 96, 640, 200, 0.90, "f32", pattern="uniform"),
        # the plain FP32 form on a square layer
        _case("square_f32_s90", 1024, 1024, 1024, 0.90, "f32", pattern="uniform"),
        # the convolution layer of the bench sweep (im2col, post-ReLU input)
        # at an ordinary, a high and an extreme sparsity
        _case("conv_bf16_s90", 512, 4608, 3136, 0.90, "bf16", relu=True),
        _case("conv_bf16_s99", 512, 4608, 3136, 0.99, "bf16", relu=True),
        _case("conv_bf16_s998", 512, 4608, 3136, 0.998, "bf16", relu=True),
        # the same layer quantised, with the FP32 activations that the next
        # layer reads
        _case("conv_i8_dequant_s90", 512, 4608, 3136, 0.90, "i8f", relu=True),
        # transformer feed-forward layers over 2048 tokens (prefill)
        _case("ffn_up_bf16_s70", 11008, 4096, 2048, 0.70, "bf16"),
        _case("ffn_down_i8_s90", 4096, 11008, 2048, 0.90, "i8"),
        # the same weight on the 16 tokens of one decoding step of a batch
        _case("ffn_decode_bf16_s90", 11008, 4096, 16, 0.90, "bf16"),
        # odd sizes, rows of very uneven length, added into a residual whose
        # rows are not 16-byte aligned
        _case("ragged_bf16_powerlaw", 1000, 700, 333, 0.97, "bf16", pattern="powerlaw", relu=True,
              residual=True),
        # many uneven pruned layers in one call
        _case("batch16_bf16", 4096, 4096, 12544, 0.0, "bf16", kind="batch", pattern="uniform",
              relu=True, count=16, shapes=3),
        # training: after a pruning step, pack the weight and its transpose,
        # forward product and input gradient
        _case("prune_step_bf16_s95", 512, 4608, 3136, 0.95, "bf16", kind="prune", relu=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["spmm", "batch", "prune"], [8, 1, 1])[0]
    pattern = rng.choice(["magnitude", "uniform", "powerlaw", "block4x1"])
    relu = rng.random() < 0.5
    while kind == "batch":
        c = _case("", 4096, 4096, 12544, 0.0, "bf16", kind=kind, pattern=pattern, relu=relu,
                  count=rng.randint(2, 16), shapes=rng.randint(100, 1 << 20))
        # no dearer than the feed-forward layer
        if sum(M * K * N for M, K, N, _ in _problems(c)) <= 11008 * 4096 * 2048:
            return c
    form = "bf16" if kind == "prune" else rng.choice(["f32", "bf16", "bf16", "i8", "i8f"])
    while True:
        # from one small layer to the feed-forward layers, any odd size
        M, K = _log_int(rng, 64, 11008), _log_int(rng, 64, 11008)
        N = _log_int(rng, 8, 12544)
        s = 1.0 - math.exp(rng.uniform(math.log(0.002), math.log(0.5)))
        if kind == "prune" and M * K > 512 * 4608:
            continue
        # no dearer than the feed-forward layer, nor (where each nonzero is
        # multiplied by itself) than the convolution layer at 90 %
        if M * K * N > 11008 * 4096 * 2048 or M * K > 11008 * 4096:
            continue
        if (1.0 - s) * M * K * N <= (0.1 * 512 * 4608 * 3136 if form in ("f32", "i8f")
                                     else 0.3 * 11008 * 4096 * 2048):
            break
    return _case("", M, K, N, s, form, kind=kind, pattern=pattern, relu=relu,
                 residual=kind == "spmm" and rng.random() < 0.25)


def _problems(case):
    """(M, K, N, s) of every product in the pass."""
    if case["kind"] == "batch":
        return gen.c4_shapes(case["shapes"], case["count"])
    return [(case["M"], case["K"], case["N"], case["s"])]


def _weight(M, K, s, pattern, g):
    """A pruned FP32 weight with N(0, 1) entries."""
    W = torch.randn((M, K), device="cuda", generator=g)
    if pattern == "magnitude":
        return W * (W.abs() > math.sqrt(2.0) * float(torch.erfinv(torch.tensor(s, dtype=torch.float64))))
    if pattern == "powerlaw":
        w = torch.rand((M, 1), device="cuda", generator=g).clamp_min(1e-12) ** (-1.0 / 1.5)
        keep = torch.rand((M, K), device="cuda", generator=g) < w * ((1.0 - s) * M / w.sum())
    elif pattern == "block4x1":
        keep = torch.rand(((M + 3) // 4, K), device="cuda", generator=g) < 1.0 - s
        keep = keep.repeat_interleave(4, 0)[:M]
    else:
        keep = torch.rand((M, K), device="cuda", generator=g) < 1.0 - s
    return W * keep


def _padded(x, dtype):
    """x as `dtype`, its rows padded to 16 bytes (the library's rule for B)."""
    per = 16 // torch.empty((), dtype=dtype).element_size()
    out = torch.zeros((x.shape[0], -(-x.shape[1] // per) * per), dtype=dtype, device="cuda")
    out[:, :x.shape[1]] = x
    return out[:, :x.shape[1]]


def _inputs(case, seed):
    """Per problem the tensors a user has: FP32 weight, B, and what the form
    and the options add."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    out = []
    for M, K, N, s in _problems(case):
        p = {"W": _weight(M, K, s, case["pattern"], g)}
        B = torch.randn((K, N), device="cuda", generator=g)
        if case["relu"]:
            B = B.relu()
        if case["form"] in ("i8", "i8f"):
            t = B.abs().amax(0).clamp_min(1e-6) / 127.0
            p["B"] = _padded((B / t).round().clamp(-127, 127), torch.int8)
            if case["form"] == "i8f":
                p["t"] = t
        else:
            p["B"] = _padded(B, torch.bfloat16 if case["form"] == "bf16" else torch.float32)
        if case["kind"] == "prune":
            p["dO"] = _padded(torch.randn((M, N), device="cuda", generator=g), torch.bfloat16)
        c_type = torch.int32 if case["form"] == "i8" else torch.float32
        if case["residual"]:
            R = torch.randn((M, N), device="cuda", generator=g)
            p["R"] = (R * 1000.0).round().to(c_type) if c_type == torch.int32 else R
        out.append(p)
    return out


def prepare(case, seed):
    state = {"case": case, "p": _inputs(case, seed)}
    c_type = torch.int32 if case["form"] == "i8" else torch.float32
    for p, (M, K, N, _) in zip(state["p"], _problems(case)):
        p["C"] = torch.empty((M, N), dtype=c_type, device="cuda")
        if case["kind"] == "prune":
            p["dX"] = torch.empty((K, N), device="cuda")
        else:
            # the packed weight is kept for as long as the layer lives
            p["h"] = rosko.rosko_pack(p["W"], FORMS[case["form"]])
            del p["W"]
    return state


def run(state):
    case, ps = state["case"], state["p"]
    if case["kind"] == "batch":
        return rosko.rosko_spmm_batched([p["h"] for p in ps], [p["B"] for p in ps],
                                        [p["C"] for p in ps])
    p = ps[0]
    if case["kind"] == "prune":
        h = rosko.rosko_pack(p["W"], rosko.BF16)
        rosko.rosko_spmm(h, p["B"], p["C"])
        ht = rosko.rosko_pack_transposed(p["W"], rosko.BF16)
        rosko.rosko_spmm(ht, p["dO"], p["dX"])
        return [p["C"], p["dX"]]
    if case["residual"]:
        p["C"].copy_(p["R"])
    return rosko.rosko_spmm(p["h"], p["B"], p["C"], col_scale=p.get("t"),
                            accumulate=case["residual"])


def work(case):
    el = {"f32": 4, "bf16": 2, "i8": 1, "i8f": 1}[case["form"]]
    nbytes = flops = 0.0
    for M, K, N, s in _problems(case):
        nnz = (1.0 - s) * M * K
        flops += 2.0 * nnz * N
        # a nonzero is its value and a 16-bit index; B rows that no nonzero
        # meets are not read
        rows = K * (1.0 - s ** M)
        nbytes += nnz * (el + 2) + rows * N * el + M * N * 4.0
        if case["residual"]:
            nbytes += M * N * 4.0
        if case["kind"] == "prune":
            # both products, and the FP32 weight read once
            flops += 2.0 * nnz * N
            nbytes += M * K * 4.0 + nnz * (el + 2) + M * N * 2.0 + K * N * 4.0
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """The products of the values that the kernels are given, in 64 bits."""
    if case["form"] == "i8":
        return None
    outs = []
    for p in _inputs(case, seed):
        A = p["W"]
        if case["form"] == "bf16":
            A = A.to(torch.bfloat16)
        if case["form"] == "i8f":
            # symmetric codes per row: q = rint(a / s), s = max |a| / 127
            sc = A.abs().amax(1, keepdim=True) / torch.tensor(127.0, device="cuda")
            sc = torch.where(sc == 0, torch.ones_like(sc), sc)
            A = (A / sc).round().clamp(-127, 127).double() * sc.double()
        C = A.double() @ p["B"].double()
        if case["form"] == "i8f":
            C *= p["t"].double()
        if case["residual"]:
            C += p["R"].double()
        outs.append(C)
        if case["kind"] == "prune":
            outs.append(A.double().t() @ p["dO"].double())
    return outs if case["kind"] in ("batch", "prune") else outs[0]
