"""The work a user has this library do, as measurable cases.

A decoder keeps every pruned projection as a `celty.Matrix` bound to the GPU and calls it once per token with that
token's activations; everything below is such a call (or a short chain of them) through the public binding.  Sizes
are those of the configured LLaMA layers, the small layer of the smoke test, and ragged ones; weights are
N(0, 0.02^2) with unstructured masks (Bernoulli, per-column magnitude, row-clustered power law), activations Laplace,
normal or SiLU(gate) * up, thresholds set for an activation density, as in `paper_2608_01536_b200.synth`.
"""
from __future__ import annotations

import math

import torch

from paper_2608_01536_b200 import celty, synth

# kinds of call:
#   product      y = W . threshold(x, tau), FP32 result: what every projection of a decode step is
#   fp16         the same with an FP16 copy of y in the same launch (the consumer of a projection is FP16)
#   chain        MLP of a decode step: stacked [gate; up] product, SiLU(gate) * up and its survivor list in the same
#                launch, then the down projection from that list
#   swiglu_down  down projection that makes SiLU(gate) * up itself from the FP32 gate/up result
#   batch        N activation vectors against one matrix (a few sequences decoded together)
#   host         activations and result in pinned host memory, copies inside the call
#   static       the entry point for callers that cannot give the library a workspace
#   column       whole-column packing (the paper's own layout) instead of the lane tiles
#   load         a layer from its dense weights and mask: packed, put on the GPU, first product


def listed():
    return [
        # smallest configured layer: launch and set-up latency
        dict(name="small_1024x1024", kind="product", M=1024, K=1024, mask="bernoulli", d_w=0.5, dist="normal", d_a=0.5),
        # attention projection of a 7B decoder, magnitude pruned
        dict(name="attn_4096x4096", kind="product", M=4096, K=4096, mask="magnitude", d_w=0.5, dist="laplace", d_a=0.5),
        # ragged sizes, heavily pruned with clustered rows, few activations: work is small and uneven
        dict(name="ragged_3001x5003", kind="product", M=3001, K=5003, mask="powerlaw", d_w=0.3, dist="laplace", d_a=0.3),
        # gate or up projection of a 7B decoder with the FP16 result its consumer takes
        dict(name="gateup_11008x4096_fp16", kind="fp16", M=11008, K=4096, mask="magnitude", d_w=0.5, dist="laplace", d_a=0.5),
        # tallest configured layer (70B-shaped MLP): bandwidth
        dict(name="mlp_28672x8192", kind="product", M=28672, K=8192, mask="bernoulli", d_w=0.5, dist="laplace", d_a=0.5),
        # whole MLP of a smaller decoder: two dependent calls, list passed on the device
        dict(name="mlp_chain_5504x2048", kind="chain", M=5504, K=2048, mask="bernoulli", d_w=0.5, dist="laplace", d_a=0.4),
        # down projection of a 7B decoder from the raw gate/up result
        dict(name="down_4096x11008_swiglu", kind="swiglu_down", M=4096, K=11008, mask="magnitude", d_w=0.5, dist="normal", d_a=0.5),
        # four sequences decoded together
        dict(name="batch4_4096x4096", kind="batch", M=4096, K=4096, mask="bernoulli", d_w=0.5, dist="laplace", d_a=0.5, N=4),
        # vectors that live on the host
        dict(name="host_5120x5120", kind="host", M=5120, K=5120, mask="bernoulli", d_w=0.5, dist="laplace", d_a=0.4),
        # no workspace
        dict(name="static_4096x4096", kind="static", M=4096, K=4096, mask="bernoulli", d_w=0.5, dist="laplace", d_a=0.5),
        # the published layout
        dict(name="column_4096x4096", kind="column", M=4096, K=4096, mask="bernoulli", d_w=0.5, dist="laplace", d_a=0.5),
        # start-up: every layer of a model goes through this once
        dict(name="load_2048x4096", kind="load", M=2048, K=4096, mask="magnitude", d_w=0.5, dist="laplace", d_a=0.5),
    ]


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["fp16", "chain", "swiglu_down", "batch", "host", "static", "column", "load"])
    # sizes by area (kept below what the largest listed case costs), each side from a few hundred to 28672
    top = {"load": 2 ** 23, "column": 2 ** 24, "static": 2 ** 24, "batch": 2 ** 25, "chain": 2 ** 25}.get(kind, 2 ** 26.5)
    area = math.exp(rng.uniform(math.log(2 ** 20), math.log(top)))
    aspect = math.exp(rng.uniform(-1.3, 1.3))
    M = int(min(28672, max(300, math.sqrt(area * aspect))))
    K = int(min(28672, max(300, area / M)))
    if rng.random() < 0.5:                                   # as model dimensions are: multiples of 64
        M, K = max(320, M // 64 * 64), max(320, K // 64 * 64)
    case = dict(kind=kind, M=M, K=K, mask=rng.choice(["bernoulli", "magnitude", "powerlaw"]),
                d_w=round(rng.uniform(0.3, 0.7), 2), dist=rng.choice(["laplace", "normal", "swiglu"]),
                d_a=round(rng.uniform(0.1, 0.7), 2))
    if kind == "batch":
        case["N"] = rng.randint(2, 8)
    return case


# ----------------------------------------------------------------------------- inputs
def _activations(gen, shape, dist):
    def normal():
        return torch.randn(shape, generator=gen, device="cuda")
    if dist == "laplace":
        u = torch.rand(shape, generator=gen, device="cuda") - 0.5
        v = -torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999))
    elif dist == "normal":
        v = normal()
    else:
        v = torch.nn.functional.silu(normal()) * normal()
    return v.half()


def _threshold(x, d_a):
    """The magnitude below (or at) which a share 1 - d_a of x lies."""
    k = int((1.0 - d_a) * x.numel())
    return float(torch.sort(x.float().abs().reshape(-1))[0][k - 1]) if k > 0 else 0.0


def _threshold_in_gap(h, d_a):
    """A threshold near the same quantile that lies in the middle of a gap between two magnitudes, so that values which
    are themselves results of FP32 sums fall on the same side of it whatever the order of the additions."""
    a = torch.sort(h.float().abs().reshape(-1))[0]
    k, w = int((1.0 - d_a) * a.numel()), max(8, a.numel() // 50)
    lo, hi = max(1, min(k, a.numel() - 1) - w), min(a.numel(), max(k, 1) + w)
    g = lo + int(torch.argmax(a[lo:hi] - a[lo - 1:hi - 1]))
    return float((a[g] + a[g - 1]) * 0.5)


def _layer(gen, M, K, mask, d_w):
    """Dense FP16 weights and their keep mask, both on the GPU."""
    W = torch.randn((M, K), generator=gen, device="cuda", dtype=torch.float16).mul_(0.02)
    if mask == "bernoulli":
        keep = torch.rand((M, K), generator=gen, device="cuda") < d_w
    elif mask == "powerlaw":
        p = torch.from_numpy(synth.powerlaw_row_probability(M, d_w)).to("cuda", torch.float32)
        keep = torch.rand((M, K), generator=gen, device="cuda") < p[:, None]
    else:                                                     # per column, the largest magnitudes
        n_drop = int((1.0 - d_w) * M)
        a = W.abs()
        keep = torch.ones((M, K), dtype=torch.bool, device="cuda")
        keep.scatter_(0, torch.topk(a, n_drop, dim=0, largest=False)[1], False)
    return W, keep


def _host(W, keep):
    return W.cpu().numpy(), keep.to(torch.uint8).cpu().numpy()


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, M, K, d_a = case["kind"], case["M"], case["K"], case["d_a"]
    s = {"kind": kind}
    if kind == "chain":                                       # M = inner size I of the MLP, K = model size
        Wg, kg = _layer(gen, 2 * M, K, case["mask"], case["d_w"])
        Wd, kd = _layer(gen, K, M, case["mask"], case["d_w"])
        x = _activations(gen, (K,), case["dist"])
        s["x"], s["tau"] = x, _threshold(x, d_a)
        xs = torch.where(x.float().abs() > s["tau"], x.float(), torch.zeros((), device="cuda"))
        gu = (Wg.float() * kg) @ xs
        h = (torch.nn.functional.silu(gu[:M]) * gu[M:]).half()
        s["gate_up"] = celty.Matrix(*_host(Wg, kg), device="cuda")
        s["down"] = celty.Matrix(*_host(Wd, kd), device="cuda")
        s["mid"] = celty.SwigluOut(M, _threshold_in_gap(h, d_a), "cuda")
        return s
    W, keep = _layer(gen, M, K, case["mask"], case["d_w"])
    if kind == "swiglu_down":
        s["x"] = torch.randn(2 * K, generator=gen, device="cuda")
        h = (torch.nn.functional.silu(s["x"][:K]) * s["x"][K:]).half()
        s["tau"] = _threshold_in_gap(h, d_a)
        s["h"] = torch.empty(K, dtype=torch.float16, device="cuda")
    elif kind == "batch":
        s["x"] = _activations(gen, (case["N"], K), case["dist"])
        if K % 8:                                             # a batch sits in rows of an aligned buffer
            wide = torch.zeros((case["N"], (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
            wide[:, :K] = s["x"]
            s["x"] = wide[:, :K]
        s["y"] = torch.empty((case["N"], (M + 3) // 4 * 4), dtype=torch.float32, device="cuda")[:, :M]
        s["tau"] = _threshold(s["x"], d_a)
    else:
        s["x"] = _activations(gen, (K,), case["dist"])
        s["tau"] = _threshold(s["x"], d_a)
    if kind == "load":
        s["W"], s["keep"] = _host(W, keep)
        return s
    layout = celty.LAYOUT_COLUMN if kind == "column" else celty.LAYOUT_LANE_TILE
    s["m"] = celty.Matrix(*_host(W, keep), layout=layout, device="cuda")
    if kind == "fp16":
        s["y"] = torch.empty(M, dtype=torch.float32, device="cuda")
        s["y16"] = torch.empty(M, dtype=torch.float16, device="cuda")
    if kind == "host":
        s["x_host"] = s["x"].cpu().pin_memory()
        s["y_host"] = torch.empty(M, dtype=torch.float32).pin_memory()
        s["x_stage"] = torch.empty(K, dtype=torch.float16, device="cuda")
        s["y_stage"] = torch.empty(M, dtype=torch.float32, device="cuda")
    return s


# ----------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "product" or kind == "column":
        return s["m"].spmspv(s["x"], s["tau"])
    if kind == "fp16":
        return s["m"].spmspv_ex(s["x"], s["tau"], s["y"], fp16_out=s["y16"]), s["y16"]
    if kind == "chain":
        mid = s["mid"]
        y = s["gate_up"].spmspv_ex(s["x"], s["tau"], swiglu=mid)
        return y, mid.h, mid.count, s["down"].spmspv_list(mid.idx, mid.val, mid.count)
    if kind == "swiglu_down":
        return s["m"].spmspv_swiglu(s["x"], s["tau"], h_out=s["h"]), s["h"]
    if kind == "batch":
        return s["m"].spmspv_batch(s["x"], s["tau"], y=s["y"])
    if kind == "host":
        return s["m"].spmspv_host(s["x_host"], s["tau"], s["y_host"], s["x_stage"], s["y_stage"])
    if kind == "static":
        return s["m"].spmspv_static(s["x"], s["tau"])
    return celty.Matrix(s["W"], s["keep"], device="cuda").spmspv(s["x"], s["tau"])


# ----------------------------------------------------------------------------- what it cannot do without
def work(case):
    M, K, d_w, d_a, kind = case["M"], case["K"], case["d_w"], case["d_a"], case["kind"]
    N = case.get("N", 1)
    entries = M * K * d_w                                     # 2.5 bytes each: FP16 value and 4-bit run
    fetched = 2.5 * entries * (1.0 - (1.0 - d_a) ** N)        # a batch needs a column when any vector does
    b, f = fetched + N * (2 * K + 4 * M), 2.0 * entries * d_a * N
    if kind == "fp16":
        b += 2 * M
    elif kind == "swiglu_down":
        b += 8 * K                                            # FP32 gate and up in, FP16 h out (in place of x)
    elif kind == "chain":                                     # stacked gate and up, then down
        b, f = 3 * fetched + 2 * K + 8 * M + 2 * M + 6 * d_a * M + 4 * K, 3 * f
    elif kind == "load":
        b += 3 * M * K + 2.5 * entries                        # weights and mask in, packed layer out
    return {"bytes": b, "flops": f}


def tolerance(case):
    # Measured against FP64 evaluations of the same product, and between two runs (whose FP32 additions come in another
    # order): 1.1e-7 to 2.7e-7 in the 2-norm and up to 1.8e-6 in one row (5.6e-7 and 2.1e-6 for whole columns, which are
    # summed with fewer accumulators).  Where an FP16 value made from such a sum is returned, a few of them fall on the
    # neighbouring FP16 number: 7.7e-6 in the 2-norm, one unit in the last place (2^-10 of the value at most) in one row.
    if case["kind"] in ("fp16", "chain", "swiglu_down"):
        return {"rel": 3e-5, "max": 2.2e-3}
    if case["kind"] == "column":
        return {"rel": 2.2e-6, "max": 1e-5}
    return {"rel": 1e-6, "max": 7e-6}
