"""The workloads whose speed this library is judged by, each through a public
entry point: one spike projection, a decode step (44 projections in one
launch, plain and with its spike producer), a batch of rows sharing one weight
matrix (column gather and tensor cores), the prompt prefill of one projection
and of a whole stack, the continuous-input projections, and the vocabulary
head.  Widths are the paper's decoder (22 blocks, residual 1536, feed-forward
6144, vocabulary 57,344) and ragged sizes around it.

A case is a dict of plain values; "kind" names the path.  Inputs follow the
distributions of paper_2606_03026_gb300/synth.py (quantised normal weights,
Bernoulli spikes, log-normal column rates in prefill, N(0, 1) activations),
drawn on the GPU from the seed.
"""
import ctypes
import math

import torch

from paper_2606_03026_gb300 import spikeproj as sp

D, FF, BLOCKS, VOCAB = 1536, 6144, 22, 57344
BETA, THETA = 0.9, 1.0                       # the producer's leak and threshold
FMT_BYTES = {"u8": 1, "bool8": 1}


def listed():
    return [
        # the smallest call: one token through one mixer projection
        dict(name="decode", kind="decode", N=D, K=D, p=0.1, fmt="bits"),
        # one token through every binary-input projection of the decoder
        dict(name="step", kind="step", blocks=BLOCKS, d=D, ff=FF, p=0.1, fmt="bits"),
        # the same step with its spikes produced from membrane states
        dict(name="step_lif", kind="step_lif", blocks=BLOCKS, d=D, ff=FF),
        # a few concurrent requests sharing the weights: too few rows for the
        # tensor cores
        dict(name="batched_rows8", kind="batched", N=D, K=FF, B=8, p_lo=0.05, p_hi=0.2, fmt="bits",
             strategy="gather"),
        # 64 concurrent requests
        dict(name="batched_rows64", kind="batched", N=D, K=FF, B=64, p_lo=0.05, p_hi=0.2, fmt="bits",
             strategy="gemm"),
        # a 512-token prompt through one feed-forward down projection, spikes
        # as torch.bool
        dict(name="prefill", kind="prefill", N=D, K=FF, T=512, p=0.15, fmt="bool8",
             strategy="gemm"),
        # a short prompt of odd length and width as byte spikes, the strategy
        # left to the library
        dict(name="prefill_ragged", kind="prefill", N=1040, K=1990, T=173, p=0.15, fmt="u8",
             strategy="auto"),
        # a 512-token prompt through the down projections of every block
        dict(name="prefill_step", kind="prefill_step", blocks=BLOCKS, N=D, K=FF, T=512, p=0.15,
             fmt="bool8"),
        # the continuous-input projections of a decode step (query/key/value,
        # attention output, feed-forward up), one token
        dict(name="dense_step", kind="dense", blocks=BLOCKS, d=D, ff=FF, B=1),
        # the same for four tokens (concurrent requests or speculated tokens)
        dict(name="dense_step_rows4", kind="dense", blocks=BLOCKS, d=D, ff=FF, B=4),
        # the vocabulary head for one token, the paper's trace gate
        dict(name="head", kind="head", V=VOCAB, K=D, B=1, tau=0.5, k_sel=64),
        # and for four, the paper's power gate
        dict(name="head_rows4", kind="head", V=VOCAB, K=D, B=4, tau=4.0, k_sel=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _n(rng, lo, hi):
    """Output channels: any multiple of 16."""
    return max(1, _log(rng, lo, hi) // 16) * 16


def draw(rng):
    kind = rng.choice(["decode", "step", "step_lif", "batched", "batched", "prefill", "prefill",
                       "prefill_step", "dense", "dense", "head"])
    if kind == "decode":
        return dict(kind=kind, N=_n(rng, 256, 4096), K=_log(rng, 200, FF), p=rng.choice([0.02, 0.05, 0.1, 0.2, 0.5]),
                    fmt=rng.choice(["bits", "bits", "u8"]))
    if kind == "step":
        d = _n(rng, 512, D)
        return dict(kind=kind, blocks=rng.randint(2, BLOCKS), d=d, ff=4 * d,
                    p=rng.choice([0.05, 0.1, 0.2]), fmt=rng.choice(["bits", "bits", "u8"]))
    if kind == "step_lif":
        d = _n(rng, 512, D)
        return dict(kind=kind, blocks=rng.randint(2, BLOCKS), d=d, ff=4 * d)
    if kind == "batched":
        B = _log(rng, 2, 64)
        strategy = rng.choice(["gather", "gemm"]) if B <= 16 else "gemm"
        return dict(kind=kind, N=_n(rng, 256, 2048), K=_log(rng, 512, FF), B=B, p_lo=0.05, p_hi=0.2,
                    fmt=rng.choice(["bits", "bits", "u8", "bool8"]), strategy=strategy)
    if kind == "prefill":
        return dict(kind=kind, N=_n(rng, 512, 2048), K=_log(rng, 512, FF), T=_log(rng, 65, 512), p=0.15,
                    fmt=rng.choice(["bool8", "bool8", "u8", "bits"]),
                    strategy=rng.choice(["gemm", "gemm", "auto"]))
    if kind == "prefill_step":
        return dict(kind=kind, blocks=rng.randint(2, BLOCKS), N=_n(rng, 512, D), K=_log(rng, 512, FF),
                    T=_log(rng, 64, 512), p=0.15, fmt=rng.choice(["bool8", "bool8", "u8", "bits"]))
    if kind == "dense":
        d = rng.choice([_log(rng, 256, D), 64 * rng.randint(4, 24)])
        return dict(kind=kind, blocks=rng.randint(1, BLOCKS), d=d, ff=4 * d, B=rng.randint(1, 4))
    return dict(kind=kind, V=_log(rng, 4000, VOCAB), K=rng.choice([_log(rng, 512, D), D]), B=rng.randint(1, 4),
                tau=rng.choice([0.0, 0.5, 4.0]), k_sel=rng.choice([16, 32, 64]))


# --- inputs ------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _weights(g, rows, cols, ld=None):
    """INT8 [rows][ld] of quantised N(0, 1) values (127 at about 4 sigma)."""
    ld = cols if ld is None else ld
    W = torch.randn(rows, ld, generator=g, device="cuda", dtype=torch.bfloat16)
    return W.mul_(127 / 4).round_().clamp_(-127, 127).to(torch.int8)


def _scales(g, n):
    return torch.rand(n, generator=g, device="cuda").mul_(0.02).add_(0.02)


def _pack(x):
    """bool [R][K] -> int32 words [R][ceil(K / 32)], bit k % 32 of word k / 32."""
    R, K = x.shape
    w = -(-K // 32)
    pad = torch.zeros(R, 32 * w, dtype=torch.int64, device="cuda")
    pad[:, :K] = x
    words = (pad.view(R, w, 32) << torch.arange(32, device="cuda")).sum(-1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)


def _spikes(g, R, K, p):
    """bool [R][K]; p a number or a tensor that broadcasts to [R][K]."""
    return torch.rand(R, K, generator=g, device="cuda") < p


def _as_fmt(x, fmt, g):
    """The rows of x in a spike format: (tensor, row stride in its elements)."""
    if fmt == "bits":
        t = _pack(x)
    elif fmt == "u8":                        # any nonzero byte is a spike
        t = torch.where(x, torch.randint(1, 256, x.shape, generator=g, device="cuda"), 0).to(torch.uint8)
    else:                                    # torch.bool rows, padded to 16 bytes
        t = torch.zeros(x.shape[0], -(-x.shape[1] // 16) * 16, dtype=torch.bool, device="cuda")
        t[:, :x.shape[1]] = x
    return t, t.shape[1]


def _outputs(*shape):
    return (torch.zeros(*shape, dtype=torch.int32, device="cuda"),
            torch.zeros(*shape, dtype=torch.float32, device="cuda"))


def _prefill_rates(g, K, p):
    return (p * torch.exp(0.5 * torch.randn(K, generator=g, device="cuda"))).clamp_(max=1.0)


def _dense_shapes(case):
    d = case["d"]
    return [(n, d) for _ in range(case["blocks"]) for n in (3 * d, d, case["ff"])]


def _draw_inputs(case, seed):
    """The inputs of a case, before they are put into a plan or a format:
    a dict that both prepare() and exact() start from."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("decode", "batched", "prefill", "prefill_step"):
        N, K = case["N"], case["K"]
        n = case.get("blocks", 1)
        W = [_weights(g, K, N) for _ in range(n)]                 # column-major [K][N]
        s = [_scales(g, N) for _ in range(n)]
        if kind == "decode":
            x = [_spikes(g, 1, K, case["p"])]
        elif kind == "batched":
            p = case["p_lo"] + (case["p_hi"] - case["p_lo"]) * torch.rand(case["B"], 1, generator=g, device="cuda")
            x = [_spikes(g, case["B"], K, p)]
        else:
            x = [_spikes(g, case["T"], K, _prefill_rates(g, K, case["p"])) for _ in range(n)]
        return dict(g=g, W=W, s=s, x=x)
    if kind in ("step", "step_lif"):
        d, ff = case["d"], case["ff"]
        Ks = [d, ff] * case["blocks"]
        W = [_weights(g, K, d) for K in Ks]
        s = [_scales(g, d) for _ in Ks]
        if kind == "step":
            return dict(g=g, W=W, s=s, x=_spikes(g, len(Ks), ff, case["p"]), Ks=Ks)
        # states of a running layer and one step's currents: about 10% fire
        v = torch.rand(len(Ks), ff, generator=g, device="cuda").mul_(1.2).sub_(0.2)
        I = torch.randn(len(Ks), ff, generator=g, device="cuda").mul_(0.3).add_(0.135)
        return dict(g=g, W=W, s=s, v=v, I=I, Ks=Ks)
    if kind == "dense":
        d = case["d"]
        shapes = _dense_shapes(case)
        W = [_weights(g, n, k, -(-k // 16) * 16) for n, k in shapes]
        s = [_scales(g, n) for n, _ in shapes]
        x = torch.randn(case["blocks"], case["B"], -(-d // 4) * 4, generator=g, device="cuda")
        return dict(g=g, W=W, s=s, x=x, shapes=shapes)
    V, K = case["V"], case["K"]
    W = _weights(g, V, K, -(-K // 16) * 16)
    # logits with a standard deviation near 2.5
    s = (2.5 / math.sqrt(K) / (127 / 4)) * (0.8 + 0.4 * torch.rand(V, generator=g, device="cuda"))
    h = torch.randn(case["B"], -(-K // 4) * 4, generator=g, device="cuda")
    return dict(g=g, W=W, s=s, h=h)


def prepare(case, seed):
    i = _draw_inputs(case, seed)
    kind = case["kind"]
    st = dict(kind=kind, **i)
    if kind in ("decode", "batched", "prefill", "prefill_step"):
        N, K = case["N"], case["K"]
        rows = case.get("B", case.get("T", 1))
        gemm = kind != "decode" and case.get("strategy", "gemm") != "gather"
        st["plans"] = [sp.Plan(W, s, N, K, max_batch=rows, gemm=gemm) for W, s in zip(i["W"], i["s"])]
        st["rows"], st["fmt"], st["strategy"] = rows, case["fmt"], case.get("strategy")
        xs = [_as_fmt(x, case["fmt"], i["g"]) for x in i["x"]]
        st["x"], st["ld"] = [t for t, _ in xs], xs[0][1]
        st["acc"], st["y"] = _outputs(len(xs), rows, N)
        if kind == "prefill_step":
            st["group"] = sp.Group(st["plans"])
            st["accs"], st["ys"] = list(st["acc"]), list(st["y"])
    elif kind in ("step", "step_lif"):
        st["plans"] = [sp.Plan(W, s, case["d"], K) for W, s, K in zip(i["W"], i["s"], i["Ks"])]
        st["group"] = sp.Group(st["plans"])
        st["ld_out"] = case["d"]
        st["acc"], st["y"] = _outputs(len(i["Ks"]), case["d"])
        if kind == "step":
            st["fmt"] = case["fmt"]
            st["x"], st["ld"] = _as_fmt(i["x"], case["fmt"], i["g"])
        else:
            st["v_out"] = torch.zeros_like(i["v"])
            st["bits"] = torch.zeros(len(i["Ks"]), -(-case["ff"] // 32), dtype=torch.int32, device="cuda")
    elif kind == "dense":
        per = 4 * case["d"] + case["ff"]
        st["B"] = B = case["B"]
        st["y"] = torch.zeros(case["blocks"], B, per, device="cuda")
        # the problem table of the call, kept as a program keeps it
        table = (sp.SpDense * len(i["shapes"]))()
        off = 0
        for j, (n, k) in enumerate(i["shapes"]):
            b, off = j // 3, 0 if j % 3 == 0 else off
            W, x = i["W"][j], i["x"][b]
            table[j] = sp.SpDense(W.data_ptr(), W.shape[1], i["s"][j].data_ptr(), x.data_ptr(), x.shape[1],
                                  st["y"][b].data_ptr() + 4 * off, per, n, k)
            off += n
        st["table"], st["count"] = table, len(i["shapes"])
    else:
        B, k = case["B"], case["k_sel"]
        st["head"] = sp.Head(i["W"], i["s"], case["K"])
        st["tau"], st["k_sel"] = case["tau"], k
        st["token"], st["gap"] = _outputs(B)
        st["verified"] = torch.zeros(B, dtype=torch.int32, device="cuda")
        st["cand"], st["r"] = _outputs(B, k)
        st["z"] = torch.zeros(B, case["V"], device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind == "decode":
        st["plans"][0].decode(st["x"][0], st["fmt"], st["acc"], st["y"])
    elif kind in ("batched", "prefill"):
        st["plans"][0].batched(st["x"][0], st["fmt"], st["rows"], st["ld"], st["acc"], st["y"], st["strategy"])
    elif kind == "prefill_step":
        st["group"].prefill(st["x"], st["fmt"], st["rows"], st["ld"], st["accs"], st["ys"])
    elif kind == "step":
        st["group"].decode(st["x"], st["fmt"], st["ld"], st["acc"], st["y"], st["ld_out"])
    elif kind == "step_lif":
        st["group"].decode_lif(st["v"], st["v_out"], st["I"], BETA, THETA, st["bits"], st["acc"], st["y"],
                               st["ld_out"])
        return {"acc": st["acc"], "y": st["y"], "v": st["v_out"], "bits": st["bits"]}
    elif kind == "dense":
        status = sp.lib().spike_proj_dense(ctypes.addressof(st["table"]), st["count"], st["B"],
                                           torch.cuda.current_stream().cuda_stream)
        if status != sp.SP_OK:
            raise sp.SpikeProjError(status, "spike_proj_dense")
        return {"y": st["y"]}
    else:
        st["head"](st["h"], st["tau"], st["k_sel"], st["token"], st["verified"], st["gap"], st["cand"], st["r"],
                   st["z"])
        return {k: st[k] for k in ("token", "verified", "gap", "cand", "r", "z")}
    return {"acc": st["acc"], "y": st["y"]}


def _project(W, s, x):
    """acc and y of bool rows x [R][K] over column-major W [K][N], in 64 bits."""
    acc = x.double() @ W.double()
    return acc, acc * s.double()


def exact(case, seed):
    i = _draw_inputs(case, seed)
    kind = case["kind"]
    if kind in ("decode", "batched", "prefill", "prefill_step"):
        out = [_project(W, s, x) for W, s, x in zip(i["W"], i["s"], i["x"])]
        return {"acc": None, "y": torch.stack([y for _, y in out])}
    if kind == "step":
        out = [_project(W, s, i["x"][j:j + 1, :K]) for j, (W, s, K) in enumerate(zip(i["W"], i["s"], i["Ks"]))]
        return {"acc": None, "y": torch.cat([y for _, y in out])}
    if kind == "step_lif":
        # the fused multiply-add rounds once to FP32; the spikes follow from it
        u = (torch.tensor(BETA, dtype=torch.float32).double().item() * i["v"].double() + i["I"].double()).float()
        x = u >= THETA
        v = torch.where(x, u.double() - THETA, u.double())
        for j, K in enumerate(i["Ks"]):
            v[j, K:] = 0                     # columns past a projection's own are not written
        out = [_project(W, s, x[j:j + 1, :K]) for j, (W, s, K) in enumerate(zip(i["W"], i["s"], i["Ks"]))]
        return {"acc": None, "y": torch.cat([y for _, y in out]), "v": v, "bits": None}
    if kind == "dense":
        d, y = case["d"], []
        for b in range(case["blocks"]):
            x = i["x"][b, :, :d].double()
            y.append(torch.cat([x @ i["W"][j][:, :d].double().T * i["s"][j].double()
                                for j in range(3 * b, 3 * b + 3)], dim=1))
        return {"y": torch.stack(y)}
    # the head: the activation codes are defined in FP32, the rest in 64 bits
    K, k = case["K"], case["k_sel"]
    h, W, s = i["h"][:, :K], i["W"][:, :K].double(), i["s"]
    sx = h.abs().amax(1, keepdim=True).clamp_(min=1e-8) / 127.0
    a = torch.round(h / sx).clamp_(-127, 127).double() @ W.T
    z32 = s * (sx * a.float())               # the order of the rows is FP32's
    z = s.double() * (sx.double() * a)
    order = torch.sort(z32, dim=1, descending=True, stable=True)
    top = order.indices[:, :k]
    gap = order.values[:, 0] - order.values[:, 1]
    r = torch.gather(h.double() @ W.T, 1, top) * s.double()[top]
    r = torch.where((gap < case["tau"])[:, None], r, torch.zeros_like(r))   # unverified rows stay unwritten
    return {"token": None, "verified": None, "gap": gap.double(), "cand": None, "r": r, "z": z}


def work(case):
    kind = case["kind"]
    if kind in ("decode", "batched", "prefill", "prefill_step"):
        N, K, n = case["N"], case["K"], case.get("blocks", 1)
        R = case.get("B", case.get("T", 1))
        p = case.get("p", (case.get("p_lo", 0) + case.get("p_hi", 0)) / 2)
        row = K if case["fmt"] in FMT_BYTES else -(-K // 32) * 4
        cols = 1 - (1 - p) ** R              # share of the columns that any row needs
        return {"bytes": n * (cols * K * N + R * row + 4 * N + 8 * R * N), "flops": n * 2 * p * R * K * N}
    if kind in ("step", "step_lif"):
        d, ff, n = case["d"], case["ff"], case["blocks"]
        p = case.get("p", 0.1)
        row = 12 + 1 / 8 if kind == "step_lif" else (1 if case["fmt"] in FMT_BYTES else 1 / 8)
        return {"bytes": n * ((d + ff) * (p * d + row) + 2 * 12 * d), "flops": n * 2 * p * (d + ff) * d}
    if kind == "dense":
        B = case["B"]
        w = sum(n * k for n, k in _dense_shapes(case))
        rows = sum(n for n, _ in _dense_shapes(case))
        return {"bytes": w + 4 * rows + 4 * B * (rows + case["blocks"] * case["d"]), "flops": 2 * B * w}
    V, K, B = case["V"], case["K"], case["B"]
    return {"bytes": V * K + 4 * V + 4 * B * (K + V), "flops": 2 * B * V * K}


def tolerance(case):
    # FP32 sums of K products, which another order of the sum changes: four
    # times the 1.4e-7 measured against exact().  Integer sums and their one
    # FP32 multiply leave nothing to choose.
    if case["kind"] in ("dense", "head"):
        return {"rel": 6e-7, "max": 3e-6}
    return "exact"
