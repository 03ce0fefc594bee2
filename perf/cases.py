"""The measured workloads: what a decoding program asks of this library, through the Python binding.

A case is one pass of one of these paths, with the sizes of the models the repository is configured for (LLaMA-2-7B and
Mixtral-8x7B feed-forward layers, MPT-7B's plain FFN, Mamba2-2.7B projections, the 1024 x 1024 layer of the smoke test):

  fc         scap_sparse_fc, one decode step through `layers` layers of one shape (the layers hold different weights, so the
             weights come from memory as they do in a model, not from L2)
  dense      scap_dense_fc, the unpruned layer, likewise
  host       scap_sparse_fc_host: activations in pinned host memory, result back in host memory
  ffn        scap_glu_ffn (gated) or scap_gelu_ffn, `layers` blocks
  moe        scap_moe_ffn, one layer
  q8, q4     scap_sparse_fc_q8 / scap_sparse_fc_q4, `layers` layers
  grouped    scap_sparse_fc_grouped: rows of several contexts in one call
  calibrate  scap_calibrate / scap_calibrate_ex: mode and threshold of one layer from calibration activations

Thresholds and modes come from the library's own calibration in prepare(), as they do for a user; weights are random with
the scale of trained ones, activations follow the distributions of the repository's input recipes.
"""
import math

import numpy as np
import torch

import paper_2412_07174_b200 as scap

NBINS = 2048
T_CALIB = 512  # calibration rows behind the thresholds of the decode cases


def listed():
    return [
        # a small fp16 layer, one token: nothing but latency and launches
        {"name": "fc_small_fp16_b1", "op": "fc", "K": 1024, "N": 1024, "B": 1, "dt": "fp16", "sparsity": 0.5, "act": "laplace", "layers": 1},
        # the headline: LLaMA-2-7B down projection, one token, 60 % pruned
        {"name": "fc_down_bf16_b1", "op": "fc", "K": 11008, "N": 4096, "B": 1, "dt": "bf16", "sparsity": 0.6, "act": "gated", "layers": 6},
        # Mamba2 in-projection (columns that fill no tile) at the paper's 30 %, three sequences
        {"name": "fc_inproj_bf16_b3", "op": "fc", "K": 2560, "N": 10576, "B": 3, "dt": "bf16", "sparsity": 0.3, "act": "laplace", "layers": 4},
        # Mixtral-sized down projection at the largest batch a call takes
        {"name": "fc_wide_bf16_b16", "op": "fc", "K": 14336, "N": 4096, "B": 16, "dt": "bf16", "sparsity": 0.5, "act": "laplace", "layers": 3},
        # the same layer for a caller whose activations live on the host
        {"name": "host_down_bf16_b1", "op": "host", "K": 11008, "N": 4096, "B": 1, "dt": "bf16", "sparsity": 0.65, "act": "gated", "layers": 6},
        # LLaMA-2-7B SwiGLU block, one token, the paper's 40 % / 70 % targets
        {"name": "swiglu_bf16_b1", "op": "ffn", "gated": True, "D": 4096, "F": 11008, "B": 1, "dt": "bf16", "s1": 0.4, "s2": 0.7, "layers": 2},
        # MPT-7B FFN (dense up projection, GELU, pruned down projection) in fp16, eight sequences
        {"name": "gelu_fp16_b8", "op": "ffn", "gated": False, "D": 4096, "F": 16384, "B": 8, "dt": "fp16", "s1": 0.0, "s2": 0.5, "layers": 2},
        # Mixtral-8x7B expert layer, four tokens
        {"name": "moe_bf16_b4", "op": "moe", "D": 4096, "F": 14336, "E": 8, "top_k": 2, "B": 4, "dt": "bf16", "s1": 0.4, "s2": 0.6},
        # 8-bit weights, eight sequences
        {"name": "q8_down_b8", "op": "q8", "K": 11008, "N": 4096, "B": 8, "dt": "bf16", "sparsity": 0.5, "act": "gated", "layers": 3},
        # 4-bit weights, one token
        {"name": "q4_down_b1", "op": "q4", "K": 11008, "N": 4096, "B": 1, "dt": "fp16", "sparsity": 0.5, "act": "gated", "layers": 6, "group": 128},
        # eight beams of each of four prompts: the rows of a prompt mostly share their pattern
        {"name": "grouped_bf16_b32", "op": "grouped", "K": 11008, "N": 4096, "B": 32, "contexts": 4, "overlap": 0.9, "dt": "bf16", "sparsity": 0.6, "layers": 1},
        # offline calibration of one wide layer
        {"name": "calibrate_2048x14336", "op": "calibrate", "T": 2048, "K": 14336, "dt": "bf16", "sparsity": 0.6, "estimator": 0, "scope": 0},
    ]


def _spread(rng, lo, hi, step):
    """A multiple of `step` between lo and hi, evenly spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi, max(lo, round(v / step) * step)))


def draw(rng):
    op = rng.choice(["fc", "fc", "fc", "dense", "host", "ffn", "ffn", "moe", "q8", "q4", "grouped", "calibrate"])
    dt = rng.choice(["bf16", "fp16"])
    if op == "calibrate":
        est, scope = rng.choice([(0, 0), (0, 0), (0, 0), (2, 0), (1, 0), (0, 1), (2, 1)])
        return {"op": op, "T": _spread(rng, 128, 2048, 1), "K": _spread(rng, 1024, 14336, 8), "dt": dt,
                "sparsity": round(rng.uniform(0.3, 0.9), 3), "estimator": est, "scope": scope}
    if op == "ffn":
        gated = rng.random() < 0.6
        return {"op": op, "gated": gated, "D": _spread(rng, 1024, 4096, 8), "F": _spread(rng, 2048, 14336 if gated else 16384, 8),
                "B": rng.choice([1, 1, 2, 3, 4, 5, 8, 12, 16]), "dt": dt, "s1": rng.choice([0.3, 0.4, 0.5]) if gated else 0.0,
                "s2": round(rng.uniform(0.4, 0.8), 3), "layers": rng.choice([1, 2])}
    if op == "moe":
        return {"op": op, "D": _spread(rng, 1024, 4096, 8), "F": _spread(rng, 2048, 14336, 8), "E": rng.choice([4, 8]), "top_k": rng.choice([1, 2]),
                "B": rng.choice([1, 2, 3, 4]), "dt": dt, "s1": rng.choice([0.3, 0.4, 0.5]), "s2": round(rng.uniform(0.5, 0.7), 3)}
    K = _spread(rng, 1024, 14336, 1 if op in ("fc", "dense") and rng.random() < 0.3 else 8)
    N = _spread(rng, 1024, 11008, 16 if op in ("q8", "q4") else 8)
    if op == "grouped":
        n_ctx = rng.choice([2, 3, 4, 8])
        return {"op": op, "K": K, "N": min(N, 4096), "B": n_ctx * rng.choice([2, 4, 6, 8]), "contexts": n_ctx, "overlap": rng.choice([0.5, 0.9, 1.0]),
                "dt": dt, "sparsity": round(rng.uniform(0.5, 0.8), 3), "layers": 1}
    case = {"op": op, "K": K, "N": N, "B": rng.choice([1, 1, 1, 2, 3, 4, 5, 8, 11, 16]), "dt": dt,
            "sparsity": 0.0 if op == "dense" else round(rng.uniform(0.3, 0.9), 3), "act": rng.choice(["laplace", "gated"])}
    if op in ("q8", "q4"):
        case["layers"] = 1
        if op == "q4":
            case["group"] = rng.choice([32, 64, 128, 128])
    else:
        case["layers"] = rng.choice([1, 2, 4])
    return case


# ---- inputs -------------------------------------------------------------------------------------------------------

def _dtype(case):
    return torch.float16 if case["dt"] == "fp16" else torch.bfloat16


class _Maker:
    """Random tensors on the GPU, from the seed alone."""

    def __init__(self, case, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
        self.dt = _dtype(case)

    def normal(self, *shape, std=1.0, dtype=torch.float32):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=self.g)

    def uniform(self, *shape, lo=0.0, hi=1.0):
        return torch.empty(shape, dtype=torch.float32, device="cuda").uniform_(lo, hi, generator=self.g)

    def laplace(self, *shape, scale):
        v = self.uniform(*shape, lo=-0.499999, hi=0.499999)
        return -scale * torch.sign(v) * torch.log1p(-2.0 * v.abs())

    def weight(self, K, N):
        return self.normal(K, N, std=0.02, dtype=self.dt)

    def rows(self, kind, K, counts):
        """Activations of one layer, `counts` rows each: silu(g) u, or Laplace around a mode per channel."""
        mode = self.uniform(K, lo=-0.5, hi=0.5)
        out = []
        for n in counts:
            if kind == "gated":
                out.append((torch.nn.functional.silu(self.normal(n, K)) * self.normal(n, K)).to(self.dt))
            else:
                out.append((mode + self.laplace(n, K, scale=0.3)).to(self.dt))
        return out


def _calibrated(x_calib, sparsity):
    """m [K] and tau [1] of one layer, by the library's calibration."""
    T, K = x_calib.shape
    m = torch.empty(K, dtype=torch.float32, device="cuda")
    tau = torch.empty(1, dtype=torch.float32, device="cuda")
    pad = x_calib if K % 8 == 0 else torch.nn.functional.pad(x_calib, (0, 8 - K % 8))  # calibration takes multiples of eight channels
    mp = m if K % 8 == 0 else torch.empty(pad.shape[1], dtype=torch.float32, device="cuda")
    ws = torch.empty(scap.scap_calibrate_workspace(T, pad.shape[1], NBINS), dtype=torch.uint8, device="cuda")
    scap.scap_calibrate(pad.contiguous(), sparsity, NBINS, mp, tau, ws)
    if K % 8:
        m.copy_(mp[:K])
    return m, tau


def _f32(*shape):
    return torch.empty(shape, dtype=torch.float32, device="cuda")


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    mk, op = _Maker(case, seed), case["op"]
    st = {"case": case}
    if op == "calibrate":
        T, K = case["T"], case["K"]
        st["x"] = mk.rows("laplace", K, (T,))[0]
        st["m"], st["tau"] = _f32(K), _f32(1)
        st["ws"] = _bytes(scap.scap_calibrate_workspace(T, K, NBINS))
        return st
    B = case["B"]
    if op == "ffn":
        D, F = case["D"], case["F"]
        size = scap.scap_glu_workspace if case["gated"] else scap.scap_gelu_ffn_workspace
        st["ws"] = _bytes(size(B, D, F))
        st["blocks"] = []
        for _ in range(case["layers"]):
            b = {"W1": mk.weight(D, 2 * F if case["gated"] else F), "W2": mk.weight(F, D), "y": _f32(B, D)}
            gamma = torch.exp(0.5 * mk.normal(D))
            hc, b["h"] = ((gamma * mk.normal(n, D)).to(mk.dt) for n in (T_CALIB, B))
            if case["s1"] > 0:
                b["m1"], b["tau1"] = _calibrated(hc, case["s1"])
                b["b1"] = _f32(b["W1"].shape[1])
                scap.scap_fold_bias(b["W1"], b["m1"], None, b["b1"], st["ws"])
            else:
                b["m1"], b["tau1"], b["b1"] = None, torch.zeros(1, device="cuda"), None
            u = hc[:256].float() @ b["W1"].float()
            z = torch.nn.functional.silu(u[:, :F]) * u[:, F:] if case["gated"] else torch.nn.functional.gelu(u)
            b["m2"], b["tau2"] = _calibrated(z.to(mk.dt), case["s2"])
            b["b2"] = _f32(D)
            scap.scap_fold_bias(b["W2"], b["m2"], None, b["b2"], _bytes(scap.scap_fold_bias_workspace(F, D)))
            st["blocks"].append(b)
        return st
    if op == "moe":
        D, F, E = case["D"], case["F"], case["E"]
        st["h"] = mk.normal(B, D).to(mk.dt)
        st["logits"] = mk.normal(B, E)
        st["experts"] = []
        for _ in range(E):
            e = {"Wgu": mk.weight(D, 2 * F), "Wd": mk.weight(F, D), "bgu_fused": _f32(2 * F), "bd_fused": _f32(D)}
            hc = mk.normal(T_CALIB, D).to(mk.dt)
            e["m1"], e["tau1"] = _calibrated(hc, case["s1"])
            u = (hc[:128] @ e["Wgu"]).float()
            e["m2"], e["tau2"] = _calibrated((torch.nn.functional.silu(u[:, :F]) * u[:, F:]).to(mk.dt), case["s2"])
            scap.scap_fold_bias(e["Wgu"], e["m1"], None, e["bgu_fused"], _bytes(scap.scap_fold_bias_workspace(D, 2 * F)))
            scap.scap_fold_bias(e["Wd"], e["m2"], None, e["bd_fused"], _bytes(scap.scap_fold_bias_workspace(F, D)))
            st["experts"].append(e)
        st["y"] = _f32(B, D)
        st["ws"] = _bytes(scap.scap_moe_workspace(B, D, F, E, case["top_k"]))
        return st
    K, N = case["K"], case["N"]
    if op == "grouped":
        C = case["contexts"]
        st["groups"] = [r % C for r in range(B)]
        st["ws"] = _bytes(scap.scap_grouped_workspace())
        ctx_of = lambda n: torch.arange(n, device="cuda") % C  # noqa: E731
        mode, active = mk.uniform(K, lo=-0.5, hi=0.5), mk.uniform(C, K) < 0.5

        def rows(n):
            on = torch.where(mk.uniform(n, K) < case["overlap"], active[ctx_of(n)], mk.uniform(n, K) < 0.5)
            return (mode + mk.laplace(n, K, scale=1.0) * torch.where(on, 0.3, 0.01)).to(mk.dt)
        xc, x = rows(T_CALIB), rows(B)
        m, tau = _calibrated(xc, case["sparsity"])
        W, bf = mk.weight(K, N), _f32(N)
        scap.scap_fold_bias(W, m, None, bf, _bytes(scap.scap_fold_bias_workspace(K, N)))
        st["layers"] = [{"W": W, "x": x, "m": m, "tau": tau, "bf": bf, "y": _f32(B, N)}]
        return st
    st["ws"] = _bytes(scap.scap_fc_host_workspace(B, K, N) if op == "host" else scap.scap_fc_workspace(B, K, N))
    st["layers"] = []
    for _ in range(case["layers"]):
        a = {"y": _f32(B, N), "bf": _f32(N)}
        xc, a["x"] = mk.rows(case["act"], K, (T_CALIB, B))
        if op == "dense":
            a["W"] = mk.weight(K, N)
            a["bf"].normal_(0.0, 0.01, generator=mk.g)
            st["layers"].append(a)
            continue
        a["m"], a["tau"] = _calibrated(xc, case["sparsity"])
        fold_ws = _bytes(scap.scap_fold_bias_workspace(K, N))
        if op == "q8":
            # per-input-channel symmetric quantisation: the largest weight of a row of N normals sits near 3.9 sigma
            a["Wq"] = torch.clamp(torch.round(mk.normal(K, N, std=127.0 / 3.9, dtype=torch.float32)), -127, 127).to(torch.int8)
            a["scale"] = mk.uniform(K, lo=0.8, hi=1.2) * (0.02 * 3.9 / 127.0)
            scap.scap_fold_bias_q8(a["Wq"], a["scale"], a["m"], None, a["bf"], fold_ws)
        elif op == "q4":
            # asymmetric, groups of input channels: the extremes of a group lie near 2.6 sigma on either side
            G = -(-K // case["group"])
            q = torch.clamp(torch.round(mk.normal(K, N, std=15.0 / 5.2, dtype=torch.float32) + 7.5), 0, 15).to(torch.uint8)
            a["Wq"] = (q[:, 0::2] | (q[:, 1::2] << 4)).contiguous()
            a["scale"] = mk.uniform(G, N, lo=0.8, hi=1.2) * (0.02 * 5.2 / 15.0)
            a["zero"] = torch.round(mk.uniform(G, N, lo=5.6, hi=9.4)).to(torch.uint8)
            scap.scap_fold_bias_q4(a["Wq"], a["scale"], a["zero"], case["group"], a["m"], None, a["bf"], fold_ws)
        else:
            a["W"] = mk.weight(K, N)
            scap.scap_fold_bias(a["W"], a["m"], None, a["bf"], fold_ws)
        if op == "host":
            a["x"] = a["x"].cpu().pin_memory()
            a["y"] = torch.empty((B, N), dtype=torch.float32).pin_memory()
        st["layers"].append(a)
    return st


# ---- one pass -----------------------------------------------------------------------------------------------------

def run(state):
    case, ws = state["case"], state["ws"]
    op = case["op"]
    if op == "calibrate":
        if case["estimator"] == 0 and case["scope"] == 0:
            scap.scap_calibrate(state["x"], case["sparsity"], NBINS, state["m"], state["tau"], ws)
        else:
            scap.scap_calibrate_ex(state["x"], case["sparsity"], case["estimator"], case["scope"], NBINS, state["m"], state["tau"], ws)
        return [state["m"], state["tau"]]
    if op == "ffn":
        ffn = scap.scap_glu_ffn if case["gated"] else scap.scap_gelu_ffn
        for b in state["blocks"]:
            ffn(b["h"], b["W1"], b["W2"], b["m1"], b["tau1"], b["b1"], b["m2"], b["tau2"], b["b2"], b["y"], ws)
        return [b["y"] for b in state["blocks"]]
    if op == "moe":
        scap.scap_moe_ffn(state["h"], state["logits"], state["experts"], case["top_k"], state["y"], ws)
        return state["y"]
    for a in state["layers"]:
        if op == "fc":
            scap.scap_sparse_fc(a["x"], a["W"], a["m"], a["tau"], a["bf"], a["y"], ws)
        elif op == "dense":
            scap.scap_dense_fc(a["x"], a["W"], a["bf"], a["y"], ws)
        elif op == "host":
            scap.scap_sparse_fc_host(a["x"], a["W"], a["m"], a["tau"], a["bf"], a["y"], ws)
        elif op == "q8":
            scap.scap_sparse_fc_q8(a["x"], a["Wq"], a["scale"], a["m"], a["tau"], a["bf"], a["y"], ws)
        elif op == "q4":
            scap.scap_sparse_fc_q4(a["x"], a["Wq"], a["scale"], a["zero"], case["group"], a["m"], a["tau"], a["bf"], a["y"], ws)
        else:
            scap.scap_sparse_fc_grouped(a["x"], a["W"], a["m"], a["tau"], a["bf"], a["y"], state["groups"], ws)
    return [a["y"] for a in state["layers"]]


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def _fc_work(B, K, N, kept, union, weight_bytes, x_bytes=2.0):
    """Rows that some batch row keeps, activations, modes, threshold, bias and result; multiply-adds of the kept entries."""
    return np.array([union * K * N * weight_bytes + B * K * x_bytes + 4.0 * K + 4 + 4.0 * N + 4.0 * B * N, 2.0 * B * kept * K * N])


def work(case):
    op = case["op"]
    if op == "calibrate":
        return {"bytes": 2.0 * case["T"] * case["K"] + 4.0 * case["K"] + 4, "flops": 0.0}
    B, L = case["B"], case.get("layers", 1)
    union = lambda s, n: 1.0 - s ** n  # rows keep their entries independently of one another  # noqa: E731
    if op in ("ffn", "moe"):
        D, F, s1, s2 = case["D"], case["F"], case["s1"], case["s2"]
        width = F if op == "ffn" and not case["gated"] else 2 * F
        block = lambda n: _fc_work(n, D, width, 1 - s1, union(s1, n), 2.0) + _fc_work(n, F, D, 1 - s2, union(s2, n), 2.0, 0.0)  # noqa: E731
        if op == "ffn":
            w = L * block(B)
        else:  # an expert has n of the B rows with binomial probability
            E, p = case["E"], case["top_k"] / case["E"]
            w = sum(E * math.comb(B, n) * p ** n * (1 - p) ** (B - n) * block(n) for n in range(1, B + 1)) + np.array([4.0 * B * E, 0.0])
        return {"bytes": float(w[0]), "flops": float(w[1])}
    K, N, s = case["K"], case["N"], case["sparsity"]
    wb = {"q8": 1.0, "q4": 0.5}.get(op, 2.0)
    if op == "grouped":  # a weight row is needed once, whichever contexts keep it: union over contexts of (shared set, then own draws)
        n, ov, p = B // case["contexts"], case["overlap"], min(1.0, 2.0 * (1 - s))
        in_set, off_set = 1 - (1 - p * (ov + 0.5 * (1 - ov))) ** n, 1 - (1 - p * 0.5 * (1 - ov)) ** n
        w = _fc_work(B, K, N, 1 - s, 1 - (1 - 0.5 * (in_set + off_set)) ** case["contexts"], wb)
    else:
        w = _fc_work(B, K, N, 1 - s, union(s, B), wb)
        w[0] += {"q8": 4.0 * K, "q4": 5.0 * N * -(-K // case.get("group", 128))}.get(op, 0.0)
    return {"bytes": float(L * w[0]), "flops": float(L * w[1])}


def tolerance(case):
    if case["op"] == "calibrate":
        return "exact"  # every operation of the definition is rounded on its own: one right answer
    if case["op"] in ("ffn", "moe"):
        # The second mask is taken on fp32 values of the first product: a value within rounding of the threshold may fall on
        # either side of it, which changes a row by about its threshold over the norm of the kept values (1 % for one row).
        return {"rel": 5e-3, "max": 0.2}
    # fp32 sums of exact products, up to 14336 of them: 1e-7 to 1.6e-6 from the same sum in 64 bits (largest entry 4.4e-6)
    return {"rel": 6e-6, "max": 2e-5}


# ---- the same pass in 64 bits -------------------------------------------------------------------------------------

def _pruned(x, m, tau):
    """Eq. 2: the difference to the mode where it reaches the threshold (decided in binary32, as the definition says), else 0."""
    x = x.cuda()
    if m is None:
        return torch.where(x.float().abs() >= tau, x.double(), 0.0)
    return torch.where((x.float() - m).abs() >= tau, x.double() - m.double(), 0.0)


def _block64(h, Win, Wout, m1, tau1, b1, m2, tau2, b2, gated):
    u = _pruned(h, m1, tau1) @ Win.double()
    if b1 is not None:
        u = u + b1.double()
    F = Wout.shape[0]
    z = torch.nn.functional.silu(u[:, :F]) * u[:, F:] if gated else torch.nn.functional.gelu(u)
    z32 = z.float()
    kept = z32.abs() >= tau2 if m2 is None else (z32 - m2).abs() >= tau2
    d = torch.where(kept, z if m2 is None else z - m2.double(), 0.0)
    return d @ Wout.double() + b2.double()


def exact(case, seed):
    st, op = prepare(case, seed), case["op"]
    if op == "calibrate":
        if case["estimator"] != 0 or case["scope"] != 0:
            return None
        # mode: the centre of the fullest of NBINS bins between a channel's extremes, each operation rounded in binary32
        x = st["x"].float()
        lo, hi = x.amin(0), x.amax(0)
        n = torch.full((), float(NBINS), device="cuda")
        bins = torch.clamp(((x - lo) * (n / (hi - lo))).floor().long(), 0, NBINS - 1)
        count = torch.zeros(NBINS, case["K"], dtype=torch.int64, device="cuda").scatter_add_(0, bins, torch.ones_like(bins))
        best = (count == count.amax(0)).to(torch.uint8).argmax(0)  # the lowest of the fullest
        m = torch.where(hi == lo, lo, lo + (best.float() + 0.5) * ((hi - lo) * (1.0 / NBINS)))
        # threshold: the pooled quantile, between neighbours in proportion
        v = (x - m).abs().flatten().sort().values
        pos = case["sparsity"] * (v.numel() - 1)
        j = min(int(pos), v.numel() - 2)
        return [m.double(), (v[j].double() + (pos - j) * (v[j + 1].double() - v[j].double())).reshape(1)]
    if op == "ffn":
        return [_block64(b["h"], b["W1"], b["W2"], b["m1"], b["tau1"], b["b1"], b["m2"], b["tau2"], b["b2"], case["gated"]) for b in st["blocks"]]
    if op == "moe":
        p = torch.softmax(st["logits"].double(), -1)
        top, idx = p.topk(case["top_k"], -1)
        top = top / top.sum(-1, keepdim=True)
        y = torch.zeros(case["B"], case["D"], dtype=torch.float64, device="cuda")
        for e, w in enumerate(st["experts"]):
            rows, slot = (idx == e).nonzero(as_tuple=True)
            if rows.numel():
                out = _block64(st["h"][rows], w["Wgu"], w["Wd"], w["m1"], w["tau1"], w["bgu_fused"], w["m2"], w["tau2"], w["bd_fused"], True)
                y[rows] += top[rows, slot, None] * out
        return y
    out = []
    for a in st["layers"]:
        if op in ("q8", "q4"):
            if op == "q8":
                W = a["Wq"].double() * a["scale"].double()[:, None]
            else:
                q = torch.stack((a["Wq"] & 15, a["Wq"] >> 4), -1).flatten(1).double()
                g = torch.arange(case["K"], device="cuda") // case["group"]
                W = a["scale"].double()[g] * (q - a["zero"].double()[g])
        else:
            W = a["W"].double()
        d = a["x"].double() if op == "dense" else _pruned(a["x"], a["m"], a["tau"])
        out.append(d @ W + a["bf"].double())
    return out
