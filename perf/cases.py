"""The work a user of this library has it do, as cases that can be timed and compared.

A case names an operation and its sizes.  `prepare` draws its inputs on the GPU and makes the
descriptor, workspace and output buffers a program would keep between calls; `run` is one pass
through the C ABI by way of `paper_2609_39813_b200.binding`; its outputs are everything the pass
leaves for the caller: per-use statistics and verdicts, gradients, shifted sums.

  check        bsp_mc_check: the per-use check of normalisation -> FP8 store -> linear, all six reads
  step         the same layer as single operators, once: store forward, incoming gradient, weight
               gradient under one read and normalisation backward under another
  attn_check   bsp_mc_check_attn: the check of attention's D use, BF16 or FP8 operands
  attn_step    attention once: forward statistics, output store, backward under a read at D
  store_check  bsp_mc_check_store: the check with the b-bit per-token store
  coupling     bsp_coupling_check: averages over the forward's own rounding
  probs        bsp_probs_mc: rounded softmax probabilities as the saved tensor
  lsm          bsp_lsm_check: log-softmax with an error in its saved output
"""
import numpy as np
import torch

from paper_2609_39813_b200 import binding as b

POLICIES_ALL = 0x3F
TENSOR = 1


def listed():
    return [
        # the smallest check, as in unit tests and for trying a policy: launches and latency
        dict(name="check_tiny", op="check", norm="rms", dtype="f32", x="normal", T=64, C=128, O=128, K=256),
        # one layer of a 390M-parameter model with outlier channels: the ordinary check
        dict(name="check_390m", op="check", norm="rms", dtype="bf16", x="outliers", T=4096, C=1024, O=4096, K=64),
        # unbiasedness sweep: many draws, LayerNorm with bias, FP32 storage, heavy tails
        dict(name="check_sweep", op="check", norm="layer", dtype="f32", x="student", T=8192, C=2048, O=2048, K=1024),
        # a large MLP layer, few draws: the headline workload of bench.py
        dict(name="check_mlp", op="check", norm="rms", dtype="bf16", x="normal", T=16384, C=4096, O=11008, K=16),
        # one layer evaluated once under a policy, at a ragged token count (a packed batch)
        dict(name="step_ragged", op="step", norm="layer", dtype="f32", x="normal", T=3001, C=1552, O=4112, gain_read=2, w_read=1),
        # the check of attention's D use at the benchmark's shape, both operand modes
        dict(name="attn_check", op="attn_check", B=8, H=16, S=2048, causal=True, fp8=False, K=32),
        dict(name="attn_check_fp8", op="attn_check", B=8, H=16, S=2048, causal=True, fp8=True, K=32),
        # attention forward and backward once, at a ragged sequence length
        dict(name="attn_step_ragged", op="attn_step", B=4, H=16, S=1000, causal=True, fp8=False, read=1),
        # the paper's own store, six bits per entry, at the 390M layer's shape
        dict(name="store_check", op="store_check", norm="rms", dtype="bf16", x="outliers", T=4096, C=1024, O=4096, K=16, bits=6),
        # averages over the forward's rounding, eight pairs of forwards, same shape
        dict(name="coupling", op="coupling", norm="rms", dtype="bf16", x="outliers", T=4096, C=1024, O=4096, pairs=8),
        # rounded probabilities of an attention key block: 128 keys at head width 64
        dict(name="probs", op="probs", rows=16384, n=128, d=64, law=0, param=1.0 / 64, K=256),
        # log-softmax, the paper's case
        dict(name="lsm", op="lsm", rows=64, classes=128, eps=0.1, trials=4096),
    ]


def draw(rng):
    def log(lo, hi, step=1):
        return max(lo, min(hi, int(round((lo * (hi / lo) ** rng.random()) / step)) * step))

    op = rng.choice(["check", "check", "check", "step", "step", "attn_check", "attn_step", "store_check", "coupling", "probs", "lsm"])
    if op in ("check", "step", "store_check", "coupling"):
        c = dict(op=op, norm=rng.choice(["rms", "layer"]), dtype=rng.choice(["f32", "bf16"]),
                 x=rng.choice(["normal", "outliers", "student"]), T=log(64, 16384), C=log(64, 4096, 16), O=log(64, 11008, 16))
        if op == "step":
            c["gain_read"], c["w_read"] = rng.choice([0, 1, 2]), rng.choice([0, 1])
            return c
        if op == "coupling":
            while c["T"] * c["O"] > 1 << 25:
                c["T"] = max(64, c["T"] * 2 // 3)
            c["pairs"] = log(1, 8)
            return c
        c["K"] = log(4, 1024)
        if op == "store_check":
            c["K"], c["bits"] = min(c["K"], 64), rng.choice([5, 6])
        most = min(5.0e12 / (c["T"] * c["C"] * c["O"]), 3.0e9 / (c["T"] * c["C"]))
        c["K"] = max(4, min(c["K"], int(most)))
        return c
    if op in ("attn_check", "attn_step"):
        c = dict(op=op, B=rng.randint(1, 8), H=rng.randint(1, 16), S=log(64, 2048), causal=rng.random() < 0.75,
                 fp8=rng.random() < 0.4)
        c.update(dict(K=log(4, 32)) if op == "attn_check" else dict(read=rng.choice([0, 1, 2])))
        return c
    if op == "probs":
        n, d = (128, 64) if rng.random() < 0.5 else (log(16, 256), log(8, 64))
        rows = log(256, 16384)
        K = max(8, min(log(8, 256), int(16384 * 128 * 64 * 64 / (rows * n * d))))
        return dict(op=op, rows=rows, n=n, d=min(n, d), law=rng.randint(0, 1), param=rng.choice([1.0 / 64, 1.0 / 128]), K=K)
    rows, classes = log(16, 256), log(32, 8192, 4)
    return dict(op=op, rows=rows, classes=classes, eps=rng.choice([0.05, 0.1]), trials=max(2, min(log(64, 4096), int(5.0e8 / (rows * classes)))))


# ---------------------------------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, shape, std, dtype):
    return torch.randn(shape, generator=g, device="cuda").mul_(std).to(dtype)


def _layer_inputs(case, seed):
    """x, gamma, beta, W, dY of one normalisation -> linear layer."""
    g = _gen(seed)
    T, C, O = case["T"], case["C"], case["O"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    x = torch.randn((T, C), generator=g, device="cuda")
    if case["x"] == "outliers":          # one feature in a hundred twenty times as large
        x[:, torch.randperm(C, generator=g, device="cuda")[: max(1, C // 100)]] *= 20.0
    elif case["x"] == "student":         # four degrees of freedom
        chi = sum(torch.randn((T, C), generator=g, device="cuda").square_() for _ in range(4))
        x.div_(chi.mul_(0.25).sqrt_())
    gamma = 1.0 + 0.1 * torch.randn(C, generator=g, device="cuda")
    beta = 0.1 * torch.randn(C, generator=g, device="cuda") if case["norm"] == "layer" else None
    W = _normal(g, (O, C), C ** -0.5, dt)
    dY = _normal(g, (T, O), 0.1 if dt == torch.bfloat16 else 1.0, dt)
    return x.to(dt), gamma, beta, W, dY


def _fill(desc, case, s):
    desc.norm_kind = b.RMSNORM if case["norm"] == "rms" else b.LAYERNORM
    desc.dtype = b.BF16 if case["dtype"] == "bf16" else b.F32
    desc.T, desc.C, desc.O = case["T"], case["C"], case["O"]
    desc.x, desc.gamma, desc.beta, desc.W = (b.ptr(s[k]) for k in ("x", "gamma", "beta", "W"))
    desc.eps = 1e-6 if case["norm"] == "rms" else 1e-5
    desc.tensor_id = TENSOR
    return desc


def _zeros(n, dtype=torch.float32):
    return torch.zeros(n, dtype=dtype, device="cuda")


def prepare(case, seed):
    s = dict(case=case, op=case["op"], seed=int(seed), diag=b.new_diag())
    op = case["op"]
    if op in ("check", "step", "store_check", "coupling"):
        s["x"], s["gamma"], s["beta"], s["W"], s["dY"] = _layer_inputs(case, seed)
        T, C, O = case["T"], case["C"], case["O"]
    if op == "check":
        d = s["desc"] = _fill(b.NormLinearDesc(), case, s)
        d.dY, d.store_fmt, d.grad_fmt, d.forward_mode = b.ptr(s["dY"]), b.E4M3, b.E5M2, b.ROUND_STOCHASTIC
        d.seed, d.policy_mask = s["seed"], POLICIES_ALL
        s["ws"] = b.workspace(b.bsp_mc_check_workspace_bytes(d, case["K"]))
        lay = b.bsp_mc_check_layout(d, case["K"])
        sizes = dict(dgamma_ref=C, dbeta_ref=C, dgamma_forward=C, dgamma_S1=C, dgamma_S2=C, dW_ref=O * C, dW_S1=O * C,
                     dW_S2=O * C, dx=T * C)
        s["arrays"] = {k: b.ws_view(s["ws"], getattr(lay, k), n) for k, n in sizes.items()}
    elif op == "store_check":
        d = s["desc"] = _fill(b.StoreDesc(), case, s)
        d.dY, d.bits, d.grad_fmt, d.seed, d.policy_mask = b.ptr(s["dY"]), case["bits"], b.E5M2, s["seed"], 0x7F
        s["ws"] = b.workspace(b.bsp_mc_check_store_workspace_bytes(d, case["K"]))
    elif op == "coupling":
        d = s["desc"] = _fill(b.CouplingDesc(), case, s)
        d.store_fmt, d.forward_mode, d.seed = b.E4M3, b.ROUND_STOCHASTIC, s["seed"]
        s["ws"] = b.workspace(b.bsp_coupling_check_workspace_bytes(d, case["pairs"]))
        lay = b.bsp_coupling_layout(d, case["pairs"])
        sizes = dict(gain_total=C, gain_mean_part=C, gain_fresh=C, X=C * O, X_sq=C * O)
        s["arrays"] = {k: b.ws_view(s["ws"], getattr(lay, k), n) for k, n in sizes.items()}
    elif op == "step":
        s["kind"] = b.RMSNORM if case["norm"] == "rms" else b.LAYERNORM
        ld = s["ld"] = (T + 15) // 16 * 16
        s["rstd"], s["mean"], s["amax"], s["scale"], s["amax_dy"], s["scale_dy"] = _zeros(T), _zeros(T), _zeros(1), _zeros(1), _zeros(1), _zeros(1)
        s["q"] = b.quant(b.E4M3, b.ROUND_STOCHASTIC, 1.0, s["scale"])
        s["q_dy"] = b.quant(b.E5M2, b.ROUND_NEAREST, 1.0, s["scale_dy"])
        s["codes"], s["codes_t"] = _zeros(T * C, torch.uint8), _zeros(C * ld, torch.uint8)
        s["u_bf16_t"] = _zeros(C * ld, torch.bfloat16) if case["w_read"] == b.READ_ORIGINAL else None
        s["dy_codes"], s["dy_codes_t"] = _zeros(T * O, torch.uint8), _zeros(O * ld, torch.uint8)
        s["du"] = _zeros(T * C, s["x"].dtype)
        s["dW"], s["dgamma"], s["dbeta"], s["dx"] = _zeros(O * C), _zeros(C), _zeros(C), _zeros(T * C)
        s["ws_w"] = b.workspace(b.bsp_linear_wgrad_workspace_bytes(T, O, C, case["w_read"]))
        s["ws_d"] = b.workspace(b.bsp_linear_dgrad_workspace_bytes(T, O, C))
        s["ws_n"] = b.workspace(b.bsp_norm_bwd_workspace_bytes(T, C))
    elif op in ("attn_check", "attn_step"):
        g, shape = _gen(seed), (case["B"], case["H"], case["S"], 64)
        s["q"], s["k"], s["v"] = (_normal(g, shape, 0.125, torch.bfloat16) for _ in range(3))
        s["dO"] = _normal(g, shape, 1.0, torch.bfloat16)
        n, rows, BH = s["q"].numel(), s["q"].numel() // 64, case["B"] * case["H"]
        if op == "attn_check":
            d = s["desc"] = b.AttnDesc()
            d.B, d.H, d.S, d.Dh, d.causal, d.softmax_scale, d.dtype = *shape, int(case["causal"]), 0.125, b.BF16
            d.q, d.k, d.v, d.dO = (b.ptr(s[k]) for k in ("q", "k", "v", "dO"))
            d.store_fmt, d.forward_mode, d.seed, d.tensor_id, d.policy_mask = b.E4M3, b.ROUND_STOCHASTIC, s["seed"], TENSOR, 7
            d.fp8_operands, d.p_scale, d.ds_scale = int(case["fp8"]), 256.0, 1024.0
            s["ws"] = b.workspace(b.bsp_mc_check_attn_workspace_bytes(d, case["K"]))
        else:
            s["o"], s["lse"], s["d"] = _zeros(n), _zeros(rows), _zeros(rows)
            s["dq"], s["dk"], s["dv"] = _zeros(n), _zeros(n), _zeros(n)
            s["o_codes"], s["o_amax"], s["o_scales"] = _zeros(n, torch.uint8), _zeros(BH), _zeros(BH)
            if case["fp8"]:
                s["f8"] = {k: (_zeros(n, torch.bfloat16), _zeros(n, torch.uint8), _zeros(BH), _zeros(BH)) for k in ("q", "k", "v", "dO")}
                f = s["f8"]
                s["fp8"] = b.attn_fp8(f["q"][3], f["k"][3], f["v"][3], f["dO"][3], 256.0, 1024.0,
                                      f["q"][1], f["k"][1], f["v"][1], f["dO"][1])
    elif op == "probs":
        g, R, n, d = _gen(seed), case["rows"], case["n"], case["d"]
        s["p"] = torch.softmax(1.5 * torch.randn((R, n), generator=g, device="cuda"), dim=1)
        s["V"] = _normal(g, (n, d), d ** -0.5, torch.float32)
        s["ds"], s["sq"], s["dV"] = _zeros(5 * R * n), _zeros(5 * R * n), _zeros(2 * R * n * d)
    else:
        g, R, n = _gen(seed), case["rows"], case["classes"]
        s["logits"] = torch.randn((R, n), generator=g, device="cuda")
        s["target"] = torch.randint(0, n, (R,), generator=g, device="cuda", dtype=torch.int32)
        s["per_trial"] = _zeros(case["trials"] * 6)
        s["ws"] = b.workspace(b.bsp_lsm_check_workspace_bytes(R, n, case["trials"]))
    return s


# ------------------------------------------------------------------------------------- one pass


def _stats(results):
    """The host-side statistics of a check, field by field, and its verdicts."""
    return dict(rel=np.array([r.rel_l2_mean_err for r in results]), R=np.array([r.R for r in results]),
                z=np.array([(r.Qprime, r.mean_z, r.rms_z, r.frac_abs_z_gt3) for r in results]),
                max_z=np.array([r.max_abs_z for r in results]), verdict=np.array([r.verdict for r in results]))


def run(s):
    return _RUN[s["op"]](s, s["case"])


def _run_check(s, case):
    return dict(s["arrays"], stats=_stats(b.bsp_mc_check(s["desc"], case["K"], s["ws"], s["diag"])))


def _run_store_check(s, case):
    return _stats(b.bsp_mc_check_store(s["desc"], case["K"], s["ws"], s["diag"]))


def _run_coupling(s, case):
    T, control = b.bsp_coupling_check(s["desc"], case["pairs"], s["ws"], s["diag"])
    return dict(s["arrays"], T=np.array(T), control=np.array(control))


def _run_attn_check(s, case):
    return _stats(b.bsp_mc_check_attn(s["desc"], case["K"], s["ws"], s["diag"]))


def _run_step(s, case):
    T, C, O, ld, kind, diag = case["T"], case["C"], case["O"], s["ld"], s["kind"], s["diag"]
    x, gamma, beta, rstd, mean = s["x"], s["gamma"], s["beta"], s["rstd"], s["mean"]
    b.bsp_norm_stats(kind, x, T, C, gamma, beta, 1e-6 if kind == b.RMSNORM else 1e-5, rstd, mean, s["amax"], diag)
    b.bsp_scale_from_amax(s["amax"], 1, b.E4M3, s["scale"])
    b.bsp_norm_fwd(kind, x, T, C, gamma, beta, rstd, mean, s["q"], b.key(s["seed"], TENSOR, b.STREAM_FORWARD),
                   s["codes"], s["codes_t"], ld, None, s["u_bf16_t"], diag)
    b.bsp_amax(s["dY"], 1, T * O, s["amax_dy"], diag)
    b.bsp_scale_from_amax(s["amax_dy"], 1, b.E5M2, s["scale_dy"])
    b.bsp_round_2d(s["dY"], T, O, s["q_dy"], b.key(0, 0, 0), s["dy_codes"], s["dy_codes_t"], ld, diag)
    b.bsp_linear_dgrad(T, O, C, s["dy_codes"], s["q_dy"], s["W"], s["du"], s["ws_d"], diag)
    x_t = s["u_bf16_t"] if case["w_read"] == b.READ_ORIGINAL else s["codes_t"]
    b.bsp_linear_wgrad(T, O, C, s["dy_codes_t"], s["q_dy"], case["w_read"], x_t, s["q"], ld, s["dW"], ws=s["ws_w"], diag=diag)
    b.bsp_norm_bwd(kind, x, T, C, gamma, beta, rstd, mean, s["du"], case["gain_read"], s["codes"], s["q"],
                   b.key(s["seed"], TENSOR, b.STREAM_GAIN), s["dgamma"], s["dbeta"], s["dx"], s["ws_n"], diag)
    return dict(codes=s["codes"], du=s["du"], dW=s["dW"], dgamma=s["dgamma"], dbeta=s["dbeta"], dx=s["dx"])


def _run_attn_step(s, case):
    B, H, S, BH, causal, diag = case["B"], case["H"], case["S"], case["B"] * case["H"], case["causal"], s["diag"]
    ops, fp8 = {k: s[k] for k in ("q", "k", "v", "dO")}, None
    if case["fp8"]:
        fp8 = s["fp8"]
        for k in ops:
            xq, codes, amax, scales = s["f8"][k]
            b.bsp_attn_quantize(s[k], BH, S * 64, b.E5M2 if k == "dO" else b.E4M3, xq, amax, scales, diag, codes=codes)
            ops[k] = xq
    b.bsp_attn_fwd_stats(B, H, S, 64, causal, 0.125, ops["q"], ops["k"], ops["v"], s["o"], s["lse"], diag, fp8=fp8)
    b.bsp_amax(s["o"], BH, S * 64, s["o_amax"], diag)
    b.bsp_scale_from_amax(s["o_amax"], BH, b.E4M3, s["o_scales"])
    b.bsp_round_grouped(s["o"], BH, S * 64, b.E4M3, b.ROUND_STOCHASTIC, s["o_scales"],
                        b.key(s["seed"], TENSOR, b.STREAM_FORWARD), s["o_codes"], diag)
    b.bsp_attn_bwd(B, H, S, 64, causal, 0.125, int(case["fp8"]), ops["q"], ops["k"], ops["v"], ops["dO"], s["lse"], s["o"],
                   s["o_codes"], s["o_scales"], b.E4M3, case["read"], b.key(s["seed"], TENSOR, b.STREAM_ATTN_D),
                   s["dq"], s["dk"], s["dv"], s["d"], diag, fp8=fp8)
    return dict(o=s["o"], lse=s["lse"], o_codes=s["o_codes"], D=s["d"], dq=s["dq"], dk=s["dk"], dv=s["dv"])


def _run_probs(s, case):
    b.bsp_probs_mc(s["p"], s["V"], case["rows"], case["n"], case["d"], case["law"], case["param"], s["seed"], TENSOR, 0,
                   case["K"], s["ds"], s["sq"], s["dV"])
    return dict(ds=s["ds"], sq=s["sq"], dV=s["dV"])


def _run_lsm(s, case):
    st = b.bsp_lsm_check(s["logits"], s["target"], case["rows"], case["classes"], case["eps"], case["trials"], s["seed"], TENSOR,
                         s["per_trial"], s["ws"])
    return dict(per_trial=s["per_trial"], stats=np.array([(t.mean, t.se) for t in st]))


_RUN = dict(check=_run_check, step=_run_step, store_check=_run_store_check, coupling=_run_coupling, attn_check=_run_attn_check,
            attn_step=_run_attn_step, probs=_run_probs, lsm=_run_lsm)


# ------------------------------------------------------------------------------ work and tolerance


def work(case):
    """Bytes of the inputs and outputs, each once, and the operations of the contractions."""
    op = case["op"]
    if op in ("check", "step", "store_check", "coupling"):
        T, C, O = case["T"], case["C"], case["O"]
        eb, prod = 2 if case["dtype"] == "bf16" else 4, 2.0 * T * C * O
        inputs, K = (T * C + O * C + T * O) * eb, case.get("K", 0)
        if op == "check":           # du; dW under U, R and K fresh reads
            return dict(bytes=inputs + 4 * (3 * O * C + T * C), flops=prod * (3 + K))
        if op == "step":
            return dict(bytes=inputs + T * C * (1 + eb + 4) + 4 * O * C, flops=prod * 2)
        if op == "store_check":     # du; dW under U, R and K draws of each of two fresh reads
            return dict(bytes=inputs, flops=prod * (3 + 2 * K))
        return dict(bytes=inputs - T * O * eb + 8 * O * C, flops=prod * 5 * case["pairs"])   # y and du twice, X once per pair
    if op in ("attn_check", "attn_step"):
        n = case["B"] * case["H"] * case["S"] * 64
        prod = 2.0 * n * case["S"] * (0.5 if case["causal"] else 1.0)
        if op == "attn_step":       # two products forward, five backward
            return dict(bytes=n * (8 + 1 + 16), flops=7 * prod)
        # BF16 operands: S, P V, dP, dV, dK, dQ, P K and one product per draw; FP8: dK and dQ per draw
        return dict(bytes=n * 8, flops=prod * (7 + case["K"] * (2 if case["fp8"] else 1)))
    if op == "probs":               # per row and draw: o, dp and two outer products
        R, n, d = case["rows"], case["n"], case["d"]
        return dict(bytes=4 * (n * d + R * n * 11 + 2 * R * n * d), flops=8.0 * R * n * d * case["K"])
    e = float(case["rows"]) * case["classes"]
    return dict(bytes=4 * (e + 6 * case["trials"]), flops=10.0 * e * case["trials"])


def tolerance(case):
    """About four times the largest distance to the same path in 64-bit arithmetic, measured at several sizes.

    check: shifted sums of the gain use 5e-5 (32-bit sums over the tokens), everything else below 1e-5; with
    fewer than eight draws the largest |z| divides by a spread that nearly vanishes: 1e-3.
    step: 2e-7 .. 1e-6 given the statistics; a last-bit difference in them moves single codes.
    store_check: bf16(dY s) enters the contraction of the draws; coupling: <du, r> is a small difference, 5e-4.
    attention: P and dS enter the products as bf16, 1.7e-3; the codes of O move with its last bits.
    probs: 32-bit sums over the draws; lsm: a mean over the classes that nearly cancels, 2e-5."""
    if case["op"] == "check" and case["K"] < 8:
        return dict(rel=4e-3)
    return dict(_TOLERANCE[case["op"]])


_TOLERANCE = dict(
    check=dict(rel=2e-4),
    step=dict(rel=1e-4, differ=1e-5),
    store_check=dict(rel=2e-3),
    coupling=dict(rel=2e-3),
    attn_check=dict(rel=7e-3),
    attn_step=dict(rel=7e-3, differ=0.01),
    probs=dict(rel=1e-5),
    lsm=dict(rel=1e-4),
)
