"""The work a user of this framework has it do, as cases of one pass each through the public entry points.

Kinds of work
  layer   a module as it arrives: initialisation (forward definition, accumulators), the inverse of the module input's
          system, then the first `iters` iterations of the ADMM loop
  step    one iteration in the middle of the loop (a loop has 10 to 50 of them): weight recoveries, scores, top-k,
          recovery on the kept support, token pass
  (`select`: the mask is re-selected in every iteration, Algorithm 2; otherwise it is fixed beforehand, Algorithm 1,
  and the unrestricted recovery and the scores are not needed)
  heads   head pruning of an attention module with its head outputs held fixed: Gram and cross products over the
          tokens, head scores, head mask, recovery of W_O on the kept heads
  mha     one outer iteration of the attention module's alternating updates: recoveries of W_Q, W_K, W_O, W_V, then
          the updates of the auxiliary variables
  plan    the mask step over the layers of a model: unit scores and importances of every layer, allocation, top-k

Shapes, distributions, sparsities and ridge are those of the repository's workloads (FFN widths 768/3072, 2048/8192,
4096/16384, 4096/11008 gated, 7168/28672; Gaussian or Laplace inputs with a few outlier channels), the token counts
from one chunk of tokens to a whole calibration set of 128 sequences of 2048.
"""
import math

import torch

from paper_2510_03246_b200 import api, pipeline

DEV = "cuda"
RHO = 0.1


def _ffn(name, kind, d, n, N, **kw):
    c = dict(name=name, kind=kind, d=d, n=n, N=N, dtype="bf16", act="relu", keep=0.5, chunk=0, laplace=False,
             out_share=0.01, out_factor=30.0, sigma=0.02, dual=False, exact=False, iters=1, select=True)
    c.update(kw)
    return c


def listed():
    return [
        # smallest module of the family, fp32 storage: a layer from its inputs through the first iterations of its loop
        _ffn("layer_f32_768", "layer", 768, 3072, 2048, dtype="f32", iters=2, out_factor=20.0),
        # the same shape in the tensor-core mode: one iteration is a chain of short kernels
        _ffn("step_768", "step", 768, 3072, 2048, out_factor=20.0),
        # odd sizes: widths that fill no tile, tokens that end inside a row tile; dual variable, exact select rule
        _ffn("step_ragged_dual", "step", 1096, 4376, 9973, keep=0.37, dual=True, exact=True),
        # a module of the 1.3B shape on one chunk of tokens (a small calibration set)
        _ffn("step_2048", "step", 2048, 8192, 32768, out_share=0.005),
        # the same module over the whole calibration set, 128 sequences of 2048 tokens, chunk by chunk
        _ffn("step_2048_full", "step", 2048, 8192, 262144, chunk=32768, out_share=0.005),
        # a gated module (SiLU gate) of the 7B shape, mask fixed beforehand
        _ffn("step_gated_4096", "step", 4096, 11008, 16384, act="swiglu", keep=0.3, out_factor=50.0, select=False),
        # the 6.7B shape with the mask fixed beforehand: set-up and first iteration of a layer
        _ffn("layer_4096", "layer", 4096, 16384, 32768, keep=0.4, laplace=True, out_share=0.005, out_factor=40.0,
             sigma=0.015, select=False),
        # the widest module (30B shape), where the factorisation of the 28672-wide system rules
        _ffn("step_7168", "step", 7168, 28672, 8192, keep=0.2, sigma=0.01),
        # head pruning of an attention module over a quarter of the calibration set
        dict(name="heads_2048", kind="heads", d=2048, heads=32, N=65536, keep_heads=16, chunk=32768),
        # attention module of the smallest model, 16 sequences of 128 tokens, 12 heads of width 64
        dict(name="mha_768", kind="mha", d=768, heads=12, T=128, seqs=16, keep_heads=6, a_steps=4, z_steps=4, chunk=8),
        # attention module of the 1.3B shape, sequences of 1024 tokens
        dict(name="mha_2048", kind="mha", d=2048, heads=32, T=1024, seqs=8, keep_heads=16, a_steps=2, z_steps=2, chunk=8),
        # scores, allocation and masks of the 24 layers of the 1.3B shape
        dict(name="plan_24_layers", kind="plan", layers=24, d=2048, n=8192, keep=0.5),
    ]


def _log(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step, int(round(v / step)) * step)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "layer", "f32", "gated", "heads", "mha", "plan"])
    share, factor = rng.choice([0.005, 0.01]), rng.choice([20.0, 30.0, 40.0, 50.0])
    common = dict(out_share=share, out_factor=factor, keep=round(rng.uniform(0.2, 0.7), 3),
                  laplace=rng.random() < 0.25, sigma=rng.choice([0.01, 0.015, 0.02]))
    if kind == "f32":        # fp32 storage: any widths
        d = _log(rng, 96, 1024)
        c = _ffn("", rng.choice(["layer", "step"]), d, int(d * rng.uniform(2.5, 4.0)), _log(rng, 256, 4096),
                 dtype="f32", exact=rng.random() < 0.3, dual=rng.random() < 0.2, **common)
    elif kind == "gated":
        d = _log(rng, 512, 4096, 8)
        c = _ffn("", "step", d, int(d * rng.uniform(2.5, 3.5)) // 8 * 8, _log(rng, 1024, 16384), act="swiglu", select=False,
                 **common)
    elif kind in ("step", "layer"):
        d = _log(rng, 256, 4096, 8)
        n = int(d * rng.uniform(3.0, 4.0)) // 8 * 8
        N = _log(rng, 512, min(262144, 3.0e12 / (n * n)))
        c = _ffn("", kind, d, n, N, chunk=32768 if N > 32768 else 0, exact=rng.random() < 0.25,
                 dual=rng.random() < 0.2, select=kind == "step", **common)
    elif kind == "heads":
        heads = rng.choice([8, 12, 16, 24, 32])
        c = dict(name="", kind="heads", d=heads * 64, heads=heads, N=_log(rng, 1024, 65536),
                 keep_heads=rng.randint(heads // 4, heads - 2), chunk=32768)
    elif kind == "mha":
        heads, dh = rng.choice([8, 12, 16, 24, 32]), rng.choice([64, 64, 128])
        heads = min(heads, 2048 // dh)
        T = _log(rng, 64, 1024, 8)
        c = dict(name="", kind="mha", d=heads * dh, heads=heads, T=T, seqs=rng.randint(2, max(2, min(16, 8192 // T))),
                 keep_heads=rng.randint(heads // 4, heads - 2), a_steps=rng.randint(1, 4), z_steps=rng.randint(1, 4),
                 chunk=rng.choice([2, 4, 8]))
    else:
        d = _log(rng, 512, 4096, 8)
        c = dict(name="", kind="plan", layers=rng.randint(6, 32), d=d, n=int(d * rng.uniform(2.5, 4.0)),
                 keep=round(rng.uniform(0.3, 0.7), 3))
        c["layers"] = min(c["layers"], max(4, int(8e8 / (c["d"] * c["n"]))))
    c.pop("name")
    return c


# ------------------------------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _activations(g, N, d, dtype, share, factor, laplace=False):
    x = torch.randn(N, d, generator=g, device=DEV)
    if laplace:      # unit-variance Laplace: a Gaussian times the root of an exponential variable
        x.mul_(torch.empty_like(x).exponential_(generator=g).sqrt_())
    cols = torch.randperm(d, generator=g, device=DEV)[:max(1, math.ceil(share * d))]
    x[:, cols] *= factor
    return x.to(dtype)


def _weight(g, rows, cols, sigma):
    return (torch.randn(rows, cols, generator=g, device=DEV) * sigma).bfloat16()      # checkpoints are bf16


def _keep(c):
    return max(1, int(c["keep"] * c["n"]))


def _magnitude_mask(W1, W2, k):
    """A mask chosen beforehand: the k channels with the largest product of weight norms."""
    s = W1.double().square().sum(1) * W2.double().square().sum(0)
    m = torch.zeros(s.numel(), dtype=torch.uint8, device=DEV)
    m[torch.sort(s, descending=True, stable=True).indices[:k]] = 1
    return m


def _params(c, **kw):
    p = dict(rho=RHO, k_keep=_keep(c), token_chunk=c["chunk"], dual_mode=c["dual"],
             z_rule=api.SP_Z_EXACT if c["exact"] else api.SP_Z_PAPER)
    p.update(kw)
    return api.AdmmParams(**p)


def prepare(case, seed):
    g, c = _gen(seed), case
    if c["kind"] in ("layer", "step"):
        d, n, N = c["d"], c["n"], c["N"]
        X = _activations(g, N, d, torch.float32 if c["dtype"] == "f32" else torch.bfloat16, c["out_share"],
                         c["out_factor"], c["laplace"])
        W1, W2 = _weight(g, n, d, c["sigma"]), _weight(g, d, n, c["sigma"])
        Wg = _weight(g, n, d, c["sigma"]) if c["act"] == "swiglu" else None
        mod = api.FfnModule(X, W1, W2, dual_mode=c["dual"], token_chunk=c["chunk"], overlap_k=_keep(c), Wg_0=Wg)
        st = dict(kind=c["kind"], mod=mod, iters=c["iters"], select=c["select"], mask=_magnitude_mask(W1, W2, _keep(c)))
        fixed = _params(c, reselect_mask=False, skip_scores=True)
        if c["kind"] == "layer":
            st["params"] = _params(c) if c["select"] else fixed
        else:
            # the module in the middle of its loop: some iterations on a mask chosen beforehand lie behind it; after
            # four the pruned channels have faded far enough (scores of kept and pruned channels apart by 75 % and
            # more) that the re-selection of the measured iteration is no near-tie
            mod.sp_ffn_init()
            mod.mask.copy_(st["mask"])
            for _ in range(4 if c["select"] else 2):
                mod.sp_admm_step(fixed)
            st["params"] = _params(c) if c["select"] else fixed
        return st
    if c["kind"] == "heads":
        d, N = c["d"], c["N"]
        H = _activations(g, N, d, torch.bfloat16, 0.005, 8.0)
        W = _weight(g, d, d, 0.02).float()
        return dict(kind="heads", H=H, Y=(H.float() @ W.T).bfloat16(), W=W, heads=c["heads"], keep=c["keep_heads"],
                    chunk=c["chunk"])
    if c["kind"] == "mha":
        d, H = c["d"], c["heads"]
        X = _activations(g, c["seqs"] * c["T"], d, torch.bfloat16, 0.005, 5.0)
        Wq, Wk, Wv, Wo = (_weight(g, d, d, 1.0 / math.sqrt(d)) for _ in range(4))
        mod = api.MhaModule(X, Wq, Wk, Wv, Wo, n_heads=H, T=c["T"], seq_chunk=c["chunk"])
        mod.sp_mha_init(True)
        mask = torch.zeros(H, dtype=torch.uint8, device=DEV)
        mask[torch.randperm(H, generator=g, device=DEV)[:c["keep_heads"]]] = 1
        return dict(kind="mha", mod=mod, mask=mask, params=api.MhaParams(a_steps=c["a_steps"], z_steps=c["z_steps"],
                                                                         seq_chunk=c["chunk"]))
    L, d, n = c["layers"], c["d"], c["n"]
    Ws = [_weight(g, d, n, 0.02).float() * (1.0 + 0.03 * l) for l in range(L)]
    colsq = torch.rand(L, n, generator=g, device=DEV) + 0.5
    return dict(kind="plan", W=Ws, colsq=colsq, n=n, rbar=1.0 - c["keep"],
                units=torch.full((L,), n, dtype=torch.int64, device=DEV),
                T=torch.tensor([1.0], dtype=torch.float64, device=DEV))


# ------------------------------------------------------------------------------------------------------- one pass
def run(state):
    s = state
    if s["kind"] in ("layer", "step"):
        mod = s["mod"]
        if s["kind"] == "layer":
            mod.sp_ffn_init()
            if not s["select"]:
                mod.mask.copy_(s["mask"])
        for _ in range(s["iters"]):
            mod.sp_admm_step(s["params"])
        out = dict(W1=mod.W1, W2=mod.W2, Z=mod.Z, mask=mod.mask, G_A=mod.G_A, R1=mod.R1, R2=mod.R2, absA=mod.absA,
                   report=mod.report)
        if s["kind"] == "layer":
            out.update(Ypre=mod.Ypre, G_X=mod.G_X)
        if s["select"]:
            out.update(scores=mod.scores, importance=mod.importance)
        if mod.U is not None:
            out["U"] = mod.U
        return out
    if s["kind"] == "heads":
        mask, W, scores = pipeline.prune_attention_heads(s["H"], s["Y"], s["W"], s["heads"], s["keep"], rho=RHO,
                                                         token_chunk=s["chunk"])
        return dict(mask=mask, W=W, scores=scores)
    if s["kind"] == "mha":
        mod = pipeline.mha_outer_iterations(s["mod"], s["mask"], 1, s["params"], rho=RHO)
        return dict(Wq=mod.Wq, Wk=mod.Wk, Wv=mod.Wv, Wo=mod.Wo, Zq=mod.Zq, Zk=mod.Zk, P=mod.P, Aattn=mod.Aattn,
                    R_Q=mod.R_Q, R_K=mod.R_K, G_attn=mod.G_attn, R_O=mod.R_O)
    L, n = len(s["W"]), s["n"]
    scores, imp = zip(*(api.sp_struct_scores(api.SP_SCORE_WANDA_L2, n, W=s["W"][l], colsq=s["colsq"][l])[:2]
                        for l in range(L)))
    I = torch.cat(imp)
    r, k = api.sp_allocate_sparsity_grid(I, s["units"], s["rbar"], s["T"])
    scores = torch.stack(scores)
    mask, tau, _ = api.sp_apply_mask_batched(scores, k[0])
    return dict(importance=I, r=r, k_keep=k, scores=scores, mask=mask, tau=tau)


# ------------------------------------------------------------------------------------------------------- work
def _solve(n, m):
    return n ** 3 / 3.0 + 2.0 * m * n * n


def work(case):
    c = case
    if c["kind"] in ("layer", "step"):
        d, n, N, k = float(c["d"]), float(c["n"]), float(c["N"]), float(_keep(c))
        esz = 4.0 if c["dtype"] == "f32" else 2.0
        gated = c["act"] == "swiglu"
        # weight phase: W1 from the kept inverse, W2 on all channels (unless the mask is fixed) and on the kept ones,
        # the d x d system of the a-update; token pass: E, D, z1 on the kept channels, then G_A (triangle), R1, R2.
        # Where pruned channels only fade (ReLU without the dual variable, an unchanged mask) their parts of the
        # accumulators follow from the last iteration's.
        kk = k if c["kind"] == "step" and not gated and not c["dual"] and c["dtype"] == "bf16" else n
        step = (_solve(n, d) if c["select"] else 0.0) + _solve(k, d) + 2 * n * d * d + _solve(d, k) + 2 * k * d * d
        step += N * (6 * k * d + 4 * kk * d + (2 * n * kk - kk * kk))
        byte = N * (2 * d * esz + (8 * n) + (8 * n if c["dual"] else 0) + (4 * n if gated else 0))
        byte += 4.0 * (2 * n * d + 2 * (n * n + 2 * n * d) + d * d)
        flops, bytes_ = step * c["iters"], byte * c["iters"]
        if c["kind"] == "layer":
            flops += N * (2 * n * d * 4 + d * d + n * n) + _solve(d, d)
            bytes_ += N * (2 * d * esz + 4 * n) + 4.0 * (n * n + 4 * n * d + 2 * d * d)
        return {"bytes": bytes_, "flops": flops}
    if c["kind"] == "heads":
        d, N, k = float(c["d"]), float(c["N"]), c["d"] * c["keep_heads"] / c["heads"]
        return {"bytes": N * d * 4 + 8 * d * d, "flops": N * 3 * d * d + _solve(k, d)}
    if c["kind"] == "mha":
        d, T, S, H = float(c["d"]), float(c["T"]), float(c["seqs"]), float(c["heads"])
        kh, dh = float(c["keep_heads"]), d / H
        pairs = S * H
        # recoveries: W_Q, W_K, W_O and one system of size d per kept head with its regressors P X; then the products
        # of width d_h on the T x T tensors (logits, P V and its gradient, the softmax gradients) and the projections
        flops = 2 * _solve(d, d) + _solve(dh * kh, d) + kh * _solve(d, dh)
        flops += kh * S * (2 * T * T * d + T * d * d + 2 * T * d * dh)
        flops += pairs * 2 * T * T * dh * (2 + 2 * c["a_steps"] + 3 * c["z_steps"])
        flops += S * T * d * d * (6 + 4 + 8) + _solve(d, 2 * d)
        return {"bytes": pairs * T * T * 8 + S * T * d * (2 + 2 + 24) + 4 * 12 * d * d, "flops": flops}
    return {"bytes": c["layers"] * (4.0 * c["d"] * c["n"] + 13.0 * c["n"]), "flops": 2.0 * c["layers"] * c["d"] * c["n"]}


def tolerance(case):
    # Measured: the same pass with its sums in another order (fixed instead of free) and, for the attention module,
    # against the fp32 mode; stated: about four times that.
    k = case["kind"]
    if k in ("layer", "step"):
        # The select rule branches on the sign of the old z: an entry within rounding of zero takes the other branch
        # in a share of entries that follows from the rounding (bf16 operands: 1e-5, fp32 storage: 1e-6), which shows
        # in `max` (0.4 to 0.8 of the root mean square) and rules `rel`.  The recovered weights differ by 3e-3 after
        # five iterations (the ridge systems amplify the accumulators' rounding), the dual variable by 9e-3.
        return {"rel": 2e-3 if case["dtype"] == "f32" else 2.5e-2 if case["dual"] else 1e-2, "max": 0.95, "differ": 2e-3}
    if k == "mha":       # W_O 3.3e-3 and 0.023 from the fp32 mode's
        return {"rel": 1e-2, "max": 0.1}
    if k == "heads":
        return {"rel": 5e-4, "max": 5e-3}
    return {"rel": 1e-5, "differ": 2e-3}


# ------------------------------------------------------------------------------------------------------- in 64 bits
def _ridge(R, G, ridge=None):
    """R (G + rho tr(G)/dim I)^-1."""
    ridge = RHO * G.diagonal().mean() if ridge is None else ridge
    L = torch.linalg.cholesky(G + ridge * torch.eye(G.shape[0], dtype=G.dtype, device=G.device))
    return torch.cholesky_solve(R.T, L).T


def _refit(R, G, keep):
    W = torch.zeros_like(R)
    W[:, keep] = _ridge(R[:, keep], G[keep][:, keep], RHO * G.diagonal().mean())
    return W


def _top(s, k):
    return torch.sort(torch.sort(s, descending=True, stable=True).indices[:k]).values


def _exact_ffn(c, seed):
    g, d, n, N, f64 = _gen(seed), c["d"], c["n"], c["N"], torch.float64
    iters = c["iters"] if c["kind"] == "layer" else 5 if c["select"] else 3
    if (iters + 1) * N * (2.0 * n * n + 8.0 * n * d) > 2.5e14:
        return None
    X = _activations(g, N, d, torch.float32 if c["dtype"] == "f32" else torch.bfloat16, c["out_share"], c["out_factor"],
                     c["laplace"])
    W1, W2 = _weight(g, n, d, c["sigma"]), _weight(g, d, n, c["sigma"])
    Wg = _weight(g, n, d, c["sigma"]).to(f64) if c["act"] == "swiglu" else None
    fixed = _top(W1.double().square().sum(1) * W2.double().square().sum(0), _keep(c))
    stored, X, W1, W2 = X.dtype, X.to(f64), W1.to(f64), W2.to(f64)
    chunks = [slice(t, min(N, t + 16384)) for t in range(0, N, 16384)]
    Z, U = torch.empty(N, n, dtype=f64, device=DEV), None
    Y = torch.empty(N, d, dtype=f64, device=DEV)
    if c["dual"]:
        U = torch.zeros_like(Z)
    G_X, out = X.T @ X, {}

    def sums(t, A, first):
        for name, v in (("G_A", A.T @ A), ("R1", Z[t].T @ X[t]), ("R2", Y[t].T @ A), ("absA", A.abs().sum(0))):
            out[name] = v if first else out[name].add_(v)

    def phi(t):
        return Z[t].clamp_min(0) if Wg is None else torch.nn.functional.silu(X[t] @ Wg.T) * Z[t]

    for t in chunks:
        Z[t] = X[t] @ W1.T
        A = phi(t)
        Y[t] = (A @ W2.T).to(stored).to(f64)       # the target is held in the storage type
        sums(t, A, t.start == 0)
    for i in range(iters):
        select = c["select"] and (c["kind"] == "layer" or i == iters - 1)
        keep = fixed
        if select:
            out["scores"] = (_ridge(out["R2"], out["G_A"]).square().sum(0) * out["G_A"].diagonal()).sqrt()
            out["importance"] = out["scores"].mean().reshape(1)
            keep = _top(out["scores"], _keep(c))
        out["W1"] = torch.zeros_like(W1)
        out["W1"][keep] = _ridge(out["R1"][keep], G_X)
        out["W2"] = _refit(out["R2"], out["G_A"], keep)
        w1, w2 = out["W1"], out["W2"]
        inner = torch.linalg.inv(torch.eye(d, dtype=f64, device=DEV) + w2 @ w2.T) @ w2
        for t in chunks:
            h = phi(t) if U is None else phi(t) - U[t]
            A = h + (Y[t] - h @ w2.T) @ inner
            Au, z1 = A if U is None else A + U[t], X[t] @ w1.T
            if Wg is not None:
                gate = torch.nn.functional.silu(X[t] @ Wg.T)
                Z[t] = (gate * Au + z1) / (gate * gate + 1)
            elif c["exact"]:
                zn, zp = z1.clamp_max(0), ((Au + z1) / 2).clamp_min(0)
                lower = Au.square() + (zn - z1).square() < (Au - zp).square() + (zp - z1).square()
                Z[t] = torch.where(lower, zn, zp)
            else:
                Z[t] = torch.where(Z[t] < 0, z1, (Au + z1) / 2)
            if U is not None:
                U[t] += A - phi(t)
            sums(t, A, t.start == 0)
    res = dict(W1=out["W1"], W2=out["W2"], Z=Z, mask=None, G_A=out["G_A"], R1=out["R1"], R2=out["R2"], absA=out["absA"],
               report=None)
    if c["kind"] == "layer":
        res.update(Ypre=Y, G_X=G_X)
    if c["select"]:
        res.update(scores=out["scores"], importance=out["importance"])
    if U is not None:
        res["U"] = U
    return res


def _exact_heads(c, seed):
    g, d, H = _gen(seed), c["d"], c["heads"]
    X = _activations(g, c["N"], d, torch.bfloat16, 0.005, 8.0)
    W = _weight(g, d, d, 0.02).float()
    Y, X, W = (X.float() @ W.T).bfloat16().double(), X.double(), W.double()
    G, R = X.T @ X, Y.T @ X
    scores = (W.square().sum(0) * G.diagonal()).view(H, -1).sum(1).sqrt()
    dh = d // H
    keep = (_top(scores, c["keep_heads"])[:, None] * dh + torch.arange(dh, device=DEV)).flatten()
    return dict(mask=None, W=_refit(R, G, keep), scores=scores)


def _exact_mha(c, seed):
    g, d, H, T, S = _gen(seed), c["d"], c["heads"], c["T"], c["seqs"]
    dh = d // H
    X = _activations(g, S * T, d, torch.bfloat16, 0.005, 5.0).double()
    Wq, Wk, Wv, Wo = (_weight(g, d, d, 1.0 / math.sqrt(d)).double() for _ in range(4))
    kept = torch.sort(torch.randperm(H, generator=g, device=DEV)[:c["keep_heads"]]).values
    keep = (kept[:, None] * dh + torch.arange(dh, device=DEV)).flatten()
    future = torch.ones(T, T, dtype=torch.bool, device=DEV).triu(1)

    def heads(v):                                  # [S T, d] -> [S, H, T, dh]
        return v.view(S, T, H, dh).transpose(1, 2)

    def flat(v):
        return v.transpose(1, 2).reshape(S * T, d)

    def probs(zq, zk):
        return (heads(zq) @ heads(zk).transpose(2, 3) / math.sqrt(dh)).masked_fill(future, float("-inf")).softmax(3)

    def rows(w):
        out = torch.zeros_like(w)
        out[keep] = w[keep]
        return out

    zq, zk, v = X @ Wq.T, X @ Wk.T, X @ Wv.T
    P = probs(zq, zk)
    A = flat(P @ heads(v))
    Y = (A @ Wo.T).bfloat16().double()
    G_X = X.T @ X
    Wq, Wk, Wo = rows(_ridge(zq.T @ X, G_X)), rows(_ridge(zk.T @ X, G_X)), _refit(Y.T @ A, A.T @ A, keep)
    Wv = torch.zeros_like(Wv)
    for h in kept.tolist():
        r, cols = (P[:, h] @ X.view(S, T, d)).reshape(S * T, d), slice(h * dh, (h + 1) * dh)
        Wv[cols] = _ridge(A[:, cols].T @ r, r.T @ r)
    v, target_q, target_k, F = X @ Wv.T, X @ Wq.T, X @ Wk.T, probs(zq, zk)
    step = 1.0 / (2.0 * (heads(v).square().sum((2, 3), keepdim=True) + 1.0))
    for _ in range(c["a_steps"]):
        P = P - step * (2.0 * (P @ heads(v) - heads(A)) @ heads(v).transpose(2, 3) + 2.0 * (P - F))
    A = (flat(P @ heads(v)) + Y @ Wo) @ torch.linalg.inv(Wo.T @ Wo + torch.eye(d, dtype=X.dtype, device=DEV))
    for _ in range(c["z_steps"]):
        F = probs(zq, zk)
        E = F - P
        dS = 2.0 * F * (E - (E * F).sum(3, keepdim=True)) / math.sqrt(dh)
        q, k = heads(zq), heads(zk)
        eta = 1.0 / (2.0 + (q.square().sum((2, 3), keepdim=True) + k.square().sum((2, 3), keepdim=True)) / dh)
        zq, zk = (flat(q - eta * (dS @ k + 2.0 * (q - heads(target_q)))),
                  flat(k - eta * (dS.transpose(2, 3) @ q + 2.0 * (k - heads(target_k)))))
    return dict(Wq=Wq, Wk=Wk, Wv=Wv, Wo=Wo, Zq=zq, Zk=zk, P=P, Aattn=A, R_Q=zq.T @ X, R_K=zk.T @ X, G_attn=A.T @ A,
                R_O=Y.T @ A)


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits throughout (integer and report outputs left out)."""
    kind = case["kind"]
    if kind != "plan":
        return {"heads": _exact_heads, "mha": _exact_mha}.get(kind, _exact_ffn)(case, seed)
    g, L, d, n = _gen(seed), case["layers"], case["d"], case["n"]
    sq = torch.stack([(_weight(g, d, n, 0.02).float() * (1.0 + 0.03 * l)).double().square().sum(0) for l in range(L)])
    scores = (sq * (torch.rand(L, n, generator=g, device=DEV) + 0.5)).sqrt()
    I = scores.mean(1)
    raw = (1.0 - case["keep"]) * L * torch.softmax(-I / I.abs().mean(), 0)
    r = raw.clamp(0, 0.95)
    if not bool((raw > 0.95).any()):
        r = (r * ((1.0 - case["keep"]) / r.mean())).clamp(0, 0.95)
    return dict(importance=I, r=r[None], k_keep=None, scores=scores, mask=None, tau=None)
