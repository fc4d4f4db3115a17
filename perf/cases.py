"""The work that a training program has this library do, as timed cases.

A program built on the library makes, per optimisation step: the continuation
probabilities of its candidate groups (pair_allocate), the per-rollout
coefficients of the completed ones (pair_coeffs, or a weighting variant, or
the product form), and the head's objective and gradients (pair_grad, or the
clipped surrogate of later epochs). Offline it audits a design over many draws
(pair_audit) and forms estimates from explicit scores (pair_estimate_dense).
Each case is one such call, or the coefficients and the head together, through
`paper_2608_11368_gb300.binding`, with the sizes of the package's named
workloads, of its tests, or between them.

Inputs are drawn on the device from the seed alone, with the distributions of
`paper_2608_11368_gb300.synth`: success rates U(0, 1) or Beta(1/2, 1/2),
binary rewards, p_i ~ U(floor, 1), J_i ~ Bernoulli(p_i), rho_ij = p_i p_j or a
general symmetric matrix capped by min(p_i, p_j), H ~ N(0, 1), W ~ N(0, 1/d),
uniform targets, segments padded to 8 tokens. In the head cases the first two
rollouts of every group are completed with different rewards: a trainer drops
a group without a contrast before it runs the head, so none is drawn here (and
the expected number of active tokens is the same for every seed).
"""
import math

import numpy as np
import torch

from paper_2608_11368_gb300 import binding as L

DEV = "cuda"
WMODES = ("ht", "unweighted", "marginal", "clipped", "hajek")
W_MAX = 12.0      # clipping constant of the clipped weighting (as in the tests)
CLIP_EPS = 0.2    # clip range of the trajectory ratio
# pair_grad_workspace_size by default, or the minimum (no logit-sized tensor kept).
WORKSPACES = ("default", "min")


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # Coefficients of one training step of 8 prompts x 8 rollouts: a few
        # kilobytes, so the call's latency is all there is.
        dict(name="coeffs_8x8", kind="coeffs", B=8, G=8, rho="product", floor=0.2, flags=0),
        # The coefficient stress workload: 4096 groups of 64, general rho.
        dict(name="coeffs_4096x64", kind="coeffs", B=4096, G=64, rho="general", floor=0.05,
             flags=0),
        # A stabilised weighting with its diagnostics, for a group size that
        # is no multiple of 4 (1000 logged groups of 50).
        dict(name="weighted_1000x50", kind="weighted", B=1000, G=50, rho="general", floor=0.05,
             flags=0, wmode="clipped"),
        # The dense estimator over explicit scores, at the stress workload's
        # size: the largest amount of memory one call streams.
        dict(name="dense_4096x64x4096", kind="dense", B=4096, G=64, D=4096, floor=0.05),
        # Frozen-population audit: 50,000 draws of one group of 16.
        dict(name="audit_50000x16", kind="audit", N=50000, G=16, D=4096, wmode="ht"),
        # Allocation before a step of 64 prompts x 16 candidates, and for a
        # whole logged set of 4096 x 64.
        dict(name="allocate_64x16", kind="allocate", B=64, G=16, frac=0.5, pi_min=0.08,
             norms=False),
        dict(name="allocate_4096x64", kind="allocate", B=4096, G=64, frac=0.5, pi_min=0.08,
             norms=True),
        # The fp32 reference head: 4 prompts x 8 rollouts, d = 256, V = 4096.
        dict(name="grad_f32_4x8", kind="grad", dtype="f32", B=4, G=8, d=256, V=4096, floor=0.2,
             len_lo=32, len_hi=64, ws="default", clipped=False),
        # A small bf16 head whose hidden size is no multiple of 512.
        dict(name="grad_d768_4x8", kind="grad", dtype="bf16", B=4, G=8, d=768, V=32000, floor=0.2,
             len_lo=64, len_hi=512, ws="default", clipped=False),
        # One prompt's micro-batch on the 1.7B head (d = 2048, V = 151,936),
        # where reading W and writing dW weigh as much as the contractions.
        dict(name="grad_1p7b_1x8", kind="grad", dtype="bf16", B=1, G=8, d=2048, V=151936,
             floor=0.2, len_lo=64, len_hi=512, ws="default", clipped=False),
        # The full step on that head: 4 prompts x 8 rollouts of 256 to 2048
        # tokens, coefficients and head.
        dict(name="grad_1p7b_4x8", kind="grad", dtype="bf16", B=4, G=8, d=2048, V=151936,
             floor=0.2, len_lo=256, len_hi=2048, ws="default", clipped=False),
        # A clipped-surrogate epoch on the 4B head (d = 2560), 1 prompt x 16.
        dict(name="clipped_4b_1x16", kind="grad", dtype="bf16", B=1, G=16, d=2560, V=151936,
             floor=0.1, len_lo=64, len_hi=512, ws="default", clipped=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("coeffs", "weighted", "product", "dense", "audit", "allocate", "grad",
                       "grad", "grad", "grad"))
    # Group sizes of the configurations and tests, and any other up to 128.
    G = rng.choice((rng.choice((8, 16, 64)), rng.randint(2, 128)))
    if kind in ("coeffs", "weighted", "product"):
        c = dict(kind=kind, B=_log_int(rng, 1, min(4096, 4096 * 64 * 64 // (G * G))), G=G,
                 floor=rng.choice((0.05, 0.1, 0.2)), flags=rng.choice((0, 0, 1, 2, 3)))
        if kind != "product":
            c["rho"] = rng.choice(("product", "general"))
        if kind == "weighted":
            c["wmode"] = rng.choice(WMODES)
        return c
    if kind == "dense":
        D = _log_int(rng, 16, 16384)
        return dict(kind=kind, B=_log_int(rng, 1, max(1, min(4096, (1 << 30) // (G * D)))), G=G,
                    D=D, floor=rng.choice((0.05, 0.2)))
    if kind == "audit":
        return dict(kind=kind, N=_log_int(rng, 500, 50000 * 256 // max(256, G * G)), G=G,
                    D=_log_int(rng, 16, 4096), wmode=rng.choice(WMODES))
    if kind == "allocate":
        return dict(kind=kind, B=_log_int(rng, 1, max(1, min(4096, 4096 * 64 ** 3 // G ** 3))), G=G,
                    frac=round(rng.uniform(0.15, 0.9), 3), pi_min=rng.choice((0.05, 0.08)),
                    norms=rng.random() < 0.5)
    f32 = rng.random() < 0.25
    c = dict(kind="grad", dtype="f32" if f32 else "bf16", floor=rng.choice((0.1, 0.2)),
             G=rng.choice((4, 8, 16)))
    if f32:
        c.update(d=16 * _log_int(rng, 2, 64), V=_log_int(rng, 200, 32000))
        limit, most = 2e11, 8192
    else:
        c.update(d=rng.choice((64 * _log_int(rng, 2, 64), 512 * rng.randint(1, 6))),
                 V=rng.choice((_log_int(rng, 1000, 151936), 151936)))
        limit, most = 3e13, 65536
    tokens = _log_int(rng, 64, max(64, min(most, limit / (6.0 * c["d"] * c["V"]))))
    c["B"] = rng.choice((1, 2, 4)) if tokens >= 1024 else 1
    hi = max(4, int(1.25 * tokens / (c["B"] * c["G"])))
    c.update(len_lo=max(1, hi // rng.choice((2, 8))), len_hi=hi,
             ws="min" if rng.random() < 0.2 else "default", clipped=rng.random() < 0.25)
    return c


# ----------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape):
    return torch.rand(shape, generator=g, device=DEV)


def _groups(g, B, G, floor, rho_kind, contrast=False):
    q = _uniform(g, B, 1)
    r = (_uniform(g, B, G) < q).float()
    p = floor + (1.0 - floor) * (1.0 - _uniform(g, B, G))
    J = (_uniform(g, B, G) < p).to(torch.uint8)
    if contrast:
        r[:, 0], r[:, 1] = 1.0, 0.0
        J[:, :2] = 1
    if rho_kind == "general":
        u = torch.triu(0.05 + 0.95 * (1.0 - _uniform(g, B, G, G)), 1)
        rho = torch.minimum(u + u.transpose(1, 2), torch.minimum(p[:, :, None], p[:, None, :]))
    else:
        rho = p[:, :, None] * p[:, None, :]
    rho.diagonal(dim1=1, dim2=2).copy_(p)
    return dict(r=r, p=p, J=J, rho=rho.contiguous())


def _scale(G):
    return 2.0 / (G * (G - 1))  # 1 / C(G, 2): the paper's coefficients


def _normal(g, rows, cols, std, dtype):
    out = torch.empty(rows, cols, dtype=dtype, device=DEV)
    for s in range(0, rows, 16384):
        e = min(rows, s + 16384)
        out[s:e] = torch.randn(e - s, cols, generator=g, device=DEV) * std
    return out


def _head(case, seed):
    """Group inputs and the packed head batch of a grad case."""
    g = _gen(seed)
    B, G, d, V = case["B"], case["G"], case["d"], case["V"]
    st = _groups(g, B, G, case["floor"], "product", contrast=True)
    R = B * G
    # Lengths spread evenly over their range, dealt to the rollouts by the
    # seed: every batch of a case then has the same number of packed tokens.
    L_ = np.rint(np.linspace(case["len_lo"], case["len_hi"], R)).astype(np.int64)
    np.random.default_rng(seed).shuffle(L_)
    cu = np.zeros(R + 1, np.int64)
    np.cumsum((L_ + 7) // 8 * 8, out=cu[1:])
    T = int(cu[-1])
    mask = np.zeros(T, np.uint8)
    for i in range(R):
        mask[cu[i]:cu[i] + L_[i]] = 1
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    mask = torch.from_numpy(mask).to(DEV)
    H = _normal(g, T, d, 1.0, dt)
    H[mask == 0] = 0
    y = torch.randint(0, V, (T,), generator=g, device=DEV, dtype=torch.int32)
    y[mask == 0] = -100
    # Log-probabilities of an earlier policy (clipped cases): about those of
    # this one, so that some ratios are clipped and some are not. The target
    # logit of a random head is N(0, 1) and its log-sum-exp ln V + 1/2.
    st.update(T=T, H=H, W=_normal(g, V, d, 1.0 / math.sqrt(d), dt), y=y, mask=mask,
              cu=torch.from_numpy(cu.astype(np.int32)).to(DEV), B=B, G=G, d=d, V=V, R=R)
    return st


def _logp_old(case, seed, st):
    """Old per-rollout log-probabilities: this head's, from plain torch in
    fp32 blocks of the vocabulary, off by the ratio that earlier epochs moved
    them by: up to 1.4 for a rewarded rollout, down to 0.65 for the others, and
    0.02 away from the clip range's ends (rounding decides no clip)."""
    rows = torch.nonzero(st["mask"]).squeeze(1)
    Hf = st["H"][rows].float()
    lse = torch.full((rows.numel(),), -math.inf, device=DEV)
    for s in range(0, case["V"], 8192):
        z = Hf @ st["W"][s:s + 8192].float().t()
        lse = torch.logaddexp(lse, torch.logsumexp(z, 1))
    zy = (Hf * st["W"][st["y"][rows].long()].float()).sum(1)
    seg = torch.searchsorted(st["cu"], rows.to(torch.int32), right=True) - 1
    lp = torch.stack([(zy - lse)[seg == i].double().sum() for i in range(st["R"])])
    g = _gen(seed + 7919)
    lo = torch.tensor((0.65, 0.82, 1.02, 1.22), device=DEV)
    hi = torch.tensor((0.78, 0.98, 1.18, 1.40), device=DEV)
    part = torch.randint(0, 2, (st["R"],), generator=g, device=DEV)
    part = part + 2 * st["r"].reshape(-1).long()
    ratio = lo[part] + (hi - lo)[part] * torch.rand(st["R"], generator=g, device=DEV)
    return (lp - torch.log(ratio)).float()


def prepare(case, seed):
    k = case["kind"]
    st = dict(case=case)
    if k in ("coeffs", "weighted", "product"):
        st.update(_groups(_gen(seed), case["B"], case["G"], case["floor"],
                          case.get("rho", "product")))
    elif k == "dense":
        g = _gen(seed)
        st.update(_groups(g, case["B"], case["G"], case["floor"], "general"))
        st["S"] = torch.randn(case["B"], case["G"], case["D"], generator=g, device=DEV)
        st["g"] = torch.empty(case["B"], case["D"], device=DEV)
        st["a"] = torch.empty(case["B"], case["G"], device=DEV)
    elif k == "audit":
        g = _gen(seed)
        N, G, D = case["N"], case["G"], case["D"]
        st["r"] = (_uniform(g, G) < 0.5).float()
        st["r"][0], st["r"][1] = 1.0, 0.0
        p = 0.1 + 0.85 * _uniform(g, G)
        st["rho"] = torch.outer(p, p)
        st["rho"].diagonal().copy_(p)
        st["S"] = torch.randn(G, D, generator=g, device=DEV)
        st["Jd"] = (_uniform(g, N, G) < p).to(torch.uint8)
        st["ws"] = torch.empty(int(L.lib().pair_audit_workspace_size(N, G, D)), dtype=torch.uint8,
                               device=DEV)
    elif k == "allocate":
        g = _gen(seed)
        B, G = case["B"], case["G"]
        st["p_hat"] = 0.02 + 0.96 * _uniform(g, B, G)
        st["c_hat"] = torch.exp(0.6 * torch.randn(B, G, generator=g, device=DEV))
        st["m_hat"] = 0.3 + 2.7 * _uniform(g, B, G) if case["norms"] else None
        st["budget"] = (case["frac"] * st["c_hat"].double().sum(1)).float()
    else:
        st.update(_head(case, seed))
        dt = L.PAIR_BF16 if case["dtype"] == "bf16" else L.PAIR_F32
        size = (L.pair_grad_workspace_size if case["ws"] == "default"
                else L.pair_grad_workspace_min_size)
        # What a trainer keeps from step to step: the workspace and the
        # gradient buffers.
        st["ws"] = torch.empty(size(st["T"], st["d"], st["V"], st["R"], dt), dtype=torch.uint8,
                               device=DEV)
        st["dH"] = torch.empty(st["T"], st["d"], device=DEV)
        st["dW"] = torch.empty(st["V"], st["d"], device=DEV)
        if case["clipped"]:
            st["logp_old"] = _logp_old(case, seed, st)
    st["err"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    return st


def run(st):
    c = st["case"]
    k = c["kind"]
    if k == "coeffs":
        a, act, e, ce = L.pair_coeffs(st["r"], st["J"], st["rho"], scale=_scale(c["G"]),
                                      flags=c["flags"], dev_err=st["err"])
        return dict(a=a, active=act, edges=e, contrast=ce)
    if k == "weighted":
        a, act, e, ce, ess, mw = L.pair_coeffs_weighted(
            st["r"], st["J"], st["rho"], wmode=WMODES.index(c["wmode"]), w_max=W_MAX,
            scale=_scale(c["G"]), flags=c["flags"], dev_err=st["err"])
        return dict(a=a, active=act, edges=e, contrast=ce, ess=ess, max_w=mw)
    if k == "product":
        a, act, e, ce, ess, mw = L.pair_coeffs_product(
            st["r"], st["J"], st["p"], scale=_scale(c["G"]), flags=c["flags"], dev_err=st["err"])
        return dict(a=a, active=act, edges=e, contrast=ce, ess=ess, max_w=mw)
    if k == "dense":
        g, a = L.pair_estimate_dense(st["r"], st["J"], st["rho"], st["S"], scale=_scale(c["G"]),
                                     g=st["g"], a=st["a"], dev_err=st["err"])
        return dict(g=g, a=a)
    if k == "audit":
        stats, bias = L.pair_audit(st["r"], st["rho"], st["S"], st["Jd"],
                                   wmode=WMODES.index(c["wmode"]), w_max=W_MAX,
                                   scale=_scale(c["G"]), ws=st["ws"], dev_err=st["err"])
        return dict(bias_norm=stats[0], mse=stats[1], cos=stats[2], counts=stats[3:6],
                    target_sq=stats[6], weight=stats[7], bias=bias)
    if k == "allocate":
        pi, stats = L.pair_allocate(st["c_hat"], st["budget"], c["pi_min"], p_hat=st["p_hat"],
                                    m_hat=st["m_hat"], dev_err=st["err"])
        # Objective, expected cost and status. The other two columns say how
        # the solver got there (its duality-gap bound, its Newton steps) and
        # have no value of their own: the gap's bound is part of the contract
        # (at most 1e-12 of the objective) and is tested as such.
        return dict(pi=pi, phi=stats[:, 0], spent=stats[:, 1], status=stats[:, 4])
    # The head: this step's coefficients, then its objective and gradients.
    a = L.pair_coeffs(st["r"], st["J"], st["rho"], scale=_scale(c["G"]), dev_err=st["err"])[0]
    args = (st["H"], st["W"], st["y"], st["mask"], st["cu"], a.view(-1))
    if c["clipped"]:
        J, dH, dW, lp, coef = L.pair_grad_clipped(*args, st["logp_old"], CLIP_EPS, dH=st["dH"],
                                                  dW=st["dW"], ws=st["ws"], dev_err=st["err"])
        return dict(J=J, dH=dH, dW=dW, logp_seq=lp, a=a, coef=coef)
    J, dH, dW, lp = L.pair_grad(*args, dH=st["dH"], dW=st["dW"], ws=st["ws"], dev_err=st["err"])
    return dict(J=J, dH=dH, dW=dW, logp_seq=lp, a=a)


# ------------------------------------------------------- work and tolerance
def _mean_p(case):
    return 0.5 * (1.0 + case["floor"])


def _active_tokens(case):
    """Expected active tokens: every completed rollout has a contrast."""
    done = 2.0 + (case["G"] - 2) * _mean_p(case)
    return case["B"] * done * 0.5 * (case["len_lo"] + case["len_hi"])


def work(case):
    k = case["kind"]
    B, G = case.get("B", 1), case["G"]
    if k in ("coeffs", "weighted", "product"):
        # r, J and the outputs; of rho the edges between completed vertices.
        K = _mean_p(case) * G
        edge_bytes = 0.0 if k == "product" else 4.0 * K * K / 2
        out = 5.0 * G + 8 + (0 if k == "coeffs" else 8)
        return dict(bytes=B * (5.0 * G + edge_bytes + out + (4.0 * G if k == "product" else 0.0)),
                    flops=B * 3.0 * K * K / 2)
    if k == "dense":
        K = _mean_p(case) * G
        return dict(bytes=B * (5.0 * G + 2.0 * K * K + 4.0 * K * case["D"] + 4.0 * case["D"]
                               + 4.0 * G),
                    flops=B * (2.0 * K * case["D"] + 1.5 * K * K))
    if k == "audit":
        N, D = case["N"], case["D"]
        return dict(bytes=N * G + 4.0 * G * (D + G + 1) + 8.0 * D + 64.0,
                    flops=N * (2.0 * G * G + 1.5 * G * G / 2) + G * G * D)
    if k == "allocate":
        # Inputs and outputs; a dense symmetric solve for each of some twenty
        # interior-point steps (a path-following method's usual number).
        return dict(bytes=B * (4.0 * G * (3 + case["norms"]) + 4 + 40),
                    flops=B * 20.0 * (G ** 3 / 3.0 + 8.0 * G * G))
    d, V = case["d"], case["V"]
    Te = _active_tokens(case)
    T = B * G * (0.5 * (case["len_lo"] + case["len_hi"]) + 3.5)
    es = 2.0 if case["dtype"] == "bf16" else 4.0
    return dict(bytes=es * d * (Te + V) + 4.0 * d * (T + V) + 5.0 * T,
                flops=6.0 * d * V * Te)


def tolerance(case):
    # About four times what the library's results differ by from 64 bits.
    k = case["kind"]
    if k in ("coeffs", "weighted", "product"):
        return dict(rel=4e-7, max=2e-5)
    if k == "dense":
        return dict(rel=6e-7, max=4e-5)
    if k == "audit":  # the bias is what is left of sums a hundred times as large
        return dict(rel=1e-5, max=1e-4)
    if k == "allocate":  # fp32 rounding of pi; a bound that hardly binds moves more
        return dict(rel=4e-7, max=2e-6)
    if case["clipped"]:  # the ratio exponentiates a summed log-probability
        return dict(rel=3e-3, max=2e-2)
    if case["dtype"] == "f32":
        return dict(rel=1e-5, max=1e-3)
    # The one-hot parts are exact; the softmax parts, rounded to bf16, are
    # about 1 / sqrt(V) of them.
    return dict(rel=1.2e-2 / math.sqrt(case["V"]), max=1.2 / math.sqrt(case["V"]))


# ------------------------------------------------------------- in 64 bits
def _coeffs64(r, J, rho, scale, flags, mode="ht"):
    """Coefficients, counts and weight diagnostics [..., G] from rho's strict
    upper triangle (batched)."""
    r, rho, on = r.double(), rho.double(), J != 0
    G = r.shape[-1]
    live = on[..., :, None] & on[..., None, :]
    live = live & ~torch.eye(G, dtype=torch.bool, device=r.device)
    up = torch.triu(rho, 1)
    sym = up + up.transpose(-1, -2)
    if mode == "unweighted":
        w = torch.ones_like(sym)
    elif mode == "marginal":
        pi = torch.diagonal(rho, dim1=-2, dim2=-1)
        w = 1.0 / (pi[..., :, None] * pi[..., None, :])
    else:
        w = 1.0 / torch.where(live, sym, torch.ones_like(sym))
        if mode == "clipped":
            w = w.clamp(max=W_MAX)
    w = torch.where(live, w.expand(live.shape), torch.zeros((), dtype=w.dtype, device=w.device))
    dr = r[..., :, None] - r[..., None, :]
    a = 0.5 * (w * dr).sum(-1)
    W, W2 = w.sum((-1, -2)) / 2, (w * w).sum((-1, -2)) / 2
    if mode == "hajek":
        a = torch.where(W[..., None] > 0, a / W[..., None].clamp(min=1e-300), 0.0)
    K = on.sum(-1)
    Kd = K.double()[..., None]
    if flags & 2:
        mean = (r * on).sum(-1, keepdim=True) / Kd.clamp(min=1)
        sd = ((((r - mean) * on) ** 2).sum(-1, keepdim=True) / (Kd - 1).clamp(min=1)).sqrt()
        a = torch.where(Kd >= 2, torch.where(sd > 0, a / sd.clamp(min=1e-300), 0.0), a)
    if flags & 1:
        a = torch.where(on, a - a.sum(-1, keepdim=True) / Kd.clamp(min=1), a)
    contrast = live & (dr != 0)
    return dict(a=a * scale, active=contrast.any(-1).to(torch.uint8),
                edges=(K * (K - 1) // 2).int(), contrast=(contrast.sum((-1, -2)) // 2).int(),
                ess=torch.where(W2 > 0, W * W / W2.clamp(min=1e-300), 0.0),
                max_w=w.amax((-1, -2)), K=K)


def _audit64(case, st):
    N, G = case["N"], case["G"]
    S, r = st["S"].double(), st["r"].double()
    scale = _scale(G)
    abar = scale * 0.5 * (G * r - r.sum())
    g = abar @ S
    K = S @ S.t()
    mse = cos = vert = edge = ess = 0.0
    asum = torch.zeros(G, dtype=torch.float64, device=DEV)
    for s in range(0, N, 4096):
        Jd = st["Jd"][s:s + 4096]
        n = Jd.shape[0]
        o = _coeffs64(st["r"].expand(n, G), Jd, st["rho"].expand(n, G, G), scale, 0, case["wmode"])
        a = o["a"]
        e = a - abar
        aa = ((a @ K) * a).sum(1)
        ag = (a @ K) @ abar
        gg = float(g @ g)
        mse += float(((e @ K) * e).sum())
        cos += float(torch.where((aa > 0) & (gg > 0), ag / (aa * gg).clamp(min=1e-300).sqrt(),
                                 0.0).sum())
        vert += float(o["K"].sum())
        edge += float(o["edges"].sum())
        ess += float(o["ess"].sum())
        asum += a.sum(0)
    bias = (asum / N - abar) @ S
    f = lambda v: torch.tensor(v, dtype=torch.float64)  # noqa: E731
    return dict(bias_norm=f(float(bias.norm())), mse=f(mse / N), cos=f(cos / N),
                counts=f([vert / N, edge / N, ess / N]), target_sq=f(float(g @ g)), weight=f(1.0),
                bias=bias)


def _allocate64(case, st):
    """min sum_{i<j} a_ij / (pi_i pi_j) + sum_i b_i / pi_i over pi_min <= pi <= 1
    and sum c pi = budget (the objective falls in every pi_i, so the budget is
    spent), by a batched primal-dual interior-point method."""
    G = case["G"]
    p, c = st["p_hat"].double(), st["c_hat"].double()
    bud = st["budget"].double()[:, None]
    pmin = float(torch.tensor(case["pi_min"], dtype=torch.float32))
    A = p[:, :, None] * (1 - p[:, None, :]) + (1 - p[:, :, None]) * p[:, None, :]
    if st["m_hat"] is not None:
        m = st["m_hat"].double()
        A = A * (0.5 * (m[:, :, None] + m[:, None, :])) ** 2
    A = A * (1 - torch.eye(G, dtype=torch.float64, device=p.device))
    b = A.sqrt().sum(2) ** 2 - A.sum(2)

    def terms(pi):
        v = 1.0 / pi
        w = (A @ v[:, :, None])[:, :, 0]
        return v, w + b, (v * (0.5 * w + b)).sum(1, keepdim=True)

    lo = bud / c.sum(1, keepdim=True) - pmin + torch.zeros_like(c)
    hi = 1.0 - pmin - lo
    v, wb, phi = terms(pmin + lo)
    zl, zh = 0.1 * phi / (2 * G) / lo, 0.1 * phi / (2 * G) / hi
    y = (v * v * wb / c).mean(1, keepdim=True)
    for _ in range(60):
        pi = torch.where(hi < lo, 1.0 - hi, pmin + lo)
        v, wb, phi = terms(pi)
        eta = (zl * lo + zh * hi).sum(1, keepdim=True)
        res = ((-v * v * wb + y * c - zl + zh) * pi).abs().sum(1, keepdim=True)
        if bool(((eta <= 1e-14 * phi) & (res <= 1e-12 * phi)).all()):
            break
        mu = torch.maximum(0.1 * eta, 5e-16 * phi) / (2 * G)
        H = A * (v * v)[:, :, None] * (v * v)[:, None, :]
        H = H + torch.diag_embed(2 * v ** 3 * wb + zl / lo + zh / hi)
        Lc = torch.linalg.cholesky(H)
        rhs = torch.stack((v * v * wb - y * c + mu / lo - mu / hi, c), 2)
        h = torch.cholesky_solve(rhs, Lc)
        rp = bud - (c * pi).sum(1, keepdim=True)
        dy = (((c * h[:, :, 0]).sum(1, keepdim=True) - rp)
              / (c * h[:, :, 1]).sum(1, keepdim=True))
        d = h[:, :, 0] - dy * h[:, :, 1]
        dzl, dzh = (mu - zl * d) / lo - zl, (mu + zh * d) / hi - zh
        step = torch.ones_like(bud)
        for q, dq in ((lo, d), (hi, -d), (zl, dzl), (zh, dzh)):
            t = torch.where(dq < 0, -q / dq.clamp(max=-1e-300), 1e300).amin(1, keepdim=True)
            step = torch.minimum(step, 0.995 * t)
        lo, hi, y = lo + step * d, hi - step * d, y + step * dy
        zl, zh = zl + step * dzl, zh + step * dzh
    pi = torch.where(hi < lo, 1.0 - hi, pmin + lo)
    return dict(pi=pi, phi=terms(pi)[2][:, 0], spent=(c * pi).sum(1),
                status=torch.zeros(case["B"], dtype=torch.float64, device=p.device))


def _grad64(case, st):
    a = _coeffs64(st["r"], st["J"], st["rho"], _scale(case["G"]), 0)["a"].reshape(-1)
    T, d, V, R = st["T"], st["d"], st["V"], st["R"]
    t = torch.arange(T, device=DEV, dtype=torch.int32)
    seg = (torch.searchsorted(st["cu"], t, right=True) - 1).long()
    rows = torch.nonzero((st["mask"] != 0) & (a[seg] != 0)).squeeze(1)
    sg, yt = seg[rows], st["y"][rows].long()
    H = st["H"][rows].double()
    n, step = rows.numel(), 8192
    lse = torch.full((n,), -math.inf, dtype=torch.float64, device=DEV)
    for s in range(0, V, step):
        lse = torch.logaddexp(lse, torch.logsumexp(H @ st["W"][s:s + step].double().t(), 1))
    zy = (H * st["W"][yt].double()).sum(1)
    lp = torch.zeros(R, dtype=torch.float64, device=DEV).index_add_(0, sg, zy - lse)
    out = dict(logp_seq=lp, a=a.reshape(st["r"].shape))
    if case["clipped"]:
        ratio = torch.exp(torch.where(a != 0, lp - st["logp_old"].double(), 0.0))
        lim = ratio.clamp(1.0 - CLIP_EPS, 1.0 + CLIP_EPS)
        out["J"] = torch.minimum(ratio * a, lim * a).sum().reshape(1)
        keep = torch.where(a > 0, ratio <= 1.0 + CLIP_EPS, ratio >= 1.0 - CLIP_EPS) & (a != 0)
        coef = torch.where(keep, a * ratio, 0.0)
        out["coef"] = coef
    else:
        out["J"] = (a * lp).sum().reshape(1)
        coef = a
    c = coef[sg]
    dHr = torch.zeros(n, d, dtype=torch.float64, device=DEV)
    dW = torch.zeros(V, d, dtype=torch.float64, device=DEV)
    for s in range(0, V, step):
        Wd = st["W"][s:s + step].double()
        Gs = torch.exp(H @ Wd.t() - lse[:, None]) * -c[:, None]
        dHr += Gs @ Wd
        dW[s:s + step] = Gs.t() @ H
    dHr += c[:, None] * st["W"][yt].double()
    dW.index_add_(0, yt, c[:, None] * H)
    dH = torch.zeros(T, d, dtype=torch.float64, device=DEV)
    dH[rows] = dHr
    out.update(dH=dH, dW=dW)
    return out


def exact(case, seed):
    k = case["kind"]
    if k == "grad" and work(case)["flops"] > 8e12:
        return None  # over 20 s in 64 bits
    st = prepare(dict(case, ws="min") if k == "grad" else case, seed)
    if k in ("coeffs", "weighted", "product"):
        rho = st["rho"]
        if k == "product":
            p = st["p"].double()
            rho = p[:, :, None] * p[:, None, :]
        out = {}
        for s in range(0, case["B"], 1024):
            o = _coeffs64(st["r"][s:s + 1024], st["J"][s:s + 1024], rho[s:s + 1024],
                          _scale(case["G"]), case["flags"], case.get("wmode", "ht"))
            for n, v in o.items():
                out.setdefault(n, []).append(v)
        keys = ["a", "active", "edges", "contrast"] + ([] if k == "coeffs" else ["ess", "max_w"])
        return {n: torch.cat(out[n]) for n in keys}
    if k == "dense":
        a, g = [], []
        for s in range(0, case["B"], 64):
            o = _coeffs64(st["r"][s:s + 64], st["J"][s:s + 64], st["rho"][s:s + 64],
                          _scale(case["G"]), 0)["a"]
            a.append(o)
            g.append((o[:, None, :] @ st["S"][s:s + 64].double())[:, 0])
        return dict(g=torch.cat(g), a=torch.cat(a))
    if k == "audit":
        return _audit64(case, st)
    if k == "allocate":
        return _allocate64(case, st)
    return _grad64(case, st)
