"""Cases for timing the framework: the work a program that fits adapters gives it, through the
public entry points of ``paper_2608_03020_gb300.loca``.

A case is one of six kinds.

* ``pass``    one outer iteration through ``loca.Pass`` (head error, targets, Gram / cross
  statistics per mini-batch, ridge solves), bf16 or fp32 activations;
* ``chain``   the same iteration for a single mini-batch from the separate entry points: the cross
  product at alpha = 1, the step from the trace of the Gram matrix, alpha applied in the solve;
* ``fused``   the iteration without a stored T: ``loca_targets_sq``, ``loca_gram_cross_fused``, the
  step, the solve;
* ``kspace``  the iteration with the statistics kept in adapter space (k x k);
* ``solve``   the ridge solves alone from statistics at hand (another candidate set of lambdas);
* ``calib``   the one-shot feedback fit from probe pairs and its alignment diagnostic, either
  label-restricted (``loca_calib_fit``) or d-wide (``loca_calib_fit_rsvd``).

Shapes are those of ``synth.inputs.WORKLOADS``, of the tests, or generic ones between them.
Activations are Gaussian with log-normal channel scales and, for bf16, four outlier channels at
20x; logits come from the last block's activations when only the label columns exist (V == C), else
they are a full vocabulary row that gives the label columns about half the softmax mass.
"""

import math

import torch

from paper_2608_03020_gb300 import loca

DEV = "cuda"
F32 = torch.float32
F64 = torch.float64
ETA = 0.01
LAMBDAS = (1e-4, 1e-3, 1e-2)


def _case(kind, name, **sizes):
    return dict(kind=kind, name=name, **sizes)


def listed():
    return [
        # the smallest pass in fp32 (the tiny workload): launches and latency
        _case("pass", "pass_tiny_f32", dtype="f32", L=2, d=64, N=512, C=4, V=4, r=4, k=4, nl=1, mb=1),
        # a few ragged sequences of a small model, ranks that are no multiple of 4, two uneven mini-batches
        _case("pass", "pass_ragged_bf16", dtype="bf16", L=6, d=328, N=3001, C=3, V=3, r=5, k=6, nl=3, mb=2),
        # the Qwen2.5-0.5B workload: one mini-batch of 64 sequences of 256 tokens
        _case("pass", "pass_qwen0.5b", dtype="bf16", L=24, d=896, N=16384, C=4, V=4, r=8, k=8, nl=3, mb=1),
        # the Qwen2.5-1.5B workload: 8 streamed mini-batches of 8192 tokens, statistics accumulated
        _case("pass", "pass_qwen1.5b_stream", dtype="bf16", L=28, d=1536, N=65536, C=4, V=4, r=16, k=16, nl=3, mb=8),
        # the Qwen2.5-7B workload, the headline: every block, every token
        _case("chain", "chain_qwen7b", L=28, d=3584, N=131072, C=4, V=4, r=16, k=16, nl=3),
        # 7B width where T (as large as X) is not to be stored
        _case("fused", "fused_7b_width", L=8, d=3584, N=32768, C=4, V=4, r=16, k=16, nl=3),
        # one small batch through the k-space path: latency
        _case("kspace", "kspace_small", L=24, d=896, N=1000, C=4, V=4, r=8, k=8, nl=3),
        # the Qwen2.5-7B workload in adapter space
        _case("kspace", "kspace_qwen7b", L=28, d=3584, N=131072, C=4, V=4, r=16, k=16, nl=3),
        # SmolLM2-1.7B: full vocabulary row for the head error, r = k = 32
        _case("kspace", "kspace_smollm2_vocab", L=24, d=2048, N=65536, C=4, V=49152, r=32, k=32, nl=3),
        # the Qwen2.5-14B solves from statistics at hand, second iteration (B_prev)
        _case("solve", "solve_qwen14b", L=48, d=5120, k=32, nl=3),
        # label-restricted calibration (C = 16 error columns) at 1.5B width over all blocks
        _case("calib", "calib_label_1.5b", wide=False, L=28, d=1536, Np=8192, m=16, r=16),
        # d-wide calibration at 1.5B width over all blocks: ell = 2 r, two power iterations
        _case("calib", "calib_wide_1.5b", wide=True, L=28, d=1536, Np=8192, m=1536, r=16, ell=32, q=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi, step=1):
    return max(lo, min(hi, int(round(_log(rng, lo, hi) / step)) * step))


def draw(rng):
    kind = rng.choice(["pass", "pass", "pass", "chain", "fused", "kspace", "kspace", "solve", "calib", "calib"])
    C = rng.choice([2, 3, 4, 4, 5, 8])
    nl = rng.choice([1, 3, 3, 4])
    if kind == "calib":
        wide = rng.random() < 0.5
        r = rng.choice([4, 8, 12, 16])
        L, d, Np = rng.randint(2, 28), _size(rng, 128, 2048, rng.choice([1, 8, 64])), _size(rng, 512, 8192)
        if wide:
            c = dict(kind=kind, wide=True, L=L, d=d, Np=Np, m=d, r=r, ell=2 * r, q=rng.choice([1, 2]))
        else:
            c = dict(kind=kind, wide=False, L=L, d=d, Np=Np, m=rng.choice([r, r + 1, 24, 32]), r=r)
        while c["L"] > 1 and c["L"] * c["Np"] * c["d"] > 28 * 8192 * 1536:
            c["L"] = max(1, c["L"] // 2)
        return c
    k = rng.choice([4, 6, 8, 12, 16, 20, 32])
    if kind == "solve":
        return dict(kind=kind, L=rng.randint(1, 32), d=_size(rng, 64, 5120, rng.choice([1, 4, 8, 128])), k=k, nl=nl)
    r = rng.choice([1, 4, 5, 8, 16, 24, 32])
    L, N = rng.randint(1, 28), _size(rng, 64, 65536, rng.choice([1, 1, 64, 256]))
    d = _size(rng, 64, 4096, rng.choice([8, 8, 64, 256]))
    c = dict(kind=kind, L=L, d=d, N=N, C=C, V=C, r=r, k=k, nl=nl)
    if kind == "pass":
        if rng.random() < 0.25:
            c.update(dtype="f32", mb=1, L=rng.randint(1, 4), d=_size(rng, 17, 128), N=_size(rng, 64, 1024))
            c.update(k=min(c["k"], c["d"]))
        else:
            c.update(dtype="bf16", mb=rng.choice([1, 1, 2, 4]))
    elif rng.random() < 0.4:
        c["V"] = _size(rng, 1024, 151936)
    while c["N"] > 64 and (c["L"] * c["N"] * c["d"] ** 2 > 28 * 16384 * 1536 ** 2 or c["N"] * c["V"] > 1 << 31):
        c["N"] = c["N"] // 2
    return c


def _lambdas(c):
    return (1e-2,) if c["nl"] == 1 else tuple((1e-4, 1e-3, 1e-2, 1e-1)[: c["nl"]])


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _normal(g, *shape, scale=1.0):
    return torch.randn(shape, generator=g, device=DEV, dtype=F32).mul_(scale)


def _channel_scales(g, d, outliers):
    s = torch.exp(0.5 * _normal(g, d))
    if outliers:
        s[torch.randperm(d, generator=g, device=DEV)[:4]] *= 20.0
    return s


def _activations(g, L, N, d, dtype):
    X = torch.empty((L, N, d), device=DEV, dtype=dtype)
    for l in range(L):
        s = _channel_scales(g, d, dtype == torch.bfloat16)
        for n0 in range(0, N, 32768):
            n1 = min(N, n0 + 32768)
            X[l, n0:n1] = _normal(g, n1 - n0, d).mul_(s)
    return X


def _logits(g, c, X_last):
    N, C, V, d = c["N"], c["C"], c["V"], c["d"]
    if V == C:
        head = _normal(g, d, C, scale=1.0 / math.sqrt(d))
        return X_last.float() @ head, torch.arange(C, device=DEV, dtype=torch.int32)
    cols = torch.randperm(V, generator=g, device=DEV)[:C].sort().values
    z = torch.empty((N, V), device=DEV, dtype=torch.bfloat16)
    for n0 in range(0, N, 8192):
        n1 = min(N, n0 + 8192)
        part = _normal(g, n1 - n0, V)
        part[:, cols] += math.log(V / C)
        z[n0:n1] = part
    return z, cols.to(torch.int32)


def _down(g, L, d, k):
    """Orthonormal down-projections (L x d x k)."""
    return torch.linalg.qr(_normal(g, L, d, k).double())[0].float().contiguous()


def _batches(c):
    nb = -(-c["N"] // c.get("mb", 1))
    return [(n0, min(c["N"], n0 + nb)) for n0 in range(0, c["N"], nb)]


def _buf(*shape, dtype=F32):
    return torch.empty(shape, device=DEV, dtype=dtype)


def _inputs(c, seed):
    """Inputs of a pass: activations, logits, labels, feedback factors, down-projections."""
    g = _gen(seed)
    L, N, d, C, r, k = c["L"], c["N"], c["d"], c["C"], c["r"], c["k"]
    s = dict(case=c, lam=_lambdas(c))
    s["X"] = _activations(g, L, N, d, F32 if c.get("dtype") == "f32" else torch.bfloat16)
    s["z"], s["cols"] = _logits(g, c, s["X"][L - 1])
    s["y"] = torch.randint(0, C, (N,), generator=g, device=DEV, dtype=torch.int32)
    s["P"] = _normal(g, L, C, r, scale=1.0 / math.sqrt(r))
    s["Q"] = _normal(g, L, r, d, scale=1.0 / math.sqrt(r))
    s["A"] = _down(g, L, d, k)
    return s


def _probe_pairs(c, seed):
    """Probe errors with anisotropic columns and gradients E M_l + noise, M_l of rank r with a
    decaying spectrum."""
    g = _gen(seed)
    L, d, Np, m, r = c["L"], c["d"], c["Np"], c["m"], c["r"]
    E = _normal(g, Np, m).mul_(torch.exp(0.5 * _normal(g, m)) if c["wide"] else 1.0)
    G = _buf(L, Np, d)
    decay = 0.8 ** torch.arange(r, device=DEV, dtype=F32)
    for l in range(L):
        clean = (E @ (_normal(g, m, r) * decay)) @ _normal(g, r, d, scale=1.0 / math.sqrt(r * m))
        G[l] = clean + 0.1 * clean.square().mean().sqrt() * _normal(g, Np, d)
    s = dict(case=c, E=E, G=G, beta=float(1e-3 * E.square().sum() / m))
    if c["wide"]:
        s["Omega"] = _normal(g, d, c["ell"])
    return s


def _statistics(c, seed):
    """Gram and cross products as a pass leaves them (512 tokens plus the channel variances)."""
    g = _gen(seed)
    L, d, k = c["L"], c["d"], c["k"]
    s = dict(case=c, lam=_lambdas(c), gram=_buf(L, d, d), cross=_buf(L, d, d))
    for l in range(L):
        scale = _channel_scales(g, d, True)
        X = _normal(g, 512, d).mul_(scale)
        s["gram"][l] = X.t() @ X
        s["gram"][l].diagonal().add_(512.0 * scale * scale)
        s["cross"][l] = ((_normal(g, 512, 4) @ _normal(g, 4, d)).t() @ X).mul_(-1e-2)
    s["xsq"] = s["gram"].diagonal(dim1=1, dim2=2).double().sum(1)
    s["A"] = _down(g, L, d, k)
    s["B_prev"] = _normal(g, L, d, k, scale=0.01)
    return s


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "solve":
        s = _statistics(c, seed)
        L, d, k, nl = c["L"], c["d"], c["k"], c["nl"]
        s.update(B=_buf(nl, L, d, k), info=_buf(nl, L, dtype=torch.int32), G=_buf(L, k, k), C_out=_buf(L, d, k),
                 ws=_buf(max(1, loca.ridge_solve_workspace_size(L, d, k)), dtype=torch.uint8))
        return s
    if kind == "calib":
        s = _probe_pairs(c, seed)
        L, d, m, r = c["L"], c["d"], c["m"], c["r"]
        s.update(P=_buf(L, m, r), Q=_buf(L, r, d), sigma=_buf(L, r), alpha=_buf(L, dtype=F64))
        return s
    s = _inputs(c, seed)
    L, N, d, C, r, k, nl = c["L"], c["N"], c["d"], c["C"], c["r"], c["k"], c["nl"]
    if kind == "pass":
        s["X"] = [s["X"]] if c["mb"] == 1 else [s["X"][:, n0:n1].contiguous() for n0, n1 in _batches(c)]
        s["pass"] = loca.Pass(L, N, d, C, r, k, s["X"][0].dtype, s["lam"], ETA, micro_batches=len(s["X"]))
        return s
    s.update(E=_buf(N, C), ce=_buf(N), xsq=_buf(L, dtype=F64), alpha=_buf(L), B=_buf(nl, L, d, k),
             info=_buf(nl, L, dtype=torch.int32))
    if kind == "kspace":
        s.update(G=_buf(L, k, k), SC=_buf(L, C, k), C_out=_buf(L, d, k),
                 ws=_buf(max(1, loca.kspace_workspace_size(L, N, d, k, C, r)), dtype=torch.uint8))
        return s
    s.update(tsq=_buf(L, dtype=F64), ones=torch.ones((L,), device=DEV), gram=_buf(L, d, d), cross=_buf(L, d, d),
             ws_s=_buf(max(1, loca.ridge_solve_workspace_size(L, d, k)), dtype=torch.uint8))
    if kind == "chain":
        s.update(T=_buf(L, N, d, dtype=torch.bfloat16),
                 ws_t=_buf(max(1, loca.targets_workspace_size(N, L, d)), dtype=torch.uint8),
                 ws_g=_buf(max(1, loca.gram_cross_workspace_size()), dtype=torch.uint8))
    else:
        s.update(ws_t=_buf(max(1, loca.targets_sq_workspace_size(N, C)), dtype=torch.uint8),
                 ws_g=_buf(max(1, loca.gram_cross_fused_workspace_size(L, N, r)), dtype=torch.uint8))
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "pass":
        p = s["pass"]
        p.run(s["z"], s["cols"], s["y"], s["X"][0] if len(s["X"]) == 1 else s["X"], s["P"], s["Q"], s["A"])
        n0, n1 = _batches(c)[-1]
        T = p.T.view(-1)[: c["L"] * (n1 - n0) * c["d"]].view(c["L"], n1 - n0, c["d"])
        return dict(E=p.E, ce=p.ce, T=T, gram=p.gram, cross=p.cross, xsq=p.xsq, B=p.B, info=p.info)
    if kind == "solve":
        loca.loca_ridge_solve(s["gram"], s["cross"], s["A"], s["lam"], s["B"], s["info"], xsq_total=s["xsq"],
                              B_prev=s["B_prev"], G_out=s["G"], C_out=s["C_out"], workspace=s["ws"])
        return dict(B=s["B"], info=s["info"], G=s["G"], C=s["C_out"])
    if kind == "calib":
        if c["wide"]:
            loca.loca_calib_fit_rsvd(s["E"], s["G"], s["beta"], c["r"], s["Omega"], c["q"], s["P"], s["Q"],
                                     sigma=s["sigma"])
        else:
            loca.loca_calib_fit(s["E"], s["G"], s["beta"], c["r"], s["P"], s["Q"], sigma=s["sigma"])
        loca.loca_alignment(s["E"], s["G"], s["P"], s["Q"], s["alpha"])
        return dict(P=s["P"], Q=s["Q"], sigma=s["sigma"], alpha=s["alpha"])
    loca.loca_error(s["z"], s["cols"], s["y"], s["E"], ce=s["ce"])
    if kind == "kspace":
        loca.loca_kspace_accumulate(s["X"], s["A"], s["E"], s["P"], s["Q"], ETA, s["G"], s["SC"], s["xsq"],
                                    zero_first=True, alpha=s["alpha"], workspace=s["ws"])
        loca.loca_kspace_solve(s["G"], s["SC"], s["P"], s["Q"], s["lam"], s["B"], s["info"], xsq_total=s["xsq"],
                               C_out=s["C_out"])
        return dict(E=s["E"], ce=s["ce"], G=s["G"], SC=s["SC"], xsq=s["xsq"], alpha=s["alpha"], B=s["B"],
                    info=s["info"], C=s["C_out"])
    if kind == "chain":
        loca.loca_targets(s["E"], s["P"], s["Q"], s["T"], tsq=s["tsq"], workspace=s["ws_t"])
        loca.loca_gram_cross(s["X"], s["T"], s["ones"], s["gram"], s["cross"], zero_first=True, workspace=s["ws_g"])
    else:
        loca.loca_targets_sq(s["E"], s["P"], s["Q"], s["tsq"], workspace=s["ws_t"])
        loca.loca_gram_cross_fused(s["X"], s["E"], s["P"], s["Q"], s["ones"], s["gram"], s["cross"], zero_first=True,
                                   workspace=s["ws_g"])
    loca.loca_step_from_gram(s["gram"], s["tsq"], ETA, s["xsq"], s["alpha"])
    loca.loca_ridge_solve(s["gram"], s["cross"], s["A"], s["lam"], s["B"], s["info"], xsq_total=s["xsq"],
                          cross_scale=s["alpha"], workspace=s["ws_s"])
    return dict(E=s["E"], ce=s["ce"], tsq=s["tsq"], gram=s["gram"], cross=s["cross"], xsq=s["xsq"],
                alpha=s["alpha"], B=s["B"], info=s["info"])


def work(case):
    c = case
    kind = c["kind"]
    L, d = c["L"], c["d"]
    if kind == "calib":
        Np, m, r = c["Np"], c["m"], c["r"]
        # the probe pairs are read by the fit and, with the fitted factors, by the diagnostic; the
        # fit's last product needs the factors of the whole probe set, so G is counted once for each
        byt = 4 * (2 * (Np * m + L * Np * d) + 2 * L * r * (m + d))
        if c["wide"]:
            ell, q = c["ell"], c["q"]
            flops = Np * m * (m + 1) + m ** 3 / 3 + (2 * q + 2) * L * ell * (2 * Np * (m + d) + 2 * m * m)
        else:
            flops = Np * m * (m + 1) + 2 * L * Np * m * d + L * (m * m * d * 2)
        flops += 2 * L * Np * r * (m + d)
        return dict(bytes=byt, flops=flops)
    k, nl = c["k"], c["nl"]
    solve_b = 4 * (L * d * k * (1 + nl))
    solve_f = L * nl * (k ** 3 / 3 + 2 * d * k * k)
    if kind == "solve":
        return dict(bytes=4 * (2 * L * d * d + 2 * L * d * k + L * k * k) + solve_b,
                    flops=4 * L * d * d * k + 4 * L * d * k * k + solve_f)
    N, C, V, r = c["N"], c["C"], c["V"], c["r"]
    el = 4 if c.get("dtype") == "f32" else 2
    byt = L * N * d * el + N * V * (4 if V == C else 2) + 4 * N * (C + 2) + 4 * L * r * (C + d) + solve_b
    if kind == "kspace":
        byt += 4 * L * (k * k + C * k + d * k)
        return dict(bytes=byt, flops=L * N * (2 * d * k + k * k + 2 * C * k + 2 * d) + 4 * L * d * C * k + solve_f)
    byt += 4 * 2 * L * d * d
    stats = L * N * d * (d + 1)
    if kind == "fused":  # T^T X = Q^T ((E P)^T X): T need not exist
        stats += 2 * L * N * r * (C + d) + 2 * L * d * d * r
    else:  # T is an output (one mini-batch of it in a streamed pass), rounded to the activations' type
        byt += L * (_batches(c)[0][1]) * d * el if kind == "pass" else L * N * d * el
        stats += 2 * L * N * r * (C + d) + 2 * L * N * d * d
    return dict(bytes=byt, flops=stats + 4 * L * d * d * k + solve_f)


def tolerance(case):
    """About four times the error against 64 bits that the listed and drawn cases show."""
    c = case
    if c["kind"] in ("calib", "solve") or c.get("dtype") == "f32":
        return {"rel": 1e-5}  # fp32 sums, fp64 solves; 3e-7 measured
    if c["kind"] == "kspace":
        return {"rel": 3e-5}  # A split into two bf16 parts (2^-16 each entry): 7e-6 measured
    # T is rounded to bf16 once, 1.7e-3 of T; up to 1.6e-3 of a cross product and of B
    return {"rel": 7e-3}


# ------------------------------------------------------------------------------ the same in 64 bits

def _head_error64(s):
    c = s["case"]
    N, C = c["N"], c["C"]
    E, ce = _buf(N, C, dtype=F64), _buf(N, dtype=F64)
    cols, y = s["cols"].long(), s["y"].long()
    for n0 in range(0, N, 4096):
        n1 = min(N, n0 + 4096)
        z = s["z"][n0:n1].double()
        lse = torch.logsumexp(z, dim=1)
        zc = z[:, cols]
        onehot = torch.nn.functional.one_hot(y[n0:n1], C).double()
        E[n0:n1] = torch.exp(zc - lse[:, None]) - onehot
        ce[n0:n1] = lse - (zc * onehot).sum(1)
    return E, ce


def _solve64(Gk, Ck, lam):
    """B[j, l] = C_l (G_l + lam_jl I)^-1, lam: nl x L."""
    eye = torch.eye(Gk.shape[1], device=DEV, dtype=F64)
    M = Gk[None] + lam[:, :, None, None] * eye
    return torch.linalg.solve(M, Ck.transpose(1, 2)[None].expand(M.shape[0], -1, -1, -1)).transpose(2, 3).contiguous()


def _signed(u, sv, vt, r):
    """P = U S, Q = V^T with the entry of largest magnitude in each row of Q positive."""
    u, sv, vt = u[:, :r], sv[:r], vt[:r]
    at = vt.abs().argmax(dim=1, keepdim=True)
    sign = torch.sign(torch.gather(vt, 1, at))[:, 0]
    return u * (sv * sign)[None, :], vt * sign[:, None], sv


def _calib64(s):
    c = s["case"]
    E = s["E"].double()
    m, r = c["m"], c["r"]
    chol = torch.linalg.cholesky(E.t() @ E + s["beta"] * torch.eye(m, device=DEV, dtype=F64))
    out = dict(P=[], Q=[], sigma=[], alpha=[])
    for l in range(c["L"]):
        G = s["G"][l].double()
        if c["wide"]:
            def ft(x):
                return torch.cholesky_solve(E.t() @ (G @ x), chol)

            def f(x):
                return G.t() @ (E @ torch.cholesky_solve(x, chol))

            basis = torch.linalg.qr(ft(s["Omega"].double()))[0]
            for _ in range(c["q"]):
                basis = torch.linalg.qr(ft(torch.linalg.qr(f(basis))[0]))[0]
            u, sv, vt = torch.linalg.svd(f(basis).t(), full_matrices=False)
            u = basis @ u
        else:
            u, sv, vt = torch.linalg.svd(torch.cholesky_solve(E.t() @ G, chol), full_matrices=False)
        P, Q, sv = _signed(u, sv, vt, r)
        T = (E @ P) @ Q
        for key, v in zip(("P", "Q", "sigma", "alpha"), (P, Q, sv, (G * T).sum() / (G.norm() * T.norm()))):
            out[key].append(v)
    return {key: torch.stack(v) for key, v in out.items()}


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    # 64-bit Gram matrices above this size take over 20 s; everything else of such a pass is still given
    gram_fits = kind in ("solve", "calib", "kspace") or c["L"] * c["N"] * c["d"] ** 2 <= 1.3 * 28 * 65536 * 1536 ** 2
    if kind == "calib":
        return _calib64(_probe_pairs(c, seed))
    if kind == "solve":
        s = _statistics(c, seed)
        A, Bp = s["A"].double(), s["B_prev"].double()
        lam = torch.tensor(s["lam"], device=DEV, dtype=F32).double()[:, None] * s["xsq"][None] / c["d"]
        Gk, Ck = _buf(c["L"], c["k"], c["k"], dtype=F64), _buf(c["L"], c["d"], c["k"], dtype=F64)
        for l in range(c["L"]):
            Gk[l] = A[l].t() @ (s["gram"][l].double() @ A[l])
            Ck[l] = Bp[l] @ Gk[l] + s["cross"][l].double() @ A[l]
        return dict(B=_solve64(Gk, Ck, lam), info=None, G=Gk, C=Ck)
    s = _inputs(c, seed)
    L, N, d, C, k = c["L"], c["N"], c["d"], c["C"], c["k"]
    E, ce = _head_error64(s)
    P, Q, A = s["P"].double(), s["Q"].double(), s["A"].double()
    gram = _buf(L, d, d, dtype=F32) if kind != "kspace" and gram_fits else None
    cross = _buf(L, d, d, dtype=F32) if kind != "kspace" else None
    xsq, tsq, alpha = (torch.zeros(L, device=DEV, dtype=F64) for _ in range(3))
    Gk, SC, Ck = (torch.zeros(shape, device=DEV, dtype=F64) for shape in ((L, k, k), (L, C, k), (L, d, k)))
    batches = _batches(c)
    T = _buf(L, batches[-1][1] - batches[-1][0], d) if kind == "pass" else None
    for l in range(L):
        g64 = torch.zeros((d, d), device=DEV, dtype=F64) if gram is not None else None
        c64 = torch.zeros((d, d), device=DEV, dtype=F64) if cross is not None else None
        for n0, n1 in batches:
            U = E[n0:n1] @ P[l]
            xb = torch.zeros((), device=DEV, dtype=F64)
            S, Sk, ua = (torch.zeros(shape, device=DEV, dtype=F64) for shape in ((c["r"], d), (C, k), (c["r"], c["r"])))
            for m0 in range(n0, n1, 16384):
                m1 = min(n1, m0 + 16384)
                x = s["X"][l, m0:m1].double()
                u = U[m0 - n0:m1 - n0]
                xb += x.square().sum()
                ua += u.t() @ u
                p = x @ A[l]
                Gk[l] += p.t() @ p
                Sk += E[m0:m1].t() @ p
                if c64 is not None:
                    S += u.t() @ x
                if g64 is not None:
                    g64 += x.t() @ x
            tb = (ua * (Q[l] @ Q[l].t())).sum()
            step = -ETA * torch.sqrt(xb / tb)
            xsq[l] += xb
            tsq[l], alpha[l] = tb, step
            SC[l] += step * Sk
            if c64 is not None:
                c64 += (1.0 if kind in ("chain", "fused") else step) * (Q[l].t() @ S)
        if T is not None:
            T[l] = U @ Q[l]
        Ck[l] = Q[l].t() @ (P[l].t() @ SC[l])
        if gram is not None:
            gram[l] = g64
        if cross is not None:
            cross[l] = c64
    lam = torch.tensor(s["lam"], device=DEV, dtype=F32).double()[:, None] * xsq[None] / d
    B = _solve64(Gk, Ck, lam)
    if kind == "kspace":
        return dict(E=E, ce=ce, G=Gk, SC=SC, xsq=xsq, alpha=alpha, B=B, info=None, C=Ck)
    if kind == "pass":
        return dict(E=E, ce=ce, T=T, gram=gram, cross=cross, xsq=xsq, B=B, info=None)
    return dict(E=E, ce=ce, tsq=tsq, gram=gram, cross=cross, xsq=xsq, alpha=alpha, B=B, info=None)
