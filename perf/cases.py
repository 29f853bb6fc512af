"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one call of a public entry point of ``paper_2609_36835_gb300``:

``layer``   ``compact_layer`` deciding for itself: scoring, top-t, assignment, merge and both fits
``given``   ``compact_layer`` on anchors and groups that the caller brings (anchors_in and assign_in)
``anchors`` ``compact_layer`` on anchors that the caller brings (anchors_in)
``attend``  ``attend``: queries against one layer's fp32 compact cache
``joint``   ``attend_joint``: decode attention, a compact block, an uncompressed block or both
``error``   ``truncated_error``: the held-out error of anchor sets

Sizes are those of the benchmark's workloads and of the tests, and odd ones between them.
"""
import math

import torch

import paper_2609_36835_gb300 as arckv

D = 128  # head width: the only one the library takes


# ------------------------------------------------------------------ the cases

def _compact(kind, H, T, n_pos, t, selector="indexer", chunk_len=0, d_x=4096, H_I=8):
    return {"kind": kind, "H": H, "T": T, "n_pos": n_pos, "t": t, "selector": selector, "chunk_len": chunk_len,
            "d_x": d_x, "H_I": H_I}


def _joint(H, n, t, F, compact="bf16"):
    return {"kind": "joint", "H": H, "n": n, "t": t, "F": F, "compact": compact}


def listed():
    return [
        # one short prompt's single head: the smallest call, all latency and launches
        {"name": "layer_1head_T1024", **_compact("layer", 1, 1024, 64, 102)},
        # one Llama-3.1-8B layer of an ordinary context, the call that is made 32 times per context
        {"name": "layer_T8192_r10", **_compact("layer", 8, 8192, 256, 819)},
        # the same layer by highest attention, for models without a trained indexer
        {"name": "layer_T8192_r05_ha", **_compact("layer", 8, 8192, 256, 409, selector="ha")},
        # a 32K context, its anchors chosen chunk by chunk
        {"name": "layer_T32768_r05_chunked", **_compact("layer", 8, 32768, 512, 1638, chunk_len=8192)},
        # a 128K context: the largest call and the benchmark's default workload (t above n)
        {"name": "layer_T131072_r10", **_compact("layer", 8, 131072, 512, 13107)},
        # a ragged context whose anchors and groups an earlier pass fixed: merge and fits alone
        {"name": "given_T5003_t251", **_compact("given", 4, 5003, 150, 251)},
        # the same with few reference queries and many anchors (t above n)
        {"name": "given_T20011_t2001", **_compact("given", 8, 20011, 128, 2001)},
        # held-out queries against a layer's compact cache: checking a compaction, or a prefill on top of it
        {"name": "attend_n1024_t819", "kind": "attend", "H": 8, "n": 1024, "t": 819},
        # one decode step of 64 sequences on full caches: the largest decode call
        {"name": "joint_full_b64_T8192", **_joint(512, 4, 0, 8192)},
        # the same step on compact caches with the tokens generated since
        {"name": "joint_compact_b64_t1638", **_joint(512, 4, 1638, 200)},
        # one sequence's decode step on the fits' own fp32 output: the smallest decode call
        {"name": "joint_fp32_b1_t819", **_joint(8, 4, 819, 37, compact="fp32")},
        # choosing a selector: the held-out error of a layer's anchor sets
        {"name": "error_T8192_n64", "kind": "error", "H": 8, "n": 64, "T": 8192, "t": 819},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "anchors", "given", "given", "attend", "joint", "joint", "error"])
    if kind in ("layer", "anchors", "given"):
        T = _log_int(rng, 512, 131072 if kind == "layer" else 32768)
        H = rng.choice([1, 2, 4, 8])
        n_pos = _log_int(rng, 32, 512)
        t = max(8, int(T * rng.choice([0.02, 0.05, 0.1]) * rng.uniform(0.8, 1.0)))
        selector = rng.choice(["indexer", "indexer", "ha", "vi"]) if kind == "layer" else "indexer"
        chunk = rng.choice([0, 0, 4096, 8192]) if kind == "layer" and T > 10000 else 0
        return _compact(kind, H, T, n_pos, t, selector, chunk)
    if kind == "attend":
        return {"kind": kind, "H": rng.choice([1, 2, 8]), "n": _log_int(rng, 1, 2048), "t": _log_int(rng, 16, 13107)}
    if kind == "error":
        T = _log_int(rng, 512, 32768)
        return {"kind": kind, "H": rng.choice([1, 8]), "n": rng.randint(16, 256), "T": T, "t": max(8, T // rng.randint(10, 50))}
    H = 8 * _log_int(rng, 1, 64)
    t = rng.choice([0, _log_int(rng, 64, 6553)])
    F = _log_int(rng, 512, 32768) if t == 0 else rng.choice([0, _log_int(rng, 1, 1024)])
    while H * (t + F) > 512 * 8192:  # no more than the largest listed step
        H = max(8, H // 2)
    return _joint(H, rng.choice([1, 4, 4, 8]), t, F, rng.choice(["bf16", "bf16", "fp32"]))


# ----------------------------------------------------------------- the inputs

def _rope(x):
    """Llama's rotation (theta = 500000) at positions 0..T-1 of x [H, T, 128]."""
    half = D // 2
    inv = 500000.0 ** (-torch.arange(half, device=x.device, dtype=torch.float32) / half)
    ang = torch.arange(x.shape[1], device=x.device, dtype=torch.float32)[:, None] * inv[None]
    c, s = ang.cos(), ang.sin()
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], dim=-1)


class _Draw:
    def __init__(self, seed):
        self.dev = torch.device("cuda")
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(int(seed))

    def normal(self, *shape, scale=1.0):
        return torch.randn(*shape, device=self.dev, generator=self.g) * scale

    def bf(self, *shape, scale=1.0):
        return self.normal(*shape, scale=scale).to(torch.bfloat16)

    def keys(self, H, T):
        """Unit-normal keys with four channels eight times as large, rotated, the first key an attention sink."""
        out = torch.empty(H, T, D, dtype=torch.bfloat16, device=self.dev)
        for h in range(H):  # head by head: the rotation's fp32 intermediates stay small
            k = self.normal(1, T, D)
            k[..., torch.randperm(D, device=self.dev, generator=self.g)[:4]] *= 8.0
            k = _rope(k)
            k[:, 0] *= 10.0
            out[h] = k[0].to(torch.bfloat16)
        return out

    def queries(self, K, n):
        """Random keys of each head with noise of half a unit."""
        H, T, _ = K.shape
        j = torch.randint(T, (H, n), device=self.dev, generator=self.g)
        q = torch.gather(K, 1, j[..., None].expand(-1, -1, D)).float()
        return (q + self.normal(H, n, D, scale=0.5)).to(torch.bfloat16)

    def anchors(self, H, T, t):
        return torch.stack([torch.randperm(T, device=self.dev, generator=self.g)[:t].sort().values
                            for _ in range(H)]).to(torch.int32)

    def compact(self, H, t):
        """A compact cache as the fits leave it: keys, biases with the projected-out entries at -20, values."""
        beta = self.normal(H, t)
        beta[torch.rand(H, t, device=self.dev, generator=self.g) < 0.2] = -20.0
        return self.keys(H, t).float() + self.normal(H, t, D, scale=0.05), beta, self.normal(H, t, D)


def _groups(K, Q, anchors):
    """The group of each key: the anchor whose response to the queries is most like its own, itself for an anchor."""
    H, T, _ = K.shape
    out = torch.empty(H, T, dtype=torch.int32, device=K.device)
    for h in range(H):
        logits = Q[h].float() @ K[h].float().T / math.sqrt(D)
        u = torch.exp(logits - logits.max(dim=0).values)
        u = u / u.norm(dim=0)
        a = anchors[h].long()
        out[h] = torch.cat([(u[:, j:j + 4096].T @ u[:, a]).argmax(dim=1) for j in range(0, T, 4096)]).int()
        out[h, a] = torch.arange(a.numel(), dtype=torch.int32, device=K.device)
    return out


def _config(case):
    sel = {"indexer": arckv.SELECTOR_INDEXER, "ha": arckv.SELECTOR_HA, "vi": arckv.SELECTOR_VI}[case["selector"]]
    return arckv.Config(H_kv=case["H"], T=case["T"], n_pos=case["n_pos"], t=case["t"], d_x=case["d_x"],
                        H_I=case["H_I"], chunk_len=case["chunk_len"], selector=sel)


def _workspace(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    r = _Draw(seed)
    kind, H = case["kind"], case["H"]
    s = {"case": case}
    if kind in ("layer", "anchors", "given"):
        cfg = s["cfg"] = _config(case)
        s["K"], s["V"] = r.keys(H, case["T"]), r.bf(H, case["T"], D)
        s["Q"] = r.queries(s["K"], cfg.n)
        s["X"] = s["idx"] = s["anchors_in"] = s["assign_in"] = None
        if kind == "layer" and case["selector"] == "indexer":
            w, d_x = case["H_I"] * D, case["d_x"]
            s["X"] = r.bf(case["n_pos"], d_x)
            s["idx"] = {f: r.bf(H, w, D, scale=D ** -0.5) for f in ("L_q", "L_k", "L_c", "L_v")}
            s["idx"].update({f: r.bf(H, D, D, scale=D ** -0.5) for f in ("U_q", "U_k", "U_v")})
            s["idx"].update(L_x=r.bf(H, case["H_I"], d_x, scale=d_x ** -0.5), b_x=r.bf(H, case["H_I"], scale=0.1))
        if kind != "layer":
            s["anchors_in"] = r.anchors(H, case["T"], case["t"])
        if kind == "given":
            s["assign_in"] = _groups(s["K"], s["Q"], s["anchors_in"])
        s["ws"] = _workspace(arckv.workspace_bytes(cfg))  # a serving program keeps one per stream
    elif kind == "attend":
        s["C_k"], s["beta"], s["C_v"] = r.compact(H, case["t"])
        s["Q"] = r.queries(s["C_k"].to(torch.bfloat16), case["n"])
        s["ws"] = _workspace(arckv.attend_workspace_bytes(H, case["n"], case["t"]))
    elif kind == "joint":
        t, F = case["t"], case["F"]
        s["C_k"] = s["beta"] = s["C_v"] = s["K"] = s["V"] = None
        if t:
            s["C_k"], s["beta"], s["C_v"] = r.compact(H, t)
            if case["compact"] == "bf16":
                s["C_k"], s["C_v"] = s["C_k"].to(torch.bfloat16), s["C_v"].to(torch.bfloat16)
        if F:
            s["K"], s["V"] = r.keys(H, F), r.bf(H, F, D)
        s["Q"] = r.queries((s["C_k"] if t else s["K"]).to(torch.bfloat16), case["n"])
        s["ws"] = _workspace(arckv.attend_joint_workspace_bytes(H, case["n"], t, F))
    else:
        s["K"], s["V"] = r.keys(H, case["T"]), r.bf(H, case["T"], D)
        s["Q"] = r.queries(s["K"], case["n"])
        s["anchors"] = r.anchors(H, case["T"], case["t"])
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind in ("layer", "anchors", "given"):
        out = arckv.compact_layer(s["cfg"], s["K"], s["V"], s["Q"], s["X"], s["idx"], ws=s["ws"],
                                  anchors_in=s["anchors_in"], assign_in=s["assign_in"])
        return {k: out[k] for k in ("C_k", "beta", "C_v", "anchors")}
    if kind == "attend":
        return arckv.attend(s["Q"], s["C_k"], s["beta"], s["C_v"], ws=s["ws"])
    if kind == "joint":
        return arckv.attend_joint(s["Q"], s["C_k"], s["beta"], s["C_v"], s["K"], s["V"], ws=s["ws"])
    return arckv.truncated_error(s["Q"], s["K"], s["V"], s["anchors"])


# ------------------------------------------------------------------- the work

def work(case):
    kind, H = case["kind"], case["H"]
    if kind in ("layer", "anchors", "given"):
        T, t, n_pos = case["T"], case["t"], case["n_pos"]
        n, m, w = 4 * n_pos, min(4 * n_pos, t), case["H_I"] * D
        nbytes = 2 * T * D * 2 + n * D * 2 + t * (2 * D + 1) * 4 + t * 4
        flops = 4 * n * T * D                                   # reference attention and its output
        flops += 2 * T * D                                      # merge
        flops += 2 * n * t * D + 2 * n * t * m + 2 * n * t * D  # compact logits, both Grams, the right-hand sides
        flops += 2 * m ** 3 // 3 + 2 * m * m * (D + 1)          # both factorisations, their substitutions
        if t > n:
            flops += 2 * n * t * D                              # back from the dual solution
        if kind == "given":
            nbytes += T * 4
        else:
            flops += 2 * n * (T - t) * t                        # assignment
        if kind == "layer" and case["selector"] == "indexer":
            nbytes += (4 * w * D + 3 * D * D + case["H_I"] * (case["d_x"] + 1)) * 2 + n_pos * case["d_x"] * 2 // H
            flops += 2 * T * 2 * D * w + 4 * n * T * D + 2 * n * 2 * D * w + 2 * n_pos * case["d_x"] * case["H_I"]
            flops += 2 * n * T * w                              # index logits
        if kind == "layer" and case["selector"] == "vi":
            flops += 4 * n * T * D                              # the output without the largest key, its distances
        return {"bytes": H * nbytes, "flops": H * flops}
    n = case["n"]
    if kind == "attend":
        t = case["t"]
        return {"bytes": H * (n * D * 6 + t * (2 * D + 1) * 4), "flops": H * 4 * n * t * D}
    if kind == "joint":
        t, F = case["t"], case["F"]
        row = 2 * D * (2 if case["compact"] == "bf16" else 4) + 4
        return {"bytes": H * (n * D * 6 + t * row + F * 4 * D), "flops": H * 4 * n * (t + F) * D}
    T = case["T"]
    return {"bytes": H * (n * D * 2 + T * 4 * D + case["t"] * 4 + 4), "flops": H * 4 * n * T * D}


# ------------------------------------------------------------ 64-bit reference

def _softmax_v(Q, K, bias, V):
    x = Q @ K.T / math.sqrt(D)
    return torch.softmax(x if bias is None else x + bias, dim=-1) @ V


def _exact_given(s):
    """Merge and fits of the given anchors and groups (ridge_w = 1e-4, ridge_v = 1e-3, lambda_m = 0.25)."""
    cfg, out = s["cfg"], {"C_k": [], "beta": [], "C_v": []}
    for h in range(cfg.H_kv):
        K, V, Q = s["K"][h].double(), s["V"][h].double(), s["Q"][h].double()
        a, g, t, n = s["anchors_in"][h].long(), s["assign_in"][h].long(), cfg.t, cfg.n
        x = Q @ K.T / math.sqrt(D)
        z = x.max(dim=1).values
        p = torch.exp(x - z[:, None])
        mass = p.sum(dim=1)
        Y = (p / mass[:, None]) @ V
        del p
        logphi = torch.logsumexp(x, dim=0)
        top = torch.full((t,), -math.inf, dtype=torch.float64, device=K.device).scatter_reduce(0, g, logphi, "amax")
        wt = torch.exp(logphi - top[g])
        den = torch.zeros(t, dtype=torch.float64, device=K.device).index_add(0, g, wt)
        mu = torch.zeros(t, D, dtype=torch.float64, device=K.device).index_add(0, g, wt[:, None] * K) / den[:, None]
        C_k = 0.75 * K[a] + 0.25 * mu
        del x
        xc = Q @ C_k.T / math.sqrt(D)

        def ridge(A, rhs, lam):
            lam = lam * A.square().sum() / t
            if t <= n:
                return torch.linalg.solve(A.T @ A + lam * torch.eye(t, dtype=A.dtype, device=A.device), A.T @ rhs)
            return A.T @ torch.linalg.solve(A @ A.T + lam * torch.eye(n, dtype=A.dtype, device=A.device), rhs)

        w = ridge(torch.exp(xc - z[:, None]), mass[:, None], cfg.ridge_w)[:, 0]
        beta = torch.log(w.clamp_min(0.0).clamp_min(cfg.eps_w)).clamp(cfg.b_min, cfg.b_max)
        C_v = ridge(torch.softmax(xc + beta, dim=1), Y, cfg.ridge_v)
        for k, v in (("C_k", C_k), ("beta", beta), ("C_v", C_v)):
            out[k].append(v)
    return {k: torch.stack(v) for k, v in out.items()}


def exact(case, seed):
    """64-bit values. A call that decides for itself has none: near-ties among its keys may go either way."""
    kind = case["kind"]
    if kind in ("layer", "anchors"):
        return None
    s = prepare(case, seed)
    if kind == "given":
        return {**_exact_given(s), "anchors": None}
    H, out = case["H"], []
    for h in range(H):
        Q = s["Q"][h].double()
        if kind == "attend":
            out.append(_softmax_v(Q, s["C_k"][h].double(), s["beta"][h].double(), s["C_v"][h].double()))
        elif kind == "joint":
            zero = torch.zeros(case["F"], dtype=torch.float64, device=Q.device)
            parts = [(s["C_k"][h], s["C_v"][h], s["beta"][h])] if case["t"] else []
            parts += [(s["K"][h], s["V"][h], zero)] if case["F"] else []
            K, V, b = (torch.cat([p[i].double() for p in parts]) for i in range(3))
            out.append(_softmax_v(Q, K, b, V))
        else:
            V = s["V"][h].double()
            p = torch.softmax(Q @ s["K"][h].double().T / math.sqrt(D), dim=-1)
            a = s["anchors"][h].long()
            O = p @ V
            out.append(((O - p[:, a] @ V[a]).norm(dim=1) / (O.norm(dim=1) + 1e-6)).mean())
    return torch.stack(out)
