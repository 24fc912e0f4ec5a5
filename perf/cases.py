"""The work a user of this library has it do, as measurable cases.

Every case is one call of a public entry point on sizes of the library's own
benchmark, tests and documented limits: traces of seeded circuit pairs
(``Ensemble.trace_batch``, ``trace_brick_static``), the Monte Carlo driver
(``Ensemble.frame_potential``), the bootstrap of stored traces, the exact
Weingarten sweep and the control variate's dense layer.

``exact`` restates the same quantities in 64-bit torch: the random numbers from
the published Philox4x64-10 keying, Haar gates by Gram-Schmidt, and the trace
networks contracted qubit by qubit without any of the library's code.

Outputs of paths whose boundaries are FP32 are handed on as FP32 values (the
library writes them into float64 arrays): FP32 rounding is what they carry.
"""
import math

import numpy as np
import torch

import paper_2205_09900_gb300 as fp

KINDS = {"brickwork": fp.PARALLEL, "local": fp.LOCAL, "hea": fp.HEA, "hea_paper": fp.HEA_PAULI}
PRECS = {"fp64": fp.PREC_FP64, "fp32": fp.PREC_FP32, "fp32_raw": fp.PREC_FP32_RAW}


def listed():
    return [
        # the smallest call: a plugin tracing a handful of shallow pairs without allocating; launches count
        dict(name="static_n8_l3", call="static", n=8, l=3, count=64, prec="fp32_raw"),
        # the FP64 configuration of the benchmark: n = 8, 4 layers, 10^4 pairs, traces with kappa
        dict(name="brick_n8_l4_fp64", call="traces", kind="brickwork", n=8, dmin=4, dmax=4, count=10_000,
             prec="fp64", q=2),
        # a shallow depth of a depth sweep on an odd chain: many pairs, small boundaries
        dict(name="brick_n51_l5", call="traces", kind="brickwork", n=51, dmin=5, dmax=5, count=20_001,
             prec="fp32", q=2),
        # the headline workload: n = 50, depths 2..10 mixed, Monte Carlo moments k = 1..4
        dict(name="brick_n50_l2_10", call="potential", kind="brickwork", n=50, dmin=2, dmax=10, count=16_000,
             prec="fp32", k_max=4, q=2),
        # the paper's largest case, n = 50, l = 11: boundaries of 2^20 amplitudes
        dict(name="brick_n50_l11", call="traces", kind="brickwork", n=50, dmin=11, dmax=11, count=96,
             prec="fp32", q=2),
        # hardware-efficient ansatz (RY RZ + CZ ladder), n = 50, L = 1..8 mixed
        dict(name="hea_n50_L1_8", call="potential", kind="hea", n=50, dmin=1, dmax=8, count=100_000,
             prec="fp32", k_max=4, q=2),
        # the paper's hardware-efficient ansatz (Pauli rotations, CNOT walls), n = 50, L = 1..8 mixed
        dict(name="hea_paper_n50_L1_8", call="potential", kind="hea_paper", n=50, dmin=1, dmax=8, count=16_000,
             prec="fp32", k_max=4, q=2),
        # local random circuits, n = 20, T = 20, 40, .., 100 gates: a topology per pair, uneven boundaries
        dict(name="local_n20_T20_100", call="traces", kind="local", n=20, tmin=20, tmax=100, tstep=20, count=4_000,
             prec="fp32", q=2),
        # qutrit brickwork, n = 50, l = 2..5 mixed
        dict(name="qutrit_n50_l2_5", call="potential", kind="brickwork", n=50, dmin=2, dmax=5, count=2_000,
             prec="fp32", k_max=2, q=3),
        # the variance-free F^(3) beside a Monte Carlo run: n = 50, l = 6, a state of 6^10 entries
        dict(name="exact_f3_n50_l6", call="exact_fk", n=50, l=6, k=3, q=2),
        # 300 bootstrap resamples of 200,000 stored traces in 9 depth groups
        dict(name="bootstrap_200k", call="bootstrap", groups=9, count=200_000, k_max=4, resamples=300),
        # the control variate's input layer on one chunk of surrogate pairs (HEA n = 50, L = 4: 2400 features)
        dict(name="mlp_layer_65536x256x2400", call="gemm", m=65_536, n=256, k=2_400, mode=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _flops_pair(c, d):
    """Real flops of one pair of depth d (8 per complex multiply-add)."""
    n, q = c["n"], c.get("q", 2)
    if c["kind"] == "brickwork":
        return 8.0 * q * q * (n - 1) * max(d - 1, 0) * float(q) ** (2 * (d - 1)) if d > 1 else 8.0 * 16 * (n - 1)
    if c["kind"] == "hea":      # per qubit and amplitude: 2L-2 phases (complex products) and as many Hadamard adds
        return 8.0 * n * max(2 * d - 2, 1) * 2.0 ** (2 * d - 2)
    return 8.0 * 2 * n * max(2 * d - 1, 1) * 2.0 ** (2 * d - 1)


def draw(rng):
    call = rng.choice(["traces", "traces", "traces", "potential", "potential", "static", "exact_fk", "bootstrap", "gemm"])
    if call == "static":
        return dict(call=call, n=rng.randint(2, 20), l=rng.randint(2, 5), count=_log(rng, 1, 300),
                    prec=rng.choice(["fp32_raw", "fp64"]))
    if call == "exact_fk":
        k = rng.choice([2, 3])
        return dict(call=call, n=rng.randint(3, 50), l=rng.randint(2, 10 if k == 2 else 5), k=k, q=rng.choice([2, 3]))
    if call == "bootstrap":
        return dict(call=call, groups=rng.randint(1, 9), count=_log(rng, 1_000, 200_000), k_max=rng.randint(1, 6),
                    resamples=_log(rng, 30, 300))
    if call == "gemm":
        return dict(call=call, m=_log(rng, 100, 65_536), n=16 * rng.randint(1, 24), k=8 * rng.randint(2, 300),
                    mode=rng.randint(0, 2))
    kind = rng.choice(["brickwork", "brickwork", "hea", "hea_paper", "local"])
    prec = rng.choice(["fp32", "fp32", "fp32_raw", "fp64"])
    c = dict(call=call, kind=kind, n=rng.randint(4, 51), q=2, prec=prec)
    if kind == "local":
        c["n"] = rng.randint(4, 20)
        c["tmin"] = rng.randint(5, 20)
        c["tstep"] = rng.randint(1, 20)
        c["tmax"] = c["tmin"] + c["tstep"] * rng.randint(0, 3)
        c["count"] = _log(rng, 20, 2_000)
    else:
        if kind == "brickwork" and rng.random() < 0.2:
            c["q"] = rng.choice([3, 4])
        top = 4 if c["q"] > 2 else 9 if kind == "brickwork" else 8
        lo = rng.randint(2, top)
        hi = rng.randint(lo, top)
        c["dmin"], c["dmax"] = lo, hi
        # as many pairs as a fixed amount of arithmetic allows, spread over the logarithm below that
        per = sum(_flops_pair(c, d) for d in range(lo, hi + 1)) / (hi - lo + 1) + 2e5 * c["q"] ** 2
        most = max(2, min(20_000, (1.5e11 if prec == "fp64" else 3e12 if c["q"] == 2 else 2e11) / per))
        c["count"] = _log(rng, max(1, most / 50), most)
    if call == "potential":
        c["k_max"] = rng.randint(1, 4)
    return c


# ---------------------------------------------------------------------------
# inputs, the call, its work
# ---------------------------------------------------------------------------
def _bootstrap_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    group = torch.randint(0, c["groups"], (c["count"],), generator=g, device="cuda", dtype=torch.int32)
    # traces of deep circuits are complex Gaussian with E|Tr|^2 = 1; shallow groups have heavier tails
    z = torch.randn(c["count"], 2, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(0.5)
    heavy = torch.randn(c["count"], 1, generator=g, device="cuda", dtype=torch.float64) / (group[:, None] + 2.0)
    return (z * torch.exp(heavy)).reshape(-1).contiguous(), group


def _gemm_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, n, k = c["m"], c["n"], c["k"]
    phase = torch.rand(m, k, generator=g, device="cuda") * (2 * math.pi)   # features are cosines and sines of angles
    a = torch.cos(phase).to(torch.bfloat16)
    del phase
    b = (torch.randn(n, k, generator=g, device="cuda") * math.sqrt(2.0 / k)).to(torch.bfloat16)
    bias = torch.randn(n, generator=g, device="cuda") * 0.1
    z = torch.randn(m, n, generator=g, device="cuda") if c["mode"] == 2 else None
    return a, b, bias, z


def prepare(case, seed):
    c = dict(case)
    s = {"case": c, "seed": seed}
    call = c["call"]
    if call in ("traces", "potential"):
        flags = fp.FLAG_SKIP_INFEASIBLE if c["kind"] == "local" else 0
        s["ens"] = fp.Ensemble(KINDS[c["kind"]], c["n"], c.get("dmin", 1), c.get("dmax", 1), c.get("tmin", 0),
                               c.get("tmax", 0), c.get("tstep", 1), seed=seed, flags=flags, q=c["q"])
        if call == "traces":
            s["tr"] = torch.zeros(2 * c["count"], dtype=torch.float64, device="cuda")
            s["group"] = torch.zeros(c["count"], dtype=torch.int32, device="cuda")
            s["kappa"] = torch.zeros(c["count"], dtype=torch.float64, device="cuda") if c["prec"] == "fp64" else None
    elif call == "static":
        s["tr"] = torch.zeros(2 * c["count"], dtype=torch.float64, device="cuda")
    elif call == "bootstrap":
        s["ens"] = fp.Ensemble(fp.PARALLEL, 50, 2, 1 + c["groups"], seed=1)
        s["tr"], s["group"] = _bootstrap_inputs(c, seed)
        s["out"] = torch.zeros(c["groups"] * c["k_max"] * c["resamples"], dtype=torch.float64, device="cuda")
    elif call == "gemm":
        s["a"], s["b"], s["bias"], s["z"] = _gemm_inputs(c, seed)
        s["c"] = torch.zeros(c["m"], c["n"], dtype=torch.bfloat16, device="cuda")
    elif call == "exact_fk":
        # the sweep has no random input: another chain length of the same cost stands for another input
        s["n"] = _chain(c, seed)
    return s


def _chain(c, seed):
    return c["n"] + seed % 7


def _as(x, prec):
    return x if prec == "fp64" else x.to(torch.float32)


def run(state):
    c, call = state["case"], state["case"]["call"]
    if call == "traces":
        tr, kappa, group = state["ens"].trace_batch(0, c["count"], PRECS[c["prec"]], state["tr"], state["kappa"],
                                                    state["group"])
        out = {"tr": _as(tr, c["prec"]), "group": group}
        if kappa is not None:
            out["kappa"] = kappa
        return out
    if call == "potential":
        F, se, st = state["ens"].frame_potential(0, c["count"], c["k_max"], 0.0, PRECS[c["prec"]])
        t = np.float64 if c["prec"] == "fp64" else np.float32
        return {"F": F.astype(t), "stderr": se.astype(t), "pairs": int(st.pairs)}
    if call == "static":
        tr, _ = fp.trace_brick_static(c["n"], c["l"], state["seed"], 0, c["count"], PRECS[c["prec"]], state["tr"])
        return {"tr": _as(tr, c["prec"])}
    if call == "bootstrap":
        return {"F": state["ens"].bootstrap(state["tr"], state["group"], c["count"], c["k_max"], c["resamples"],
                                            seed=11, out=state["out"])}
    if call == "gemm":
        fp.gemm_bf16(state["a"], state["b"], state["bias"], c["mode"], Z=state["z"], C_bf16=state["c"])
        return {"C": state["c"]}
    return {"F": fp.exact_brickwork_fk(state["n"], c["l"], c["k"], q=c["q"])}


def work(case):
    c = case
    call = c["call"]
    if call in ("traces", "potential"):
        # the inputs are a seed: what has to move is the results
        out = 24.0 * c["count"] if call == "traces" else 16.0 * c["k_max"] * (c.get("dmax", 1) - c.get("dmin", 1) + 1)
        if c["kind"] == "local":
            # boundaries differ by pair: a 2^t-like growth with the light cone, counted at its typical width
            ts = range(c["tmin"], c["tmax"] + 1, c["tstep"])
            fl = sum(8.0 * 4 * 2 * t * 2.0 ** min(20, 0.14 * t * 20 / c["n"]) for t in ts) / len(ts)
        else:
            ds = range(c["dmin"], c["dmax"] + 1)
            fl = sum(_flops_pair(c, d) for d in ds) / len(ds)
        return {"bytes": out, "flops": fl * c["count"]}
    if call == "static":
        return {"bytes": 16.0 * c["count"], "flops": _flops_pair(dict(c, kind="brickwork"), c["l"]) * c["count"]}
    if call == "bootstrap":
        return {"bytes": 20.0 * c["count"] + 8.0 * c["groups"] * c["k_max"] * c["resamples"],
                "flops": 2.0 * c["k_max"] * c["count"] * c["resamples"]}
    if call == "gemm":
        m, n, k = c["m"], c["n"], c["k"]
        return {"bytes": 2.0 * (m * k + n * k + m * n) + (4.0 * m * n if c["mode"] == 2 else 0) + 4.0 * n,
                "flops": 2.0 * m * n * k}
    s = 2 if c["k"] == 2 else 6
    slots = 2 * (c["l"] - 1)
    return {"bytes": 8.0, "flops": 2.0 * (c["n"] - 2) * slots * s * float(s) ** slots + 8.0}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _s64(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _mulhi(a, x):
    """High 64 bits of the unsigned product of the constant a and the tensor x (bit patterns in int64)."""
    a0, a1 = a & _M32, a >> 32
    x0, x1 = x & _M32, (x >> 32) & _M32
    mid = x0 * a1 + (((x0 * a0) >> 32) & _M32)
    mid2 = x1 * a0 + (mid & _M32)
    return x1 * a1 + ((mid >> 32) & _M32) + ((mid2 >> 32) & _M32)


def _philox(seed, c0, c1, pair, stream):
    """Philox4x64-10, key {seed, 0}, counter {c0, c1, pair, stream} (int64 tensors that broadcast)."""
    c0, c1, pair, stream = torch.broadcast_tensors(c0, c1, pair, stream)
    c = [c0, c1, pair, stream]
    m0, m1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    k0, k1 = seed, 0
    for _ in range(10):
        hi0, lo0 = _mulhi(m0, c[0]), c[0] * _s64(m0)
        hi1, lo1 = _mulhi(m1, c[2]), c[2] * _s64(m1)
        c = [hi1 ^ c[1] ^ _s64(k0), lo1, hi0 ^ c[3] ^ _s64(k1), lo0]
        k0 = (k0 + 0x9E3779B97F4A7C15) & ((1 << 64) - 1)
        k1 = (k1 + 0xBB67AE8584CAA73B) & ((1 << 64) - 1)
    return c


def _unit(x):
    """The top 53 bits as an integer."""
    return ((x >> 11) & ((1 << 53) - 1)).to(torch.float64)


def _i(x):
    return torch.as_tensor(x, dtype=torch.int64, device="cuda")


def _pick(x, choices):
    return (((x >> 32) & _M32) * choices) >> 32


def _depths(seed, count, choices):
    x = _philox(seed, _i(0), _i(0), torch.arange(count, device="cuda"), _i(4))
    return _pick(x[0], choices)


def _haar(seed, pairs, which, gates, d):
    """Haar U(d) gates [len(pairs), len(gates), d, d]: Q of the Gaussian matrix with R's diagonal positive."""
    k = torch.arange((d * d + 1) // 2, device="cuda")
    x = _philox(seed, k[None, None, :], gates[None, :, None], pairs[:, None, None], _i(which))
    z = []
    for a, b in ((x[0], x[1]), (x[2], x[3])):
        rad = torch.sqrt(-torch.log((_unit(a) + 1.0) * 2.0 ** -53))
        ang = _unit(b) * (2.0 ** -53 * 2 * math.pi)
        z.append(torch.polar(rad, ang))
    z = torch.stack(z, -1).reshape(len(pairs), len(gates), -1)[..., :d * d].reshape(-1, d, d)
    q = torch.zeros_like(z)
    for j in range(d):
        v = z[:, :, j].clone()
        for _ in range(2):      # Gram-Schmidt twice is orthogonal to rounding
            if j:
                h = torch.einsum("bri,br->bi", q[:, :, :j].conj(), v)
                v = v - torch.einsum("bri,bi->br", q[:, :, :j], h)
        q[:, :, j] = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
    return q.reshape(len(pairs), len(gates), d, d)


def _apply(M, x, post):
    """x [B, pre, D, post] -> sum_e M[b, o, e] x[b, :, e, :] for small D."""
    B, D = M.shape[0], M.shape[1]
    x = x.reshape(B, -1, D, post)
    if D > 4:
        return torch.einsum("boe,bpeq->bpoq", M, x)
    y = torch.empty_like(x)
    for o in range(D):
        acc = M[:, o, 0, None, None] * x[:, :, 0]
        for e in range(1, D):
            acc = torch.addcmul(acc, M[:, o, e, None, None], x[:, :, e])
        y[:, :, o] = acc
    return y


def _brick_traces(seed, n, l, pairs, q):
    """Tr(U^dagger V) of brickwork pairs of depth l: bond by bond along the chain, the state over the wire
    segments of one qudit (digit t: its value before time position t of the cyclic circuit)."""
    D, B = q * q, len(pairs)
    if l == 1:
        g = torch.arange(n // 2, device="cuda")
        U, V = _haar(seed, pairs, 0, g, D), _haar(seed, pairs, 1, g, D)
        return (U.conj() * V).sum((-1, -2)).prod(1) * (q if n % 2 else 1)
    c0, c1 = n // 2, (n - 1) // 2
    n_raw = ((l + 1) // 2) * c0 + (l // 2) * c1
    g = torch.arange(n_raw, device="cuda")
    U, V = _haar(seed, pairs, 0, g, D), _haar(seed, pairs, 1, g, D)
    index = lambda t, b: ((t + 1) // 2) * c0 + (t // 2) * c1 + (b - t % 2) // 2   # noqa: E731  layer t (0-based)
    P = 2 * (l - 1)
    digits = torch.arange(q ** P, device="cuda")
    digit = lambda t: (digits // q ** (P - 1 - t)) % q   # noqa: E731  digit 0 most significant

    def idle(par):   # wire ends at positions without a gate
        ok = torch.ones(q ** P, dtype=torch.bool, device="cuda")
        for t in range(par, P, 2):
            ok &= digit(t) == digit((t + 1) % P)
        return ok.to(torch.complex128)

    x = idle(0).expand(B, -1).contiguous()
    for b in range(n - 1):
        for t in range((b + 1) % 2, P, 2):
            if t < l - 2:
                G = V[:, index(t + 1, b)]
            elif t == l - 2:
                G = U[:, index(l - 1, b)].mH @ V[:, index(l - 1, b)]
            elif t == P - 1:
                G = V[:, index(0, b)] @ U[:, index(0, b)].mH
            else:
                G = U[:, index(P - 1 - t, b)].mH
            # G[(out_b, out_b1), (in_b, in_b1)] -> M[(in_b1, out_b1), (in_b, out_b)]
            M = G.reshape(B, q, q, q, q).permute(0, 4, 2, 3, 1).reshape(B, D, D).contiguous()
            if t < P - 1:
                x = _apply(M, x, q ** (P - 2 - t)).reshape(B, -1)
            else:   # the pair (last, first) of the ring
                y = x.reshape(B, q, -1, q).permute(0, 3, 1, 2).reshape(B, D, -1)
                y = _apply(M, y, y.shape[-1]).reshape(B, q, q, -1)
                x = y.permute(0, 2, 3, 1).reshape(B, -1)
    return (x * idle(n % 2)).sum(1)


def _ry(th):
    c, s = torch.cos(th / 2), torch.sin(th / 2)
    return torch.stack([torch.stack([c, -s], -1), torch.stack([s, c], -1)], -2).to(torch.complex128)


def _angles(seed, n, L, pairs, which):
    t = torch.arange(L, device="cuda")[None, :, None]
    return _philox(seed, t, torch.arange(n, device="cuda")[None, None, :], pairs[:, None, None], _i(which))


def _hea_slots(R, L):
    """The cyclic rotations of U^dagger V with the last and the first layer's merged."""
    U, V = R
    s = [V[:, 0] @ U[:, 0].mH] + [V[:, t] for t in range(1, L - 1)]
    s += [U[:, L - 1].mH @ V[:, L - 1]] + [U[:, t].mH for t in range(L - 2, 0, -1)]
    return s


def _hea_traces(seed, n, L, pairs):
    B, R = len(pairs), []
    for w in range(2):
        x = _angles(seed, n, L, pairs, w)
        half = _unit(x[1]) * (2.0 ** -53 * math.pi)
        rz = torch.diag_embed(torch.stack([torch.polar(torch.ones_like(half), -half),
                                           torch.polar(torch.ones_like(half), half)], -1))
        R.append(_ry(_unit(x[0]) * (2.0 ** -53 * 2 * math.pi)) @ rz)
    if L == 1:
        return torch.einsum("bqij,bqij->bq", R[0][:, 0].conj(), R[1][:, 0]).prod(1)
    N = 2 * L - 2
    slots = _hea_slots(R, L)      # slot s acts between segment s-1 and segment s; a CZ ladder follows each
    x = torch.ones(B, 2 ** N, dtype=torch.complex128, device="cuda")
    for q in range(n):
        for s in range(N):        # digit s (0 most significant): the wire after slot s
            M = slots[s][:, q]
            if s:
                x = x.reshape(B, 2 ** (s - 1), 2, 2, -1) * M.mT[:, None, :, :, None]    # [in, out]
            else:
                x = x.reshape(B, 2, -1, 2) * M[:, :, None, :]                            # [out, .., in]
        if q == n - 1:
            return x.reshape(B, -1).sum(1)
        for s in range(N):
            y = x.reshape(B, 2 ** s, 2, -1)
            x = torch.stack([y[:, :, 0] + y[:, :, 1], y[:, :, 0] - y[:, :, 1]], 2)
        x = x.reshape(B, -1)


def _hea_paper_traces(seed, n, L, pairs):
    """The paper's ansatz: the fixed wall cancels; every CNOT is a sum over its control's value."""
    B, R = len(pairs), []
    for w in range(2):
        x = _angles(seed, n, L, pairs, w)
        half = _unit(x[0]) * (2.0 ** -53 * math.pi)
        c, s, zero = torch.cos(half), torch.sin(half), torch.zeros_like(half)
        axis = _pick(x[1], 3)
        z = torch.complex
        X = [z(c, zero), z(zero, -s), z(zero, -s), z(c, zero)]
        Y = [z(c, zero), z(-s, zero), z(s, zero), z(c, zero)]
        Z = [z(c, -s), z(zero, zero), z(zero, zero), z(c, s)]
        m = [torch.where(axis == 0, a, torch.where(axis == 1, b, e)) for a, b, e in zip(X, Y, Z)]
        R.append(torch.stack(m, -1).reshape(*c.shape, 2, 2))
    U, V = R
    ops = []                       # in time order: a rotation or a wall of CNOTs (parity of its bonds)
    for t in range(L - 1):
        ops += [V[:, t], 0, 1]
    ops.append(U[:, L - 1].mH @ V[:, L - 1])
    for t in range(L - 2, -1, -1):
        ops += [1, 0, U[:, t].mH]
    x = torch.eye(2, dtype=torch.complex128, device="cuda").expand(B, 1, 2, 2).contiguous()
    for q in range(n):
        # x [B, left CNOT values still open (time order), right ones (time order), wire at start, wire now]
        x = x.reshape(B, -1, 2, 2)
        for op in ops:
            if not isinstance(op, int):
                M = op[:, q]
                x = torch.stack([M[:, a, 0, None, None] * x[..., 0] + M[:, a, 1, None, None] * x[..., 1]
                                 for a in range(2)], -1)
            elif op == q % 2:
                if q < n - 1:      # control: its value becomes a new index
                    y = torch.zeros(*x.shape[:2], 2, 2, 2, dtype=x.dtype, device="cuda")
                    y[:, :, 0, :, 0], y[:, :, 1, :, 1] = x[..., 0], x[..., 1]
                    x = y.reshape(B, -1, 2, 2)
            elif q > 0:            # target: flipped where the left control is 1, which is summed
                y = x.reshape(B, 2, -1, 2, 2)
                x = y[:, 0] + y[:, 1].flip(-1)
        x = x[..., 0, 0] + x[..., 1, 1]
        if q < n - 1:
            x = (x.reshape(B, -1, 1, 1) * torch.eye(2, dtype=x.dtype, device="cuda")).contiguous()
    return x.reshape(B)


def _local_traces(seed, n, T, pairs):
    """Dense matrices (small n only)."""
    g = torch.arange(T, device="cuda")
    mats = []
    for w in range(2):
        G = _haar(seed, pairs, w, g, 4)
        x = _philox(seed, _i(0), g[None, :], pairs[:, None], _i(2 + w))
        bond = _pick(x[0], n - 1).cpu().tolist()
        A = torch.eye(2 ** n, dtype=torch.complex128, device="cuda").expand(len(pairs), -1, -1).clone()
        for p in range(len(pairs)):
            for t in range(T):
                A[p] = torch.matmul(G[p, t], A[p].reshape(2 ** bond[p][t], 4, -1)).reshape(2 ** n, 2 ** n)
        mats.append(A.reshape(len(pairs), -1))
    return (mats[0].conj() * mats[1]).sum(1)


def _seconds_exact(c, d):
    """About the time of one pair's exact trace (measured at the deepest depths)."""
    q, n = c.get("q", 2), c["n"]
    if c["kind"] == "brickwork":
        return 2.2e-10 * n * max(d - 1, 1) * float(q) ** (2 * (d - 1)) * (q * q / 4) + 2e-7 * n * d * (q / 2) ** 6
    return 1.2e-9 * n * 2 * d * 2.0 ** (2 * d - 2) * (0.045 if c["kind"] == "hea" else 0.25) + 1e-7 * n * d


def _traces(c, seed):
    """complex128 traces of all pairs and the group of each; None where they would take too long."""
    count = c["count"]
    lo, step = (c["tmin"], c["tstep"]) if c["kind"] == "local" else (c["dmin"], 1)
    ng = ((c["tmax"] if c["kind"] == "local" else c["dmax"]) - lo) // step + 1
    if c["kind"] == "local":
        if c["n"] > 9 or count * (c["tmin"] + c["tmax"]) > 60_000:
            return None
    elif sum(_seconds_exact(c, lo + g) for g in range(ng)) / ng * count > 18:
        return None
    group = _depths(seed, count, ng)
    tr = torch.zeros(count, dtype=torch.complex128, device="cuda")
    for g in range(ng):
        d = lo + g * step
        members = torch.nonzero(group == g).flatten()
        if c["kind"] == "local":
            f, chunk = (lambda p: _local_traces(seed, c["n"], d, p)), 64
        else:
            if c["kind"] == "brickwork":
                f, size = (lambda p: _brick_traces(seed, c["n"], d, p, c["q"])), c["q"] ** (2 * (d - 1))
            elif c["kind"] == "hea":
                f, size = (lambda p: _hea_traces(seed, c["n"], d, p)), 2 ** (2 * d)
            else:
                f, size = (lambda p: _hea_paper_traces(seed, c["n"], d, p)), 2 ** (2 * d + 1)
            chunk = int(max(1, 2 ** 33 // (size * 16 * 6 + c["n"] * d * c.get("q", 2) ** 4 * 160)))
        for p in members.split(chunk):
            tr[p] = f(p)
    return tr, group.to(torch.int32)


def _moments(tr, group, ng, k_max):
    F = torch.full((ng, k_max), float("nan"), dtype=torch.float64, device="cuda")
    se = F.clone()
    a2 = tr.abs() ** 2
    for g in range(ng):
        v = a2[group == g]
        for k in range(1, k_max + 1):
            if len(v):
                F[g, k - 1] = (v ** k).mean()
            if len(v) > 1:
                se[g, k - 1] = (v ** k).std() / math.sqrt(len(v))
    return F, se


def _exact_fk(n, l, k, q):
    """The Haar average bond by bond: every gate a sum over pairings with Weingarten weights."""
    import itertools
    S = list(itertools.permutations(range(k)))
    s = len(S)

    def cycles(a, b):
        inv = [a.index(i) for i in range(k)]
        seen, c = set(), 0
        for i in range(k):
            c += i not in seen
            while i not in seen:
                seen.add(i)
                i = inv[b[i]]
        return c

    gram = lambda d: torch.tensor([[float(d) ** cycles(a, b) for b in S] for a in S], dtype=torch.float64)   # noqa: E731
    wg = torch.linalg.inv(gram(q * q)).cuda()      # the Weingarten matrix inverts the Gram matrix of pairings
    link = gram(q).cuda()
    P = 2 * (l - 1)
    if s ** P > 7e7:
        return None

    def pair_factor(v, t, u, M):     # v[.. digit t = a .., digit u = b ..] *= M[a, b], digit 0 most significant
        shape = [1] * P
        shape[t] = shape[u] = s
        return v * (M if t < u else M.T).reshape(shape)

    v = torch.ones([s] * P, dtype=torch.float64, device="cuda")
    scale = 0.0
    for t in range(1, P, 2):
        v = pair_factor(v, t, (t - 1) % P, wg)
        v = pair_factor(v, t, (t + 1) % P, link)
    for b in range(1, n - 1):
        for t in range(P):           # all links of qubit b
            v = (link.T @ v.reshape(s ** t, s, -1)).reshape([s] * P)
        for t in range((b + 1) % 2, P, 2):
            v = pair_factor(v, t, (t - 1) % P, wg)
        m = float(v.abs().max())
        scale += math.log2(m)
        v = v / m
    for t in range((n - 1) % 2, P, 2):
        v = pair_factor(v, t, (t + 1) % P, link)
    return float(v.sum()) * 2.0 ** scale


def exact(case, seed):
    c = dict(case)
    call = c["call"]
    if call == "static":
        c.update(kind="brickwork", dmin=c["l"], dmax=c["l"], q=2)
    if call in ("traces", "static", "potential"):
        got = _traces(c, seed)
        if got is None:
            return None
        tr, group = got
        if call == "potential":
            ng = (c["tmax"] - c["tmin"]) // c["tstep"] + 1 if c["kind"] == "local" else c["dmax"] - c["dmin"] + 1
            F, se = _moments(tr, group, ng, c["k_max"])
            return {"F": F, "stderr": se, "pairs": c["count"]}
        out = {"tr": torch.view_as_real(tr).reshape(-1)}
        if call == "traces":
            out["group"] = group
            if c["prec"] == "fp64":
                out["kappa"] = None
        return out
    if call == "bootstrap":
        tr, group = _bootstrap_inputs(c, seed)
        a2 = tr[0::2] ** 2 + tr[1::2] ** 2
        F = torch.zeros(c["groups"], c["k_max"], c["resamples"], dtype=torch.float64, device="cuda")
        for g in range(c["groups"]):
            v = a2[group == g]
            draws = torch.arange((len(v) + 3) // 4, device="cuda")
            for b in range(c["resamples"]):
                x = torch.stack(_philox(11, _i(b), draws, _i(g), _i(5)), -1).reshape(-1)[:len(v)]
                w = v[_pick(x, len(v))]
                for k in range(1, c["k_max"] + 1):
                    F[g, k - 1, b] = (w ** k).mean()
        return {"F": F}
    if call == "gemm":
        a, b, bias, z = _gemm_inputs(c, seed)
        y = a.double() @ b.double().T + bias.double()
        if c["mode"] == 1:
            y = 0.5 * y * (1 + torch.erf(y / math.sqrt(2)))
        elif c["mode"] == 2:
            t = z.double()
            y = y * (0.5 * (1 + torch.erf(t / math.sqrt(2))) + t * torch.exp(-0.5 * t * t) / math.sqrt(2 * math.pi))
        return {"C": y}
    F = _exact_fk(_chain(c, seed), c["l"], c["k"], c["q"])
    return None if F is None else {"F": F}
