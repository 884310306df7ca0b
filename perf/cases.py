"""The work this library's performance is measured on.

Every case calls the public binding (paper_2505_24256_gb300.zr) as a program
would: it keeps a context and its buffers, and one pass is one call (or one
full reconstruction).  Results are exact residues modulo p = 2^63 - 25, so
every output is an integer and has one right value: the hidden function the
inputs were made from, or the definition evaluated here in plain torch.

listed() names the cases, draw(rng) gives more of the same ranges, prepare()
makes a case's inputs from a seed, run() is one pass, work() what a pass
cannot do without and exact() the right outputs.
"""
import math

import numpy as np
import torch

from paper_2505_24256_gb300 import zr

P = 2**63 - 25


def listed():
    return [
        # One Zippel step of a small reconstruction (the size of the plain
        # three-variable, 200-term polynomial): latency and launches.
        dict(name="step_T200_S11", kind="step", T=200, nv=3, maxexp=20, S=11, offset=0, fill=1.0),
        # Many small uneven steps in one call, as a program that drives
        # several reconstructions at once issues them.
        dict(name="steps_batch64_T20_66_S11", kind="batch", n=64, tmin=20, tmax=66, nv=3, maxexp=10, S=11, offset=0),
        # An ordinary step with odd sizes, probes from y^1, and a hidden
        # function whose terms do not use every power of the new variable.
        dict(name="step_T1531_S6", kind="step", T=1531, nv=4, maxexp=20, S=6, offset=1, fill=0.5),
        # The batched step the library quotes its throughput on.
        dict(name="step_T10000_S21", kind="step", T=10000, nv=6, maxexp=20, S=21, offset=0, fill=1.0),
        # The smallest skeleton size of the paper's data sets (125k terms).
        dict(name="step_T125000_S9", kind="step", T=125000, nv=6, maxexp=20, S=9, offset=0, fill=0.7),
        # The largest step: 2^20 terms in seven variables, degree 8.
        dict(name="step_T1048576_S9", kind="step", T=1 << 20, nv=8, maxexp=12, S=9, offset=0, fill=1.0),
        # Transposed Vandermonde systems of uneven sizes and right-hand
        # sides in one call, for a program with its own nodes and values.
        dict(name="solve_uneven10", kind="solve", n=10, tmin=97, tmax=4099, smax=21, offset=0),
        # The built-in black box's probes for one step, ordinary and large:
        # every step of every reconstruction of a built-in function needs them.
        dict(name="probes_T1200_Tf3000_S11", kind="probes", T=1200, Tf=3000, nv=5, k=2, maxexp=20, S=11, offset=0),
        dict(name="probes_T10000_Tf10000_S21", kind="probes", T=10000, Tf=10000, nv=6, k=5, maxexp=20, S=21, offset=0),
        # Full reconstructions from host arrays: the plain three-variable
        # polynomial, a polynomial of the serving mix, and the balanced
        # rational function.
        dict(name="recon_poly_n3_T200", kind="poly", nv=3, T=200, shape="simplex", deg=10),
        dict(name="recon_poly_n4_T6000", kind="poly", nv=4, T=6000, shape="box", deg=20),
        dict(name="recon_rational_n5_N5000_D3000", kind="rational", nv=5, TN=5000, TD=3000, shape="simplex", deg=15),
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "solve", "probes", "probes", "poly", "rational"])
    offset = rng.randint(0, 1)
    if kind == "step":
        T, S = _log_uniform(rng, 100, 1 << 20), rng.randint(4, 21)
        S = max(2, min(S, 9 * (1 << 20) // T))
        nv = rng.randint(6, 8) if T > 8000 else rng.randint(4, 8) if T > 150 else rng.randint(3, 8)
        return dict(kind="step", T=T, nv=nv, maxexp=20 if nv < 8 else 12, S=S, offset=offset,
                    fill=rng.choice([1.0, 0.7, 0.5]))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(8, 64), tmin=20, tmax=_log_uniform(rng, 40, 400), nv=rng.randint(4, 5),
                    maxexp=20, S=rng.randint(4, 21), offset=offset)
    if kind == "solve":
        return dict(kind="solve", n=rng.randint(1, 12), tmin=_log_uniform(rng, 17, 1000),
                    tmax=_log_uniform(rng, 1500, 5000), smax=rng.randint(1, 21), offset=offset)
    if kind == "probes":
        T = _log_uniform(rng, 200, 20000)
        Tf = min(60000, int(T * rng.uniform(1.0, 4.0)))
        nv = rng.randint(5, 8)
        return dict(kind="probes", T=T, Tf=Tf, nv=nv, k=rng.randint(1, nv - 1), maxexp=20, S=rng.randint(3, 21),
                    offset=offset)
    if kind == "poly":
        nv = rng.randint(3, 6)
        return dict(kind="poly", nv=nv, T=_log_uniform(rng, 50, 4000 if nv == 3 else 12000), shape="box",
                    deg=rng.randint(8, 20) if nv > 4 else 20)
    T = _log_uniform(rng, 60, 8000)
    TN = max(1, (T * 3 + 4) // 5)
    return dict(kind="rational", nv=rng.randint(4, 5), TN=TN, TD=max(1, T - TN), shape="box", deg=rng.randint(9, 15))


# --------------------------------------------------------------- arithmetic
# Residues modulo P as int64 tensors; products in three 21-bit pieces of one
# factor, the quotient from doubles (at most 2^22, so it is exact to less
# than one unit in the last place of the remainder's range) and the remainder
# in wrapping 64-bit integers.

def _mul(a, b):
    r = torch.zeros((), dtype=torch.int64, device=a.device)
    for sh in (42, 21, 0):
        x = (b >> sh) & 0x1FFFFF
        q = torch.round((r.double() * 2097152.0 + a.double() * x.double()) / float(P)).long()
        r = r * 2097152 + a * x - q * P
        r = torch.where(r < 0, r + P, r)
    return r


def _add(a, b):
    d = a - (P - b)
    return torch.where(d < 0, d + P, d)


def _sum(x, dim):
    hi, lo = (x >> 32).sum(dim), (x & 0xFFFFFFFF).sum(dim)
    return _add(_mul(hi, torch.full_like(hi, 1 << 32)), lo)


def _pow(a, e):
    """a^e for tensors a, e of small nonnegative exponents."""
    r = torch.ones((), dtype=torch.int64, device=a.device)
    top = int(e.max()) if e.numel() else 0
    while top:
        r = torch.where((e & 1) == 1, _mul(a, r), r)
        a, e, top = _mul(a, a), e >> 1, top >> 1
    return r + torch.zeros_like(e)


# ------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _residues(g, *shape):
    return torch.randint(1, P, shape, generator=g, device="cuda", dtype=torch.int64)


def _monomials(g, n, nv, maxexp):
    """n distinct exponent rows with entries in [0, maxexp], in lexicographic order."""
    base = maxexp + 1
    total = base**nv
    if n * 4 >= total:
        codes = torch.randperm(total, generator=g, device="cuda")[:n]
    else:
        codes = torch.empty(0, dtype=torch.int64, device="cuda")
        while codes.numel() < n:
            codes = torch.unique(torch.cat([codes, torch.randint(0, total, (n,), generator=g, device="cuda")]))
        codes = codes[torch.randperm(codes.numel(), generator=g, device="cuda")[:n]]
    codes = codes.sort().values
    rows = [(codes // base ** (nv - 1 - m)) % base for m in range(nv)]
    return torch.stack(rows, 1).to(torch.uint8)


def _hidden(g, T, nv, maxexp, S, fill):
    """A skeleton of T monomials in x_0..x_{nv-2} and a hidden function on it:
    G[j, e] is the coefficient of the j-th monomial times x_{nv-1}^e.  A
    share `fill` of them is nonzero, at least one for every monomial."""
    skel = torch.zeros((T, nv), dtype=torch.uint8, device="cuda")
    skel[:, :nv - 1] = _monomials(g, T, nv - 1, maxexp)
    G = _residues(g, T, S)
    if fill < 1.0:
        rank = torch.rand((T, S), generator=g, device="cuda")
        rank.scatter_(1, torch.randint(0, S, (T, 1), generator=g, device="cuda"), 2.0)
        drop = rank.view(-1).argsort(descending=True)[max(T, round(fill * T * S)):]
        G.view(-1)[drop] = 0
    return skel, G


def _terms(skel, G):
    """The hidden function's terms in the order of the skeleton, then of the new variable's power."""
    j, e = torch.nonzero(G, as_tuple=True)
    exps = skel[j]
    exps[:, -1] = e.to(torch.uint8)
    return exps.contiguous(), G[j, e].contiguous()


def _step_inputs(ctx, g, T, nv, maxexp, S, offset, fill):
    k = nv - 1
    skel, G = _hidden(g, T, nv, maxexp, S, fill)
    exps, coef = _terms(skel, G)
    y, cs = _residues(g, k), _residues(g, S)
    b = torch.empty((S, T), dtype=torch.int64, device="cuda")
    f = ctx.poly(nv, exps.shape[0], exps, coef)
    ctx.zippel_probes(f, k, y, S, cs, None, T, offset, b, T)
    return skel, G, y, cs, b


def _sizes(case):
    """The uneven sizes of a batch, fixed by the case alone."""
    n, lo, hi = case["n"], case["tmin"], case["tmax"]
    if case["kind"] == "batch":
        return [(lo + (i * 37) % (hi - lo + 1), case["S"]) for i in range(n)]
    out = []
    for i in range(n):
        t = lo * (hi / lo) ** (i / max(n - 1, 1))
        out.append((min(hi, int(t)), 1 + (i * 8 + 4) % case["smax"]))
    return out


def _host_monomials(rng, n, nv, shape, deg):
    base = deg + 1
    if shape == "simplex":
        grid = np.indices((base,) * nv).reshape(nv, -1).T
        rows = grid[grid.sum(1) <= deg]
        return rows[np.sort(rng.choice(rows.shape[0], n, replace=False))].astype(np.uint8)
    codes = np.empty(0, np.int64)
    while codes.size < n:
        codes = np.unique(np.concatenate([codes, rng.integers(0, base**nv, n)]))
    codes = np.sort(rng.choice(codes, n, replace=False))
    return np.stack([(codes // base ** (nv - 1 - m)) % base for m in range(nv)], 1).astype(np.uint8)


def _host_function(case, seed):
    rng = np.random.default_rng(seed)
    nv, shape, deg = case["nv"], case["shape"], case["deg"]
    if case["kind"] == "poly":
        return _host_monomials(rng, case["T"], nv, shape, deg), rng.integers(1, P, case["T"], dtype=np.uint64)
    Ne, De = (_host_monomials(rng, case[n], nv, shape, deg) for n in ("TN", "TD"))
    low = np.minimum(Ne.min(0), De.min(0))            # no common monomial factor: N/D in lowest terms
    Ne, De = Ne - low, De - low
    Nc, Dc = (rng.integers(1, P, case[n], dtype=np.uint64) for n in ("TN", "TD"))
    Dc[0] = 1                                         # the normalisation of the result
    return Ne, Nc, De, Dc


def prepare(case, seed):
    kind = case["kind"]
    ctx = zr.Context(P)
    st = dict(kind=kind, ctx=ctx, case=case)
    if kind in ("poly", "rational"):
        st["f"] = _host_function(case, seed)
        st["deg"] = [case["deg"]] * case["nv"]
        st["seed"] = seed
        return st
    g = _gen(seed)
    offset = case["offset"]
    if kind == "step":
        T, nv, S = case["T"], case["nv"], case["S"]
        skel, _, y, cs, b = _step_inputs(ctx, g, T, nv, case["maxexp"], S, offset, case["fill"])
        st.update(skel=ctx.poly(nv, T, skel), keep=skel, y=y, cs=cs, b=b, cap=T * S,
                  oe=torch.empty((T * S, nv), dtype=torch.uint8, device="cuda"),
                  oc=torch.empty(T * S, dtype=torch.int64, device="cuda"))
    elif kind == "batch":
        nv, sizes = case["nv"], _sizes(case)
        total = sum(T * S for T, S in sizes)
        st.update(oe=torch.empty((total, nv), dtype=torch.uint8, device="cuda"),
                  oc=torch.empty(total, dtype=torch.int64, device="cuda"),
                  on=torch.empty(len(sizes), dtype=torch.int64, device="cuda"), keep=[], steps=[])
        o = 0
        for i, (T, S) in enumerate(sizes):
            skel, _, y, cs, b = _step_inputs(ctx, g, T, nv, case["maxexp"], S, offset, 1.0)
            st["keep"].append(skel)
            st["steps"].append(dict(skel=ctx.poly(nv, T, skel), newvar=nv - 1, S=S, offset=offset, y=y, samples=cs,
                                    probes=b, ldb=T, out_exps=st["oe"][o:o + T * S], out_coef=st["oc"][o:o + T * S],
                                    out_cap=T * S, out_count=st["on"][i:i + 1]))
            o += T * S
    elif kind == "solve":
        st["systems"], st["out"] = [], []
        for T, S in _sizes(case):
            nv = 5
            skel, _, y, cs, b = _step_inputs(ctx, g, T, nv, 20, S, offset, 1.0)
            v = torch.empty(T, dtype=torch.int64, device="cuda")
            ctx.anchor_values(T, nv, skel, nv - 1, y, offset, v)
            c = torch.empty((S, T), dtype=torch.int64, device="cuda")
            st["systems"].append(dict(T=T, S=S, offset=offset, v=v, b=b, ldb=T, c=c, ldc=T))
            st["out"].append(c)
    else:
        nv, k, T, Tf, S = (case[n] for n in ("nv", "k", "T", "Tf", "S"))
        exps, coef, y, cs, z = _probe_function(case, g)
        st.update(f=ctx.poly(nv, Tf, exps, coef), keep=(exps, coef), y=y, cs=cs, z=z,
                  out=torch.empty((S, T), dtype=torch.int64, device="cuda"))
    torch.cuda.synchronize()
    return st


def _probe_function(case, g):
    nv, Tf = case["nv"], case["Tf"]
    exps, coef = _monomials(g, Tf, nv, case["maxexp"]), _residues(g, Tf)
    return exps, coef, _residues(g, case["k"]), _residues(g, case["S"]), _residues(g, nv)


def run(st):
    kind, ctx, case = st["kind"], st["ctx"], st["case"]
    if kind == "step":
        n = ctx.zippel_step(st["skel"], case["nv"] - 1, st["y"], case["S"], st["cs"], st["b"], case["T"],
                            case["offset"], st["oe"], st["oc"], st["cap"])
        return [st["oe"][:n], st["oc"][:n]]
    if kind == "batch":
        ctx.zippel_step_batched(st["steps"])
        return [st["oe"], st["oc"], st["on"]]
    if kind == "solve":
        ctx.vandermonde_solve(st["systems"])
        return st["out"]
    if kind == "probes":
        ctx.zippel_probes(st["f"], case["k"], st["y"], case["S"], st["cs"], st["z"], case["T"], case["offset"],
                          st["out"], case["T"])
        return st["out"]
    if kind == "poly":
        (e, c), _, _ = ctx.reconstruct(case["nv"], st["deg"], st["seed"], *st["f"])
        return [e, c.view(np.int64)]
    Ne, Nc, De, Dc = st["f"]
    (ne, nc), (de, dc), _ = ctx.reconstruct(case["nv"], st["deg"], st["seed"], Ne, Nc, De, Dc, degD=st["deg"])
    return [ne, nc.view(np.int64), de, dc.view(np.int64)]


# --------------------------------------------------------------------- work
# flops: two per modular multiply-accumulate of the cheaper of the two known
# ways, the dense one (S T^2) and the quasi-linear one ((S + 1) T log2(T)^2).

def _solve_macs(T, S):
    return min((S + 2.5) * T * T, (S + 1) * T * max(math.log2(T), 1.0) ** 2)


def _probe_macs(T, Tf, S):
    n = max(T, Tf)
    return min(float(S) * T * Tf, (S + 1) * n * max(math.log2(n), 1.0) ** 2)


def work(case):
    kind = case["kind"]
    if kind == "step" or kind == "batch":
        nv, fill = case["nv"], case.get("fill", 1.0)
        sizes = [(case["T"], case["S"])] if kind == "step" else _sizes(case)
        return dict(bytes=sum(T * nv + 8 * S * T + fill * T * S * (nv + 8) for T, S in sizes),
                    flops=sum(2 * (_solve_macs(T, S) + S * S * T) for T, S in sizes))
    if kind == "solve":
        return dict(bytes=sum(8 * T * (1 + 2 * S) for T, S in _sizes(case)),
                    flops=sum(2 * _solve_macs(T, S) for T, S in _sizes(case)))
    if kind == "probes":
        T, Tf, S = case["T"], case["Tf"], case["S"]
        return dict(bytes=Tf * (case["nv"] + 8) + 8 * S * T, flops=2 * _probe_macs(T, Tf, S))
    # a reconstruction: its last step at the full skeleton size, probes and
    # solve, and the function in and out
    nv, S = case["nv"], case["deg"] + 1
    if kind == "poly":
        T = case["T"]
        return dict(bytes=2 * T * (nv + 8), flops=2 * (_probe_macs(T, T, S) + _solve_macs(T, S)))
    TN, TD = case["TN"], case["TD"]
    return dict(bytes=2 * (TN + TD) * (nv + 8),
                flops=2 * (_probe_macs(TN, TN, 2 * S) + _probe_macs(TN, TD, 2 * S) + _solve_macs(TN, S) +
                           _solve_macs(TD, S)))


# -------------------------------------------------------------------- exact

def _horner(G, x):
    """The polynomials with coefficient rows G[j, :] at the points x[s]: out[s, j]."""
    acc = torch.zeros((x.numel(), G.shape[0]), dtype=torch.int64, device=G.device)
    for e in range(G.shape[1] - 1, -1, -1):
        acc = _add(_mul(acc, x[:, None].expand_as(acc)), G[:, e][None, :].expand_as(acc))
    return acc


def exact(case, seed):
    kind = case["kind"]
    if kind in ("poly", "rational"):
        f = _host_function(case, seed)
        return [a if a.dtype == np.uint8 else a.view(np.int64) for a in f]
    g = _gen(seed)
    if kind == "step":
        return list(_terms(*_hidden(g, case["T"], case["nv"], case["maxexp"], case["S"], case["fill"])))
    if kind == "batch":
        es, cs, ns = [], [], []
        for T, S in _sizes(case):
            e, c = _terms(*_hidden(g, T, case["nv"], case["maxexp"], S, 1.0))
            _residues(g, case["nv"] - 1), _residues(g, S)
            es.append(e), cs.append(c), ns.append(c.numel())
        return [torch.cat(es), torch.cat(cs), torch.tensor(ns, dtype=torch.int64)]
    if kind == "solve":
        out = []
        for T, S in _sizes(case):
            _, G = _hidden(g, T, 5, 20, S, 1.0)
            _residues(g, 4)
            out.append(_horner(G, _residues(g, S)))
        return out
    # out[s, i] = sum_t coef_t prod_{m<k} y_m^(e_m (i + offset)) c_s^(e_k) prod_{m>k} z_m^(e_m):
    # w[s, t] u_t^(i + offset), 64 consecutive powers at a time
    T, S, k, nv = case["T"], case["S"], case["k"], case["nv"]
    if T * case["Tf"] * S > 6e9:
        return None
    exps, coef, y, cs, z = _probe_function(case, g)
    ex = exps.long()
    u = torch.ones_like(coef)
    for m in range(k):
        u = _mul(u, _pow(y[m].expand_as(coef), ex[:, m]))
    for m in range(k + 1, nv):
        coef = _mul(coef, _pow(z[m].expand_as(coef), ex[:, m]))
    w = _mul(coef[None, :].expand(S, -1), _pow(cs[:, None].expand(S, coef.numel()), ex[None, :, k].expand(S, -1)))
    if case["offset"]:
        w = _mul(w, u[None, :].expand_as(w))
    out = torch.empty((S, T), dtype=torch.int64, device="cuda")
    B = 16
    pw = torch.ones((B, u.numel()), dtype=torch.int64, device="cuda")
    for b in range(1, B):
        pw[b] = _mul(pw[b - 1], u)
    step = _mul(pw[B - 1], u)
    for i in range(0, T, B):
        n = min(B, T - i)
        out[:, i:i + n] = _sum(_mul(w[:, None, :].expand(S, n, -1), pw[None, :n].expand(S, n, -1)), 2)
        w = _mul(w, step[None, :].expand_as(w))
    return out
