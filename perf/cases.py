"""Timed cases of the displacement-probed estimator of Tr(P A^{-1}).

A case is one call that a user's program makes: a probed trace (every colour
of one or several colourings, every noise set, every spin-colour component,
in one batched solve), a batch of solves, an adjoint gradient, or a greedy
colouring.  `prepare` makes what such a program has in hand before the call
(context, gauge links, operator, colouring, right-hand sides), `run` is the
call.  `exact` restates the same quantity in plain torch / numpy in 64 bits.

Workload sizes are those of this repository's benchmark and tests: the 16^4
shifted Laplacian with m2 = 0.01, Wilson-Dirac on 24^3 x 48 and 16^3 x 32
with kappa = 0.124 and links exp(i 0.3 H), the clover term with c_sw = 1,
ragged lattices with odd sides, and a 4^4 lattice for the shortest call.
"""
import itertools
import math

import numpy as np
import torch

from paper_2106_01275_gb300 import ptrace as pt

TOL = 1e-10
MAXIT = 20000


def listed():
    return [
        # the first call of a new user and the check before a long run: a
        # handful of probes on a tiny lattice, where latency is everything
        dict(name="lap_trace_4", call="trace", op="lap", dims="4x4x4x4", m2=0.1, mu=0, pk="1,2", p="1", noise="z2",
             sets=2, prec="mixed_fp32"),
        # a study of several displacements on a lattice whose sides are odd
        # and unequal (no even-odd split, no vector path)
        dict(name="lap_trace_odd", call="trace", op="lap", dims="9x7x11x15", m2=0.05, mu=2, pk="2,2", p="0,1,2,3",
             noise="z2", sets=8, prec="mixed_fp32"),
        # the method's headline use: the twenty (p, k) colourings of p = 0..4
        # and k = 1..4 on 16^4, eight noise sets each, in one call
        dict(name="lap_trace_16", call="trace", op="lap", dims="16x16x16x16", m2=0.01, mu=3,
             pk="0,1 1,1 2,1 3,1 4,1 0,2 1,2 2,2 3,2 4,2 0,3 1,3 2,3 3,3 4,3 0,4 1,4 2,4 3,4 4,4", p="0,1,2,3,4",
             noise="z2", sets=8, prec="mixed_fp32"),
        # few probes on a large volume (the paper's 32^3 x 64), its colouring
        # repeated from a tile
        dict(name="lap_trace_32", call="trace", op="lap", dims="32x32x32x64", m2=0.01, mu=2, pk="4,1", p="0,4",
             noise="z2", sets=8, prec="mixed_fp32", tiled=True),
        # solves for a user's own right-hand sides in plain FP64
        dict(name="lap_solve_16_fp64", call="solve", op="lap", dims="16x16x16x16", m2=0.05, nrhs=24, prec="fp64"),
        # one (p, k) colouring, one Z4 set, twelve-fold spin-colour dilution
        # on a mid-size gauge configuration
        dict(name="wilson_trace_16", call="trace", op="wilson", dims="16x16x16x32", kappa=0.124, mu=2, pk="4,2",
             p="0,2,4,8", noise="z4", sets=1, prec="mixed_fp32"),
        # the same on the largest configuration of the benchmark
        dict(name="wilson_trace_24", call="trace", op="wilson", dims="24x24x24x48", kappa=0.124, mu=2, pk="4,2",
             p="0,2,4,8", noise="z4", sets=1, prec="mixed_fp32"),
        # the paper's operator class: with the clover term
        dict(name="clover_trace_16", call="trace", op="wilson", dims="16x16x16x32", kappa=0.124, csw=1.0, mu=2,
             pk="4,2", p="0,2,4,8", noise="z4", sets=1, prec="mixed_fp32"),
        # BF16 storage of the inner vectors, chosen by the caller
        dict(name="wilson_trace_8_bf16", call="trace", op="wilson", dims="8x8x8x16", kappa=0.12, mu=2, pk="2,2",
             p="0,2", noise="z4", sets=1, prec="mixed_bf16"),
        # propagators for a user's own sources on a lattice with odd sides
        dict(name="wilson_solve_odd", call="solve", op="wilson", dims="9x9x9x20", kappa=0.12, nrhs=12,
             prec="mixed_fp32"),
        # adjoint gradient with respect to kappa and every link
        dict(name="wilson_grad_8", call="grad", op="wilson", dims="8x8x8x16", kappa=0.12, mu=2, pk="4,2", p="4",
             noise="z4", sets=1, prec="mixed_fp32"),
        # a displaced distance-4 colouring, as a program without stored
        # colourings makes before its first trace
        dict(name="colour_16", call="colour", dims="16x16x16x16", mu=3, pk="2,4", order="redblack"),
    ]


def draw(rng):
    """One more case; its work stays below the 24^3 x 48 trace's."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sides(lo, hi, most, even):
        while True:
            d = [log_int(lo, hi) for _ in range(4)]
            if even:
                d = [max(2, 2 * ((x + 1) // 2)) for x in d]
            if math.prod(d) <= most:
                return d

    kind = rng.choice(["lap_trace"] * 4 + ["lap_solve"] * 2 + ["wilson_trace"] * 3 + ["clover_trace"] +
                      ["wilson_solve"] * 2 + ["wilson_grad"] + ["colour"])
    prec = rng.choice(["mixed_fp32"] * 4 + ["fp64", "mixed_bf16"])
    if kind == "colour":
        d = sides(6, 20, 70000, False)
        return dict(call="colour", dims=_x(d), mu=rng.randrange(4), pk="%d,%d" % (rng.randint(1, 4), rng.randint(1, 4)),
                    order=rng.choice(["natural", "redblack"]))
    if kind.startswith("lap"):
        even = rng.random() < 0.7
        d = sides(4, 26, 160000, even)
        m2 = round(math.exp(rng.uniform(math.log(0.01), math.log(0.2))), 4)
        if kind == "lap_solve":
            return dict(call="solve", op="lap", dims=_x(d), m2=max(m2, 0.05), nrhs=log_int(1, 64), prec=prec)
        mu, k = rng.randrange(4), rng.randint(1, 3)
        pk = " ".join("%d,%d" % (rng.randrange(5), k) for _ in range(rng.choice([1, 1, 2, 4])))
        p = ",".join(str(q) for q in sorted(rng.sample(range(9), rng.randint(1, 5))))
        return dict(call="trace", op="lap", dims=_x(d), m2=m2, mu=mu, pk=pk, p=p, noise="z2", sets=rng.randint(1, 8),
                    prec=prec)
    if kind == "clover_trace":
        d = sides(4, 16, 66000, True)
        return dict(call="trace", op="wilson", dims=_x(d), kappa=round(rng.uniform(0.11, 0.124), 4),
                    csw=round(rng.uniform(0.5, 1.2), 2), mu=rng.randrange(4), pk="%d,1" % rng.randrange(5),
                    p="0,%d" % rng.randint(1, 6), noise="z4", sets=1, prec="mixed_fp32")
    even = rng.random() < 0.7
    d = sides(4, 16, 33000 if prec == "fp64" or kind == "wilson_grad" else 66000, even)
    kappa = round(rng.uniform(0.11, 0.124), 4)
    if kind == "wilson_solve":
        return dict(call="solve", op="wilson", dims=_x(d), kappa=kappa, nrhs=log_int(1, 24), prec=prec)
    pk = "%d,1" % rng.randrange(5)
    if kind == "wilson_grad":
        return dict(call="grad", op="wilson", dims=_x(d), kappa=kappa, mu=rng.randrange(4), pk=pk,
                    p=str(rng.randint(0, 4)), noise=rng.choice(["z2", "z4"]), sets=1, prec="mixed_fp32")
    return dict(call="trace", op="wilson", dims=_x(d), kappa=kappa, mu=rng.randrange(4), pk=pk,
                p=",".join(str(q) for q in sorted(rng.sample(range(7), rng.randint(1, 4)))),
                noise=rng.choice(["z2", "z4"]), sets=rng.randint(1, 2), prec=prec)


# ------------------------------------------------------------------ a program's side
def prepare(case, seed):
    dims, N = _dims(case), _volume(case)
    ctx = pt.Context(0)
    if case["call"] == "colour":
        # the walk takes no random input: the seed turns the lattice by
        # choosing the dimension along which the displacement runs
        return dict(case=case, ctx=ctx, mu=(case["mu"] + int(seed)) % 4)
    s = dict(case=case, ctx=ctx, seed=int(seed))
    if case["op"] == "lap":
        op = pt.laplacian(ctx, dims, case["m2"])
    else:
        ctx.set_memory_budget(48 << 30)
        op = pt.wilson(ctx, dims, _links(dims, seed), case["kappa"], True)
        if case.get("csw"):
            pt.set_clover(op, case["csw"])
    s["op"] = op
    if case["call"] == "solve":
        s["B"] = _sources(case, seed)
        return s
    cols, m = [], []
    for p, k in _pk(case):
        if case.get("tiled"):
            c, n, _ = pt.colour_tiled(ctx, dims, case["mu"], [p], k)
        else:
            c, n = pt.colour(ctx, dims, case["mu"], [p], k)
        cols.append(c)
        m.append(n)
    s["cols"], s["m"] = torch.stack(cols).contiguous(), m
    torch.cuda.synchronize()
    return s


def run(state):
    c = state["case"]
    if c["call"] == "colour":
        p, k = _pk(c)[0]
        col, m = pt.colour(state["ctx"], _dims(c), state["mu"], [p], k, c["order"])
        return {"col": col, "m": m}
    op = state["op"]
    if c["call"] == "solve":
        return {"x": pt.solve(op, state["B"], c["prec"], TOL, MAXIT)[0]}
    if c["call"] == "grad":
        est, dk, G, Gb, _ = pt.grad(op, state["cols"][0], state["m"][0], c["mu"], _p(c)[0], c["noise"], state["seed"], 0,
                                    c["sets"], True, c["prec"], TOL, MAXIT, links=True)
        return {"est": est, "dkappa": np.array([dk]), "G": G, "Gbar": Gb}
    est, _ = pt.trace_multi(op, state["cols"], state["m"], c["mu"], _p(c), c["noise"], state["seed"], 0, c["sets"], True,
                            c["prec"], TOL, MAXIT)
    return {"est": est}


def work(case):
    """Inputs and outputs once; operations of the Krylov iterations that the
    operator's spectrum asks for on its even Schur complement (on the full
    system twice as many), to a residual of 1e-10."""
    N = _volume(case)
    if case["call"] == "colour":
        p, k = _pk(case)[0]
        return {"bytes": 4.0 * N, "flops": float(N) * _stencil_size(p, k)}
    lap = case["op"] == "lap"
    field = N * (8.0 if lap else 192.0)
    links = 0.0 if lap else N * 576.0
    if case["call"] == "solve":
        n, io = case["nrhs"], case["nrhs"] * 2 * field
    else:
        n = sum(_colours_about(p, k, N) for p, k in _pk(case)) * case["sets"] * (1 if lap else 12)
        io = 4.0 * N * len(_pk(case)) + 16.0 * len(_pk(case)) * case["sets"] * len(_p(case))
    if case["call"] == "grad":
        n, io = 2 * n, io + 2 * links
    even = all(d % 2 == 0 for d in _dims(case))
    if lap:
        low = case["m2"] + 4 * math.sin(math.pi / max(max(_dims(case)), 2)) ** 2
        d = 8 + case["m2"]
        cond = d * d / max(d * d - (d - low) ** 2, 1e-9) if even else (16 + case["m2"]) / low
        its = 0.5 * math.sqrt(cond) * math.log(2 / TOL)
        per_it = 20.0 * N
    else:
        its = 26.0 if even else 52.0
        per_it = 2 * 1320.0 * N + 700.0 * N
    return {"bytes": io + links, "flops": n * its * per_it}


# ------------------------------------------------------------------ 64-bit values, plain torch / numpy
def exact(case, seed):
    N = _volume(case)
    if case["call"] == "colour":
        return None                                    # whole numbers
    lap = case["op"] == "lap"
    if case["call"] == "solve":
        B = _sources(case, seed)
        if lap:
            return {"x": _lap_solve(case, B)}
        if case["nrhs"] * N > 3.5e6:
            return None
        A = _Wilson(case, seed)
        return {"x": A.from_field(A.solve(A.to_field(B)))}
    pk = _pk(case)
    if N * len(pk) > 400000 or (not lap and N * 12 * case["sets"] * sum(_colours_about(p, k, N) for p, k in pk) > 7e6):
        return None
    cols, m = _greedy(_dims(case), case["mu"], pk)
    site = _coords(_dims(case))
    ps = _p(case)
    shift = [_index(_dims(case), site + np.eye(4, dtype=np.int64)[case["mu"]] * p) for p in ps]
    shift = [torch.as_tensor(s).cuda() for s in shift]
    est = np.zeros((len(pk), case["sets"], len(ps)), dtype=np.complex128)
    if lap:
        for i, s in itertools.product(range(len(pk)), range(case["sets"])):
            z = torch.as_tensor(_noise(case, int(seed), s)).real.cuda()
            c = torch.as_tensor(cols[i]).cuda()
            for c0 in range(0, m[i], 64):
                n = min(64, m[i] - c0)
                v = z * (c[None] == torch.arange(c0, c0 + n, device="cuda")[:, None])
                x = _lap_solve(case, v)
                for j in range(len(ps)):
                    est[i, s, j] += float((v * x[:, shift[j]]).sum())
        return {"est": est}
    A = _Wilson(case, seed)
    grad = case["call"] == "grad"
    if grad:
        back = torch.as_tensor(_index(_dims(case), site - np.eye(4, dtype=np.int64)[case["mu"]] * ps[0])).cuda()
        G = torch.zeros(N, 4, 3, 3, dtype=torch.complex128, device="cuda")
        Gb = torch.zeros_like(G)
        dk = 0.0
    for i, s in itertools.product(range(len(pk)), range(case["sets"])):
        z = torch.as_tensor(_noise(case, int(seed), s)).cuda()
        c = torch.as_tensor(cols[i]).cuda()
        for q in range(m[i]):
            v = torch.zeros(N, 12, 12, dtype=torch.complex128, device="cuda")      # [site, component, right-hand side]
            v[:, torch.arange(12), torch.arange(12)] = (z * (c == q))[:, None]
            x = A.solve(v)
            if grad:
                g5 = torch.tensor([1.0] * 6 + [-1.0] * 6, dtype=torch.float64, device="cuda")[None, :, None]
                y = g5 * A.solve(g5 * v[back])
                est[i, s, 0] += complex((y.conj() * v).sum())
                dk += complex((y.conj() * A.hop(x)).sum())
                for mu in range(4):
                    w = A.kappa * A.eta(mu)[:, None, None]
                    f = A.fwd[mu]
                    X, Y = x.view(N, 4, 3, 12), y.view(N, 4, 3, 12)
                    P = torch.einsum("st,nbtr->nbsr", A.proj[mu][0], X[f].transpose(1, 2))
                    G[:, mu] += w * torch.einsum("nsar,nbsr->nab", Y.conj(), P)
                    P = torch.einsum("st,natr->nasr", A.proj[mu][1], X.transpose(1, 2))
                    Gb[:, mu] += w * torch.einsum("nsbr,nasr->nab", Y[f].conj(), P)
            else:
                for j in range(len(ps)):
                    est[i, s, j] += complex((v.conj() * x[shift[j]]).sum())
    if grad:
        return {"est": est[0, :, 0], "dkappa": np.array([dk]), "G": G, "Gbar": Gb}
    return {"est": est}


# ------------------------------------------------------------------ helpers
def _x(d):
    return "x".join(str(v) for v in d)


def _dims(case):
    return [int(v) for v in case["dims"].split("x")]


def _volume(case):
    return math.prod(_dims(case))


def _pk(case):
    return [tuple(int(v) for v in t.split(",")) for t in case["pk"].split()]


def _p(case):
    return [int(v) for v in case["p"].split(",")]


def _stencil_size(p, k):
    n = 0
    for o in itertools.product(range(-k, k + 1), repeat=3):
        r = k - sum(abs(v) for v in o)
        if r >= 0:
            n += len(set(range(p - r, p + r + 1)) | set(range(-p - r, -p + r + 1)))
    return n


def _colours_about(p, k, N):
    """Size of a greedy displaced colouring, from the clique bound's growth."""
    if p > k:
        return min(N, {1: 2, 2: 4, 3: 8}.get(k, 16))
    return min(N, {1: 4, 2: 10, 3: 16, 4: 64}.get(k, 64))


def _links(dims, seed):
    """exp(i 0.3 H), H the traceless Hermitian part of complex Gaussians:
    [N, 4, 3, 3], by the exponential's series (the norm of 0.3 H is of order 1)."""
    N = math.prod(dims)
    g = torch.Generator(device="cuda").manual_seed(4000 + int(seed))
    A = torch.randn(2, 9, N * 4, generator=g, device="cuda", dtype=torch.float64)
    A = torch.complex(A[0], A[1]).view(3, 3, N * 4)
    H = 0.5 * (A + A.transpose(0, 1).conj())
    H = H - (H[0, 0] + H[1, 1] + H[2, 2]) / 3 * torch.eye(3, device="cuda", dtype=H.dtype)[:, :, None]
    X = (0.3j / 16) * H

    def mul(a, b):
        return torch.stack([torch.stack([a[i, 0] * b[0, j] + a[i, 1] * b[1, j] + a[i, 2] * b[2, j] for j in range(3)])
                            for i in range(3)])

    U = torch.eye(3, device="cuda", dtype=H.dtype)[:, :, None].expand(3, 3, N * 4).clone()
    for n in range(14, 0, -1):
        U = torch.eye(3, device="cuda", dtype=H.dtype)[:, :, None] + mul(X, U) / n
    for _ in range(4):
        U = mul(U, U)
    return U.permute(2, 0, 1).reshape(N, 4, 3, 3).contiguous()


def _sources(case, seed):
    g = torch.Generator(device="cuda").manual_seed(9000 + int(seed))
    N, n = _volume(case), case["nrhs"]
    if case["op"] == "lap":
        return torch.randn(n, N, generator=g, device="cuda", dtype=torch.float64)
    r = torch.randn(n, N, 4, 3, 2, generator=g, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(r)


def _coords(dims):
    i = np.arange(math.prod(dims), dtype=np.int64)
    out = []
    for d in dims:
        out.append(i % d)
        i = i // d
    return np.stack(out, axis=1)


def _index(dims, x):
    idx, s = np.zeros(len(x), dtype=np.int64), 1
    for n, d in enumerate(dims):
        idx += s * (x[:, n] % d)
        s *= d
    return idx


def _noise(case, seed, s):
    """SplitMix64 noise of one set, one value per site."""
    def mix(z):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    with np.errstate(over="ignore"):
        gamma = np.uint64(0x9E3779B97F4A7C15)
        key = mix(np.array([seed], dtype=np.uint64) + np.uint64(s + 1) * gamma)
        h = mix(key + (np.arange(_volume(case), dtype=np.uint64) + np.uint64(1)) * gamma)
    if case["noise"] == "z2":
        return (1.0 - 2.0 * (h >> np.uint64(63)).astype(np.float64)).astype(np.complex128)
    return np.array([1, 1j, -1, -1j])[(h >> np.uint64(62)).astype(np.int64)]


def _greedy(dims, mu, pk):
    """First-fit colourings in storage order, all of them in one walk."""
    N, site = math.prod(dims), _coords(dims)
    stride = np.cumprod([1] + list(dims[:3]))
    offs = []
    for p, k in pk:
        o = np.array([o for o in itertools.product(*[range(-(p * (n == mu) + k), p * (n == mu) + k + 1) for n in range(4)])
                      if any(sum(abs(v - s * p * (n == mu)) for n, v in enumerate(o)) <= k for s in (1, -1))])
        offs.append(np.unique(o % np.array(dims), axis=0))
    width = max(len(o) for o in offs)
    rows = len(pk)
    off = np.zeros((rows, width, 4), dtype=np.int64)           # padding: the node itself, never coloured yet
    for i, o in enumerate(offs):
        off[i, : len(o)] = o
    most = min(N, width) + 2
    col = np.full((rows, N), most - 1, dtype=np.int64)         # most - 1: not coloured
    used = np.zeros((rows, most), dtype=np.int64)
    row = np.arange(rows)[:, None]
    for x in range(N):
        y = ((site[x] + off) % np.array(dims)) @ stride
        c = col[row, y]
        used[row, c] = x + 1
        used[:, most - 1] = x + 1
        col[:, x] = np.argmax(used != x + 1, axis=1)
    return col, [int(c.max()) + 1 for c in col]


def _lap_solve(case, B):
    """(8 + m2 - hops)^{-1} by the discrete Fourier transform."""
    dims = _dims(case)
    lam = 8.0 + case["m2"]
    for n, d in enumerate(dims):
        w = 2 * torch.cos(2 * math.pi * torch.arange(d, device="cuda", dtype=torch.float64) / d)
        lam = lam - w.view([-1 if 3 - n == a else 1 for a in range(4)])
    out = []
    for b in B.split(16):
        f = torch.fft.fftn(b.view(-1, *dims[::-1]), dim=(1, 2, 3, 4)) / lam
        out.append(torch.fft.ifftn(f, dim=(1, 2, 3, 4)).real.reshape(b.shape))
    return torch.cat(out)


class _Wilson:
    """Wilson-Dirac operator (clover term where the case has one) on fields
    [site, 12 components, right-hand sides]."""

    def __init__(self, case, seed):
        self.dims, self.kappa = _dims(case), case["kappa"]
        self.N = math.prod(self.dims)
        site = _coords(self.dims)
        e = np.eye(4, dtype=np.int64)
        self.fwd = [torch.as_tensor(_index(self.dims, site + e[n])).cuda() for n in range(4)]
        self.bwd = [torch.as_tensor(_index(self.dims, site - e[n])).cuda() for n in range(4)]
        self.site = site
        self.U = _links(self.dims, seed)
        s = [np.array(v, dtype=np.complex128) for v in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
        Z, I2 = np.zeros((2, 2)), np.eye(2)
        g = [np.block([[Z, -1j * v], [1j * v, Z]]) for v in s] + [np.block([[Z, I2], [I2, Z]])]
        self.spin = [[np.eye(4) - v, np.eye(4) + v] for v in g]
        self.proj = [[torch.as_tensor(P.astype(np.complex128)).cuda() for P in q] for q in self.spin]
        self.C = None
        if case.get("csw"):
            C = torch.zeros(self.N, 12, 12, dtype=torch.complex128, device="cuda")
            for a, b in itertools.combinations(range(4), 2):
                sig = torch.as_tensor(0.5j * (g[a] @ g[b] - g[b] @ g[a])).cuda()
                Q = self._leaves(a, b)
                F = (Q - Q.mH) / 8j
                C += torch.einsum("st,nab->nsatb", sig, F).reshape(self.N, 12, 12)
            self.C = -self.kappa * case["csw"] * C

    def _leaves(self, a, b):
        Ua, Ub = self.U[:, a], self.U[:, b]
        pa, pb, ma, mb = self.fwd[a], self.fwd[b], self.bwd[a], self.bwd[b]
        q = Ua @ Ub[pa] @ Ua[pb].mH @ Ub.mH
        q = q + Ub @ Ua[ma[pb]].mH @ Ub[ma].mH @ Ua[ma]
        q = q + Ua[ma].mH @ Ub[mb[ma]].mH @ Ua[mb[ma]] @ Ub[mb]
        return q + Ub[mb].mH @ Ua[mb] @ Ub[pa[mb]] @ Ua.mH

    def eta(self, mu, back=False):
        x = self.site[:, mu]
        edge = x == (0 if back else self.dims[mu] - 1)
        return torch.as_tensor(np.where(edge & (mu == 3), -1.0, 1.0)).cuda()

    def hop(self, v):
        R = v.shape[2]
        out = torch.zeros_like(v).view(self.N, 4, 3, R)
        v = v.view(self.N, 4, 3, R)
        for mu in range(4):
            for back in (False, True):
                y = self.bwd[mu] if back else self.fwd[mu]
                u = self.U[:, mu][y].mH if back else self.U[:, mu]
                u = u * self.eta(mu, back)[:, None, None]
                f = v[y]
                w = torch.stack([sum(u[:, a, b, None, None] * f[:, :, b] for b in range(3)) for a in range(3)], dim=2)
                P = self.spin[mu][int(back)]
                for s in range(4):
                    for t in range(4):
                        if P[s, t]:
                            out[:, s].add_(w[:, t], alpha=complex(P[s, t]))
        return out.view(self.N, 12, R)

    def apply(self, v):
        out = v - self.kappa * self.hop(v)
        return out if self.C is None else out + self.C @ v

    def solve(self, b, tol=1e-13):
        """BiCGStab, every right-hand side with its own scalars."""
        def dot(u, w):
            return (u.conj() * w).sum(dim=(0, 1))

        x = torch.zeros_like(b)
        r = b.clone()
        r0, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b)
        one = torch.ones(b.shape[2], dtype=b.dtype, device=b.device)
        rho, alpha, om = one, one, one
        bn = dot(b, b).real.clamp_min(1e-300)
        safe = lambda q: torch.where(q.abs() > 0, q, torch.ones_like(q))  # noqa: E731
        for _ in range(400):
            live = (dot(r, r).real / bn > tol * tol).to(b.dtype)
            if not bool(live.abs().sum() > 0):
                break
            rho1 = dot(r0, r)
            beta = rho1 / safe(rho) * (alpha / safe(om))
            rho = rho1
            p = r + beta * (p - om * v)
            v = self.apply(p)
            alpha = live * rho / safe(dot(r0, v))
            s = r - alpha * v
            t = self.apply(s)
            om = live * dot(t, s) / safe(dot(t, t))
            x = x + alpha * p + om * s
            r = s - om * t
        return x

    def to_field(self, B):
        return B.reshape(B.shape[0], self.N, 12).permute(1, 2, 0).contiguous()

    def from_field(self, x):
        return x.permute(2, 0, 1).reshape(x.shape[2], self.N, 4, 3).contiguous()
