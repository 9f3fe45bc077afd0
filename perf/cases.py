"""Performance cases: the calls a user of the screening library makes, over the sizes they make them.

The networks are those of the synthetic study and of its tests: the 118-bus study network (``synth.case118``,
186 branches, 54 generators, load levels 70 % and 90 %), the 300-bus serving network (``synth.case_scaled``) and
the 14-bus network of the smoke and serving tests.  What the seed draws is the work itself: which outages are asked
about, in which order, and the failure rates.

Pairs of outages are asked about at the 70 % level.  At 90 % load about ten of the study's 28,680 pairs have Newton
systems that FP64 cannot resolve: whether and when they converge is decided by rounding (the CPU oracle's own solve
variants disagree on them), so a record of them says nothing about a change.  The 90 % level is measured by its
single outages, none of which is of that kind.  So is the 300-bus network, at 60 % load for the same reason (at 70 %
three of its 525 single outages are of that kind), and in the FP64 form: its mixed form returns eigenvalues as the
FP32 screen gives them, good to about 1e-5 and different with any change of rounding in the OPF.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_08465_gb300 import cs, synth

DEV = "cuda:0"
_NETS = {}
_STUDY = {}


def listed():
    return [
        # an operator's question: one pair of outages, answered alone (latency of one scenario)
        dict(name="whatif_mixed", kind="evaluate", net="118", form="mixed", level=0, order=2, n=1, island=False),
        # the hourly N-1 scan of the heavier operating point: every single outage, far fewer than the GPU holds
        dict(name="n1_mixed_90", kind="evaluate", net="118", form="mixed", level=1, order=1, n=240, island=False),
        # the same scan in the FP64 form
        dict(name="n1_fp64", kind="evaluate", net="118", form="fp64", level=0, order=1, n=240, island=False),
        # a short list of pairs (a protection scheme's, a maintenance plan's): about one wave of the GPU
        dict(name="pairs_mixed_501", kind="evaluate", net="118", form="mixed", level=0, order=2, n=501, island=False),
        # the N-2 study itself, a third of one load level: more than one internal batch, the second one ragged
        dict(name="pairs_mixed_10000", kind="evaluate", net="118", form="mixed", level=0, order=2, n=10000,
             island=False),
        # the N-2 study in the FP64 form
        dict(name="pairs_fp64_2000", kind="evaluate", net="118", form="fp64", level=0, order=2, n=2000, island=False),
        # the main-island option with the severity indices: split networks get the OPF of their main island too
        dict(name="island_mixed_1000", kind="evaluate", net="118", form="mixed", level=0, order=2, n=1000,
             island=True),
        # the serving path: requests of several sizes from host arrays, records back in host arrays
        dict(name="serve_mixed_1500", kind="serve", net="118", form="mixed", level=0, requests=5, n=1500),
        # the large serving network: a share of its single outages, in the FP64 form
        dict(name="net300_fp64_200", kind="evaluate", net="300", form="fp64", level=0, order=1, n=200, island=False),
        # a small network, every pair and every single outage of it
        dict(name="net14_fp64_325", kind="evaluate", net="14", form="fp64", level=0, order=2, n=325, island=False),
        # Risk Index of one set of severity tables (one rank's reduction after the merge)
        dict(name="risk_240", kind="risk", n_elem=240),
        # Monte-Carlo Risk Index: sampled failure rates against the study's tables
        dict(name="risk_mc_10000", kind="risk_mc", samples=10000),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pairs", "pairs", "fp64", "n1", "island", "serve", "net300", "net14", "risk", "risk_mc"])
    ev = dict(kind="evaluate", net="118", form="mixed", level=0, order=2, island=False)
    if kind == "pairs":
        return dict(ev, n=_log_uniform(rng, 1, 10000))
    if kind == "fp64":
        return dict(ev, form="fp64", n=_log_uniform(rng, 1, 2000))
    if kind == "n1":
        return dict(ev, form=rng.choice(["mixed", "fp64"]), level=rng.choice([0, 1]), order=1,
                    n=rng.randint(60, 240))
    if kind == "island":
        return dict(ev, island=True, n=_log_uniform(rng, 10, 2000))
    if kind == "serve":
        return dict(kind="serve", net="118", form=rng.choice(["mixed", "mixed", "fp64"]), level=0,
                    requests=rng.randint(1, 5), n=_log_uniform(rng, 16, 1500))
    if kind == "net300":
        return dict(ev, net="300", form="fp64", order=1, n=_log_uniform(rng, 8, 400))
    if kind == "net14":
        return dict(ev, net="14", form=rng.choice(["mixed", "fp64"]), n=rng.randint(20, 325))
    if kind == "risk":
        return dict(kind="risk", n_elem=_log_uniform(rng, 25, 3250))
    return dict(kind="risk_mc", samples=_log_uniform(rng, 100, 20000))


def _net(name):
    if name not in _NETS:
        if name == "118":
            _NETS[name] = synth.case118()
        elif name == "300":
            _NETS[name] = synth.case_scaled(300, seed=300, levels=(0.6,), vband=(0.85, 1.15))
        else:
            _NETS[name] = synth.make_network(14, 20, 5, 11, 1, seed=3, levels=(0.5,))
    return _NETS[name]


def _connected(net, out):
    """Whether the bus graph without the branches in ``out`` is in one piece."""
    root = list(range(net.n_bus))

    def find(u):
        while root[u] != u:
            u = root[u]
        return u

    for b in range(net.n_branch):
        if b not in out:
            root[find(int(net.f[b]))] = find(int(net.t[b]))
    return len({find(u) for u in range(net.n_bus)}) == 1


def _outages(case, seed):
    """The outages asked about: n of the network's single elements or pairs, in a drawn order."""
    net = _net(case["net"])
    rng = np.random.default_rng(seed)
    if case.get("order") == 1:
        ei = rng.permutation(net.n_elem)[:case["n"]].astype(np.int32)
        return ei, np.full(ei.size, -1, np.int32)
    ii, jj = synth.all_pairs(net.n_elem)
    if case["net"] == "14":                       # a complete list: the single outages come with the pairs
        one = np.arange(net.n_elem, dtype=np.int32)
        ii, jj = np.concatenate([one, ii]), np.concatenate([np.full(one.size, -1, np.int32), jj])
    sel = rng.permutation(ii.size)
    if case["n"] == 1:                            # a question worth asking: the network stays in one piece
        sel = [next(q for q in sel if _connected(net, {int(ii[q]), int(jj[q])}))]
    sel = sel[:case["n"]]
    return ii[sel].astype(np.int32), jj[sel].astype(np.int32)


def _form(case):
    return cs.PREC_MIXED if case["form"] == "mixed" else cs.PREC_FP64


def _rates(seed, shape):
    return np.random.default_rng(seed).uniform(0.01, 1.0, shape)


def _tables(case, seed):
    """Severity tables with the study's share of severe scenarios (17 % of the pairs, 9 % of the singles)."""
    E = case["n_elem"]
    rng = np.random.default_rng([seed, 1])
    s1 = (rng.random(E) < 0.09).astype(np.uint8)
    s2 = (rng.random(E * (E - 1) // 2) < 0.17).astype(np.uint8)
    return s1, s2


def _study():
    """A context that has evaluated the 70 % level of the study: rates are sampled against its tables."""
    if not _STUDY:
        net = _net("118")
        ctx = cs.Context(precision=cs.PREC_MIXED)
        nid = ctx.load_network(net)
        ii, jj = synth.all_pairs(net.n_elem)
        one = np.arange(net.n_elem, dtype=np.int32)
        ei = torch.as_tensor(np.concatenate([one, ii]), device=DEV)
        ej = torch.as_tensor(np.concatenate([np.full(one.size, -1, np.int32), jj]), device=DEV)
        ctx.evaluate_device(nid, 0, ei, ej, ctx.alloc_results(ei.numel(), DEV))
        ctx.sync()
        _STUDY.update(ctx=ctx, nid=nid)
    return _STUDY["ctx"], _STUDY["nid"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "risk":
        s1, s2 = _tables(case, seed)
        lam = _rates(seed, case["n_elem"])
        return dict(kind=kind, n_elem=case["n_elem"], s1=torch.as_tensor(s1, device=DEV),
                    s2=torch.as_tensor(s2, device=DEV), lam=torch.as_tensor(lam, device=DEV),
                    R=torch.empty(case["n_elem"], dtype=torch.float64, device=DEV))
    if kind == "risk_mc":
        ctx, nid = _study()
        lam = torch.as_tensor(_rates(seed, (case["samples"], _net("118").n_elem)), device=DEV)
        return dict(kind=kind, ctx=ctx, nid=nid, lam=lam, R=torch.empty_like(lam))
    net = _net(case["net"])
    ctx = cs.Context(precision=_form(case), main_island=int(case.get("island", False)))
    nid = ctx.load_network(net)
    ei, ej = _outages(case, seed)
    if kind == "serve":
        rng = np.random.default_rng(case["n"])     # the sizes are the case's, the outages the seed's
        cuts = np.sort(rng.choice(np.arange(1, case["n"]), case["requests"] - 1, replace=False))
        lists = list(zip(np.split(ei, cuts), np.split(ej, cuts)))
        return dict(kind=kind, ctx=ctx, nid=nid, level=case["level"], lists=lists)
    return dict(kind=kind, ctx=ctx, nid=nid, level=case["level"], ei=torch.as_tensor(ei, device=DEV),
                ej=torch.as_tensor(ej, device=DEV),
                out=ctx.alloc_results(ei.size, DEV, indices=case["island"], main_island=case["island"]))


def run(state):
    kind = state["kind"]
    if kind == "risk":
        cs.risk_reduce_device(state["n_elem"], state["s1"], state["s2"], state["lam"], state["R"])
        return state["R"]
    if kind == "risk_mc":
        state["ctx"].risk_index_batch(state["nid"], 0, state["lam"], state["R"])
        return state["R"]
    ctx, nid = state["ctx"], state["nid"]
    if kind == "serve":
        ids = [ctx.submit(nid, state["level"], ei, ej) for ei, ej in state["lists"]]
        return [ctx.poll(i, 60_000_000) for i in ids]
    ctx.evaluate_device(nid, state["level"], state["ei"], state["ej"], state["out"])
    return state["out"]


# Per network: interior-point iterations of an ordinary scenario, FP64 operations of one of them (factorisation and
# solve on the network's fill pattern, residual, branch derivatives), order of the state matrix, bytes of its data.
_WORK = {"118": (33, 6.3e5, 269, 1.4e5), "300": (34, 2.1e6, 374, 4.0e5), "14": (18, 5.5e4, 24, 1.5e4)}


def work(case):
    if case["kind"] == "risk":
        E = case["n_elem"]
        return dict(bytes=E * (E - 1) / 2 + 17 * E, flops=float(E * E))
    if case["kind"] == "risk_mc":
        E, s = 240, case["samples"]
        return dict(bytes=16.0 * E * s + E * E / 2, flops=0.2 * E * E * s)
    iters, per_iter, order, data = _WORK[case["net"]]
    n = case["n"]
    return dict(bytes=data + n * (8 + (55 if case.get("island") or case["kind"] == "serve" else 30)),
                flops=n * 0.83 * (iters * per_iter + 10.0 * order ** 3))


# ------------------------------------------------------------------------------- the same in plain numpy ----
def exact(case, seed):
    """Records of the evaluation cases small enough for dense numpy, and the Risk Index of given tables."""
    if case["kind"] == "risk":
        E = case["n_elem"]
        s1, s2 = _tables(case, seed)
        lam = _rates(seed, E)
        ii, jj = np.triu_indices(E, k=1)
        S = np.zeros((E, E))
        S[ii, jj] = s2
        S = S + S.T
        return np.array([math.fsum([lam[i] * s1[i]] + list(2.0 * (lam[i] * lam[S[i] != 0]))) for i in range(E)])
    if case["kind"] != "evaluate" or case["island"] or case["n"] > {"118": 8, "300": 0, "14": 400}[case["net"]]:
        return None                               # the main island's OPF, and what would take minutes
    net = _net(case["net"])
    rows = [_scenario(net, case["level"], int(i), int(j)) for i, j in zip(*_outages(case, seed))]
    out = {k: None for k in ("klass", "severe", "n_islands", "opf_iters")}
    for k, name in enumerate(("cost", "max_re", "min_zeta")):
        out[name] = np.array([r[k] for r in rows])
    return out


def _scenario(net, level, i, j):
    """(cost, largest real part, smallest damping ratio) of one scenario; NaN where it has none."""
    nan3 = (math.nan, math.nan, math.nan)
    gone = {e for e in (i, j) if e >= 0}
    br = np.array([b for b in range(net.n_branch) if b not in gone])
    gen = np.array([g for g in range(net.n_gen) if g + net.n_branch not in gone])
    if not _connected(net, gone):
        return nan3
    point = _opf(net, level, br, gen)
    if point is None:
        return nan3
    cost, V, Sg, Y = point
    lam = np.linalg.eigvals(_state_matrix(net, level, gen, V, Sg, Y))
    return cost, lam.real.max(), (-lam.real / np.abs(lam)).min()


def _opf(net, level, br, gen, tol=1e-8, max_it=50):
    """Primal-dual interior-point AC optimal power flow in polar coordinates, dense."""
    B, nb, ng, nl = net.base_mva, net.n_bus, len(gen), len(br)
    f, t, rows = net.f[br], net.t[br], np.arange(nl)
    ys, tap = 1.0 / (net.r[br] + 1j * net.x[br]), net.tap[br]
    ytt = ys + 0.5j * net.b[br]
    Cf, Ct = np.zeros((nl, nb)), np.zeros((nl, nb))
    Cf[rows, f], Ct[rows, t] = 1.0, 1.0
    Yf = (ytt / tap ** 2)[:, None] * Cf - (ys / tap)[:, None] * Ct
    Yt = ytt[:, None] * Ct - (ys / tap)[:, None] * Cf
    Y = Cf.T @ Yf + Ct.T @ Yt + np.diag((net.Gs + 1j * net.Bs) / B)
    Cg = np.zeros((nb, ng))
    Cg[net.gbus[gen], np.arange(ng)] = 1.0
    Sd = (net.Pd[level] + 1j * net.Qd[level]) / B
    smax2 = (net.rate[br] / B) ** 2
    hi = np.concatenate([net.Vmax, net.Pmax[gen] / B, net.Qmax[gen] / B])
    lo = np.concatenate([net.Vmin, net.Pmin[gen] / B, net.Qmin[gen] / B])
    c2, c1, c0 = net.c2[gen] * B * B, net.c1[gen] * B, net.c0[gen]
    nx, box = 2 * nb + 2 * ng, np.arange(nb, 2 * nb + 2 * ng)
    pg = np.arange(2 * nb, 2 * nb + ng)

    def flow(C, Yx, V, E):                        # S = (C V) conj(Yx V) and its derivatives by (Va, Vm)
        I, U = Yx @ V, C @ V
        d = [np.conj(I)[:, None] * C * D + U[:, None] * np.conj(Yx * D) for D in (1j * V, E)]
        return U * np.conj(I), np.hstack(d)

    def curvature(W, V, E, Vm):                   # second derivatives of Re(V^T W conj(V)) by (Va, Vm)
        a, b = V * (W @ np.conj(V)), np.conj(V) * (W.T @ V)
        G = V[:, None] * W * np.conj(V)
        aa = np.diag(-a - b) + G + G.T
        am = (1j * (np.diag(a) - np.diag(b) + G - G.T)) / Vm
        mm = (G + G.T) / np.outer(Vm, Vm)
        return np.block([[aa.real, am.real], [am.real.T, mm.real]])

    def look(x):
        Va, Vm, P, Q = np.split(x, [nb, 2 * nb, 2 * nb + ng])
        E = np.exp(1j * Va)
        V = Vm * E
        (Sb, dSb), (Sf, dSf), (St, dSt) = (flow(C, M, V, E) for C, M in ((np.eye(nb), Y), (Cf, Yf), (Ct, Yt)))
        g = Sb - Cg @ (P + 1j * Q) + Sd
        Jg = np.zeros((2 * nb + 1, nx))
        Jg[:nb, :2 * nb], Jg[nb:2 * nb, :2 * nb] = dSb.real, dSb.imag
        Jg[:nb, 2 * nb:2 * nb + ng] = Jg[nb:2 * nb, 2 * nb + ng:] = -Cg
        Jg[2 * nb, net.ref_bus] = 1.0
        g = np.concatenate([g.real, g.imag, [Va[net.ref_bus]]])
        h = np.concatenate([np.abs(Sf) ** 2 - smax2, np.abs(St) ** 2 - smax2, x[box] - hi, lo - x[box]])
        Jh = np.zeros((h.size, nx))
        Jh[:nl, :2 * nb] = 2.0 * (np.conj(Sf)[:, None] * dSf).real
        Jh[nl:2 * nl, :2 * nb] = 2.0 * (np.conj(St)[:, None] * dSt).real
        k = 2 * nl + np.arange(box.size)
        Jh[k, box], Jh[k + box.size, box] = 1.0, -1.0
        df = np.zeros(nx)
        df[pg] = 2.0 * c2 * P + c1
        return float(np.sum(c2 * P ** 2 + c1 * P + c0)), df, g, h, Jg, Jh, (V, E, Vm, Sf, dSf, St, dSt)

    x = np.concatenate([np.zeros(nb), np.ones(nb), (net.Pmin + net.Pmax)[gen] / (2 * B), np.zeros(ng)])
    cost, df, g, h, Jg, Jh, at = look(x)
    lam, z, gamma, before = np.zeros(2 * nb + 1), np.maximum(-h, 1.0), 1.0, cost
    mu = gamma / z
    for it in range(max_it + 1):
        Lx = df + Jg.T @ lam + Jh.T @ mu
        top = np.abs(x).max()
        if max(max(np.abs(g).max(), h.max()) / (1 + max(top, np.abs(z).max())),
               np.abs(Lx).max() / (1 + max(np.abs(lam).max(), np.abs(mu).max())), z @ mu / (1 + top),
               abs(cost - before) / (1 + abs(before))) < tol:
            return cost, at[0], x[2 * nb:2 * nb + ng] + 1j * x[2 * nb + ng:], Y
        if it == max_it:
            return None
        V, E, Vm, Sf, dSf, St, dSt = at
        H = curvature((lam[:nb] - 1j * lam[nb:2 * nb])[:, None] * np.conj(Y), V, E, Vm)
        for S, dS, C, Yx, m in ((Sf, dSf, Cf, Yf, mu[:nl]), (St, dSt, Ct, Yt, mu[nl:2 * nl])):
            H += curvature(C.T @ ((2 * m * np.conj(S))[:, None] * np.conj(Yx)), V, E, Vm)
            H += 2 * (np.conj(dS).T @ (m[:, None] * dS)).real
        M = Jh.T @ ((mu / z)[:, None] * Jh)
        M[:2 * nb, :2 * nb] += H
        M[pg, pg] += 2 * c2
        N = Lx + Jh.T @ ((mu * h + gamma) / z)
        K = np.block([[M, Jg.T], [Jg, np.zeros((g.size, g.size))]])
        try:
            step = np.linalg.solve(K, -np.concatenate([N, g]))
        except np.linalg.LinAlgError:
            return None
        if not np.isfinite(step).all():
            return None
        dx, dl = step[:nx], step[nx:]
        dz = -h - z - Jh @ dx
        dm = -mu + (gamma - mu * dz) / z
        ap = min(0.99995 * np.min(-z[dz < 0] / dz[dz < 0], initial=np.inf), 1.0)
        ad = min(0.99995 * np.min(-mu[dm < 0] / dm[dm < 0], initial=np.inf), 1.0)
        x, z, lam, mu = x + ap * dx, z + ap * dz, lam + ad * dl, mu + ad * dm
        gamma, before = 0.1 * (z @ mu) / h.size, cost
        cost, df, g, h, Jg, Jh, at = look(x)


def _state_matrix(net, level, gen, V, Sg, Y):
    """Linearised machines and regulators at the OPF point, angles referred to the first machine."""
    B, m = net.base_mva, len(gen)
    zb = B / net.Pmax[gen]
    xd, xq, xp = net.xd[gen] * zb, net.xq[gen] * zb, net.xdp[gen] * zb
    H, D = net.H[gen] / zb, net.D[gen] / zb
    gb, ws = net.gbus[gen], 2 * math.pi * net.f_hz
    Ybb = Y + np.diag((net.Pd[level] - 1j * net.Qd[level]) / B / np.abs(V) ** 2)
    ym = 1 / (1j * xp)
    Ybb[gb, gb] += ym
    Ybg = np.zeros((net.n_bus, m), complex)
    Ybg[gb, np.arange(m)] = -ym
    Yr = np.diag(ym) - Ybg.T @ np.linalg.solve(Ybb, Ybg)
    I0 = np.conj(Sg / V[gb])
    delta = np.angle(V[gb] + 1j * xq * I0)
    e = np.exp(1j * delta)
    idq, vdq = 1j * I0 / e, 1j * V[gb] / e
    eq, ed = vdq.imag + xp * idq.real, vdq.real - xp * idq.imag
    Ep = (eq - 1j * ed) * e
    I = Yr @ Ep
    i, Vt = 1j * I / e, Ep - 1j * xp * I
    A = np.zeros((5 * m, 5 * m))
    k = 5 * np.arange(m)
    for s, dE in ((0, 1j * Ep), (2, e), (3, -1j * e)):          # d E' by delta, e'q, e'd of each machine
        dI = Yr * dE
        di = 1j * dI / e[:, None]
        dV = -1j * xp[:, None] * dI + np.diag(dE)
        dPe = ed[:, None] * di.real + eq[:, None] * di.imag
        if s == 0:                                              # the frame turns with delta
            turn = np.diag(-1j * i)
            di = di + turn
            dPe = dPe + np.diag(ed * np.diag(turn).real + eq * np.diag(turn).imag)
        dPe = dPe + (np.diag(i.imag) if s == 2 else np.diag(i.real) if s == 3 else 0.0)
        c = k + s
        A[np.ix_(k + 1, c)] = -dPe / (2 * H)[:, None]
        A[np.ix_(k + 2, c)] = -((xd - xp) / net.Td0p[gen])[:, None] * di.real
        A[np.ix_(k + 3, c)] = ((xq - xp) / net.Tq0p[gen])[:, None] * di.imag
        A[np.ix_(k + 4, c)] = -(net.KA[gen] / net.TA[gen] / np.abs(Vt))[:, None] * (np.conj(Vt)[:, None] * dV).real
    A[k, k + 1] = ws
    A[k + 1, k + 1] -= D / (2 * H)
    A[k + 2, k + 2] -= 1 / net.Td0p[gen]
    A[k + 2, k + 4] += 1 / net.Td0p[gen]
    A[k + 3, k + 3] -= 1 / net.Tq0p[gen]
    A[k + 4, k + 4] -= 1 / net.TA[gen]
    A[k[1:]] -= A[0]                                            # angles relative to the first machine's
    return A[1:, 1:]
