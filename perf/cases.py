"""What a user of the CC3 triples library runs, as cases to be timed and checked.

A case is one call of the public entry points on a problem of the seeded
synthetic kind that the tests and the benchmark use: orbital energies in the
usual ranges, integrals from Cholesky-like vectors, MP2 doubles, normalised
trial vectors.  The context (the staged problem) is what a program keeps
between calls; `run` is one evaluation on it.  `exact` is the same quantity
from plain FP64 torch tensor algebra, one occupied triple at a time.

Kinds: `omega` (triples residual), `jacobian` (right transformation), `left`
(its transpose), `density` (one-electron densities), `host` (a residual from
host arrays: upload, evaluation, download), `serve` (a burst of mixed requests
through the serving loop).
"""
import math

import numpy as np
import torch

import paper_2007_01088_gb300 as cc3

OMEGA_W = 0.25  # frequency of the trial vectors, below every denominator


def listed():
    return [
        # the smallest residual of the configurations: latency and launches
        dict(name="omega_small", kind="omega", prec="split", no=5, nv=30),
        # the FP64 path, used to validate the split one and for small systems
        dict(name="omega_fp64", kind="omega", prec="fp64", no=6, nv=48),
        # an ordinary molecule of the serving stream (odd sizes, ragged tiles)
        dict(name="omega_medium", kind="omega", prec="split", no=11, nv=87),
        # the mid-size configuration, the whole triple loop
        dict(name="omega_mid160", kind="omega", prec="split", no=16, nv=160),
        # the L-proline-sized problem, a share of its triple loop (as a rank of
        # a sharded evaluation has it), with its near-degenerate virtual cluster
        dict(name="omega_proline_part", kind="omega", prec="split", no=22, nv=250,
             naux=700, ndeg=10, ntri=96),
        # residual with T1-transformed (non-symmetric) integrals, reproducible sums
        dict(name="omega_general", kind="omega", prec="split", no=8, nv=72, general=True,
             det=True),
        # an excited-state iteration of a small molecule: few vectors
        dict(name="jacobian_small", kind="jacobian", prec="split", no=6, nv=45, nvec=2),
        # core-excited states: the batched Jacobian under core-valence separation
        dict(name="jacobian_cvs", kind="jacobian", prec="split", no=16, nv=128, nvec=3, core=1),
        # left excited states of an ordinary molecule
        dict(name="left", kind="left", prec="split", no=9, nv=81, nvec=2),
        # densities at the benchmark's size
        dict(name="density", kind="density", prec="split", no=12, nv=120),
        # one residual end to end from host arrays (a program that hands over
        # new integrals each time)
        dict(name="host_residual", kind="host", prec="split", no=8, nv=64),
        # a burst of small and ordinary requests through the serving loop
        dict(name="serve_burst", kind="serve", prec="split", no=9, nv=66, nreq=6, slots=4),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def draw(rng):
    kind = rng.choice(["omega", "omega", "omega", "jacobian", "jacobian", "left", "density",
                       "host", "serve"])
    no = _logint(rng, 4, 18)
    nv = min(210, int(round(no * rng.uniform(6.0, 10.0))))
    c = dict(kind=kind, prec="split", no=no, nv=nv)
    if kind == "omega":
        form = rng.choice(["plain", "plain", "general", "det", "fp64"])
        if form == "general":
            c["general"] = True
        elif form == "det":
            c["det"] = True
        elif form == "fp64":
            c.update(prec="fp64", no=min(no, 8), nv=min(nv, 64))
        if no >= 14:
            c["ntri"] = rng.randint(40, 240)
    elif kind == "jacobian":
        c.update(nvec=rng.randint(1, 6))
        if no >= 11:
            c.update(core=rng.randint(1, 2), nvec=rng.randint(1, 3), nv=min(nv, 130))
    elif kind == "left":
        c.update(no=min(no, 11), nv=min(nv, 96), nvec=rng.randint(1, 3))
    elif kind == "density":
        c.update(no=min(no, 12), nv=min(nv, 120))
    elif kind == "host":
        c.update(no=min(no, 10), nv=min(nv, 90))
    else:
        c.update(no=min(no, 10), nv=min(nv, 70), nreq=rng.randint(3, 8), slots=rng.choice([2, 4]))
    return c


# ---- inputs -----------------------------------------------------------------
class Problem:
    """The fields that the library's Context and Server read."""


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _rnd(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _uni(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _block(L, p, q, r, s):
    """(pq|rs) = sum_J L[J,p,q] L[J,r,s]"""
    A, B = L[:, p, q], L[:, r, s]
    out = A.reshape(A.shape[0], -1).T @ B.reshape(B.shape[0], -1)
    return out.reshape(A.shape[1], A.shape[2], B.shape[1], B.shape[2])


def _problem(no, nv, seed, naux=None, ndeg=0):
    g = _gen(seed)
    n = no + nv
    naux = naux or 3 * n
    p = Problem()
    p.no, p.nv = no, nv
    p.eps_o = _uni(g, -1.5, -0.3, no).sort().values
    p.eps_v = _uni(g, 0.1, 3.0, nv).sort().values
    if ndeg:
        p.eps_v[:ndeg] = p.eps_v[0] + _uni(g, 0.0, 1e-3, ndeg)
        p.eps_v = p.eps_v.sort().values
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    up = torch.triu(0.05 * _rnd(g, naux, n, n) * torch.exp(-(i[:, None] - i[None, :]).abs() / 20.0))
    L = p.chol_L = (up + torch.triu(up, 1).transpose(1, 2)).contiguous()
    o, v = slice(0, no), slice(no, n)
    p.g_vvvo = _block(L, v, v, v, o).contiguous()
    p.g_ooov = _block(L, o, o, o, v).contiguous()
    p.g_ovov = _block(L, o, v, o, v).contiguous()
    p.F_ov = 1e-3 * _rnd(g, no, nv)
    d = (p.eps_o[:, None, None, None] + p.eps_o[None, :, None, None]
         - p.eps_v[None, None, :, None] - p.eps_v[None, None, None, :])
    p.t2 = (p.g_ovov.permute(0, 2, 1, 3) / d).contiguous()
    return p


def _vectors(no, nv, nvec, seed):
    g = _gen(seed + 7919)
    r1 = 0.1 * _rnd(g, nvec, no, nv)
    x = 0.01 * _rnd(g, nvec, no, no, nv, nv)
    r2 = 0.5 * (x + x.permute(0, 2, 1, 4, 3))
    s = (r1.square().sum((1, 2)) + r2.square().sum((1, 2, 3, 4))).sqrt()
    return ((r1 / s[:, None, None]).contiguous(),
            (r2 / s[:, None, None, None, None]).contiguous())


def _blocks(p, seed=None):
    """The five blocks as the residual reads them; with a seed, as a T1
    transformation with small random amplitudes leaves them (non-symmetric)."""
    no, n = p.no, p.no + p.nv
    o, v = slice(0, no), slice(no, n)
    L = p.chol_L
    F = p.F_ov
    if seed is not None:
        t1 = 0.02 * _rnd(_gen(seed + 104729), no, p.nv)
        x = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        x[v, o] = t1.T                                  # x[a, i] = t^a_i
        one = torch.eye(n, dtype=torch.float64, device="cuda")
        L = (one - x) @ L @ (one + x.T).T
        L = L.contiguous()
    return dict(vvvo=_block(L, v, v, v, o).contiguous(), oovo=_block(L, o, o, v, o).contiguous(),
                ooov=_block(L, o, o, o, v).contiguous(), ovov=_block(L, o, v, o, v).contiguous(),
                vvov=_block(L, v, v, o, v).contiguous(), F_ov=F)


def _all_triples(no):
    return [(i, j, k) for i in range(no) for j in range(i + 1) for k in range(j + 1)
            if not i == j == k]


def _triples(case):
    """The occupied triples of the loop: all, a seeded share, or those with a
    core orbital."""
    t = _all_triples(case["no"])
    if case.get("core"):
        t = [x for x in t if min(x) < case["core"]]
    n = case.get("ntri")
    if n and n < len(t):
        at = np.random.default_rng(5).choice(len(t), n, replace=False)
        t = [t[i] for i in sorted(at)]
    return t


def _weight(triples):
    return sum(6 if i != j != k else 3 for i, j, k in triples)


def _prec(case):
    return cc3.CC3_FP64 if case["prec"] == "fp64" else cc3.CC3_SPLIT_BF16


def _request_shapes(case):
    """The requests of a burst: sizes from the case's own down to about half,
    residuals and Jacobians in turn."""
    out = []
    for q in range(case["nreq"]):
        f = 1.0 - 0.1 * (q % 6)
        no = max(3, int(round(case["no"] * f)))
        nv = max(12, int(round(case["nv"] * f)))
        out.append((no, nv, 0 if q % 2 == 0 else 1 + q % 3))
    return out


def _host(p):
    h = Problem()
    h.no, h.nv = p.no, p.nv
    for n in ("eps_o", "eps_v", "t2", "g_vvvo", "g_ooov", "g_ovov", "F_ov", "chol_L"):
        setattr(h, n, getattr(p, n).cpu().numpy())
    return h


class _State:
    ctx = None
    server = None

    def __del__(self):
        if self.ctx is not None:
            cc3.cc3_ctx_destroy(self.ctx)
            self.ctx = None
        if self.server is not None:
            self.server.stop()
            self.server = None


def prepare(case, seed):
    s = _State()
    s.case = case
    no, nv = case["no"], case["nv"]
    if case["kind"] == "serve":
        s.reqs = []
        for q, (qo, qv, nvec) in enumerate(_request_shapes(case)):
            p = _host(_problem(qo, qv, seed * 64 + q))
            R = None
            if nvec:
                R = [x.cpu().numpy() for x in _vectors(qo, qv, nvec, seed * 64 + q)]
            s.reqs.append((p, R))
        s.server = cc3.Server(hbm_budget_bytes=16 << 30, max_slots=case["slots"])
        return s
    p = _problem(no, nv, seed, case.get("naux"), case.get("ndeg", 0))
    if case["kind"] == "host":
        s.host = _host(p)
        return s
    flags = cc3.CC3_DEVICE_PTRS | (cc3.CC3_DETERMINISTIC if case.get("det") else 0)
    torch.cuda.synchronize()  # the inputs are complete before another stream reads them
    if case.get("general"):
        b = _blocks(p, seed)
        torch.cuda.synchronize()
        s.ctx = cc3.cc3_ctx_create_general(no, nv, p.eps_o, p.eps_v, p.t2, b["vvvo"], b["oovo"],
                                           b["ooov"], b["ovov"], b["vvov"], b["F_ov"], flags)
    else:
        s.ctx = cc3.cc3_ctx_create(no, nv, p.eps_o, p.eps_v, p.t2, p.g_vvvo, p.g_ooov, p.g_ovov,
                                   p.F_ov, p.chol_L, p.chol_L.shape[0], flags)
    if case.get("ntri") or case.get("core"):
        cc3.cc3_ctx_set_triples(s.ctx, _triples(case))
    if case["kind"] != "omega":
        s.x1, s.x2 = _vectors(no, nv, case.get("nvec", 1), seed)
    return s


def _new(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


def run(s):
    case, no, nv = s.case, s.case["no"], s.case["nv"]
    prec, kind = _prec(case), case["kind"]
    if kind == "omega":
        o1, o2, e = _new(no, nv), _new(no, no, nv, nv), _new(1)
        cc3.cc3_omega_triples(s.ctx, prec, o1, o2, e)
        return dict(omega1=o1, omega2=o2, energy=e)
    if kind in ("jacobian", "left"):
        n = case["nvec"]
        y1, y2 = _new(n, no, nv), _new(n, no, no, nv, nv)
        f = cc3.cc3_jacobian_triples if kind == "jacobian" else cc3.cc3_left_jacobian_triples
        f(s.ctx, prec, n, [OMEGA_W] * n, s.x1, s.x2, y1, y2)
        return dict(singles=y1, doubles=y2)
    if kind == "density":
        doo, dov, dvv = _new(no, no), _new(no, nv), _new(nv, nv)
        cc3.cc3_density_triples(s.ctx, prec, OMEGA_W, s.x1[0], s.x2[0], doo, dov, dvv)
        return dict(oo=doo, ov=dov, vv=dvv)
    if kind == "host":
        ctx = cc3.Context(s.host)
        o1, o2, e = ctx.omega(prec)
        ctx.close()
        return dict(omega1=o1, omega2=o2, energy=e)
    tickets = []
    for p, R in s.reqs:
        if R is None:
            tickets.append(s.server.submit_omega(p, prec))
        else:
            tickets.append(s.server.submit_jacobian(p, R[0], R[1], OMEGA_W, prec))
    out = []
    for t in tickets:
        status, y = s.server.wait(t)
        if status != 0:
            raise RuntimeError("request failed: %s" % cc3.cc3_strerror(status))
        out.append(y)
    return out


# ---- the work of a pass -----------------------------------------------------
def _in_values(no, nv, naux):
    return no * no * nv * nv * 2 + no * nv**3 + no**3 * nv + naux * (no + nv) ** 2


def work(case):
    no, nv, kind = case["no"], case["nv"], case["kind"]
    if kind == "serve":
        by = fl = 0.0
        for qo, qv, nvec in _request_shapes(case):
            nt2 = qo * qo * qv * qv
            by += 8.0 * (_in_values(qo, qv, 3 * (qo + qv) if nvec else 0) + max(1, 2 * nvec) * nt2)
            fl += (8.0 * nvec if nvec else 4.0) * qv**4 * (qo**3 - qo)
        return dict(bytes=by, flops=fl)
    w, nvec, nt2 = _weight(_triples(case)), case.get("nvec", 1), no * no * nv * nv
    naux = (case.get("naux") or 3 * (no + nv)) if kind in ("jacobian", "left") else 0
    vals = _in_values(no, nv, naux)
    if case.get("general"):  # vvov and oovo are blocks of their own
        vals += no * nv**3 + no**3 * nv
    if kind in ("omega", "host"):
        return dict(bytes=8.0 * (vals + nt2), flops=4.0 * nv**4 * w)
    if kind in ("jacobian", "left"):
        return dict(bytes=8.0 * (vals + 2 * nvec * nt2), flops=8.0 * nvec * nv**4 * w)
    # densities: the occupied loop, and the occupied-occupied block by pairs
    return dict(bytes=8.0 * (vals + nt2 + nv * nv),
                flops=6.0 * nv**4 * (no**3 - no) + no**3 * (no + 1.0) * nv**3)


def tolerance(case):
    """FP64 sums of ~nv^2 terms in another order, or FP64 operands carried as
    48-bit fixed point with one scale per tensor and double-float sums."""
    if case["prec"] == "fp64":
        return {"rel": 1e-13, "max": 1e-11}
    return {"rel": 4e-11, "max": 2e-9}


# ---- the same quantities in plain FP64 --------------------------------------
_PERMS = ((0, 1, 2), (1, 0, 2), (2, 1, 0), (0, 2, 1), (1, 2, 0), (2, 0, 1))


def _inverse(m):
    return tuple(m.index(i) for i in range(3))


def _distinct(ijk):
    seen, out = set(), []
    for m in _PERMS:
        key = tuple(ijk[x] for x in m)
        if key not in seen and not ijk[0] == ijk[1] == ijk[2]:
            seen.add(key)
            out.append(m)
    return out


class _Exact:
    """Plain tensor algebra for one problem; B(p,q,r) builders are passed in."""

    def __init__(self, p, blocks):
        self.p, self.b = p, blocks
        self.no, self.nv = p.no, p.nv
        # the occupied index of each virtual-heavy block outermost
        self.vvvo = blocks["vvvo"].permute(3, 1, 0, 2).contiguous()   # [r][d][y][z]
        self.vvov = blocks["vvov"].permute(2, 0, 1, 3).contiguous()   # [r][d][y][z]

    def denom(self, ijk, w):
        v, o = self.p.eps_v, self.p.eps_o
        return w - (v[:, None, None] + v[None, :, None] + v[None, None, :]
                    - (o[ijk[0]] + o[ijk[1]] + o[ijk[2]]))

    def build(self, ijk, w, term):
        """sum over the six permutations of term(p,q,r)[x][y][z], divided."""
        tot, made = 0.0, {}
        for m in _PERMS:
            key = tuple(ijk[x] for x in m)
            if key not in made:
                made[key] = term(*key)
            tot = tot + made[key].permute(_inverse(m))
        return tot / self.denom(ijk, w)

    def w_term(self, t, vvvo_r, oovo):
        def term(p, q, r):
            nv = self.nv
            x = (t[p, q] @ vvvo_r[r].reshape(nv, nv * nv)).reshape(nv, nv, nv)
            return x - torch.einsum("lxy,lz->xyz", t[p], oovo[:, q, :, r])
        return term

    def l_term(self, l1, lt):
        b = self.b

        def term(p, q, r):
            nv = self.nv
            x = (lt[p, q] @ self.vvov[r].reshape(nv, nv * nv)).reshape(nv, nv, nv)
            x = x - torch.einsum("lxy,lz->xyz", lt[p], b["ooov"][q, :, r, :])
            x = x + l1[p][:, None, None] * b["ovov"][q, :, r, :][None]
            return x + lt[p, q][:, :, None] * b["F_ov"][r][None, None, :]
        return term

    def tau(self, ijk):
        return self.build(ijk, 0.0, self.w_term(self.p.t2, self.vvvo, self.b["oovo"]))

    @staticmethod
    def contra(t):
        return (4.0 * t - 2.0 * t.permute(0, 2, 1) - 2.0 * t.permute(2, 1, 0)
                - 2.0 * t.permute(1, 0, 2) + t.permute(2, 0, 1) + t.permute(1, 2, 0))

    def contract(self, ijk, tt, b, vvov_r, o1, ot):
        nv = self.nv
        for m in _distinct(ijk):
            p, q, r = (ijk[x] for x in m)
            v = tt.permute(m).contiguous()
            vm = v.reshape(nv, nv * nv)
            if b.get("ovov") is not None:
                o1[p] += vm @ b["ovov"][q, :, r, :].reshape(-1)
            ot[p, q] += v @ b["F_ov"][r] + vm @ vvov_r[r].reshape(nv, nv * nv).T
            ot[p] -= torch.einsum("xyz,lz->lxy", v, b["ooov"][q, :, r, :])


def _back(x):
    y = (2.0 * x + x.transpose(2, 3)) / 3.0
    return y + y.permute(1, 0, 3, 2)


def _zeros(*shape):
    return torch.zeros(*shape, dtype=torch.float64, device="cuda")


def _exact_omega(p, blocks, triples):
    X = _Exact(p, blocks)
    o1, ot = _zeros(p.no, p.nv), _zeros(p.no, p.no, p.nv, p.nv)
    for ijk in triples:
        X.contract(ijk, X.contra(X.tau(ijk)), blocks, X.vvov, o1, ot)
    return dict(omega1=o1, omega2=_back(ot), energy=(p.t2 * ot).sum().reshape(1))


def _kinds(p):
    no, n = p.no, p.no + p.nv
    o, v = slice(0, no), slice(no, n)
    L = p.chol_L
    return (_block(L, o, v, v, o), _block(L, v, v, o, o), _block(L, o, o, o, o),
            _block(L, o, o, v, v), _block(L, o, v, o, v), L[:, v, v].contiguous())


def _exact_jacobian(p, x1, x2, triples):
    """The derivative of the residual along (R1, R2), R3 with the frequency in
    its denominator: the first-order blocks of a T1 transformation."""
    g = _blocks(p)
    X = _Exact(p, g)
    ovvo, vvoo, oooo, oovv, ovov, Lvv = _kinds(p)
    E = torch.einsum
    dressed = []
    n = x1.shape[0]
    for R in x1:
        M = E("Jce,ke->Jck", Lvv, R)
        h = dict(
            vvvo=(-E("lb,ldck->bdck", R, ovvo) - E("bdlk,lc->bdck", vvoo, R)
                  + E("Jbd,Jck->bdck", Lvv, M)),
            oovo=(E("jd,ldck->ljck", R, ovvo) - E("ljmk,mc->ljck", oooo, R)
                  + E("ljcd,kd->ljck", oovv, R)),
            ooov=E("jdkc,ld->jlkc", ovov, R), vvov=-E("ld,lbkc->dbkc", R, ovov),
            F_ov=2.0 * E("kcld,ld->kc", ovov, R) - E("kdlc,ld->kc", ovov, R))
        h["vvvo_r"] = h["vvvo"].permute(3, 1, 0, 2).contiguous()
        h["vvov_r"] = h["vvov"].permute(2, 0, 1, 3).contiguous()
        dressed.append(h)
    o1, ot = _zeros(n, p.no, p.nv), _zeros(n, p.no, p.no, p.nv, p.nv)
    for ijk in triples:
        tt = X.contra(X.tau(ijk))
        for u in range(n):
            h = dressed[u]
            a = X.w_term(x2[u], X.vvvo, g["oovo"])
            b = X.w_term(p.t2, h["vvvo_r"], h["oovo"])
            r3 = X.contra(X.build(ijk, OMEGA_W, lambda *k: a(*k) + b(*k)))
            X.contract(ijk, r3, g, X.vvov, o1[u], ot[u])
            X.contract(ijk, tt, h, h["vvov_r"], o1[u], ot[u])
    return dict(singles=o1, doubles=torch.stack([_back(t) for t in ot]))


def _exact_left(p, x1, x2, triples):
    """The transpose of _exact_jacobian, factor by factor."""
    g = _blocks(p)
    X = _Exact(p, g)
    ovvo, vvoo, oooo, oovv, ovov, Lvv = _kinds(p)
    E = torch.einsum
    no, nv, n = p.no, p.nv, x1.shape[0]
    s1, s2 = _zeros(n, no, nv), _zeros(n, no, no, nv, nv)
    tts = {ijk: X.contra(X.tau(ijk)) for ijk in triples}
    for u in range(n):
        l1, lt = x1[u], _back(x2[u])
        d2, Q = _zeros(no, no, nv, nv), _zeros(no, nv)
        G, H = _zeros(nv, nv, nv, no), _zeros(no, no, nv, no)
        for ijk in triples:
            tt = tts[ijk]
            l3 = X.contra(X.build(ijk, OMEGA_W, X.l_term(l1, lt)))
            for m in _distinct(ijk):
                i, j, k = (ijk[x] for x in m)
                v = tt.permute(m).contiguous()
                Q[k] += E("xy,xyz->z", lt[i, j], v)
                s1[u] -= E("lxy,xyd->ld", lt[i], v @ ovov[j, :, k, :].T)
                s1[u] -= E("xyz,lyz->xl", v, ovov[:, :, k, :]).T @ lt[i, j]
                w = l3.permute(m).contiguous()
                wm = w.reshape(nv, nv * nv)
                d2[i, j] += wm @ X.vvvo[k].reshape(nv, nv * nv).T
                d2[i] -= E("xyz,lz->lxy", w, g["oovo"][:, j, :, k])
                G[:, :, :, k] += E("xyz,xd->ydz", w, p.t2[i, j])
                H[:, j, :, k] += E("lxy,xyz->lz", p.t2[i], w)
        s1[u] += 2.0 * E("kc,kcld->ld", Q, ovov) - E("kc,kdlc->ld", Q, ovov)
        s1[u] -= E("ldck,bdck->lb", ovvo, G) + E("bdlk,bdck->lc", vvoo, G)
        s1[u] += E("Jck,Jce->ke", E("Jbd,bdck->Jck", Lvv, G), Lvv)
        # the occupied blocks enter W with a minus sign
        s1[u] += (-E("ljck,ldck->jd", H, ovvo) + E("ljmk,ljck->mc", oooo, H)
                  - E("ljck,ljcd->kd", H, oovv))
        s2[u] = 0.5 * (d2 + d2.permute(1, 0, 3, 2))
    return dict(singles=s1, doubles=s2)


def _exact_density(p, l1, l2):
    g = _blocks(p)
    X = _Exact(p, g)
    no, nv, E = p.no, p.nv, torch.einsum
    lt = _back(l2)
    doo, dov, dvv = _zeros(no, no), _zeros(no, nv), _zeros(nv, nv)
    Y = _zeros(nv, no, no, no)
    tau, lc = {}, {}
    for i in range(no):
        for j in range(i + 1):
            for k in range(j + 1):
                ijk = (i, j, k)
                tau[ijk] = X.tau(ijk)
                lc[ijk] = X.contra(X.build(ijk, OMEGA_W, X.l_term(l1, lt)))
                tt = X.contra(tau[ijk])
                for m in _distinct(ijk):
                    a, b, c = (ijk[x] for x in m)
                    v, w = tt.permute(m).contiguous(), lc[ijk].permute(m).contiguous()
                    Y[:, :, a, c] += E("xyz,lxy->zl", w, p.t2[:, b])
                    dov[c] += E("xy,xyz->z", lt[a, b], v)
                    t = tau[ijk].permute(m).contiguous()
                    dvv += 0.5 * w.reshape(nv * nv, nv).T @ t.reshape(nv * nv, nv)

    def view(store, key):
        """store of the sorted triple, axes in the order of `key`."""
        order = sorted(range(3), key=lambda x: -key[x])
        srt = tuple(key[x] for x in order)
        return store[srt].permute(_inverse(tuple(order)))

    for i in range(no):
        for j in range(i + 1):
            lw = torch.stack([view(lc, (i, j, k)).reshape(-1) for k in range(no)])
            tw = torch.stack([view(tau, (i, j, k)).reshape(-1) for k in range(no)])
            doo -= (1.0 if i != j else 0.5) * tw @ lw.T
    dov -= E("clik,kicd->ld", Y, p.t2)
    return dict(oo=doo, ov=dov, vv=dvv)


def exact(case, seed):
    no, nv, kind = case["no"], case["nv"], case["kind"]
    if kind == "serve":
        out = []
        for q, (qo, qv, nvec) in enumerate(_request_shapes(case)):
            p = _problem(qo, qv, seed * 64 + q)
            if nvec:
                y = _exact_jacobian(p, *_vectors(qo, qv, nvec, seed * 64 + q), _all_triples(qo))
                out.append((y["singles"].cpu().numpy(), y["doubles"].cpu().numpy()))
            else:
                y = _exact_omega(p, _blocks(p), _all_triples(qo))
                out.append(tuple(y[k].cpu().numpy() for k in ("omega1", "omega2", "energy")))
        return out
    p = _problem(no, nv, seed, case.get("naux"), case.get("ndeg", 0))
    triples = _triples(case)
    if kind in ("omega", "host"):
        y = _exact_omega(p, _blocks(p, seed if case.get("general") else None), triples)
        return y if kind == "omega" else {k: v.cpu().numpy() for k, v in y.items()}
    x1, x2 = _vectors(no, nv, case.get("nvec", 1), seed)
    if kind == "jacobian":
        return _exact_jacobian(p, x1, x2, triples)
    if kind == "left":
        return _exact_left(p, x1, x2, triples)
    return _exact_density(p, x1[0], x2[0])
