"""Timed cases of the library: what its users have it do, through the public package.

Every case builds its inputs on the GPU from a seed: two sheets of the manifold-like
family the tests and the benchmark use,

    A(theta, s) = g(s) T(theta) + F(s),   T a six-term trigonometric sum, g = 1 + s or
                  4**s, F three cubic folds,
    B(theta, s) = A(theta + c0, 1 - s) + h (sin(P (theta - theta0)) n1 + sin(Q pi (s - s0)) n2),

so that B crosses A transversally near a lattice of 2P x Q sites and stays a few faces
from it in between (a hard broad phase, as in the benchmark).  Kinds:

    search     tms.search, default (mixed) or plain FP64 parameters
    host       tms.search_host: coordinates in pinned host memory, hits back to it
    batched    tms.search_batched over mesh pairs of uneven sizes
    layers     LayerSweep.search: the half-layer pairs of two globalized meshes
    backward   tms.backward: vertex and family-parameter gradients of a search's hits
    refine     tms.refine: damped Newton from approximate connections
    continue   tms.continue_branches: those connections through the family parameter
    translate  tms.theta_translate of every column of a coordinate array
    align      tms.phase_align of pairs of circles
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import torch

import paper_2109_14814_gb300 as tms

TWO_PI = 2.0 * math.pi
F64 = torch.float64
DEV = "cuda"


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------

def _search(name, na, ma, nb, mb, n_theta, n_s, manifold=True, **more):
    return dict(name=name, kind="search", na=na, ma=ma, nb=nb, mb=mb, n_theta=n_theta, n_s=n_s,
                manifold=manifold, periodic=True, plain=False, **more)


def listed():
    big = dict(na=4096, ma=512, nb=4096, mb=512, n_theta=256, n_s=46, manifold=True)
    return [
        # the smallest call: a coarse pair, as in interactive use and in tests; latency only
        _search("search 64x32", 64, 32, 64, 32, 6, 1, manifold=False),
        # an ordinary half-layer pair with few crossings
        _search("search 1024x256", 1024, 256, 1024, 256, 16, 6),
        # the benchmark's size and density: 4.19M triangles a side, about 12,000 crossings
        dict(_search("search 4096x512", 4096, 512, 4096, 512, 256, 46)),
        # the plain FP64 form (what the mixed form is checked against), on uneven, odd sizes
        dict(_search("search plain 1019x253", 1019, 253, 771, 331, 16, 6), plain=True),
        # end to end from host memory: a driver that globalizes on the CPU
        dict(big, name="host 4096x512", kind="host", periodic=True),
        # a continuation sweep: many pairs of uneven sizes in one call
        dict(name="batched 64 pairs", kind="batched", pairs=64, sizes=4, n_lo=128, n_hi=2048, m_lo=32, m_hi=512),
        # the method of layers at the paper's shapes: 112 half-layer pairs of 1024x35 against 2048x35
        dict(name="layers 14", kind="layers", na=1024, nb=2048, n_max=14, per_layer=34),
        # one differentiation step on the hits of an ordinary pair
        dict(name="backward 1024x256", kind="backward", na=1024, ma=256, nb=1024, mb=256, n_theta=64, n_s=10),
        # the refinement of a dense search's hits
        dict(name="refine 12000", kind="refine", n=12000),
        # their continuation through fifty values of the family parameter
        dict(name="continue 12000x50", kind="continue", n=12000, steps=50),
        # the globalization step: every column of a mesh translated by its own shift
        dict(name="translate 4x1025x2048", kind="translate", c=4, m=1025, n=2048, derivative=False),
        # phase alignment of a family of tori, consecutive circles
        dict(name="align 16x4x4096", kind="align", a=16, c=4, n=4096),
    ]


def _spread(rng, lo, hi):
    """A whole number, even over the logarithm of its range."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "plain", "host", "batched", "layers", "backward", "refine",
                       "continue", "translate", "align"])
    if kind in ("search", "plain", "host", "backward"):
        top_n, top_m = (4096, 512) if kind in ("search", "host") else (1200, 331)
        na, nb = _spread(rng, 64, top_n), _spread(rng, 64, top_n)
        ma, mb = _spread(rng, 24, top_m), _spread(rng, 24, top_m)
        dense = rng.random() < 0.5
        c = dict(kind=kind, na=na, ma=ma, nb=nb, mb=mb, n_theta=max(2, nb // (16 if dense else 64) & ~1),
                 n_s=max(1, (mb - 1) // (11 if dense else 42)))
        if kind != "backward":
            c.update(manifold=True, periodic=rng.random() < 0.8)
        if kind in ("search", "plain"):
            c.update(kind="search", plain=kind == "plain")
        return c
    if kind == "batched":
        return dict(kind="batched", pairs=_spread(rng, 4, 64), sizes=rng.randrange(1 << 20), n_lo=128, n_hi=2048,
                    m_lo=32, m_hi=512)
    if kind == "layers":
        return dict(kind="layers", na=_spread(rng, 200, 1024), nb=_spread(rng, 200, 2048), n_max=rng.randint(2, 14),
                    per_layer=rng.randint(9, 34))
    if kind == "refine":
        return dict(kind="refine", n=_spread(rng, 40, 12000))
    if kind == "continue":
        return dict(kind="continue", n=_spread(rng, 40, 12000), steps=_spread(rng, 5, 50))
    if kind == "translate":
        n = 1 << rng.randint(6, 12)
        c = rng.randint(1, 4)
        return dict(kind="translate", c=c, m=_spread(rng, 16, min(2050, 4 * 1025 * 2048 // (4096 * c))), n=n,
                    derivative=rng.random() < 0.4)
    return dict(kind="align", a=_spread(rng, 1, 16), c=rng.randint(2, 4), n=_spread(rng, 200, 4096))


# ----------------------------------------------------------------------------
# the sheets
# ----------------------------------------------------------------------------

def _family(seed, manifold):
    """Coefficients of the sheet pair, from the seed alone (CPU generator)."""
    g = torch.Generator().manual_seed(seed)
    f = SimpleNamespace()

    def randn(*shape):
        return torch.randn(*shape, generator=g, dtype=F64)

    def rand(*shape):
        return torch.rand(*shape, generator=g, dtype=F64)

    f.ca, f.cb = randn(6, 4), randn(6, 4)
    f.dca, f.dcb = 0.25 * randn(6, 4), 0.25 * randn(6, 4)
    folds = 3 if manifold else 0
    f.stretch, f.lam = ("exp", 4.0) if manifold else ("linear", 4.0)
    f.fold_roots = 0.8 * rand(folds, 3) + 0.1
    d = randn(folds, 4)
    f.fold_dir = d / d.norm(dim=1, keepdim=True).clamp_min(1e-12)
    f.fold_amp = 12.0 * (0.5 * rand(folds) + 0.75)
    v = randn(2, 4)
    v = v / v.norm(dim=1, keepdim=True)
    f.v1, f.v2 = v[0], v[1]
    f.c0 = float(rand(1)) * TWO_PI
    f.u_theta, f.u_s = float(rand(1)), float(rand(1))
    f.alpha, f.alpha_ref, f.reg = 0.5, 0.5, 0.25
    return f


def _trig(f, theta, alpha):
    """T, T', T'' and dT/dalpha at the angles theta, each (4, n)."""
    k = torch.arange(1, 7, dtype=F64, device=theta.device)
    c, s = torch.cos(k[:, None] * theta), torch.sin(k[:, None] * theta)
    da, db = f.dca.to(theta), f.dcb.to(theta)
    a, b = f.ca.to(theta) + alpha * da, f.cb.to(theta) + alpha * db
    kk = k[:, None]
    return ((a / kk).T @ c + (b / kk).T @ s, b.T @ c - a.T @ s, -((a * kk).T @ c + (b * kk).T @ s),
            (da / kk).T @ c + (db / kk).T @ s)


def _stretch(f, s):
    if f.stretch == "linear":
        return 1.0 + s, torch.ones_like(s), torch.zeros_like(s)
    ln = math.log(f.lam)
    g = torch.exp(ln * s)
    return g, ln * g, ln * ln * g


def _folds(f, s):
    """F, F', F'' at s, each (4, n)."""
    out = [torch.zeros(4, s.numel(), dtype=F64, device=s.device) for _ in range(3)]
    for amp, r, e in zip(f.fold_amp.tolist(), f.fold_roots.tolist(), f.fold_dir):
        d0, d1, d2 = s - r[0], s - r[1], s - r[2]
        e = amp * e.to(s)[:, None]
        out[0] += e * (d0 * d1 * d2)
        out[1] += e * (d1 * d2 + d0 * d2 + d0 * d1)
        out[2] += e * (2.0 * (d0 + d1 + d2))
    return out


def _grid_sheet(f, theta, s, alpha):
    """The sheet on a grid and its partials in theta, s and alpha, each (4, m, n)."""
    T, T1, _, Ta = _trig(f, theta, alpha)
    g, g1, _ = _stretch(f, s)
    F, F1, _ = _folds(f, s)
    g, g1 = g[None, :, None], g1[None, :, None]
    return (g * T[:, None] + F[:, :, None], g * T1[:, None], g1 * T[:, None] + F1[:, :, None], g * Ta[:, None])


def _frame(f, xt, xs):
    """The crossing term's two directions: v1 and v2 less their part along (xt, xs)."""
    g11, g12, g22 = (xt * xt).sum(0), (xt * xs).sum(0), (xs * xs).sum(0)
    eps = f.reg * 0.5 * (g11 + g22)
    a, c = g11 + eps, g22 + eps
    det = a * c - g12 * g12
    out = []
    for v in (f.v1, f.v2):
        v = v.to(xt).reshape([4] + [1] * (xt.dim() - 1))
        j1, j2 = (xt * v).sum(0), (xs * v).sum(0)
        out.append(v - xt * ((c * j1 - g12 * j2) / det) - xs * ((a * j2 - g12 * j1) / det))
    return out


def _angles(n):
    return torch.arange(n, dtype=F64, device=DEV) * (TWO_PI / n)


def _pair(f, na, ma, nb, mb, n_theta, n_s, alpha=0.5):
    """Vertex grids (4, M, N) of A and B and their alpha derivatives; sets the
    crossing term's amplitude, frequencies and origin in f."""
    sa = torch.linspace(0.0, 1.0, ma, dtype=F64, device=DEV)
    sb = torch.linspace(0.0, 1.0, mb, dtype=F64, device=DEV)
    XA, xt, xs, dA = _grid_sheet(f, _angles(na), sa, alpha)
    wide = torch.maximum(xt.norm(dim=0).mean() * (TWO_PI / na), xs.norm(dim=0).mean() / (ma - 1))
    f.P, f.Q = n_theta / 2.0, float(n_s)
    f.h_amp = float(wide) * min(nb / n_theta, (mb - 1) / n_s) / math.pi
    f.theta0 = f.u_theta * 0.5 * math.pi / f.P + 0.25 * TWO_PI / nb
    f.s0 = (0.5 + 0.5 * f.u_s) / n_s
    th = _angles(nb)
    XB, xt, xs, dB = _grid_sheet(f, th + f.c0, 1.0 - sb, alpha)
    n1, n2 = _frame(f, xt, xs)
    XB = XB + f.h_amp * (torch.sin(f.P * (th - f.theta0))[None, None, :] * n1
                         + torch.sin(f.Q * math.pi * (sb - f.s0))[None, :, None] * n2)
    return XA.contiguous(), sa.cpu(), XB.contiguous(), sb.cpu(), dA.contiguous(), dB.contiguous()


def _hits(h, st):
    """The number of hits and every field of the caller's record buffer (zero past the hits)."""
    r = tms.Hits(st["out"])
    out = dict(count=len(h), ids=r.raw.view(torch.int32)[:, :4], z=r.z, P=r.P, params=r.params, rho=r.rho,
               margin=r.margin)
    if h.offsets is not None:
        out["offsets"] = h.offsets
    return out


def _out(records, device=DEV):
    return torch.zeros((records, tms.HIT_BYTES), dtype=torch.uint8, device=device)


def _records(c):
    """Room for the hits: a few times the crossing sites."""
    if c["kind"] in ("batched", "layers"):
        return 1 << 15
    if c["kind"] == "host":
        return 3 * c["n_theta"] * c["n_s"] // 2 + 4096
    return 1 << (2 * c["n_theta"] * c["n_s"] + 8000).bit_length()


def _batch_sizes(c):
    r = random.Random(c["sizes"])
    return [(r.randint(c["n_lo"], c["n_hi"]), r.randint(c["m_lo"], c["m_hi"]), r.randint(c["n_lo"], c["n_hi"]),
             r.randint(c["m_lo"], c["m_hi"])) for _ in range(c["pairs"])]


def _layer_s(n_lo, n_max, per_layer):
    """s values of a globalized mesh: half-layers [0.01 2^(n-1), 0.01 2^n], n = n_lo..n_max,
    their mirror images, and three columns of the fundamental domain."""
    pos = [0.01 * 2.0 ** (n - 1 + j / per_layer) for n in range(n_lo, n_max + 1)
           for j in range(per_layer + (n == n_max))]
    mid = [pos[0] * (2.0 * i / 4 - 1.0) for i in range(1, 4)]
    return torch.tensor([-v for v in reversed(pos)] + mid + pos, dtype=F64)


def _plain(c):
    return dict(precision=0, narrow_filter=0) if c["plain"] else {}


# ----------------------------------------------------------------------------
# approximate connections (refine, continue)
# ----------------------------------------------------------------------------

def _evaluate(f, x, alpha_u):
    """f(x) = W_A - W_B (n, 4) and its Jacobian (n, 4, 4) at x = (theta_u, s_u, theta_s, s_s)."""
    tu, su, tb, s_ = x.unbind(1)
    T, T1, _, _ = _trig_each(f, tu, alpha_u)
    g, g1, _ = _stretch(f, su)
    F, F1, _ = _folds(f, su)
    wa, wat, was = g * T + F, g * T1, g1 * T + F1
    th, s1 = tb + f.c0, 1.0 - s_
    T, T1, T2, _ = _trig_each(f, th, f.alpha)
    g, g1, g2 = _stretch(f, s1)
    F, F1, F2 = _folds(f, s1)
    S, St, Ss = g * T + F, g * T1, g1 * T + F1
    Stt, Sts, Sss = g * T2, g1 * T1, g2 * T + F2
    # the frame and its derivatives in theta and s' by the product rule
    n, nt, ns = [], [], []
    g11, g12, g22 = (St * St).sum(0), (St * Ss).sum(0), (Ss * Ss).sum(0)

    def solve(a, b, c, r1, r2):
        det = a * c - b * b
        return (c * r1 - b * r2) / det, (a * r2 - b * r1) / det

    e = f.reg * 0.5
    a, b, c = g11 + e * (g11 + g22), g12, g22 + e * (g11 + g22)
    for v in (f.v1, f.v2):
        v = v.to(x)[:, None]
        y1, y2 = solve(a, b, c, (St * v).sum(0), (Ss * v).sum(0))
        n.append(v - St * y1 - Ss * y2)
        for dt, ds, to in ((Stt, Sts, nt), (Sts, Sss, ns)):
            d11, d22 = 2.0 * (St * dt).sum(0), 2.0 * (Ss * ds).sum(0)
            d12 = (dt * Ss).sum(0) + (St * ds).sum(0)
            da, dc = d11 + e * (d11 + d22), d22 + e * (d11 + d22)
            z1, z2 = solve(a, b, c, (dt * v).sum(0) - (da * y1 + d12 * y2), (ds * v).sum(0) - (d12 * y1 + dc * y2))
            to.append(-(dt * y1 + ds * y2) - (St * z1 + Ss * z2))
    q = f.Q * math.pi
    p1, p2 = f.P * (tb - f.theta0), q * (s_ - f.s0)
    H = f.h_amp * (torch.sin(p1) * n[0] + torch.sin(p2) * n[1])
    Ht = f.h_amp * (f.P * torch.cos(p1) * n[0] + torch.sin(p1) * nt[0] + torch.sin(p2) * nt[1])
    Hs = f.h_amp * (-torch.sin(p1) * ns[0] + q * torch.cos(p2) * n[1] - torch.sin(p2) * ns[1])
    J = torch.stack([wat.T, was.T, -(St + Ht).T, -(Hs - Ss).T], dim=2)
    return (wa - (S + H)).T, J


def _trig_each(f, theta, alpha):
    """_trig with one family parameter per angle (or one for all)."""
    T = _trig(f, theta, 0.0)
    if not torch.is_tensor(alpha):
        return _trig(f, theta, alpha)
    g = SimpleNamespace(ca=f.dca, cb=f.dcb, dca=f.dca, dcb=f.dcb)
    D = _trig(g, theta, 0.0)
    return tuple(t + alpha * d for t, d in zip(T, D))


def _rho(J):
    return torch.linalg.det(J) / J.norm(dim=1).prod(dim=1)


def _connections(c, seed):
    """A sheet pair and n approximate connections: lattice crossings of the sheets, displaced
    by about what a search's (theta, s) estimates are off.  Crossings far from a tangency
    only: from the others the damped iteration may wander, and where a wandering one ends
    is a matter of rounding."""
    f = _family(seed, True)
    _pair(f, 1024, 128, 1024, 128, 256, 46)
    g = torch.Generator().manual_seed(seed + 1)
    i, j = torch.arange(256, dtype=F64), torch.arange(46, dtype=F64)
    th, s = (f.theta0 + i * math.pi / f.P) % TWO_PI, f.s0 + j / f.Q
    s = s[(s > 0.02) & (s < 0.98)]
    th, s = (v.reshape(-1) for v in torch.meshgrid(th, s, indexing="ij"))
    x = torch.stack([(th + f.c0) % TWO_PI, 1.0 - s, th, s], dim=1).to(DEV)
    _, J = _evaluate(f, x, f.alpha)
    x = x[_rho(J).abs() > 0.15].cpu()
    pick = torch.randint(0, x.shape[0], (c["n"],), generator=g)
    x = x[pick] + 2e-4 * torch.randn(c["n"], 4, generator=g, dtype=F64)
    return f, x.to(DEV).contiguous()


STEP = 5e-5      # of the family parameter
NEWTON = dict(max_iter=60)


# ----------------------------------------------------------------------------
# prepare and run
# ----------------------------------------------------------------------------

def prepare(case, seed):
    c, kind = case, case["kind"]
    st = dict(case=c)
    if kind in ("search", "host", "backward"):
        f = _family(seed, c.get("manifold", True))
        XA, sa, XB, sb, dA, dB = _pair(f, c["na"], c["ma"], c["nb"], c["mb"], c["n_theta"], c["n_s"])
        per = c.get("periodic", True)
        st.update(A=tms.Mesh(XA, sa, per), B=tms.Mesh(XB, sb, per))
        records = _records(c)
        if kind == "search":
            st["out"] = _out(records)
        elif kind == "host":
            st.update(XA=XA.cpu().pin_memory(), XB=XB.cpu().pin_memory(),
                      out=_out(records, "cpu").pin_memory())
        else:
            h = tms.search(st["A"], st["B"], out=_out(records))
            g = torch.Generator(device=DEV).manual_seed(seed)
            n = len(h)
            st.update(hits=h, dA=dA, dB=dB, gA=torch.zeros_like(XA), gB=torch.zeros_like(XB),
                      gP=torch.randn(n, 4, generator=g, dtype=F64, device=DEV),
                      gZ=torch.randn(n, 4, generator=g, dtype=F64, device=DEV),
                      ga=torch.zeros(records, dtype=F64, device=DEV))
    elif kind == "batched":
        sizes = _batch_sizes(c)
        f = _family(seed, True)
        As, Bs = [], []
        for p, (na, ma, nb, mb) in enumerate(sizes):
            XA, sa, XB, sb, _, _ = _pair(f, na, ma, nb, mb, 8, 2, alpha=p / max(1, len(sizes) - 1))
            As.append(tms.Mesh(XA, sa))
            Bs.append(tms.Mesh(XB, sb))
        st.update(As=As, Bs=Bs, out=_out(_records(c)),
                  offsets=torch.empty(len(sizes) + 1, dtype=torch.int64, device=DEV))
    elif kind == "layers":
        f = _family(seed, True)
        sa, sb = _layer_s(1, c["n_max"], c["per_layer"]), _layer_s(0, c["n_max"], c["per_layer"])
        XA, _, XB, _, _, _ = _pair(f, c["na"], sa.numel(), c["nb"], sb.numel(), 16, 12)
        A, B = tms.Mesh(XA, sa), tms.Mesh(XB, sb)
        pairs = tms.layer_pairs(sa, 0.01, 2.0, sb, 0.01, 0.5, c["n_max"])
        st.update(A=A, B=B, sweep=tms.LayerSweep(A, B, pairs), out=_out(_records(c)),
                  offsets=torch.empty(len(pairs) + 1, dtype=torch.int64, device=DEV))
    elif kind in ("refine", "continue"):
        f, x = _connections(c, seed)
        st.update(surface=tms.surface_pair(f), x=x)
        if kind == "continue":
            st["alphas"] = _alphas(c, f)
    elif kind == "translate":
        g = torch.Generator(device=DEV).manual_seed(seed)
        X = torch.randn(c["c"], c["m"], c["n"], generator=g, dtype=F64, device=DEV)
        st.update(X=X, rho=torch.rand(c["m"], generator=g, dtype=F64, device=DEV) * 6.0 - 3.0, out=torch.empty_like(X))
    else:
        st["Wr"], st["Wp"] = _circles(c, seed)
    return st


def _alphas(c, f):
    return f.alpha + STEP * torch.arange(1, c["steps"] + 1, dtype=F64, device=DEV)


def _circles(c, seed):
    """Consecutive circles of a family: the second is the first sampled from another
    phase and slightly deformed."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    k = torch.arange(1, 7, dtype=F64, device=DEV)
    th = _angles(c["n"])
    a = torch.randn(2, c["a"], c["c"], 6, generator=g, dtype=F64, device=DEV) / k
    b = a + 1e-3 * torch.randn(a.shape, generator=g, dtype=F64, device=DEV)
    ph = torch.rand(c["a"], 1, 1, 1, generator=g, dtype=F64, device=DEV) * TWO_PI
    out = []
    for u, t in ((b, th + ph), (a, th + 0.0 * ph)):
        kt = k[:, None] * t                       # (a, 1, 6, n)
        out.append(((u[0][..., None] * torch.cos(kt)) + (u[1][..., None] * torch.sin(kt))).sum(2).contiguous())
    return out


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "search":
        return _hits(tms.search(st["A"], st["B"], out=st["out"], **_plain(c)), st)
    if kind == "host":
        h = tms.search_host(st["A"], st["B"], st["XA"], st["XB"], out=st["out"])
        st["out"][len(h):].zero_()      # the call may leave anything past the hits
        return _hits(h, st)
    if kind == "batched":
        return _hits(tms.search_batched(st["As"], st["Bs"], out=st["out"], offsets=st["offsets"]), st)
    if kind == "layers":
        return _hits(st["sweep"].search(out=st["out"], offsets=st["offsets"]), st)
    if kind == "backward":
        gA, gB = st["gA"].zero_(), st["gB"].zero_()
        tms.backward(st["A"], st["B"], st["hits"], gP=st["gP"], gZ=st["gZ"], gradA=gA, gradB=gB, dA_dalpha=st["dA"],
                     dB_dalpha=st["dB"], galpha=st["ga"])
        return dict(gA=gA, gB=gB, galpha=st["ga"])
    if kind == "refine":
        r = tms.refine(st["surface"], st["x"])
        return dict(x=r.x, fnorm=r.fnorm, rho=r.rho, iters=r.iters, status=r.status)
    if kind == "continue":
        r = tms.continue_branches(st["surface"], st["x"], st["alphas"], max_jump=0.05, **NEWTON)
        return dict(x=r.x, fnorm=r.fnorm, rho=r.rho, iters=r.iters, status=r.status)
    if kind == "translate":
        return tms.theta_translate(st["X"], st["rho"], derivative=c["derivative"], out=st["out"])
    shift, cost = tms.phase_align(st["Wr"], st["Wp"])
    return dict(shift=shift, cost=cost)


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------

EVALUATION = 695 + 128 * 6 + 66 * 3      # flops of one evaluation of f, Df and the update


def work(case):
    c, kind = case, case["kind"]
    if kind in ("search", "host"):
        # every vertex read once, every hit written once (about one per crossing site),
        # one 4 x 4 solve a hit
        hits = c["n_theta"] * c["n_s"]
        return dict(bytes=32 * (c["na"] * c["ma"] + c["nb"] * c["mb"]) + 128 * hits, flops=200 * hits)
    if kind == "batched":
        s = _batch_sizes(c)
        return dict(bytes=32 * sum(a * b + p * q for a, b, p, q in s) + 128 * 16 * len(s), flops=200 * 16 * len(s))
    if kind == "layers":
        cols_a, cols_b = 2 * c["n_max"] * c["per_layer"] + 5, 2 * (c["n_max"] + 1) * c["per_layer"] + 5
        return dict(bytes=32 * (c["na"] * cols_a + c["nb"] * cols_b) + 128 * 16 * 12, flops=200 * 16 * 12)
    if kind == "backward":
        # both gradient arrays written once; the hits, their vertices and alpha derivatives read
        hits = c["n_theta"] * c["n_s"]
        return dict(bytes=32 * (c["na"] * c["ma"] + c["nb"] * c["mb"]) + hits * (128 + 64 + 8 + 12 * 32),
                    flops=500 * hits)
    if kind == "refine":
        return dict(bytes=c["n"] * (32 + 32 + 16 + 8), flops=c["n"] * 24 * EVALUATION)
    if kind == "continue":
        return dict(bytes=c["n"] * 32 + c["n"] * (c["steps"] + 1) * 56,
                    flops=c["n"] * (24 + 20 * c["steps"]) * EVALUATION)
    if kind == "translate":
        # two real rows per complex transform, there and back, and the multiplier
        n, rows = c["n"], c["c"] * c["m"]
        return dict(bytes=16 * rows * n + 8 * c["m"], flops=rows / 2 * (2 * 5 * n * math.log2(n) + 6 * n))
    return dict(bytes=8 * c["a"] * c["n"] * (2 * c["c"] + 1), flops=c["a"] * c["n"] ** 2 * (3 * c["c"] + 1))


# ----------------------------------------------------------------------------
# the same answers in 64 bits from torch alone
# ----------------------------------------------------------------------------

def _boxes(v, per):
    """Boxes of the quads of a vertex grid (4, m, n): lo and hi (4, m - 1, quads a row)."""
    w = torch.cat([v, v[:, :, :1]], dim=2) if per else v
    a, b, c, d = w[:, :-1, :-1], w[:, :-1, 1:], w[:, 1:, :-1], w[:, 1:, 1:]
    return (torch.minimum(torch.minimum(a, b), torch.minimum(c, d)),
            torch.maximum(torch.maximum(a, b), torch.maximum(c, d)))


def _blocks(lo, hi, k, i):
    """Boxes of blocks of k x i quads; rows and columns past the end hold nothing."""
    m, n = lo.shape[1:]
    pad = (0, -n % i, 0, -m % k)
    lo = torch.nn.functional.pad(lo, pad, value=math.inf)
    hi = torch.nn.functional.pad(hi, pad, value=-math.inf)
    M, N = lo.shape[1] // k, lo.shape[2] // i
    return (lo.reshape(4, M, k, N, i).amin((2, 4)).reshape(4, -1), hi.reshape(4, M, k, N, i).amax((2, 4)).reshape(4, -1),
            lo, hi, N)


def _meet(al, ah, bl, bh):
    ok = None
    for d in range(4):
        t = (al[d] <= bh[d]) & (bl[d] <= ah[d])
        ok = t if ok is None else ok & t
    return ok


def _quad_pairs(XA, XB, per):
    """Every pair of quads whose boxes meet, as quad ids k * N + i: blocks first, then the
    quads of the blocks that meet."""
    K, I = 4, 8
    loA, hiA = _boxes(XA, per)
    loB, hiB = _boxes(XB, per)
    pa, qa, la, ha, na = _blocks(loA, hiA, K, I)
    pb, qb, lb, hb, nb = _blocks(loB, hiB, K, I)
    u, v = [], []
    step = max(1, (1 << 27) // pb.shape[1])
    for at in range(0, pa.shape[1], step):
        e = min(pa.shape[1], at + step)
        ia, ib = _meet(pa[:, at:e, None], qa[:, at:e, None], pb[:, None], qb[:, None]).nonzero(as_tuple=True)
        u.append(ia + at)
        v.append(ib)
    u, v = torch.cat(u), torch.cat(v)
    k = torch.arange(K * I, device=DEV) // I
    i = torch.arange(K * I, device=DEV) % I
    A, B = [], []
    step = 1 << 15
    for at in range(0, u.numel(), step):
        p, q = u[at:at + step, None], v[at:at + step, None]
        ka, ia, kb, ib = p // na * K + k, p % na * I + i, q // nb * K + k, q % nb * I + i
        w = _meet(la[:, ka, ia][:, :, :, None], ha[:, ka, ia][:, :, :, None], lb[:, kb, ib][:, :, None, :],
                  hb[:, kb, ib][:, :, None, :]).nonzero(as_tuple=True)
        A.append(ka[w[0], w[1]] * XA.shape[2] + ia[w[0], w[1]])
        B.append(kb[w[0], w[2]] * XB.shape[2] + ib[w[0], w[2]])
    empty = torch.zeros(0, dtype=torch.int64, device=DEV)
    return (torch.cat(A), torch.cat(B)) if A else (empty, empty)


def _vertices(X, t):
    """The three vertices (3, 4, n) of triangles t, and their quads' row and column."""
    N = X.shape[2]
    q, second = t // 2, (t % 2).bool()
    k, i = q // N, q % N
    ip = (i + 1) % N
    ii = (torch.where(second, i, ip), torch.where(second, ip, i), torch.where(second, ip, i))
    kk = (torch.where(second, k + 1, k), torch.where(second, k + 1, k), torch.where(second, k, k + 1))
    return torch.stack([X[:, b, a] for a, b in zip(ii, kk)]), k, i, second


def _estimate(s, N, k, i, second, u, v):
    d = TWO_PI / N
    lo = i.to(F64) * d
    hi = lo + d
    th = torch.where(second, u * lo + (1 - u) * hi, (1 - u) * lo + u * hi)
    sv = torch.where(second, v * s[k] + (1 - v) * s[k + 1], (1 - v) * s[k] + v * s[k + 1])
    return th % TWO_PI, sv


def _exact_search(XA, sa, XB, sb, per):
    """Sorted hits of one pair: (triA, triB, z, P, params, rho, margin)."""
    qa, qb = _quad_pairs(XA, XB, per)
    got = []
    for at in range(0, qa.numel(), 1 << 19):
        for sub in range(4):
            ta, tb = 2 * qa[at:at + (1 << 19)] + sub % 2, 2 * qb[at:at + (1 << 19)] + sub // 2
            x, ka, ia, ea = _vertices(XA, ta)
            y, kb, ib, eb = _vertices(XB, tb)
            M = torch.stack([x[0] - x[1], x[2] - x[1], y[1] - y[0], y[1] - y[2]], dim=0).permute(2, 1, 0)
            z = torch.linalg.solve_ex(M, (y[1] - x[1]).T.unsqueeze(2))[0].squeeze(2)
            a, b, c, d = z.unbind(1)
            m = torch.stack([a, b, c, d, 1 - a - b, 1 - c - d]).amin(0)
            w = (torch.isfinite(z).all(1) & (m >= -1e-12)).nonzero().squeeze(1)
            if not w.numel():
                continue
            M, z, m, x = M[w], z[w], m[w], x[:, :, w]
            a, b, c, d = z.unbind(1)
            P = (x[1] + a * (x[0] - x[1]) + b * (x[2] - x[1])).T
            tu = _estimate(sa, XA.shape[2], ka[w], ia[w], ea[w], a, b)
            ts = _estimate(sb, XB.shape[2], kb[w], ib[w], eb[w], c, d)
            got.append((ta[w], tb[w], z, P, torch.stack(tu + ts, dim=1),
                        (torch.linalg.det(M) / M.norm(dim=1).prod(1)).abs(), m))
    if not got:
        return None
    got = [torch.cat(v) for v in zip(*got)]
    order = torch.argsort(got[0] * (1 << 31) + got[1])
    return [v[order] for v in got]


def _laid_out(lists, c):
    lists = [g for g in lists if g is not None]
    out = dict(count=None, ids=None)
    for j, (name, shape) in enumerate((("z", (4,)), ("P", (4,)), ("params", (4,)), ("rho", ()), ("margin", ()))):
        out[name] = torch.zeros((_records(c),) + shape, dtype=F64, device=DEV)
        if lists:
            v = torch.cat([g[j + 2] for g in lists])
            out[name][:v.shape[0]] = v
    return out


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("search", "host"):
        f = _family(seed, c["manifold"])
        XA, sa, XB, sb, _, _ = _pair(f, c["na"], c["ma"], c["nb"], c["mb"], c["n_theta"], c["n_s"])
        return _laid_out([_exact_search(XA, sa.to(DEV), XB, sb.to(DEV), c["periodic"])], c)
    if kind == "batched":
        sizes = _batch_sizes(c)
        f = _family(seed, True)
        got = []
        for p, (na, ma, nb, mb) in enumerate(sizes):
            XA, sa, XB, sb, _, _ = _pair(f, na, ma, nb, mb, 8, 2, alpha=p / max(1, len(sizes) - 1))
            got.append(_exact_search(XA, sa.to(DEV), XB, sb.to(DEV), True))
        return _laid_out(got, c)
    if kind == "layers":
        f = _family(seed, True)
        sa, sb = _layer_s(1, c["n_max"], c["per_layer"]), _layer_s(0, c["n_max"], c["per_layer"])
        XA, _, XB, _, _, _ = _pair(f, c["na"], sa.numel(), c["nb"], sb.numel(), 16, 12)
        sa, sb = sa.to(DEV), sb.to(DEV)

        def columns(s, n, sign):
            """The vertex columns of half-layer n of that sign."""
            w = ((s * sign > 0.01 * 2.0 ** (n - 1) * (1 - 1e-9)) & (s * sign < 0.01 * 2.0 ** n * (1 + 1e-9)))
            w = w.nonzero().squeeze(1)
            return slice(int(w[0]), int(w[-1]) + 1)

        got = []
        for n in range(1, c["n_max"] + 1):
            for su in (1, -1):
                for m in (n, n - 1):
                    for ss in (1, -1):
                        a, b = columns(sa, n, su), columns(sb, m, ss)
                        got.append(_exact_search(XA[:, a], sa[a], XB[:, b], sb[b], True))
        return _laid_out(got, c)
    if kind == "backward":
        st = prepare(c, seed)
        ids = st["hits"].raw.view(torch.int32)[:, :2].to(torch.int64)
        x = _vertices(st["A"].X, ids[:, 0])[0].permute(2, 0, 1).contiguous().requires_grad_()
        y = _vertices(st["B"].X, ids[:, 1])[0].permute(2, 0, 1).contiguous().requires_grad_()
        M = torch.stack([x[:, 0] - x[:, 1], x[:, 2] - x[:, 1], y[:, 1] - y[:, 0], y[:, 1] - y[:, 2]], dim=2)
        z = torch.linalg.solve(M, (y[:, 1] - x[:, 1]).unsqueeze(2)).squeeze(2)
        P = x[:, 1] + z[:, 0:1] * (x[:, 0] - x[:, 1]) + z[:, 1:2] * (x[:, 2] - x[:, 1])
        gx, gy = torch.autograd.grad((P * st["gP"]).sum() + (z * st["gZ"]).sum(), (x, y))
        out, ga = [], 0.0
        for X, dX, t, g in ((st["A"].X, st["dA"], ids[:, 0], gx), (st["B"].X, st["dB"], ids[:, 1], gy)):
            number = torch.arange(X[0].numel(), device=DEV).reshape(X[0].shape)
            at = _vertices(number[None], t)[0].squeeze(1)                     # (3, n)
            G = torch.zeros(4, X[0].numel(), dtype=F64, device=DEV)
            for j in range(3):
                G.index_add_(1, at[j], g[:, j].T.contiguous())
                ga = ga + (dX.reshape(4, -1)[:, at[j]] * g[:, j].T).sum(0)
            out.append(G.reshape(X.shape))
        galpha = torch.zeros(_records(c), dtype=F64, device=DEV)
        galpha[:ga.numel()] = ga
        return dict(gA=out[0], gB=out[1], galpha=galpha)
    if kind in ("refine", "continue"):
        return _exact_newton(c, seed)
    if kind == "translate":
        st = prepare(c, seed)
        n = c["n"]
        k = torch.fft.fftfreq(n, 1.0 / n, dtype=F64, device=DEV)
        e = torch.exp(1j * k * st["rho"][:, None])
        nyquist = torch.cos(n / 2 * st["rho"])
        if c["derivative"]:
            e, nyquist = e * 1j * k, 0.0 * nyquist
        e[:, n // 2] = nyquist.to(e.dtype)
        return torch.fft.ifft(torch.fft.fft(st["X"], dim=-1) * e, dim=-1).real
    Wr, Wp = _circles(c, seed)
    cost = torch.stack([(torch.roll(Wr, -m, dims=2) - Wp).norm(dim=1).sum(1) for m in range(c["n"])], dim=1)
    return dict(shift=None, cost=cost)


def _wrapped(x):
    y = x.clone()
    y[:, 0::2] %= TWO_PI
    return y


def _exact_newton(c, seed):
    """The damped iteration (and the walk) of every seed at once, each at its own step."""
    f, x0 = _connections(c, seed)
    walk = c["kind"] == "continue"
    n, K = c["n"], c["steps"] if walk else 0
    alphas = torch.cat([torch.tensor([f.alpha], dtype=F64, device=DEV), _alphas(c, f)]) if walk else \
        torch.tensor([f.alpha], dtype=F64, device=DEV)
    out = dict(x=torch.full((n, K + 1, 4), math.nan, dtype=F64, device=DEV),
               fnorm=torch.full((n, K + 1), math.nan, dtype=F64, device=DEV),
               rho=torch.full((n, K + 1), math.nan, dtype=F64, device=DEV))
    most = NEWTON["max_iter"] if walk else 200
    live = torch.arange(n, device=DEV)
    j = torch.zeros(n, dtype=torch.int64, device=DEV)
    it = torch.zeros(n, dtype=torch.int64, device=DEV)
    x = x0.clone()
    while live.numel():
        xl = x[live]
        r, J = _evaluate(f, xl, alphas[j[live]] if walk else f.alpha)
        fn = r.norm(dim=1)
        done = (fn <= 1e-10) | (it[live] >= most)
        x[live] = torch.where(done[:, None], xl, xl - 0.5 * torch.linalg.solve_ex(J, r.unsqueeze(2))[0].squeeze(2))
        it[live] += 1
        if done.any():
            w = live[done]
            at = j[w]
            out["x"][w, at] = _wrapped(xl[done])
            out["fnorm"][w, at] = fn[done]
            out["rho"][w, at] = _rho(J[done])
            w = w[(at < K) & (fn[done] <= 1e-10)]
            if w.numel():                          # the next step's predictor
                j[w] += 1
                it[w] = 0
                p1 = out["x"][w, j[w] - 1]
                p2 = out["x"][w, (j[w] - 2).clamp_min(0)]
                d = p1 - p2
                d[:, 0::2] -= TWO_PI * torch.round(d[:, 0::2] / TWO_PI)
                x[w] = torch.where((j[w] >= 2)[:, None], p1 + d, p1)
            stay = ~done
            stay[done] = torch.isin(live[done], w)
            live = live[stay]
    x, fnorm, rho = out["x"], out["fnorm"], out["rho"]
    return dict(x=x if walk else x[:, 0], fnorm=fnorm if walk else fnorm[:, 0], rho=rho if walk else rho[:, 0],
                iters=None, status=None)
