"""The work that users of this framework have it do, as cases that can be timed.

Each case is one pass through the public binding (paper_2206_06495_gb300.rbffd
and .wake) on node sets of the paper's kinds: the jittered staggered
cavity (Section 5.1) and the graded cylinder wake (Section 5.2).  The kinds:

  apply      one operator application y = alpha D x + beta y (Section 2.2)
  weights    one stencil search and weight build of an operator family (Section 2)
  condition  the condition numbers of a family's local systems (Section 4.2)
  step       fractional steps of a closed cavity in one call (Section 3)
  wake       fractional steps of the open flow past a cylinder (Section 5.2)
  ensemble   fractional steps of many cavities that share one node set

A pass on the same state gives the same result each time: the calls that
advance a state in place start from copies of the prepared fields.
"""
import math

import numpy as np
import torch

from paper_2206_06495_gb300 import nodesets as ns
from paper_2206_06495_gb300 import rbffd as R
from paper_2206_06495_gb300 import wake

FAMILIES = {"vv": (R.OP_DX | R.OP_DY | R.OP_LAP), "pv": (R.OP_DX | R.OP_DY),
            "pp": (R.OP_DX | R.OP_DY | R.OP_LAP), "vp": (R.OP_DX | R.OP_DY)}


def listed():
    return [
        # a post-processing derivative of the smallest configuration (40 x 40
        # P-nodes, 4,641 V-nodes): launch latency
        dict(name="apply f64 4.6k", kind="apply", n=40, family="vv", dtype="f64",
             alpha=1.0, beta=0.0, stencil=28, m=7, q=3),
        # an FP32 operator accumulated into an existing field, ragged row count
        dict(name="apply f32 300k", kind="apply", n=317, family="vv", dtype="f32",
             alpha=-0.5, beta=1.0, stencil=28, m=7, q=3),
        # the V -> V operator of the million-P-node cavity (2,996,001 rows)
        dict(name="apply f64 3M", kind="apply", n=1000, family="vv", dtype="f64",
             alpha=1.0, beta=0.0, stencil=28, m=7, q=3),
        # the operator set-up of the smallest configuration, P -> V family
        dict(name="weights vp 4.6k", kind="weights", n=40, family="vp", stencil=28, m=7, q=3),
        # a million stencils, D_x, D_y and the Laplacian in one build
        dict(name="weights vv 1.1M", kind="weights", n=600, family="vv", stencil=28, m=7, q=3),
        # the study behind the choice of the polynomial degree (Section 4.2)
        dict(name="condition pp 100k", kind="condition", n=316, family="pp", stencil=28, m=7,
             q=3),
        # the plain method's configuration: Re 100, dt 2e-3, 1,600 P-nodes
        dict(name="step f64 1.6k", kind="step", n=40, steps=20, precision="f64", Re=100.0,
             dt=2e-3, tol=1e-12),
        # the node count of the ensemble and gradient studies, one flow
        dict(name="step f64 100k", kind="step", n=316, steps=8, precision="f64", Re=1000.0,
             dt=5e-4, tol=1e-11),
        # the large cavity at Re 10^4, FP64
        dict(name="step f64 1M", kind="step", n=1000, steps=6, precision="f64", Re=1e4,
             dt=2e-4, tol=1e-11),
        # the cavity at Re 1000 with 250,000 P-nodes, mixed precision, one step
        # per call (a program that records every step)
        dict(name="step mixed 250k", kind="step", n=500, steps=1, precision="mixed", Re=1000.0,
             dt=4e-4, tol=1e-12),
        # flow past a cylinder, the short domain, from the impulsive start
        dict(name="wake f64 2.6k", kind="wake", domain="short", h_wall=0.06, steps=4,
             precision="f64", Re=100.0, dt=5e-3, tol=1e-12),
        # 64 cavities of different Reynolds numbers and lid speeds in one call
        dict(name="ensemble 64 x 100k", kind="ensemble", n=316, members=64, steps=1, dt=2.5e-4,
             tol=1e-11),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "weights", "weights", "condition", "step", "step",
                       "step", "wake", "ensemble"])
    if kind in ("apply", "weights"):
        n, m, q = rng.choice([(28, 7, 3), (28, 7, 3), (28, 7, 4), (21, 5, 2)])
        family = rng.choice(sorted(FAMILIES))
        if kind == "weights":
            return dict(kind=kind, n=_log_int(rng, 20, 400), family=family, stencil=n, m=m, q=q)
        return dict(kind=kind, n=_log_int(rng, 20, 900), family=family,
                    dtype=rng.choice(["f64", "f32"]), alpha=round(rng.uniform(-2, 2), 3),
                    beta=rng.choice([0.0, 1.0, -0.5]), stencil=n, m=m, q=q)
    if kind == "condition":
        return dict(kind=kind, n=_log_int(rng, 20, 250), family=rng.choice(["pp", "vv"]),
                    stencil=28, m=7, q=rng.choice([3, 4]))
    if kind == "step":  # P-lattice CFL 0.08 to 0.2 at unit lid speed, cell Re up to about 20
        precision = rng.choice(["f64", "f64", "mixed"])
        n = _log_int(rng, 24, 700 if precision == "f64" else 450)
        return dict(kind=kind, n=n, steps=rng.randint(2, 6) if precision == "f64" else 1,
                    precision=precision,
                    Re=float(rng.choice([100, 400, 1000] if n < 80 else [1000, 3200, 10000])),
                    dt=round(rng.uniform(0.08, 0.2) / (n - 1), 7),
                    tol=1e-11 if precision == "f64" else 1e-12)
    if kind == "wake":
        domain, h = rng.choice([("short", 0.06), ("short", 0.07), ("long", 0.05), ("long", 0.07)])
        return dict(kind=kind, domain=domain, h_wall=h, steps=rng.randint(1, 3),
                    precision="f64", Re=100.0, dt=round(rng.uniform(3e-3, 5e-3), 5), tol=1e-12)
    n = _log_int(rng, 24, 130)
    return dict(kind="ensemble", n=n, members=rng.choice([4, 8, 16, 32, 64]),
                steps=1, dt=round(0.08 / (n - 1), 6), tol=1e-11)


# --------------------------------------------------------------- prepare
def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _node_pair(case, seed):
    """(alpha x, alpha y, beta x, beta y) of an operator family on a seeded cavity."""
    nd = ns.jittered_cavity(case["n"], seed)
    xy = {"v": (_dev(nd.vx), _dev(nd.vy)), "p": (_dev(nd.px), _dev(nd.py))}
    # "pv": V-values to P-nodes, as the flow description names its families
    a, b = case["family"]
    return (*xy[a], *xy[b])


def _velocity(nd, rng, amplitude=0.2):
    """A smooth divergence-free field that vanishes on the walls: three modes of
    the stream function sin^2(k pi x) sin^2(l pi y) with random weights."""
    x, y = nd.vx, nd.vy
    u, v = np.zeros(nd.N), np.zeros(nd.N)
    for k, l in ((1, 1), (2, 1), (1, 2)):
        c = amplitude * rng.uniform(-1.0, 1.0) / math.pi
        sx, sy = np.sin(k * math.pi * x), np.sin(l * math.pi * y)
        u += c * sx * sx * l * math.pi * np.sin(2 * l * math.pi * y)
        v -= c * k * math.pi * np.sin(2 * k * math.pi * x) * sy * sy
    return u, v


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind in ("apply", "weights", "condition"):
        ctx = R.Context(case["stencil"], case["m"], case["q"])
        s.update(ctx=ctx, nodes=_node_pair(case, seed))
        if kind == "weights":
            return s
        ops = FAMILIES[case["family"]]
        idx, w, bad = R.build_weights(ctx, *s["nodes"], ops if kind == "apply" else R.OP_LAP)
        s["idx"] = idx
        if kind == "apply":
            dt = torch.float64 if case["dtype"] == "f64" else torch.float32
            bx, by = s["nodes"][2], s["nodes"][3]
            a, b = rng.uniform(2.0, 4.0, 2) * math.pi
            s["w"] = w[0].to(dt).contiguous()
            s["x"] = (torch.sin(2 * a * bx + a * by) * torch.cos(b * by)).to(dt)
            s["y"] = torch.cos(b * s["nodes"][0]).to(dt) if case["beta"] else None
        return s
    ctx = R.Context(28, 7, 3)
    if kind == "wake":
        h = case["h_wall"]
        box = dict(x0=-3.0, x1=6.0, y0=-3.0, y1=3.0) if case["domain"] == "short" else {}
        # one mesh, as a study of a flow keeps it; the seed draws the flow
        nd = ns.cylinder_wake(h_wall=h, h_wake=4.0 * h / 3.0,
                              h_far=(8.0 if box else 10.0) * h, **box)
        prec = R.PREC_FP64 if case["precision"] == "f64" else R.PREC_MIXED
        flow = wake.wake_flow(ctx, nd, Re=case["Re"], dt=case["dt"], tol=case["tol"],
                              precision=prec)
        u_inf = 1.0 + 0.05 * float(rng.standard_normal())
        gu, gv = wake.wake_data(nd, u_inf)
        inside = _dev(~nd.v_boundary).double()
        s.update(ctx=ctx, flow=flow, gu=gu, gv=gv, u0=u_inf * inside + gu,
                 v0=torch.zeros_like(gu))
        return s
    nd = ns.jittered_cavity(case["n"], seed)
    u0, v0 = _velocity(nd, rng)
    top = nd.v_wall == ns.WALL_TOP
    if kind == "ensemble":
        E = case["members"]
        flow = R.flow_from_nodes(ctx, nd, Re=1.0, dt=case["dt"], precision=R.PREC_MIXED,
                                 tol=case["tol"])
        gu = np.zeros((nd.N, E))
        gu[top] = 1.0 + 0.05 * rng.standard_normal(E)
        amp = rng.uniform(0.5, 1.5, E)
        s.update(ctx=ctx, flow=flow, Re=[float(r) for r in rng.uniform(1000.0, 5000.0, E)],
                 gu=_dev(gu.ravel()), gv=torch.zeros(nd.N * E, dtype=torch.float64, device="cuda"),
                 u0=_dev((u0[:, None] * amp + gu).ravel()), v0=_dev((v0[:, None] * amp).ravel()))
        return s
    prec = R.PREC_MIXED if case.get("precision") == "mixed" else R.PREC_FP64
    flow = R.flow_from_nodes(ctx, nd, Re=case["Re"], dt=case["dt"], precision=prec,
                             tol=case["tol"])
    gu = np.zeros(nd.N)
    gu[top] = 1.0 + 0.05 * rng.standard_normal(int(top.sum()))
    s.update(ctx=ctx, flow=flow, gu=_dev(gu), gv=torch.zeros(nd.N, dtype=torch.float64,
                                                             device="cuda"),
             u0=_dev(u0 + gu), v0=_dev(v0))
    return s


# ------------------------------------------------------------------- run
def _fields(st):
    return {"u": st.u, "v": st.v, "cu": st.cu_prev, "cv": st.cv_prev, "pt": st.pt, "p": st.p}


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "apply":
        n_rows, n_cols = s["nodes"][0].numel(), s["nodes"][2].numel()
        y = s["y"].clone() if s["y"] is not None else None
        return R.apply_op(ctx, s["idx"], s["w"], n_rows, n_cols, s["x"], y, case["alpha"],
                          case["beta"])
    if kind == "weights":
        idx, w, bad = R.build_weights(ctx, *s["nodes"], FAMILIES[case["family"]])
        na = s["nodes"][0].numel()
        return {"idx": idx[:, :na], "w": w[:, :, :na], "bad": bad}
    if kind == "condition":
        return R.stencil_condition(ctx, *s["nodes"], s["idx"])
    flow = s["flow"]
    if kind == "ensemble":
        st = R.ensemble_zeros(flow, case["members"])
        st.u.copy_(s["u0"])
        st.v.copy_(s["v0"])
        R.ensemble_step(ctx, flow, s["Re"], st, s["gu"], s["gv"], case["steps"])
        return _fields(st)
    st = R.State.zeros(flow)
    st.u.copy_(s["u0"])
    st.v.copy_(s["v0"])
    R.step(ctx, flow, st, s["gu"], s["gv"], case["steps"])
    return _fields(st)


# ------------------------------------------------------------------ work
def _rows(case):
    """(V-nodes, P-nodes) of the case's node set, to the accuracy that a count of bytes needs."""
    if case["kind"] == "wake":
        M = int((10.0 if case["domain"] == "short" else 28.0) / case["h_wall"] ** 2)
        return 3 * M, M
    n = case["n"]
    return n * (n - 1) * 2 + (n - 1) ** 2, n * n


def work(case):
    """Inputs read once and outputs written once; for the solves one product per
    implicit system and step, since an answer needs at least that."""
    N, M = _rows(case)
    kind = case["kind"]
    if kind in ("apply", "weights", "condition"):
        k = case["stencil"]
        a, b = ({"v": N, "p": M}[f] for f in case["family"])
        if kind == "apply":
            s = 8 if case["dtype"] == "f64" else 4
            return {"bytes": a * (k * (4 + s) + s * (2 if case["beta"] else 1)) + b * s,
                    "flops": 2 * k * a}
        S = k + (case["q"] + 1) * (case["q"] + 2) // 2
        if kind == "condition":
            return {"bytes": a * (4 * k + 8) + 16 * (a + b), "flops": a * 2 * S ** 3}
        nops = len(R.ops_of(FAMILIES[case["family"]]))
        return {"bytes": a * k * (4 + 8 * nops) + 16 * (a + b),
                "flops": a * (2 * S ** 3 / 3 + 2 * nops * S * S)}
    k, E = 28, case.get("members", 1)
    w = 4 if case.get("precision") == "mixed" or kind == "ensemble" else 8
    vv = N * k * (4 + 3 * w)  # D_x, D_y, Laplacian
    ops = vv + (N + M) * k * (4 + 2 * w) + M * k * (4 + w)
    state = E * 8 * (8 * N + 4 * M)
    flops = E * 2 * k * (8 * N + 4 * M)
    return {"bytes": case["steps"] * (ops + state), "flops": case["steps"] * flops}


# ----------------------------------------------------------------- exact
MOST_NODES = 6000  # dense solves and brute-force searches up to here


def _search(ax, ay, bx, by, k):
    """The k nearest b-nodes of each a-node by (squared distance, index)."""
    out = []
    for i in range(0, ax.numel(), 1024):
        dx, dy = bx[None, :] - ax[i:i + 1024, None], by[None, :] - ay[i:i + 1024, None]
        out.append(torch.sort(dx * dx + dy * dy, dim=1, stable=True).indices[:, :k])
    return torch.cat(out)


def _systems(case, ax, ay, bx, by, idx):
    """(A, x, y, scale): the augmented matrices in local coordinates."""
    m, q, k = case["m"], case["q"], idx.shape[1]
    X, Y = bx[idx] - ax[:, None], by[idx] - ay[:, None]
    sc = (X * X + Y * Y).amax(1, keepdim=True).sqrt()
    X, Y = X / sc, Y / sc
    mono = [(d - b, b) for d in range(q + 1) for b in range(d + 1)]
    S = k + len(mono)
    A = torch.zeros(ax.numel(), S, S, dtype=torch.float64, device=ax.device)
    A[:, :k, :k] = torch.hypot(X[:, :, None] - X[:, None, :], Y[:, :, None] - Y[:, None, :]) ** m
    for t, (a, b) in enumerate(mono):
        A[:, :k, k + t] = A[:, k + t, :k] = X ** a * Y ** b
    return A, X, Y, sc[:, 0], mono


def _exact_weights(case, nodes):
    m, k, ops = case["m"], case["stencil"], R.ops_of(FAMILIES[case["family"]])
    ax, ay, bx, by = nodes
    idx = _search(*nodes, k)
    A, X, Y, sc, mono = _systems(case, *nodes, idx)
    r = torch.hypot(X, Y)
    rhs = torch.zeros(A.shape[0], A.shape[1], len(ops), dtype=torch.float64, device=ax.device)
    for o, op in enumerate(ops):
        rhs[:, :k, o] = (-m * r ** (m - 2) * X if op == R.OP_DX else
                         -m * r ** (m - 2) * Y if op == R.OP_DY else m * m * r ** (m - 2))
        for t, e in enumerate(mono):
            if op == R.OP_LAP:
                rhs[:, k + t, o] = 2.0 if e in ((2, 0), (0, 2)) else 0.0
            else:
                rhs[:, k + t, o] = 1.0 if e == ((1, 0) if op == R.OP_DX else (0, 1)) else 0.0
    w = torch.linalg.solve(A, rhs)[:, :k]
    for o, op in enumerate(ops):
        w[:, :, o] /= (sc * sc if op == R.OP_LAP else sc)[:, None]
    return {"idx": idx.T.int(), "w": w.permute(2, 1, 0), "bad": None}


def _exact_condition(case, nodes, idx):
    ax, ay, bx, by = nodes
    out = []
    for i in range(0, ax.numel(), 10000):
        a = slice(i, i + 10000)
        A = _systems(case, ax[a], ay[a], bx, by, idx[:, :ax.numel()].T[a].long())[0]
        out.append(A.abs().sum(1).amax(1) * torch.linalg.inv(A).abs().sum(1).amax(1))
    return torch.cat(out)


def _exact_steps(flow, Re, dt, u, v, gu, gv, steps):
    """Section 3's step with dense factorisations of both implicit systems."""
    t, N, M = flow.tensors, flow.N, flow.M
    a = dt / (2.0 * Re)

    def product(idx, w, n, x):
        return (t[w][:, :n] * x[t[idx][:, :n].long()]).sum(0)

    def dense(idx, w, n):
        D = torch.zeros(n, n, dtype=torch.float64, device=u.device)
        rows = torch.arange(n, device=u.device)
        for k in range(idx.shape[0]):
            D[rows, idx[k, :n].long()] += w[k, :n]
        return D

    wall, pb = t["v_bc"] != 0, t["p_bc"] != 0
    H = torch.eye(N, dtype=torch.float64, device=u.device)
    H -= torch.where(wall, 0.0, a)[:, None] * dense(t["vv_idx"], t["vv_lap"], N)
    H = torch.linalg.lu_factor(H)
    L = torch.zeros(M + 1, M + 1, dtype=torch.float64, device=u.device)
    L[:M, :M] = dense(t["pp_idx"], t["pp_lap"], M)
    rows = t["pn_rows"].long()
    nx, ny = t["p_nx"][rows], t["p_ny"][rows]
    L[rows, :] = 0.0
    for k in range(t["pn_idx"].shape[0]):
        nb = rows.numel()
        L[rows, t["pn_idx"][k, :nb].long()] += nx * t["pn_dx"][k, :nb] + ny * t["pn_dy"][k, :nb]
    L[rows, M] = 1.0
    L[M, :M] = 1.0
    size = L.abs().amax(1)
    L /= size[:, None]  # the border and the one-sided rows are far smaller than the others
    LU = torch.linalg.lu_factor(L)
    pt, cup, cvp = torch.zeros(M, dtype=torch.float64, device=u.device), None, None
    for _ in range(steps):
        cu, cv = (-(u * product("vv_idx", "vv_dx", N, c) + v * product("vv_idx", "vv_dy", N, c))
                  for c in (u, v))
        cup, cvp = (cu, cv) if cup is None else (cup, cvp)
        rhs = []
        for c, cn, cp, g, gw in ((u, cu, cup, gu, "vp_dx"), (v, cv, cvp, gv, "vp_dy")):
            s = c + dt * (1.5 * cn - 0.5 * cp)
            inner = s + a * product("vv_idx", "vv_lap", N, s)
            rhs.append(torch.where(wall, g + dt * product("vp_idx", gw, N, pt), inner))
        ss = torch.linalg.lu_solve(*H, torch.stack(rhs, 1))
        F = product("pv_idx", "pv_dx", M, ss[:, 0]) + product("pv_idx", "pv_dy", M, ss[:, 1])
        b = torch.cat([torch.where(pb, 0.0, F / dt), torch.zeros_like(F[:1])])
        b = (b / size)[:, None]
        x = torch.linalg.lu_solve(*LU, b)
        for _ in range(2):
            x = x + torch.linalg.lu_solve(*LU, b - L @ x)
        pt = x[:M, 0]
        p = pt - a * product("pp_idx", "pp_lap", M, pt)
        u, v = (torch.where(wall, g, ss[:, c] - dt * product("vp_idx", w, N, pt))
                for c, g, w in ((0, gu, "vp_dx"), (1, gv, "vp_dy")))
        cup, cvp = cu, cv
    return {"u": u, "v": v, "cu": cup, "cv": cvp, "pt": pt, "p": p}


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    if kind == "apply":
        n = s["nodes"][0].numel()
        y = torch.zeros(n, dtype=torch.float64, device="cuda")
        for k in range(case["stencil"]):
            y += s["w"][k, :n].double() * s["x"][s["idx"][k, :n].long()].double()
        return case["alpha"] * y + (case["beta"] * s["y"].double() if case["beta"] else 0.0)
    if kind == "condition":
        return _exact_condition(case, s["nodes"], s["idx"])
    N, M = _rows(case)
    if kind == "wake" or N > MOST_NODES:
        return None
    if kind == "weights":
        return _exact_weights(case, s["nodes"])
    flow = s["flow"]
    if kind == "ensemble":
        E = case["members"]
        if E * N > 8 * MOST_NODES:
            return None
        col = lambda x, e: x.view(-1, E)[:, e].contiguous()  # noqa: E731
        each = [_exact_steps(flow, s["Re"][e], case["dt"], *(col(s[k], e) for k in
                                                             ("u0", "v0", "gu", "gv")),
                             case["steps"]) for e in range(E)]
        return {k: torch.stack([f[k] for f in each], 1).reshape(-1) for k in each[0]}
    return _exact_steps(flow, case["Re"], case["dt"], *(s[k] for k in ("u0", "v0", "gu", "gv")),
                        case["steps"])
