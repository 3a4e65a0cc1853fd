"""What users of this framework have it do, as cases that can be timed.

The work is explicit marching of the compressible Navier-Stokes equations: one
TVD-RK3 step (with its CFL step size) of one grid, of a fixed batch of grids,
or of the requests a server holds at the moment, and a single right-hand side
for programs that bring their own integrator.  Every case goes through the
classes of paper_2511_18042_gb300.api with the schemes, precisions and grid
sizes of this repository's benchmark, serving mix and tests.

A marching program steps one state on and on; here each pass first restores
the state it starts from (one device copy, a few per cent of the step at most),
as a parameter study or an ensemble restart does, so that every pass does the
same work and no flow leaves its regime.

`exact` restates the method in plain torch, in 64 bits, for 1D and 2D Cartesian
grids: ghosts, gradients, sensor, characteristic reconstruction, HLLC, the
localised artificial diffusivity, the per-interface hybrid, the implicit
filter, RK3 and the CFL step.  The body-fitted 3D viscous ramp (metrics,
walls, Sutherland viscosity) is not restated: its cases have no exact value.
"""
import math

import numpy as np
import torch

from paper_2511_18042_gb300 import api, inputs

GAMMA = 1.4
PERIODIC, EXTRAP, REFLECT, INFLOW = 0, 1, 2, 3
# floating-point operations per cell and RK3 step (CFL step included): 2D from
# the operation counts of the developed triple point, the others scaled by
# interfaces, nodes and variables
FLOPS = {("MEG6", 1): 1500, ("MEG6", 2): 3373, ("MEG6", 3): 8200, ("MIG4", 2): 3426, ("LAD_E4", 2): 1289,
         ("LAD_E4", 3): 4300, ("LAD_C6", 2): 1895, ("HYBRID", 1): 800, ("HYBRID", 2): 1670, ("HYBRID", 3): 5200}


def listed():
    return [
        # the smallest interactive run: Sod's tube of Sec. 3.1, replayed as a graph; pure latency
        dict(name="sod_400_meg6_fp64", kind="tube", n=400, scheme="MEG6", precision=0, graph=True),
        # one tick of the request server: tubes and quadrant problems of its mix, stepped together
        dict(name="serve_tick_5t3q_mixed", kind="serve", tubes=5, quads=3, n_tube=2000, n_quad=363, precision=1),
        # a fixed batch of quadrant problems, sizes 64..512, one graph replay per step (parameter study)
        dict(name="batch_32_hybrid_mixed", kind="batch", members=32, n_lo=64, n_hi=512, precision=1),
        # a ragged medium grid, compact gradients
        dict(name="triple_703x301_mig4_fp64", kind="triple", nx=703, ny=301, scheme="MIG4", precision=0, graph=False),
        # periodic box for a program with its own integrator: one right-hand side
        dict(name="kh_701_lad_e4_fp64_rhs", kind="kh", n=701, scheme="LAD_E4", precision=0),
        # the paper's triple point at the benchmark's size: the exact form of the main schemes ...
        dict(name="triple_1792x768_meg6_fp64", kind="triple", nx=1792, ny=768, scheme="MEG6", precision=0, graph=False),
        dict(name="triple_1792x768_hybrid_fp64", kind="triple", nx=1792, ny=768, scheme="HYBRID", precision=0,
             graph=False),
        dict(name="triple_1792x768_lad_c6_fp64", kind="triple", nx=1792, ny=768, scheme="LAD_C6", precision=0,
             graph=False),
        # ... and the mixed form, replayed as a graph as its users march it
        dict(name="triple_1792x768_meg6_mixed", kind="triple", nx=1792, ny=768, scheme="MEG6", precision=1, graph=True),
        dict(name="triple_1792x768_lad_c6_mixed", kind="triple", nx=1792, ny=768, scheme="LAD_C6", precision=1,
             graph=True),
        # the 3D viscous compression ramp (body-fitted grid, wall, inflow profile)
        dict(name="ramp_256x96x64_meg6_fp64", kind="ramp", nx=256, ny=96, nz=64, scheme="MEG6", precision=0),
        dict(name="ramp_256x96x64_lad_e4_mixed", kind="ramp", nx=256, ny=96, nz=64, scheme="LAD_E4", precision=1),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "serve", "batch", "triple", "triple", "triple", "kh", "ramp"])
    if kind == "tube":
        return dict(kind=kind, n=_logint(rng, 200, 20000), scheme=rng.choice(["MEG6", "HYBRID"]),
                    precision=rng.choice([0, 1]), graph=rng.choice([True, False]))
    if kind == "serve":
        return dict(kind=kind, tubes=rng.randint(1, 8), quads=rng.randint(1, 4), n_tube=_logint(rng, 200, 20000),
                    n_quad=_logint(rng, 128, 700), precision=1)
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(4, 32), n_lo=64, n_hi=_logint(rng, 128, 512),
                    precision=rng.choice([0, 1, 1]))
    if kind == "kh":
        return dict(kind=kind, n=_logint(rng, 48, 1024), scheme=rng.choice(["MEG6", "MIG4", "LAD_E4", "LAD_C6"]),
                    precision=rng.choice([0, 1]))
    if kind == "ramp":
        return dict(kind=kind, nx=rng.randint(96, 256), ny=rng.randint(48, 96), nz=rng.randint(16, 64),
                    scheme=rng.choice(["MEG6", "LAD_E4", "HYBRID"]), precision=rng.choice([0, 1]))
    return dict(kind="triple", nx=_logint(rng, 112, 1792), ny=_logint(rng, 48, 768),
                scheme=rng.choice(["MEG6", "MIG4", "LAD_E4", "LAD_C6", "HYBRID"]), precision=rng.choice([0, 1]),
                graph=rng.choice([True, False]))


# ---------------------------------------------------------------- inputs
def _perturb(W, prob, seed, amp):
    """Smooth seeded variations of every primitive (positive ones by a factor),
    with wave numbers that do not line up with the grid."""
    rng = np.random.default_rng(seed)
    nd = prob["ndim"]
    n = prob["n"]
    ax = [(torch.arange(n[d], dtype=torch.float64, device=W.device) + 0.5) / n[d] for d in range(nd)]
    per = prob["bc"][0][0] == PERIODIC
    for v in range(nd + 2):
        f = torch.zeros_like(W[v])
        for _ in range(3):
            ph = 0.0
            for d in range(nd):
                k = rng.integers(1, 6) if per else rng.uniform(1.0, 6.0)
                shape = [1] * nd
                shape[nd - 1 - d] = n[d]
                ph = ph + (2.0 * math.pi * float(k) * ax[d]).reshape(shape)
            f = f + torch.sin(ph + rng.uniform(0, 2 * math.pi)) / 3.0
        W[v] = W[v] * (1.0 + amp * f) if v in (0, nd + 1) else W[v] + amp * f
    return W


def _cons(W):
    nd = W.shape[0] - 2
    U = torch.empty_like(W)
    U[0] = W[0]
    q = torch.zeros_like(W[0])
    for k in range(nd):
        U[1 + k] = W[0] * W[1 + k]
        q = q + W[1 + k] * W[1 + k]
    U[nd + 1] = W[nd + 1] / (GAMMA - 1.0) + 0.5 * W[0] * q
    return U


def _bare(ndim, n, h, bc, **kw):
    return dict(ndim=ndim, n=list(n) + [1] * (3 - ndim), h=list(h) + [1.0] * (3 - ndim), bc=bc, gamma=GAMMA,
                inflow={}, **kw)


def _tube_state(case, seed):
    """Sod's solution some way into the run (the similarity solution at a
    seeded time, its jumps spread over a cell) with small smooth variations."""
    n = case["n"]
    rng = np.random.default_rng(seed)
    h = 1.0 / n
    prob = _bare(1, [n], [h], [[INFLOW, EXTRAP]])
    prob["inflow"] = {(0, 0): (1.0, 0.0, 1.0)}
    x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h
    t = rng.uniform(0.08, 0.18)
    xi = (x - 0.5) / t
    c0 = math.sqrt(GAMMA)
    ps, us, rl, rr = 0.30313017805064707, 0.92745262004894991, 0.42631942817849544, 0.26557371170530708
    head, tail, shock = -c0, us - c0 * (ps ** ((GAMMA - 1) / (2 * GAMMA))), 1.7521557320301779
    uf = 2.0 / (GAMMA + 1.0) * (c0 + xi)
    cf = c0 - 0.5 * (GAMMA - 1.0) * uf
    fan = (xi > head) & (xi < tail)
    u = torch.where(xi <= head, 0.0, torch.where(fan, uf, torch.full_like(x, us)))
    r = torch.where(fan, (cf / c0) ** (2.0 / (GAMMA - 1.0)), torch.where(xi <= head, 1.0, torch.full_like(x, rl)))
    p = torch.where(fan, (cf / c0) ** (2.0 * GAMMA / (GAMMA - 1.0)),
                    torch.where(xi <= head, 1.0, torch.full_like(x, ps)))
    w = h / t
    sc = 0.5 * (1.0 + torch.tanh((xi - us) / w))
    ss = 0.5 * (1.0 + torch.tanh((xi - shock) / w))
    r = r + (rr - rl) * sc + (0.125 - rr) * ss
    u = u - us * ss
    p = p + (0.1 - ps) * ss
    return prob, _cons(_perturb(torch.stack([r, u, p]), prob, seed, 0.002))


def _triple_state(case, seed):
    """A developed triple-point flow in outline: a transmitted and a reflected
    front, the contact between the two lower-pressure gases rolled up into a
    wave, a shear layer along it, jumps a cell or two wide, and smooth variations."""
    nx, ny = case["nx"], case["ny"]
    rng = np.random.default_rng(seed)
    prob = _bare(2, [nx, ny], [7.0 / nx, 3.0 / ny], [[REFLECT, REFLECT], [REFLECT, REFLECT]])
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * (7.0 / nx)
    y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * (3.0 / ny)).reshape(ny, 1)
    hx, hy = 7.0 / nx, 3.0 / ny

    def front(x0, a, width):
        ph = rng.uniform(0, 2 * math.pi, 2)
        xf = x0 + a * torch.sin(2.1 * y + ph[0]) + 0.3 * a * torch.sin(5.3 * y + ph[1])
        return 0.5 * (1.0 + torch.tanh((x - xf) / (width * hx)))

    ph = rng.uniform(0, 2 * math.pi, 2)
    yc = 1.5 + 0.25 * torch.sin(1.7 * x + ph[0]) + 0.08 * torch.sin(6.1 * x + ph[1])
    up = 0.5 * (1.0 + torch.tanh((y - yc) / (1.5 * hy)))
    s1 = front(rng.uniform(1.1, 1.6), 0.1, 1.5)   # driver contact
    s2 = front(rng.uniform(3.0, 4.0), 0.15, 1.0)  # transmitted shock
    rho = (1.0 - s1) * 0.6 + s1 * (1.0 - s2) * (1.9 * (1 - up) + 0.32 * up) + s2 * (1.0 * (1 - up) + 0.125 * up)
    p = 0.28 + (0.1 - 0.28) * s2
    u = (0.45 + 0.35 * up * s1) * (1.0 - s2)
    v = 0.12 * torch.sin(1.7 * x + ph[0] + 1.0) * torch.exp(-((y - 1.5) / 0.6) ** 2) * (1.0 - s2)
    W = torch.stack([rho, u.expand_as(rho), v.expand_as(rho), p.expand_as(rho)])
    return prob, _cons(_perturb(W.contiguous(), prob, seed, 0.004))


def _kh_state(case, seed):
    p = inputs.kelvin_helmholtz(case["n"])
    prob = _bare(2, p["n"][:2], p["h"][:2], p["bc"])
    U = torch.as_tensor(p["U"], device="cuda")
    W = torch.stack([U[0], U[1] / U[0], U[2] / U[0],
                     (GAMMA - 1.0) * (U[3] - 0.5 * (U[1] * U[1] + U[2] * U[2]) / U[0])])
    return prob, _cons(_perturb(W, prob, seed, 0.01))


def _ramp_state(case, seed):
    prob = inputs.compression_ramp(case["nx"], case["ny"], case["nz"], seed=seed)
    U = torch.as_tensor(prob["U"], device="cuda")
    rng = np.random.default_rng(seed + 1)
    nz, ny, nx = U.shape[1:]
    k = (torch.arange(nz, device="cuda", dtype=torch.float64) / nz).reshape(nz, 1, 1)
    j = (torch.arange(ny, device="cuda", dtype=torch.float64) / ny).reshape(ny, 1)
    i = torch.arange(nx, device="cuda", dtype=torch.float64) / nx
    a, b, c = rng.uniform(0, 2 * math.pi, 3)
    f = torch.sin(2 * math.pi * 2 * k + a) * torch.sin(9.0 * i + b) * torch.sin(7.0 * j + c)
    U = U * (1.0 + 0.01 * f)  # density and pressure vary together, velocities kept
    wz = 0.02 * torch.sin(2 * math.pi * 3 * k + b) * torch.sin(11.0 * i + c) * j
    U[3] = U[0] * wz
    U[4] = U[4] + 0.5 * U[0] * wz * wz
    return prob, U


def _quads(rng, n):
    """A quadrant problem of the batched and served mixes (as the server gets it:
    the initial states), and its initial state."""
    p = inputs.random_quadrants(rng, n)
    return p, torch.as_tensor(p["U"], device="cuda")


def _hyb_kw(rho, p, precision):
    return dict(scheme="HYBRID", hybrid_mode=1, hybrid_sensor=1, hyb_rho=0.5 * rho, hyb_p=0.5 * p, hybrid_buffer=1,
                precision=precision, cfl=0.2)


def _members(case, seed):
    """Problems, initial states and solver options of a serving tick or a batch."""
    rng = np.random.default_rng(seed)
    out = []
    if case["kind"] == "serve":
        for t in range(case["tubes"]):
            n = max(200, case["n_tube"] // (1 + t))
            p = inputs.random_tube(rng, n)
            U = torch.as_tensor(p["U"], device="cuda")
            out.append((p, U, _hyb_kw(min(p["WL"][0], p["WR"][0]), min(p["WL"][2], p["WR"][2]), case["precision"])))
        sizes = [max(64, case["n_quad"] - 37 * t) for t in range(case["quads"])]
    else:  # sizes spread over the logarithm of their range, odd ones among them
        m = case["members"]
        lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
        sizes = [int(round(math.exp(lo + (hi - lo) * (t + 0.5) / m))) for t in range(m)]
    for n in sizes:
        p, U = _quads(rng, n)
        st = p["quad_states"]
        out.append((p, U, _hyb_kw(float(st[:, 0].min()), float(st[:, 3].min()), case["precision"])))
    return out


def _options(case):
    kw = dict(scheme=case["scheme"], precision=case["precision"])
    if case["scheme"] == "HYBRID":
        kw.update(hybrid_mode=1, hybrid_sensor=1, hyb_rho=0.0625 if case["kind"] != "ramp" else 0.3)
    kw["cfl"] = 0.5 if case["kind"] == "tube" else 0.2
    return kw


_STATE = {"tube": _tube_state, "triple": _triple_state, "kh": _kh_state, "ramp": _ramp_state}


# ---------------------------------------------------------------- one pass
def prepare(case, seed):
    if case["kind"] in ("serve", "batch"):
        mem = _members(case, seed)
        flat0 = torch.cat([U.reshape(-1) for _, U, _ in mem])
        flat = flat0.clone()
        states, solvers, at = [], [], 0
        for p, U, kw in mem:  # the members' states: parts of one allocation
            states.append(flat[at:at + U.numel()].view(U.shape))
            solvers.append(api.Solver.from_problem(p, **kw))
            at += U.numel()
        st = dict(case=case, flat=flat, flat0=flat0, states=states, solvers=solvers, stream=torch.cuda.Stream())
        if case["kind"] == "batch":
            st["batch"] = api.Batch(solvers, states)
        torch.cuda.synchronize()
        return st
    prob, U0 = _STATE[case["kind"]](case, seed)
    s = api.Solver.from_problem(prob, **_options(case))
    st = dict(case=case, solver=s, U0=U0.contiguous(), U=U0.clone(), R=torch.empty_like(U0),
              dt=torch.zeros(2, dtype=torch.float64, device="cuda"), stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "kh":
        return [state["solver"].rhs(state["U0"], state["R"])]
    if case["kind"] in ("serve", "batch") or case.get("graph"):  # graphs and forks run on the program's own stream
        cur = torch.cuda.current_stream()
        st = state["stream"]
        st.wait_stream(cur)
        with torch.cuda.stream(st):
            if case["kind"] == "serve":
                state["flat"].copy_(state["flat0"])
                api.multi_step(state["solvers"], state["states"], stream=st)
            elif case["kind"] == "batch":
                state["flat"].copy_(state["flat0"])
                state["batch"].step(st)
            else:
                state["U"].copy_(state["U0"])
                state["solver"].step_graph(state["U"], state["dt"], st)
        cur.wait_stream(st)
    else:
        state["U"].copy_(state["U0"])
        state["solver"].step(state["U"], state["dt"])
    if case["kind"] in ("serve", "batch"):
        return [state["flat"]]
    return [state["U"], state["dt"][:1]]


def _cells(case):
    if case["kind"] in ("serve", "batch"):
        nd_n = []
        if case["kind"] == "serve":
            nd_n += [(1, max(200, case["n_tube"] // (1 + t))) for t in range(case["tubes"])]
            nd_n += [(2, max(64, case["n_quad"] - 37 * t) ** 2) for t in range(case["quads"])]
        else:
            m = case["members"]
            lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
            nd_n += [(2, int(round(math.exp(lo + (hi - lo) * (t + 0.5) / m))) ** 2) for t in range(m)]
        return [(nd, n, "HYBRID") for nd, n in nd_n]
    if case["kind"] == "tube":
        return [(1, case["n"], case["scheme"])]
    if case["kind"] == "kh":
        return [(2, case["n"] ** 2, case["scheme"])]
    if case["kind"] == "ramp":
        return [(3, case["nx"] * case["ny"] * case["nz"], case["scheme"])]
    return [(2, case["nx"] * case["ny"], case["scheme"])]


def work(case):
    """The state read once and written once (a right-hand side likewise) and
    the metrics of a body-fitted grid read once; the method's operations."""
    b = f = 0
    for nd, n, scheme in _cells(case):
        b += 2 * 8 * (nd + 2) * n + (8 * (2 * nd * nd + 1) * n if case["kind"] == "ramp" else 0)
        f += FLOPS[(scheme, nd)] * n / (3 if case["kind"] == "kh" else 1)
    return {"bytes": int(b), "flops": int(f)}


# ---------------------------------------------------------------- the method in plain torch
G = 8  # ghost layers of the padded arrays


def _sh(f, d, k):
    """f at offset k along direction d (the last axis is direction 0)."""
    return torch.roll(f, -k, dims=f.ndim - 1 - d)


def _pad(F, prob, mode):
    """F (nv, [ny,] nx) or a scalar field, padded by G in every direction: mode
    "prim", "cons" (vectors negated across a reflecting wall, inflow states) or "scalar"."""
    nd = prob["ndim"]
    for d in range(nd):
        n = prob["n"][d]
        pos = torch.arange(-G, n + G, device=F.device)
        src = pos.clone()
        for side, sel in ((0, pos < 0), (1, pos >= n)):
            bc = prob["bc"][d][side]
            if bc == PERIODIC:
                src = torch.where(sel, pos % n, src)
            elif bc == REFLECT:
                src = torch.where(sel, -pos - 1 if side == 0 else 2 * n - 1 - pos, src)
            else:
                src = torch.where(sel, torch.zeros_like(pos) if side == 0 else torch.full_like(pos, n - 1), src)
        F = torch.index_select(F, F.ndim - 1 - d, src)
        if mode == "scalar":
            continue
        for side in (0, 1):
            sl = [slice(None)] * F.ndim
            sl[F.ndim - 1 - d] = slice(0, G) if side == 0 else slice(n + G, n + 2 * G)
            if prob["bc"][d][side] == REFLECT:
                sl[0] = 1 + d
                F[tuple(sl)] = -F[tuple(sl)]
            elif prob["bc"][d][side] == INFLOW:
                W = torch.tensor(prob["inflow"][(d, side)], dtype=F.dtype, device=F.device).reshape(
                    (-1,) + (1,) * nd)
                F[tuple(sl)] = _cons(W) if mode == "cons" else W
    return F


def _inner(F, prob, lead=1):
    sl = [slice(None)] * lead + [slice(G, G + prob["n"][d]) for d in reversed(range(prob["ndim"]))]
    return F[tuple(sl)]


def _prim(U):
    nd = U.shape[0] - 2
    ir = 1.0 / U[0]
    u = [U[1 + k] * ir for k in range(nd)]
    ke = sum(U[1 + k] * u[k] for k in range(nd))
    return torch.stack([U[0]] + u + [(GAMMA - 1.0) * (U[nd + 1] - 0.5 * ke)])


def _solve(a, cyclic, r, d):
    """Solutions of a x_{i-1} + x_i + a x_{i+1} = r_i along direction d (not
    cyclic: the end rows are x = r), by a dense factorisation."""
    ax = r.ndim - 1 - d
    m = r.shape[ax]
    A = torch.eye(m, dtype=r.dtype, device=r.device)
    i = torch.arange(m, device=r.device)
    if cyclic:
        A[i, (i - 1) % m] += a
        A[i, (i + 1) % m] += a
    else:
        A[i[1:-1], i[:-2]] = a
        A[i[1:-1], i[2:]] = a
    b = r.movedim(ax, 0)
    x = torch.linalg.solve(A, b.reshape(m, -1)).reshape(b.shape)
    return x.movedim(0, ax)


def _grad(f, prob, d, kind):
    """First derivative of padded fields along d: MEG6, E4, MIG4 or C6 (compact
    on [-6, n+5] with E4 end rows, cyclic on periodic lines)."""
    e4 = (2.0 / 3.0) * (_sh(f, d, 1) - _sh(f, d, -1)) - (1.0 / 12.0) * (_sh(f, d, 2) - _sh(f, d, -2))
    if kind == "MEG6":
        return 0.75 * (_sh(f, d, 1) - _sh(f, d, -1)) - 0.15 * (_sh(f, d, 2) - _sh(f, d, -2)) + (1.0 / 60.0) * (
            _sh(f, d, 3) - _sh(f, d, -3))
    if kind == "E4":
        return e4
    return _compact(f, e4, prob, d, kind, 6)


def _compact(f, e4, prob, d, kind, grow):
    n, ax = prob["n"][d], f.ndim - 1 - d
    if kind == "MIG4":
        a, r = 0.25, 0.75 * (_sh(f, d, 1) - _sh(f, d, -1))
    else:
        a = 1.0 / 3.0
        r = (7.0 / 9.0) * (_sh(f, d, 1) - _sh(f, d, -1)) + (1.0 / 36.0) * (_sh(f, d, 2) - _sh(f, d, -2))
    out = torch.zeros_like(f)
    if prob["bc"][d][0] == PERIODIC:
        x = _solve(a, True, r.narrow(ax, G, n), d)
        src = torch.arange(-G, n + G, device=f.device) % n
        return torch.index_select(x, ax, src)
    lo, m = G - grow, n + 2 * grow
    rr = r.narrow(ax, lo, m).clone()
    for row in (0, m - 1):
        rr.narrow(ax, row, 1).copy_(e4.narrow(ax, lo + row, 1))
    out.narrow(ax, lo, m).copy_(_solve(a, False, rr, d))
    return out


def _mm2(a, b):
    z = torch.zeros_like(a)
    return torch.where((a > 0) & (b > 0), torch.minimum(a, b), torch.where((a < 0) & (b < 0), torch.maximum(a, b), z))


def _mp5(a, b, c, d, e):
    ul = (2.0 * a - 13.0 * b + 47.0 * c + 27.0 * d - 3.0 * e) / 60.0
    ump = c + _mm2(d - c, 4.0 * (c - b))
    dm, d0, dp = a - 2.0 * b + c, b - 2.0 * c + d, c - 2.0 * d + e
    p4 = _mm2(_mm2(4.0 * d0 - dp, 4.0 * dp - d0), _mm2(d0, dp))
    m4 = _mm2(_mm2(4.0 * d0 - dm, 4.0 * dm - d0), _mm2(d0, dm))
    uul, umd = c + 4.0 * (c - b), 0.5 * (c + d) - 0.5 * p4
    ulc = c + 0.5 * (c - b) + (4.0 / 3.0) * m4
    mn, mx = torch.minimum, torch.maximum
    umin = mx(mn(mn(c, d), umd), mn(mn(c, uul), ulc))
    umax = mn(mx(mx(c, d), umd), mx(mx(c, uul), ulc))
    return torch.where((ul - c) * (ul - ump) <= 1e-20, ul, ul + _mm2(umin - ul, umax - ul))


def _hllc(WL, WR, d, xi):
    nd = len(WL) - 2
    g, g2, ig2, gm1 = abs(xi), xi * xi, 1.0 / (xi * xi), GAMMA - 1.0
    sd = []
    for W in (WL, WR):
        q = sum(W[1 + m] * W[1 + m] for m in range(nd))
        E = W[nd + 1] / gm1 + 0.5 * W[0] * q
        sd.append((W[0], W[1:1 + nd], W[nd + 1], xi * W[1 + d], E, torch.sqrt(GAMMA * W[nd + 1] / W[0]),
                   torch.sqrt(W[0])))
    (rL, uL, pL, UL, EL, cL, sL), (rR, uR, pR, UR, ER, cR, sR) = sd
    iden = 1.0 / (sL + sR)
    uh = [(sL * uL[m] + sR * uR[m]) * iden for m in range(nd)]
    qh = sum(u * u for u in uh)
    Hh = (sL * ((EL + pL) / rL) + sR * ((ER + pR) / rR)) * iden
    ch = torch.sqrt(gm1 * (Hh - 0.5 * qh))
    SL = torch.minimum(UL - cL * g, xi * uh[d] - ch * g)
    SR = torch.maximum(UR + cR * g, xi * uh[d] + ch * g)
    Ss = (rR * UR * (SR - UR) - rL * UL * (SL - UL) + (pL - pR) * g2) / (rR * (SR - UR) - rL * (SL - UL))
    left, star = 0.0 <= Ss, (SL < 0.0) & (0.0 <= SR)
    left = left | (0.0 <= SL)
    pick = lambda a, b: torch.where(left, a, b)
    r, p, U, E, S = pick(rL, rR), pick(pL, pR), pick(UL, UR), pick(EL, ER), pick(SL, SR)
    u = [pick(uL[m], uR[m]) for m in range(nd)]
    fac, dS = r * (S - U) / (S - Ss), Ss - U
    F = [r * U] + [r * u[m] * U + (xi * p if m == d else 0.0) for m in range(nd)] + [(E + p) * U]
    Q = [fac] + [fac * (u[m] + (xi * dS * ig2 if m == d else 0.0)) for m in range(nd)]
    Q.append(fac * (E / r + dS * (Ss * ig2 + p / (r * (S - U)))))
    K = [r] + [r * u[m] for m in range(nd)] + [E]
    return torch.stack([torch.where(star, F[v] + S * (Q[v] - K[v]), F[v]) for v in range(nd + 2)])


def _omega(W, prob, kind):
    nd = prob["ndim"]
    p = W[nd + 1]
    phi = torch.zeros_like(p)
    du = []
    for l in range(nd):
        pm, pp = _sh(p, l, -1), _sh(p, l, 1)
        phi = torch.maximum(phi, torch.abs(pp - 2.0 * p + pm) / (pp + 2.0 * p + pm))
        du.append(_grad(W[1:1 + nd], prob, l, kind) / prob["h"][l])
    div = sum(du[k][k] for k in range(nd))
    w2 = (du[0][1] - du[1][0]) ** 2 if nd == 2 else torch.zeros_like(div)
    return phi * ((div * div + 1e-32) / (div * div + w2 + 1e-32))


def _gbr_flux(W, prob, d, kind, om, xi):
    """C-GBR fluxes of the interfaces i+1/2 along d, stored at node i (padded)."""
    nd, ip = prob["ndim"], prob["ndim"] + 1
    D = _grad(W, prob, d, kind)
    DD = 2.0 * (_sh(W, d, 1) - 2.0 * W + _sh(W, d, -1)) - 0.5 * (_sh(D, d, 1) - _sh(D, d, -1))
    W1 = _sh(W, d, 1)
    rb, pb = 0.5 * (W[0] + W1[0]), 0.5 * (W[ip] + W1[ip])
    cb = torch.sqrt(GAMMA * pb / rb)
    ic2 = (1.0 / cb) * (1.0 / cb)
    ha, hb, cr = 0.5 * ic2, 0.5 * rb * (1.0 / cb), cb / rb
    tv = 1 - d  # the transverse velocity (2D); its tangent is (0, 1) along x and (-1, 0) along y
    tsg = 1.0 if d == 0 else -1.0

    def char(w):
        c = [ha * w[ip] - hb * w[1 + d], w[0] - ic2 * w[ip]]
        if nd == 2:
            c.append(tsg * w[1 + tv])
        return c + [ha * w[ip] + hb * w[1 + d]]

    C = [char(_sh(W, d, k)) for k in (-2, -1, 0, 1, 2, 3)]
    Cd, Cdd = [char(D), char(_sh(D, d, 1))], [char(DD), char(_sh(DD, d, 1))]
    omb = om
    for k in range(-3, 5):
        omb = torch.maximum(omb, _sh(om, d, k))
    disc = omb > 0.01
    CL, CR = [], []
    for b in range(nd + 2):
        v = [c[b] for c in C]
        cl = v[2] + 0.5 * Cd[0][b] + Cdd[0][b] * (1.0 / 12.0)
        cr_ = v[3] - 0.5 * Cd[1][b] + Cdd[1][b] * (1.0 / 12.0)
        cc = 0.5 * (cl + cr_)
        mL, mR = _mp5(*v[:5]), _mp5(*v[:0:-1])
        if b == 1:
            ul = v[2] + _mm2(v[3] - v[2], 4.0 * (v[2] - v[1]))
            ur = v[3] + _mm2(v[2] - v[3], 4.0 * (v[3] - v[4]))
            CL.append(torch.where((cl - v[2]) * (cl - ul) > 1e-20, mL, cc))
            CR.append(torch.where((cr_ - v[3]) * (cr_ - ur) > 1e-20, mR, cc))
        else:
            acoustic = b in (0, ip)
            CL.append(torch.where(disc, mL, cl if acoustic else cc))
            CR.append(torch.where(disc, mR, cr_ if acoustic else cc))
    out = []
    for c in (CL, CR):
        s, un = c[0] + c[ip], (c[ip] - c[0]) * cr
        w = [None] * (nd + 2)
        w[0], w[ip], w[1 + d] = c[1] + s, (cb * cb) * s, un
        if nd == 2:
            w[1 + tv] = tsg * c[2]
        out.append(torch.stack(w))
    bad = (out[0][0] <= 0) | (out[0][ip] <= 0) | (out[1][0] <= 0) | (out[1][ip] <= 0)
    return _hllc(torch.where(bad, W, out[0]), torch.where(bad, W1, out[1]), d, xi)


def _lad(W, prob, kind):
    """Node fluxes of the localised artificial diffusivity, every direction (padded)."""
    nd, ip = prob["ndim"], prob["ndim"] + 1
    rho, p = W[0], W[ip]
    T, e = GAMMA * p / rho, p / (rho * (GAMMA - 1.0))
    f = torch.stack([W[1 + k] for k in range(nd)] + [T, rho, e])
    gr = [_grad(f, prob, l, kind) / prob["h"][l] for l in range(nd)]
    div = sum(gr[k][k] for k in range(nd))
    w2 = (gr[0][1] - gr[1][0]) ** 2 if nd == 2 else torch.zeros_like(div)
    fsw = torch.where(div < 0, (div * div) / (div * div + w2 + 1e-32), torch.zeros_like(div))
    gmr = torch.sqrt(sum(gr[l][nd + 1] ** 2 for l in range(nd)))
    gme = torch.sqrt(sum(gr[l][nd + 2] ** 2 for l in range(nd)))
    sb = sk = 0.0
    for l in range(nd):
        d4 = lambda q: (_sh(q, l, -2) + _sh(q, l, 2)) - 4.0 * (_sh(q, l, -1) + _sh(q, l, 1)) + 6.0 * q
        db = torch.abs(prob["h"][l] * gr[l][nd + 1]) / (gmr + 1e-32)
        dk = torch.abs(prob["h"][l] * gr[l][nd + 2]) / (gme + 1e-32)
        sb, sk = sb + d4(div) * db * db, sk + d4(e) * dk
    co = []
    for c in (1.75 * rho * fsw * torch.abs(sb), 0.01 * (rho * torch.sqrt(GAMMA * p / rho) / T) * torch.abs(sk)):
        c = _inner(c, prob, 0)
        for l in range(nd):
            c = _pad(c, prob, "scalar")
            t = lambda k: _sh(c, l, -k) + _sh(c, l, k)
            c = _inner((3565.0 / 10368.0) * c + (3091.0 / 12960.0) * t(1) + (1997.0 / 25920.0) * t(2) +
                       (149.0 / 12960.0) * t(3) + (107.0 / 103680.0) * t(4), prob, 0)
        co.append(_pad(c, prob, "scalar"))
    tau, kap = co[0] * div, co[1]
    E = p / (GAMMA - 1.0) + 0.5 * rho * sum(W[1 + m] ** 2 for m in range(nd))
    flux = []
    for l in range(nd):
        xi = math.prod(prob["h"][:nd]) / prob["h"][l]
        U = xi * W[1 + l]
        F = [rho * U] + [rho * W[1 + m] * U for m in range(nd)] + [(E + p) * U]
        F[1 + l] = F[1 + l] + xi * p - xi * tau
        F[ip] = F[ip] - xi * (W[1 + l] * tau + kap * gr[l][nd])
        flux.append(torch.stack(F))
    return flux


def _rhs(U, prob, kw):
    nd, ip = prob["ndim"], prob["ndim"] + 1
    W = _pad(_prim(U), prob, "prim")
    J = 1.0 / math.prod(prob["h"][:nd])
    xi = [math.prod(prob["h"][:nd]) / prob["h"][l] for l in range(nd)]
    acc = torch.zeros_like(U)
    scheme = kw["scheme"]
    if scheme.startswith("LAD"):
        F = _lad(W, prob, scheme[4:])
        for l in range(nd):
            if scheme == "LAD_E4":
                D = _grad(F[l], prob, l, "E4")
            else:
                D = _compact(F[l], _grad(F[l], prob, l, "E4"), prob, l, "C6", 0)
            acc = acc + _inner(D, prob)
        return -J * acc
    kind = "MIG4" if scheme == "MIG4" else "MEG6"
    om = _omega(W, prob, kind)
    if scheme == "HYBRID":
        tr = (W[0] < kw["hyb_rho"]) | (W[ip] < kw.get("hyb_p", -math.inf)) | (om > 0.01)
        if kw.get("hybrid_buffer"):
            for l in range(nd):
                tr = tr | _sh(tr, l, 1) | _sh(tr, l, -1)
        F = _lad(W, prob, "E4")
    for d in range(nd):
        H = _gbr_flux(W, prob, d, kind, om, xi[d])
        if scheme == "HYBRID":
            f = F[d]
            h = (7.0 / 12.0) * (f + _sh(f, d, 1)) - (1.0 / 12.0) * (_sh(f, d, -1) + _sh(f, d, 2))
            H = torch.where(tr | _sh(tr, d, 1), H, h)
        acc = acc + _inner(H - _sh(H, d, -1), prob)
    return -J * acc


def _filter(U, prob):
    af = 0.45
    b = [(93.0 + 70.0 * af) / 128.0, 0.5 * ((7.0 + 18.0 * af) / 16.0), 0.5 * ((-7.0 + 14.0 * af) / 32.0),
         0.5 * ((1.0 - 2.0 * af) / 16.0), 0.5 * ((-1.0 + 2.0 * af) / 128.0)]
    for d in range(prob["ndim"]):
        Q, n = _pad(U, prob, "cons"), prob["n"][d]
        ax = Q.ndim - 1 - d
        r = b[0] * Q + sum(b[k] * (_sh(Q, d, k) + _sh(Q, d, -k)) for k in range(1, 5))
        if prob["bc"][d][0] == PERIODIC:
            x = r.clone()
            x.narrow(ax, G, n).copy_(_solve(af, True, r.narrow(ax, G, n), d))
        else:
            r = r.clone()
            for at in (G - 1, G + n):
                r.narrow(ax, at, 1).copy_(Q.narrow(ax, at, 1))
            x = r
            x.narrow(ax, G - 1, n + 2).copy_(_solve(af, False, r.narrow(ax, G - 1, n + 2).clone(), d))
        U = _inner(x, prob)
    return U


def _step(U, prob, kw):
    nd = prob["ndim"]
    W = _prim(U)
    c = torch.sqrt(GAMMA * W[nd + 1] / W[0])
    dt = kw["cfl"] / sum((torch.abs(W[1 + l]) + c) / prob["h"][l] for l in range(nd)).max()
    u1 = U + dt * _rhs(U, prob, kw)
    u2 = 0.75 * U + 0.25 * (u1 + dt * _rhs(u1, prob, kw))
    u3 = (1.0 / 3.0) * U + (2.0 / 3.0) * (u2 + dt * _rhs(u2, prob, kw))
    return (_filter(u3, prob) if kw["scheme"] == "LAD_C6" else u3), dt.reshape(1)


def exact(case, seed):
    if case["kind"] == "ramp":  # not restated here (see the top of the file)
        return None
    if case["kind"] in ("serve", "batch"):
        return [torch.cat([_step(U, p, kw)[0].reshape(-1) for p, U, kw in _members(case, seed)])]
    prob, U = _STATE[case["kind"]](case, seed)
    kw = _options(case)
    if case["kind"] == "kh":
        return [_rhs(U, prob, kw)]
    return list(_step(U, prob, kw))
