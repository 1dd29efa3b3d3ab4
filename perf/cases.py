"""Performance cases of the LABFM library: the calls a user's program makes, over the range of sizes it makes them at.

A program that uses the library finds stencils for a node set (once, or at every step if its nodes move), builds the
weights of a few differential operators at an order between 2 and 8, and then applies them, steps a PDE with them or
solves a linear system with them, many times.  Each case below is one of those calls; ``prepare`` makes what the
program holds before it (node positions, fields, and the stencils and weights that an earlier call built).

``exact`` computes the same outputs with plain torch in double precision: stencils by comparing index-lattice
candidates, weights from the moment conditions by a batched LU solve with iterative refinement on their residual.
"""
import math

import torch

from paper_1912_06441_gb300 import Labfm

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
F64 = torch.float64

# stencil half radius over node spacing by order, and the operators usually wanted at that order
H_OVER_S = {2: 1.2, 3: 1.3, 4: 1.4, 5: 1.6, 6: 1.8, 7: 2.0, 8: 2.2}
HYPER = {4: "lap2", 5: "lap2", 6: "lap3", 7: "lap3", 8: "lap4"}
# the advection-diffusion run: velocity, viscosity, and hyperviscosity coefficient over h^8
ADVECT, NU, HYPERVISC = (1.0, 0.5), 1e-3, 1e-3
REYNOLDS = 10.0


def _lattice(name, call, side, order, **more):
    case = {"name": name, "call": call, "nodes": "lattice", "side": side, "order": order, "h": H_OVER_S[order],
            "jitter": 0.3, "rbf": "wendland_c2", "form": "chain", "ops": "dx dy lap", "precision": "fp64",
            "weights": "f64", "fields": "f64", "steps": 0}
    case.update(more)
    return case


def _pde(name, call, nodes, side, **more):
    """Order 4 on nodes of spacing h/2 with quadratic ABFs in the dW0/dr form: what the PDE runs of the method use."""
    more = dict({"h": 2.0, "jitter": 0.5 / math.sqrt(2.0), "rbf": "quadratic", "form": "dw0"}, **more)
    return _lattice(name, call, side, 4, nodes=nodes, **more)


def _step8(name, call, side, **more):
    """Order 8 as the time-stepping runs use it: quadratic ABFs in the dW0/dr form on a set of little noise, where every
    stencil is well conditioned.  (On the noisier sets FP64 weights of orders 6 to 8 are off by up to 1e-6 and more;
    programs keep those in FP32, or take the refined mixed builds.)"""
    more = dict({"ops": "dx dy lap lap4", "jitter": 0.1, "rbf": "quadratic", "form": "dw0"}, **more)
    return _lattice(name, call, side, 8, **more)


def listed():
    return [
        # a program whose nodes move: stencils, weights and derivatives of a small set, as it repeats them every step;
        # launches, allocations and host round trips are most of it
        _lattice("startup_64", "startup", 64, 4),
        # the stencil search of a production-size set at the radius of order 8
        _lattice("stencils_512", "stencils", 512, 8),
        # weights of first and second derivatives at order 4: the PDE runs' setup
        _pde("weights_k4_512", "weights", "lattice", 512),
        # the headline build: order 8 with hyperviscosity, FP64
        _step8("weights_k8_512", "weights", 512),
        # the same on the noisier set for a program that stores its weights in FP32: the tensor-core mixed build
        _lattice("weights_k8_tc_512", "weights", 512, 8, ops="dx dy lap lap4", precision="mixed_tc", weights="f32",
                 fields="f32"),
        # walls, variable spacing and an order of its own for every node (2 to 6): stencils and weights together,
        # the setup of a wall-bounded program that applies FP32 weights
        _lattice("walls_500", "setup", 500, 6, nodes="walls", order_cap=6, weights="f32"),
        # derivatives of an FP64 field by order-8 FP64 weights: once a time step in a program with its own integrator
        _step8("apply_f64_k8_512", "apply", 512, precision="mixed_tc"),
        # the same for FP32 weights and fields on a larger set: first and second derivatives, which FP32 suits
        _lattice("apply_f32_k6_1000", "apply", 1000, 6, weights="f32", fields="f32", jitter=0.1, rbf="quadratic",
                 form="dw0"),
        # the heat equation with fixed walls, FP64: many cheap steps on a set that fits the cache
        _pde("heat_161", "step", "walled", 161, ops="lap", steps=100),
        # advection-diffusion with hyperviscosity at order 8: FP32 fields, FP64 weights
        _step8("advect_1024", "step", 1024, fields="f32", steps=5),
        # Burgers' equation for two velocity components
        _pde("burgers_161", "burgers", "lattice", 161, jitter=0.2 / math.sqrt(2.0), steps=50),
        # Poisson's equation with fixed walls from a zero start to a relative residual of 1e-10
        _pde("poisson_257", "solve", "walled", 257, ops="lap"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["startup", "stencils", "weights", "weights", "setup", "apply", "apply", "step", "step",
                       "burgers", "solve"])
    if call in ("startup", "stencils", "weights"):
        order = rng.randint(2, 4 if call == "startup" else 8)
        ops = "dx dy lap" if order < 4 or rng.random() < 0.5 else "dx dy lap " + HYPER[order]
        more = {"ops": ops, "h": H_OVER_S[order] * rng.uniform(1.0, 1.1)}
        if order > 5 and call == "weights":
            more.update(jitter=0.1, rbf="quadratic", form="dw0")
        elif rng.random() < 0.3:
            more.update(rbf="quadratic", form=rng.choice(["chain", "dw0"]))
        if call == "startup":
            case = _lattice("", call, _log_int(rng, 32, 128), order, **more)
        elif call == "stencils":
            case = _lattice("", call, _log_int(rng, 48, 900), order, h=more["h"], nodes=rng.choice(["lattice", "walled"]))
        elif rng.random() < 0.35:  # mixed builds store FP32 weights, at the orders they are used for
            order = rng.randint(5, 8)
            case = _lattice("", call, _log_int(rng, 48, 480), order, ops="dx dy lap " + HYPER[order],
                            precision=rng.choice(["mixed", "mixed_tc"]), weights="f32", fields="f32")
        else:
            case = _lattice("", call, _log_int(rng, 48, 440), order,
                            weights="f32" if order == 7 else rng.choice(["f64", "f64", "f32"]), **more)
    elif call == "setup":
        cap = rng.randint(3, 8)
        case = _lattice("", call, _log_int(rng, 200, 480), cap, nodes="walls", order_cap=cap, weights="f32",
                        precision="fp64" if cap < 5 else "mixed_tc" if cap > 6 else rng.choice(["fp64", "mixed_tc"]))
    elif call == "apply":
        order = rng.randint(2, 8)
        kind = rng.choice(["f64", "f64", "f32"])
        ops = "dx dy lap" if kind == "f32" or order < 4 or rng.random() < 0.5 else "dx dy lap " + HYPER[order]
        if kind == "f64" and rng.random() < 0.2:
            ops = "lap"
        more = {"jitter": rng.uniform(0.1, 0.25)} if order < 5 and kind == "f64" else \
            {"jitter": rng.uniform(0.1, 0.15), "rbf": "quadratic", "form": "dw0"}
        case = _lattice("", call, _log_int(rng, 48, 700), order, ops=ops, weights=kind, fields=kind,
                        precision="fp64" if order < 5 else "mixed_tc", **more)
    elif call == "step":
        if rng.random() < 0.5:
            case = _pde("", call, "walled", _log_int(rng, 41, 321), ops="lap", steps=rng.randint(20, 60))
        else:
            order = rng.choice([4, 6, 8])
            wf = rng.choice([("f64", "f32"), ("f32", "f32"), ("f64", "f64")])
            case = _lattice("", call, _log_int(rng, 64, 900), order, ops="dx dy lap lap4" if order == 8 else "dx dy lap",
                            jitter=0.1, rbf="quadratic", form="dw0", precision="fp64" if order < 5 else "mixed_tc",
                            weights=wf[0], fields=wf[1], steps=rng.randint(2, 6))
    elif call == "burgers":
        case = _pde("", call, "lattice", _log_int(rng, 41, 321), jitter=0.2 / math.sqrt(2.0), steps=rng.randint(10, 40))
    else:
        case = _pde("", call, "walled", _log_int(rng, 33, 201), ops="lap")
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
def _nodes(case, seed):
    """(xy [n, 2], h [n], order int8 [n] or None, periodic, wall mask [n]), node index = row * side + column."""
    m, kind = case["side"], case["nodes"]
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)
    jit = (2.0 * torch.rand((m * m, 2), dtype=F64, device=DEV, generator=g) - 1.0) * case["jitter"]
    at = torch.arange(m * m, device=DEV)
    i, j = at % m, at // m
    edge = torch.minimum(torch.minimum(i, m - 1 - i), torch.minimum(j, m - 1 - j))
    if kind == "lattice":  # periodic unit square
        s = 1.0 / m
        xy = (torch.stack([i, j], 1).to(F64) + 0.5 + jit) * s
        xy = torch.where(xy < 0.0, xy + 1.0, xy)
        xy = torch.where(xy >= 1.0, xy - 1.0, xy)
        return xy.contiguous(), torch.full((m * m,), case["h"] * s, dtype=F64, device=DEV), None, True, edge < 0
    if kind == "walled":  # nodes on the walls; they and the two rows inside them stay on the lattice
        s = 1.0 / (m - 1)
        jit = torch.where((edge > 2)[:, None], jit, torch.zeros_like(jit))
        xy = ((torch.stack([i, j], 1).to(F64) + jit) * s).clamp_(0.0, 1.0)
        return xy.contiguous(), torch.full((m * m,), case["h"] * s, dtype=F64, device=DEV), None, False, edge == 0
    # walls: spacing four times finer at the walls than in the middle, order rising with x, order 4 at most and wider
    # stencils near the walls
    t = torch.stack([i, j], 1).to(F64) / (m - 1)
    xy = t - 0.6 * torch.sin(2.0 * math.pi * t) / (2.0 * math.pi)
    sp = (1.0 - 0.6 * torch.cos(2.0 * math.pi * t)) / (m - 1)
    s = (sp[:, 0] * sp[:, 1]).sqrt()
    on = torch.stack([(i == 0) | (i == m - 1), (j == 0) | (j == m - 1)], 1)
    xy = torch.where(on, xy, xy + jit * sp).clamp_(0.0, 1.0)
    hs = torch.tensor([0.0, 0.0, 1.2, 1.3, 1.5, 1.7, 1.9, 2.1, 2.3], dtype=F64, device=DEV)
    k = (2 + (7.0 * xy[:, 0]).floor().long()).clamp(max=case["order_cap"])
    wall = torch.minimum(xy, 1.0 - xy).min(1).values
    band = wall < 2.0 * 1.4 * hs[k] * s
    k = torch.where(band, k.clamp(max=4), k)
    h = torch.where(band, 1.4 * hs[k] * s, hs[k] * s)
    return xy.contiguous(), h.contiguous(), k.to(torch.int8), False, on.any(1)


def _index(a, b):
    n = a + b
    return (n - 1) * (n + 2) // 2 + b


def _targets(case):
    """Target vectors C^d, one row per operator, in the degree-major ordering of the derivatives."""
    k = case["order"] if case["nodes"] != "walls" else 8
    rows = []
    for name in case["ops"].split():
        c = [0.0] * (k * (k + 3) // 2)
        if name in ("dx", "dy"):
            c[_index(1, 0) if name == "dx" else _index(0, 1)] = 1.0
        else:
            m = int(name[3:] or 1)
            for t in range(m + 1):
                c[_index(2 * (m - t), 2 * t)] = float(math.comb(m, t))
        rows.append(c)
    return rows


def _fourier(xy, seed):
    """Sum of 16 Fourier modes with wavenumbers up to 32 and normal amplitudes."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 2)
    kk = torch.randint(-32, 33, (16, 2), device=DEV, generator=g).to(F64)
    amp = torch.randn(16, dtype=F64, device=DEV, generator=g)
    ph = 2.0 * math.pi * torch.rand(16, dtype=F64, device=DEV, generator=g)
    f = torch.zeros(xy.shape[0], dtype=F64, device=DEV)
    for m in range(16):
        f += amp[m] * torch.cos(2.0 * math.pi * (kk[m, 0] * xy[:, 0] + kk[m, 1] * xy[:, 1]) + ph[m])
    return f


def _field(case, xy, wall, seed):
    """The field(s) a call starts from."""
    x, y = xy[:, 0], xy[:, 1]
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 3)
    a, b = (2.0 * math.pi * torch.rand(2, dtype=F64, device=DEV, generator=g)).unbind()
    if case["call"] in ("startup", "apply"):
        return _fourier(xy, seed)
    if case["call"] == "solve":  # F = lap phi inside, phi on the walls
        phi = torch.sin(2.0 * math.pi * x + a) * torch.sin(2.0 * math.pi * y + b)
        return torch.where(wall, phi, -8.0 * math.pi ** 2 * phi)
    if case["call"] == "burgers":  # a Cole-Hopf velocity: both components and all advection terms are at work
        tp, c, e = 2.0 * math.pi, -2.0 / REYNOLDS, 0.5
        phi = 1.0 + e * torch.sin(tp * x + a) * torch.sin(tp * y + b)
        return torch.stack([c * tp * e * torch.cos(tp * x + a) * torch.sin(tp * y + b) / phi,
                            c * tp * e * torch.sin(tp * x + a) * torch.cos(tp * y + b) / phi])
    if case["nodes"] == "walled":  # heat: a warm wall, and a smooth start inside
        warm = torch.where(y == 0.0, torch.sin(math.pi * x), torch.zeros_like(x))
        return torch.where(wall, warm, 0.5 * torch.sin(math.pi * x) * torch.sin(math.pi * y) * (1.0 + torch.sin(a + 3.0 * x)))
    return torch.sin(2.0 * math.pi * x + a) * torch.cos(2.0 * math.pi * y + b)


def _stepping(case):
    """(beta, dt) of a time-stepping case, within the stability region of RK4."""
    if case["nodes"] == "walled":
        h = case["h"] / (case["side"] - 1)
        return [1.0], 0.015 * h * h
    s, h = 1.0 / case["side"], case["h"] / case["side"]
    if case["call"] == "burgers":
        return [0.0, 0.0, 1.0 / REYNOLDS], min(0.1 * h, 0.03 * h * h * REYNOLDS)
    beta = [-ADVECT[0], -ADVECT[1], NU]
    if "lap4" in case["ops"]:
        beta.append(-HYPERVISC * h ** 8)
    return beta, min(0.08 * s, 1.2e-4)


def _capacity(case):
    """Stencil entries that the program's own buffers hold: somewhat more than a node set of this kind has."""
    n = case["side"] ** 2
    if case["nodes"] == "walls":
        return 70 * n
    return int(1.05 * n * math.pi * (2.0 * case["h"]) ** 2) + 1024


def _build(case, lib, order, status):
    return lib.build_weights(_targets(case), order=order, uniform_order=case["order"], rbf=case["rbf"],
                             precision=case["precision"], weight_dtype=case["weights"], node_status=status,
                             abf_form=case["form"])


def prepare(case, seed):
    xy, h, order, periodic, wall = _nodes(case, seed)
    ft = torch.float32 if case["fields"] == "f32" else F64
    st = {"case": case, "xy": xy, "h": h, "order": order, "periodic": periodic, "lib": Labfm(0), "targets": _targets(case)}
    call = case["call"]
    n = xy.shape[0]
    if call in ("weights", "setup"):
        st["status"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        wt = torch.float32 if case["weights"] == "f32" else F64
        st["w"] = torch.zeros((_capacity(case), len(st["targets"])), dtype=wt, device=DEV)
    if call in ("stencils", "setup"):
        st["row_ptr"] = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        st["col"] = torch.zeros(_capacity(case), dtype=torch.int32, device=DEV)
    if call in ("startup", "apply", "step", "burgers", "solve"):
        st["f"] = _field(case, xy, wall, seed).to(ft).contiguous()
    if call in ("weights", "apply", "step", "burgers", "solve"):  # the stencils, and below the weights, of an earlier call
        st["lib"].build_neighbours(xy, h, periodic)
    if call in ("apply", "step", "burgers", "solve"):
        _build(case, st["lib"], order, torch.zeros(n, dtype=torch.int32, device=DEV))
    if call == "apply":
        st["out"] = torch.empty((len(st["targets"]), n), dtype=ft, device=DEV)
    if call in ("step", "burgers"):
        st["beta"], st["dt"] = _stepping(case)
        st["frozen"] = wall.to(torch.uint8) if case["nodes"] == "walled" else None
    if call == "burgers":
        st["u"], st["v"] = st["f"][0].clone(), st["f"][1].clone()
    if call == "solve":
        st["phi"] = torch.zeros(n, dtype=F64, device=DEV)
        st["dirichlet"] = wall.to(torch.uint8)
    return st


def _kept(buf, view):
    """The library's view, valid until its next build, copied to the program's own buffer (which is larger)."""
    buf[: view.shape[0]].copy_(view)
    return buf


def run(state):
    case, lib = state["case"], state["lib"]
    call = case["call"]
    if call == "stencils":
        lib.build_neighbours(state["xy"], state["h"], state["periodic"])
        row_ptr, col = lib.get_neighbours()
        return [_kept(state["row_ptr"], row_ptr), _kept(state["col"], col)]
    if call == "startup":
        lib.build_neighbours(state["xy"], state["h"], state["periodic"])
        _build(case, lib, state["order"], None)
        return lib.apply(state["f"])
    if call == "setup":
        lib.build_neighbours(state["xy"], state["h"], state["periodic"])
        bad = _build(case, lib, state["order"], state["status"])
        row_ptr, col = lib.get_neighbours()
        return [bad, state["status"], _kept(state["row_ptr"], row_ptr), _kept(state["col"], col),
                _kept(state["w"], lib.get_weights())]
    if call == "weights":
        bad = _build(case, lib, state["order"], state["status"])
        return [bad, state["status"], _kept(state["w"], lib.get_weights())]
    if call == "apply":
        return lib.apply(state["f"], out=state["out"])
    if call == "step":
        return lib.step(state["beta"], state["f"], state["dt"], case["steps"], frozen=state["frozen"])
    if call == "burgers":
        return lib.step_burgers(state["beta"], state["u"], state["v"], state["dt"], case["steps"])
    state["phi"].zero_()
    lib.solve(0, state["f"], state["phi"], state["dirichlet"], tol=1e-10, max_iter=20000)
    return state["phi"]


def work(case):
    """Bytes and floating-point operations of one pass, each input read and each output written once."""
    n, p = case["side"] ** 2, case["order"] * (case["order"] + 3) // 2
    nb = math.pi * (2.0 * case["h"]) ** 2  # stencil entries of a node, about
    if case["nodes"] == "walls":  # per-node orders: about the mean over orders 2 to the cap
        p, nb = p / 2.5, 0.55 * nb
    ops = len(case["ops"].split())
    nnz = n * nb
    wb, fb = (4 if case["weights"] == "f32" else 8), (4 if case["fields"] == "f32" else 8)
    search = {"bytes": n * 24 + nnz * 4 + n * 8, "flops": 8.0 * 3.0 * nnz}
    build = {"bytes": n * 24 + n * 8 + nnz * 4 + nnz * ops * wb,
             "flops": n * (nb * (2.0 * p * p + 6.0 * p + 2.0 * p * ops) + 2.0 / 3.0 * p ** 3 + 2.0 * p * p * ops)}
    apply = {"bytes": nnz * (4 + ops * wb) + n * (8 + fb + ops * fb), "flops": nnz * (1.0 + 2.0 * ops)}
    call = case["call"]
    if call == "stencils":
        return search
    if call == "weights":
        return build
    if call in ("startup", "setup"):
        got = [search, build] + ([apply] if call == "startup" else [])
        return {k: sum(w[k] for w in got) for k in ("bytes", "flops")}
    if call == "apply":
        return apply
    if call == "step":  # one combined weight per entry and stage, and the stage's fields
        st = 4 * case["steps"]
        return {"bytes": st * (nnz * (4 + wb) + n * (8 + 4 * fb)), "flops": st * nnz * 3.0}
    if call == "burgers":
        st = 4 * case["steps"]
        return {"bytes": st * (nnz * (4 + 3 * wb) + n * (8 + 8 * fb)), "flops": st * nnz * 14.0}
    it = 3.0 * case["side"]  # iterations of the linear solver, about: two products and the vector updates each
    return {"bytes": it * (2 * nnz * (4 + 8) + 24 * 8 * n), "flops": it * (4.0 * nnz + 24.0 * n)}


# ---------------------------------------------------------------------------------------------------------------------
# the same outputs in plain torch, double precision
# ---------------------------------------------------------------------------------------------------------------------
def _stencil_rows(case, xy, h, periodic, at):
    """Neighbours of the nodes `at`, ascending: (index [c, N] with -1 behind the last, dx, dy), by comparing the nodes of
    a window of the index lattice with the distance test |r_j - r_i| < 2 h_i."""
    m = case["side"]
    win = 12 if case["nodes"] == "walls" else int(math.ceil(2.0 * case["h"] + 2.0 * case["jitter"])) + 1
    o = torch.arange(-win, win + 1, device=DEV)
    ci, cj = (at % m)[:, None, None] + o[None, None, :], (at // m)[:, None, None] + o[None, :, None]
    ci, cj = torch.broadcast_tensors(ci, cj)
    inside = torch.ones_like(ci, dtype=torch.bool) if periodic else (ci >= 0) & (ci < m) & (cj >= 0) & (cj < m)
    j = ((cj % m) * m + ci % m).reshape(len(at), -1)
    inside = inside.reshape(len(at), -1) & (j != at[:, None])
    d = xy[j] - xy[at][:, None]
    if periodic:
        d = torch.where(d > 0.5, d - 1.0, torch.where(d < -0.5, d + 1.0, d))
    hit = inside & (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] < ((2.0 * h[at]) * (2.0 * h[at]))[:, None])
    order = torch.where(hit, j, torch.full_like(j, m * m)).argsort(1)[:, : int(hit.sum(1).max())]
    hit = hit.gather(1, order)
    return torch.where(hit, j.gather(1, order), torch.full_like(order, -1)), d[..., 0].gather(1, order), d[..., 1].gather(1, order)


def _r_polynomials(k):
    """P_(a,b) with d^(a,b)|r| = |r|^(1-2n) P_(a,b)(x, y), n = a + b, as {(a, b): {(s, t): coefficient of x^s y^t}}."""
    polys = {(1, 0): {(1, 0): 1.0}, (0, 1): {(0, 1): 1.0}}
    for n in range(1, k):
        for a in range(n + 1, -1, -1):
            b = n + 1 - a
            ax = 0 if a > 0 else 1  # differentiate the parent along x where there is one
            parent, got = polys[(a - 1, b) if a > 0 else (a, b - 1)], {}
            for e, c in parent.items():  # d/dx (P r^(1-2n)) = r^(-1-2n) ((x^2 + y^2) dP/dx + (1 - 2n) x P)
                for sq in ((2, 0), (0, 2)):
                    if e[ax]:
                        t = (e[0] + sq[0] - (ax == 0), e[1] + sq[1] - (ax == 1))
                        got[t] = got.get(t, 0.0) + c * e[ax]
                t = (e[0] + (ax == 0), e[1] + (ax == 1))
                got[t] = got.get(t, 0.0) + (1 - 2 * n) * c
            polys[(a, b)] = got
    return polys


def _radial(case, q):
    """First three derivatives of the radial function; the dW0/dr form drops the second and third."""
    if case["rbf"] == "quadratic":
        c = 3.0 / (16.0 * math.pi)
        d = (2.0 * c * (q - 2.0), torch.full_like(q, 2.0 * c), torch.zeros_like(q))
    else:
        c, t = 7.0 / (4.0 * math.pi), 1.0 - 0.5 * q
        d = (-5.0 * c * q * t ** 3, -5.0 * c * t * t * (1.0 - 2.0 * q), 15.0 * c * t * (1.0 - q))
    return d if case["form"] == "chain" else (d[0], torch.zeros_like(q), torch.zeros_like(q))


def _monomials_and_abfs(case, x, y, k):
    q = (x * x + y * y).sqrt()
    d1, d2, d3 = _radial(case, q)
    xs, ys = [torch.ones_like(x)], [torch.ones_like(y)]
    for _ in range(k):
        xs.append(xs[-1] * x)
        ys.append(ys[-1] * y)
    polys, X, W, r = _r_polynomials(k), [], [], {}
    for n in range(1, k + 1):
        for b in range(n + 1):
            a = n - b
            X.append(xs[a] * ys[b] / (math.factorial(a) * math.factorial(b)))
            r[a, b] = sum(c * xs[s] * ys[t] for (s, t), c in polys[a, b].items()) * q ** (1 - 2 * n)
            w = d1 * r[a, b]
            ax = [0] * a + [1] * b
            one = [r[1, 0], r.get((0, 1))]
            two = lambda u, v: r[(u == 0) + (v == 0), (u == 1) + (v == 1)]  # noqa: E731
            if n == 2:
                w = w + d2 * one[ax[0]] * one[ax[1]]
            if n == 3:
                u, v, z = ax
                w = w + d2 * (one[u] * two(v, z) + one[v] * two(u, z) + one[z] * two(u, v)) + d3 * one[u] * one[v] * one[z]
            W.append(w)
    return torch.stack(X, -1), torch.stack(W, -1)


def _exact_weights(case, seed):
    """Every node's neighbours [n, N] (-1: none) and weights [n, N, n_ops]."""
    xy, h, order, periodic, wall = _nodes(case, seed)
    n, C = xy.shape[0], torch.tensor(_targets(case), dtype=F64, device=DEV)
    idx, wts = [], []
    for s0 in range(0, n, 16384):
        at = torch.arange(s0, min(n, s0 + 16384), device=DEV)
        j, dx, dy = _stencil_rows(case, xy, h, periodic, at)
        w = torch.zeros((*j.shape, C.shape[0]), dtype=F64, device=DEV)
        ks = order[at].long() if order is not None else torch.full_like(at, case["order"])
        for k in sorted(set(ks.tolist())):
            p, on = k * (k + 3) // 2, torch.nonzero(ks == k)[:, 0]
            hi = h[at[on]]
            live = (j[on] >= 0)[..., None]
            one = torch.ones_like(hi)[:, None]
            X, W = _monomials_and_abfs(case, torch.where(live[..., 0], dx[on] / hi[:, None], one),
                                       torch.where(live[..., 0], dy[on] / hi[:, None], one), k)
            X, W = X * live, W * live
            deg = torch.tensor([t for t in range(1, k + 1) for _ in range(t + 1)], dtype=F64, device=DEV)
            Ck = C[:, :p].T if C.shape[1] >= p else torch.cat([C.T, torch.zeros((p - C.shape[1], C.shape[0]), dtype=F64, device=DEV)])
            low = torch.stack([deg[Ck[:, d] != 0].max() if bool((Ck[:, d] != 0).any()) else deg[0] for d in range(Ck.shape[1])])
            rhs = Ck[None] * hi[:, None, None] ** (low[None, None] - deg[None, :, None])  # scaled by h^low
            lu, piv = torch.linalg.lu_factor(X.mT @ W)
            psi = torch.linalg.lu_solve(lu, piv, rhs)
            ww = W @ psi
            for _ in range(4):  # refinement on the moment conditions themselves
                ww = ww + W @ torch.linalg.lu_solve(lu, piv, rhs - X.mT @ ww)
            ww = ww * hi[:, None, None] ** -low[None, None]
            w[on] = torch.where(ww.isfinite(), ww, torch.zeros_like(ww))  # a singular corner: fixed, and not used
        idx.append(j)
        wts.append(w)
    N = max(t.shape[1] for t in idx)
    idx = torch.cat([torch.nn.functional.pad(t, (0, N - t.shape[1]), value=-1) for t in idx])
    wts = torch.cat([torch.nn.functional.pad(t, (0, 0, 0, N - t.shape[1])) for t in wts])
    return xy, wall, idx, wts


def _rk4(F, u, dt, steps):
    for _ in range(steps):
        k1 = F(u)
        k2 = F(u + 0.5 * dt * k1)
        k3 = F(u + 0.5 * dt * k2)
        k4 = F(u + dt * k3)
        u = u + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return u


def _bicgstab(A, dinv, b, tol, most):
    x = torch.zeros_like(b)
    for _ in range(8):  # from the true residual again where the recurrence has drifted
        r = b - A(x)
        if float(r.norm()) <= tol * float(b.norm()):
            break
        r0, p, rho = r, r, float(r @ r)
        for _ in range(most):
            y = dinv * p
            v = A(y)
            a = rho / float(r0 @ v)
            s = r - a * v
            z = dinv * s
            t = A(z)
            om = float(t @ s) / float(t @ t)
            x = x + a * y + om * z
            r = s - om * t
            if float(r.norm()) <= 0.3 * tol * float(b.norm()):
                break
            new = float(r0 @ r)
            p = r + (new / rho) * (a / om) * (p - om * v)
            rho = new
    return x


def exact(case, seed):
    call = case["call"]
    if call == "stencils":
        return None  # indices: equal or not
    xy, wall, idx, w = _exact_weights(case, seed)
    live = idx >= 0
    if call in ("weights", "setup"):
        rows = torch.zeros((_capacity(case), w.shape[-1]), dtype=F64, device=DEV)
        rows[: int(live.sum())] = w[live]
        return [None, None, rows] if call == "weights" else [None, None, None, None, rows]
    safe = idx.clamp(min=0)
    f = _field(case, xy, wall, seed)
    if call in ("startup", "apply"):
        f = f.to(torch.float32).to(F64) if case["fields"] == "f32" else f
        return torch.einsum("nj,njd->dn", (f[safe] - f[:, None]) * live, w)
    if call == "solve":
        wl = w[..., 0]
        diag = -wl.sum(1)
        A = lambda x: torch.where(wall, x, diag * x + (wl * x[safe]).sum(1))  # noqa: E731
        return _bicgstab(A, torch.where(wall, torch.ones_like(diag), 1.0 / diag), f, 1e-12, 4000)
    beta, dt = _stepping(case)
    if call == "step":
        wc = (w * torch.tensor(beta, dtype=F64, device=DEV)).sum(-1)
        u = f.to(torch.float32).to(F64) if case["fields"] == "f32" else f
        return _rk4(lambda u: torch.where(wall, 0.0, (wc * (u[safe] - u[:, None])).sum(1)), u, dt, case["steps"])

    def rhs(uv):
        d = (uv[:, safe] - uv[..., None]) * live
        g = torch.einsum("cnj,njd->cnd", d, w)
        return -(uv[0] * g[..., 0] + uv[1] * g[..., 1]) + beta[2] * g[..., 2]

    uv = _rk4(rhs, f, dt, case["steps"])
    return uv[0], uv[1]
