"""RK4 and Burgers stages and the solver's product on double fields (the sliced stencil layout): node counts around a
slice and a block of slices, one to sixteen lanes a node, and a set whose stencils differ so much that a node gets a
whole warp, against the same sums in numpy on the library's own weights."""
import numpy as np
import pytest

import labfm_synth as S

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def _context(n, uneven, weight_dtype):
    """n random nodes in a unit box, stencils of about 24 nodes (uneven: every 40th node's about 40 times that), with
    stand-in operators of order 1 and 2 (values do not matter here, only that all come from the same weights)."""
    import torch

    from paper_1912_06441_gb300 import Labfm

    rng = np.random.default_rng(n)
    dev = torch.device("cuda", 0)
    xy = rng.random((n, 2))
    h = np.full(n, 0.5 * np.sqrt(min(24.0 / n, 0.9) / np.pi))
    if uneven:
        h[::40] *= 6.0
    L = Labfm(0)
    L.build_neighbours(torch.from_numpy(xy).to(dev), torch.from_numpy(h).to(dev), False)
    C = np.stack([S.op_c_vector(o, 2) for o in ("dx", "dy", "lap")])
    status = torch.zeros(n, dtype=torch.int32, device=dev)
    L.build_weights(C, uniform_order=2, node_status=status, weight_dtype=weight_dtype)
    rp, col = (t.cpu().numpy() for t in L.get_neighbours())
    w = L.get_weights().cpu().numpy().astype(np.float64)
    return L, rp, col, w, rng.random((2, n)) - 0.5


def _row_sums(rp, v):
    return np.add.reduceat(np.concatenate([v, [0.0]]), rp[:-1]) * (rp[1:] > rp[:-1])


def _rk4(F, u, dt, steps):
    for _ in range(steps):
        k1 = F(u)
        k2 = F(u + 0.5 * dt * k1)
        k3 = F(u + 0.5 * dt * k2)
        k4 = F(u + dt * k3)
        u = u + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return u


SETS = [(40, False), (31, False), (1000, False), (4864, False), (9728, False), (26000, False), (70000, False), (6000, True)]


@pytest.mark.parametrize("weight_dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,uneven", SETS)
def test_stages_on_double_fields(n, uneven, weight_dtype):
    import torch

    L, rp, col, w, f = _context(n, uneven, weight_dtype)
    row = np.repeat(np.arange(n), np.diff(rp))
    beta = np.array([-0.7, 0.4, 0.01])
    wc = w @ beta
    if weight_dtype == "f32":
        wc = wc.astype(np.float32).astype(np.float64)  # stored so
    most = max(_row_sums(rp, np.abs(wc)).max(), _row_sums(rp, np.abs(w[:, 0]) + np.abs(w[:, 1]) + np.abs(wc)).max())
    dt, steps, size = 0.1 / most, 3, int(np.diff(rp).max())
    # a stage's sum is off by at most (N + 3) eps dt sum |w| |du|, |du| <= 2 max |u|, and so on over 4 stages a step
    tol = 4 * steps * (size + 8) * EPS * 0.4
    frozen = (np.arange(n) % 7 == 0).astype(np.uint8)
    dev = torch.device("cuda", 0)
    u = torch.from_numpy(f[0].copy()).to(dev)
    L.step(beta, u, dt, steps, frozen=torch.from_numpy(frozen).to(dev))
    ref = _rk4(lambda s: np.where(frozen, 0.0, _row_sums(rp, wc * (s[col] - s[row]))), f[0].copy(), dt, steps)
    assert np.abs(u.cpu().numpy() - ref).max() <= tol

    lap = 0.01 * w[:, 2]
    if weight_dtype == "f32":
        lap = lap.astype(np.float32).astype(np.float64)

    def burgers(uv):
        a, b = uv
        du, dv = a[col] - a[row], b[col] - b[row]
        F = [-(a * _row_sums(rp, w[:, 0] * d) + b * _row_sums(rp, w[:, 1] * d)) + _row_sums(rp, lap * d) for d in (du, dv)]
        return np.where(frozen, 0.0, np.stack(F))

    u, v = (torch.from_numpy(x.copy()).to(dev) for x in f)
    L.step_burgers([0.0, 0.0, 0.01], u, v, dt, steps, frozen=torch.from_numpy(frozen).to(dev))
    ref = _rk4(burgers, f.copy(), dt, steps)
    assert max(np.abs(u.cpu().numpy() - ref[0]).max(), np.abs(v.cpu().numpy() - ref[1]).max()) <= 2 * tol
    L.close()


@pytest.mark.parametrize("n,uneven", SETS)
def test_solver_product(n, uneven):
    """The residual that a solve reports, of an iterate it leaves as it was (every row Dirichlet but one in ten, and an
    unreachable iteration limit of one): ||F - A phi|| / ||F|| recomputed from the weights."""
    import torch

    from paper_1912_06441_gb300 import LabfmError

    L, rp, col, w, f = _context(n, uneven, "f64")
    row = np.repeat(np.arange(n), np.diff(rp))
    fixed = np.arange(n) % 10 != 0
    rhs = np.where(fixed, f[0], 100.0 * f[0])
    dev = torch.device("cuda", 0)
    phi = torch.from_numpy(f[1].copy()).to(dev)
    try:
        L.solve(2, torch.from_numpy(rhs).to(dev), phi, torch.from_numpy(fixed.astype(np.uint8)).to(dev), tol=1e-14, max_iter=1)
    except LabfmError:
        pass
    x = phi.cpu().numpy()
    assert np.array_equal(x[fixed], rhs[fixed])
    lap = w[:, 2]
    ax = np.where(fixed, x, _row_sums(rp, lap * x[col]) - _row_sums(rp, lap) * x)
    got, ref = L.last_solve[1], np.linalg.norm(rhs - ax) / np.linalg.norm(rhs)
    size, most = int(np.diff(rp).max()), _row_sums(rp, np.abs(lap)).max()
    tol = (size + 8) * EPS * 2 * most * np.abs(x).max() * np.sqrt(n) / np.linalg.norm(rhs) + 1e-12 * ref
    assert abs(got - ref) <= tol
    L.close()
