"""Cooperative runs on double fields whose slices are cut between the warps of a block: blocks with a few more slices than
warps, sets whose rows differ a hundredfold, nodes without neighbours, and a row longer than a warp's part, against the
same sums in numpy on the library's own weights; and the time of a stage where a block has just more slices than
warps."""
import numpy as np
import pytest

import labfm_synth as S

from tests.test_gpu_sliced import EPS, _rk4, _row_sums

pytestmark = pytest.mark.gpu


def _set(kind, n):
    rng = np.random.default_rng(n)
    xy = rng.random((n, 2))
    h = np.full(n, 0.5 * np.sqrt(24.0 / n / np.pi))
    if kind == "graded":  # rows of a few entries on the left, of hundreds on the right, in this order
        xy = xy[np.argsort(xy[:, 0])]
        h *= 0.6 + 3.0 * xy[:, 0] ** 3
    elif kind == "holes":  # two thirds of the nodes, in one stretch, have no neighbours
        h[n // 6: 5 * n // 6] = 1e-9
    elif kind == "long":  # three rows of all nodes
        h[[0, n // 2, n - 1]] = 0.75
    return xy, h


SETS = [("even", 87000), ("even", 41000), ("even", 5000), ("graded", 30000), ("holes", 20000), ("holes", 90000), ("long", 3000),
        ("long", 20)]


def _context(xy, h, ops, weight_dtype):
    import torch

    from paper_1912_06441_gb300 import Labfm

    dev = torch.device("cuda", 0)
    L = Labfm(0)
    L.build_neighbours(torch.from_numpy(xy).to(dev), torch.from_numpy(h).to(dev), False)
    status = torch.zeros(len(h), dtype=torch.int32, device=dev)
    L.build_weights(np.stack([S.op_c_vector(o, 2) for o in ops]), uniform_order=2, node_status=status, weight_dtype=weight_dtype)
    rp, col = (t.cpu().numpy() for t in L.get_neighbours())
    return L, rp, col, L.get_weights().cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("kind,n", SETS)
def test_steps_of_cut_slices(kind, n):
    import torch

    L, rp, col, w = _context(*_set(kind, n), ("dx", "dy", "lap"), "f64")
    f = np.random.default_rng(1).random((2, n)) - 0.5
    row = np.repeat(np.arange(n), np.diff(rp))
    beta = np.array([-0.7, 0.4, 0.01])
    wc, lap = w @ beta, 0.01 * w[:, 2]
    most = max(_row_sums(rp, np.abs(wc)).max(), _row_sums(rp, np.abs(w[:, 0]) + np.abs(w[:, 1]) + np.abs(lap)).max())
    dt, steps, size = 0.1 / most, 3, int(np.diff(rp).max())
    tol = 4 * steps * (size + 8) * EPS * 0.4  # a stage's sum is off by at most (N + 3) eps dt sum |w| |du|
    dev = torch.device("cuda", 0)
    u = torch.from_numpy(f[0].copy()).to(dev)
    L.step(beta, u, dt, steps)
    ref = _rk4(lambda s: _row_sums(rp, wc * (s[col] - s[row])), f[0].copy(), dt, steps)
    assert np.abs(u.cpu().numpy() - ref).max() <= tol

    def burgers(uv):
        a, b = uv
        du, dv = a[col] - a[row], b[col] - b[row]
        return np.stack([-(a * _row_sums(rp, w[:, 0] * d) + b * _row_sums(rp, w[:, 1] * d)) + _row_sums(rp, lap * d) for d in (du, dv)])

    u, v = (torch.from_numpy(x.copy()).to(dev) for x in f)
    L.step_burgers([0.0, 0.0, 0.01], u, v, dt, steps)
    ref = _rk4(burgers, f.copy(), dt, steps)
    assert max(np.abs(u.cpu().numpy() - ref[0]).max(), np.abs(v.cpu().numpy() - ref[1]).max()) <= 2 * tol
    L.close()


@pytest.mark.parametrize("kind,n", SETS)
def test_products_of_cut_slices(kind, n):
    """The residual a solve reports of the iterate it leaves (nine rows in ten Dirichlet, one iteration)."""
    import torch

    from paper_1912_06441_gb300 import LabfmError

    L, rp, col, w = _context(*_set(kind, n), ("lap",), "f64")
    f = np.random.default_rng(2).random((2, n)) - 0.5
    fixed = np.arange(n) % 10 != 0
    rhs = np.where(fixed, f[0], 100.0 * f[0])
    dev = torch.device("cuda", 0)
    phi = torch.from_numpy(f[1].copy()).to(dev)
    try:
        L.solve(0, torch.from_numpy(rhs).to(dev), phi, torch.from_numpy(fixed.astype(np.uint8)).to(dev), tol=1e-14, max_iter=1)
    except LabfmError:
        pass
    x, lap = phi.cpu().numpy(), w[:, 0]
    ax = np.where(fixed, x, _row_sums(rp, lap * x[col]) - _row_sums(rp, lap) * x)
    got, ref = L.last_solve[1], np.linalg.norm(rhs - ax) / np.linalg.norm(rhs)
    size, most = int(np.diff(rp).max()), _row_sums(rp, np.abs(lap)).max()
    tol = (size + 8) * EPS * 2 * most * np.abs(x).max() * np.sqrt(n) / np.linalg.norm(rhs) + 1e-12 * ref
    assert abs(got - ref) <= tol
    L.close()


def test_stage_time_of_just_more_slices_than_warps():
    """Stages of 289^2 nodes against 257^2 (on 152 SMs 18 and 14 slices a block of 16 warps): 1.26 times the entries, 1.68
    times the time where the two last slices of a block waited for a second round."""
    import torch

    def stage_us(m):
        at = np.arange(m * m)
        xy = np.stack([(at % m + 0.5) / m, (at // m + 0.5) / m], 1)
        L = _context(xy, np.full(m * m, 1.999 / m), ("lap",), "f64")[0]
        u = torch.from_numpy(np.random.default_rng(0).random(m * m)).to("cuda")
        best = np.inf
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            L.step([0.0], u, 1e-12, 25)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 10.0)
        L.close()
        return best

    assert stage_us(289) <= 1.5 * stage_us(257)


@pytest.mark.parametrize("kind", ["step", "burgers"])
def test_the_first_step_after_a_search_does_not_wait(kind):
    """On a context that has done the same before (its buffers are there), with 50 ms of other work on the stream."""
    import time

    import torch

    m = 100
    at = np.arange(m * m)
    xy, h = np.stack([(at % m + 0.5) / m, (at // m + 0.5) / m], 1), np.full(m * m, 1.999 / m)
    X, H = torch.from_numpy(xy).to("cuda"), torch.from_numpy(h).to("cuda")
    L = _context(xy, h, ("dx", "dy", "lap"), "f64")[0]
    C = np.stack([S.op_c_vector(o, 2) for o in ("dx", "dy", "lap")])
    u, v = (torch.from_numpy(np.random.default_rng(i).random(m * m)).to("cuda") for i in (0, 1))
    run = (lambda: L.step([0.0] * 3, u, 1e-9, 1)) if kind == "step" else (lambda: L.step_burgers([0.0] * 3, u, v, 1e-9, 1))
    for _ in range(3):
        L.build_neighbours(X, H, False)
        L.build_weights(C, uniform_order=2)
        torch.cuda.synchronize()
        torch.cuda._sleep(100000000)
        t = time.perf_counter()
        run()
        t = time.perf_counter() - t
        torch.cuda.synchronize()
    assert t < 0.02
    L.close()
