"""Solves to a tolerance near the rounding of the system: the Neumann square (order 4) to 1e-13, whose residual in the
global form of the rows cannot be formed to better than about that."""
import numpy as np
import pytest

from tests import gpu_common as G
from tests import test_oracle_pins as OP

pytestmark = pytest.mark.gpu
FIELD = (lambda x, y: np.sin(2 * x + 0.3) * np.cos(3 * y - 0.2), lambda x, y: 2 * np.cos(2 * x + 0.3) * np.cos(3 * y - 0.2),
         lambda x, y: -3 * np.sin(2 * x + 0.3) * np.sin(3 * y - 0.2), lambda x, y: -13 * np.sin(2 * x + 0.3) * np.cos(3 * y - 0.2))


@pytest.mark.parametrize("nside", [37, 39, 41, 43, 45, 49, 53])
def test_solves_at_the_rounding_floor(nside):
    """It converges, and the residual it reports is that of the sums over differences in extended precision."""
    import torch

    q, rp, col, _, _, f = OP.neumann_problem(nside, 4, FIELD)
    L, _, _, w, _, _ = G.gpu_run(q.ns, 4, ("dx", "dy", "lap"), rbf="quadratic", abf_form="dw0")
    dev = torch.device("cuda", 0)
    phi = torch.zeros(q.ns.n, dtype=torch.float64, device=dev)
    nm = tuple(torch.from_numpy(a).to(dev) for a in (q.ghost, q.parent, q.normal)) + (0, 1)
    tol = 1e-13
    _, resid = L.solve(2, torch.from_numpy(f).to(dev), phi, torch.from_numpy(q.dirichlet.astype(np.uint8)).to(dev), tol=tol,
                       max_iter=20000, neumann=nm)
    assert resid <= tol
    x, w = phi.cpu().numpy().astype(np.longdouble), w.astype(np.longdouble)
    row = np.repeat(np.arange(q.ns.n), np.diff(rp))
    ax = np.add.reduceat(w[:, 2] * (x[col] - x[row]), rp[:-1])
    for g, b, nrm in zip(q.ghost, q.parent, q.normal):
        s = slice(rp[b], rp[b + 1])
        ax[g] = ((nrm[0] * w[s, 0] + nrm[1] * w[s, 1]) * (x[col[s]] - x[b])).sum()
    ax[q.dirichlet] = x[q.dirichlet]
    true = float(np.linalg.norm((f - ax).astype(float)) / np.linalg.norm(f))
    # each row's sum is off by at most (N + 2) eps sum |w| |x_j - x_i|
    absum = np.add.reduceat(np.abs(w[:, 2] * (x[col] - x[row])), rp[:-1]).astype(float)
    tol_r = (np.diff(rp).max() + 2) * np.finfo(float).eps * np.linalg.norm(absum) / np.linalg.norm(f)
    assert abs(resid - true) <= tol_r
    L.close()
