"""Waits between the blocks of a cooperative run that give up (a library compiled with a limit of one read, which all but
the last blocks to arrive use up; every wait still ends by itself): what is reported, by which call, what happens to
runs enqueued behind, and that the context goes on afterwards.  And a run longer than one launch."""
import os
import subprocess

import numpy as np
import pytest

import labfm_synth as S

from tests.test_gpu_sliced import EPS, _context, _rk4, _row_sums

pytestmark = pytest.mark.gpu
TIMEOUT = 6


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _random(n, rows=1):
    return np.random.default_rng(n).random((rows, n)) - 0.5


def _gives_up(L, call):
    import torch

    from paper_1912_06441_gb300 import LabfmError

    with pytest.raises(LabfmError) as e:
        torch.cuda.synchronize()
        call()
    assert e.value.status == TIMEOUT
    return str(e.value)


@pytest.fixture(scope="module")
def limited_library(tmp_path_factory):
    """liblabfm with LABFM_SYNC_POLLS = 1: the two files with such runs compiled again, linked with the others' objects."""
    import paper_1912_06441_gb300 as P
    from paper_1912_06441_gb300 import build as B

    B.build_library()
    out = tmp_path_factory.mktemp("limited")
    jobs = [subprocess.Popen([B._nvcc(), *B.ARCH, *B.FLAGS, "-DLABFM_SYNC_POLLS=1u", "-c", os.path.join(B.CSRC, f + ".cu"), "-o",
                              str(out / (f + ".o"))]) for f in ("apply", "solve")]
    assert [j.wait() for j in jobs] == [0, 0]
    objs = [str(out / f) if (out / f).exists() else os.path.join(B.OUT_DIR, f) for f in (s[:-3] + ".o" for s in B.SOURCES)]
    lib = str(out / "liblabfm_limited.so")
    subprocess.run([B._nvcc(), *B.ARCH, "-shared", "-o", lib, *objs, "-lcudart_static", "-ldl", "-lrt", "-lpthread"], check=True)
    return P.load_library(lib)


@pytest.fixture
def limited(limited_library, monkeypatch):
    import paper_1912_06441_gb300 as P

    with monkeypatch.context() as m:
        m.setattr(P, "_lib", limited_library)
        L = _context(5000, False, "f64")[0]
    yield L
    L.close()


@pytest.mark.parametrize("kind", ["step", "burgers"])
def test_a_run_that_gives_up_is_reported_once(limited, kind):
    import torch

    L, beta = limited, [0.0, 0.0, 1e-9]
    run = (lambda u, v: L.step(beta, u, 1e-9, 3)) if kind == "step" else (lambda u, v: L.step_burgers(beta, u, v, 1e-9, 3))
    u, v = _dev(_random(5000)[0]), _dev(_random(5000)[0])
    run(u, v)
    assert "earlier run" in _gives_up(L, lambda: L.step(beta, u, 1e-9, 0))
    assert L.step(beta, u, 1e-9, 0) is u  # reported
    f = _dev(_random(5000)[0])
    torch.cuda.synchronize()
    assert bool(L.apply(f).isfinite().all())


def test_runs_behind_it_leave_their_fields(limited):
    import torch

    from paper_1912_06441_gb300 import LabfmError

    L, beta = limited, [0.0, 0.0, 1e-9]
    u = [_dev(_random(5000)[0]) for _ in range(6)]
    before = u[0].clone()
    reported = 0
    for x in u:
        try:
            L.step(beta, x, 1e-3, 2)
        except LabfmError as e:  # the first run may have ended by now
            assert e.status == TIMEOUT
            reported += 1
            break
    torch.cuda.synchronize()
    if not reported:
        _gives_up(L, lambda: L.step(beta, u[0], 1e-9, 0))
    assert all(torch.equal(x, before) for x in u[1:])


def test_builds_report_it_and_the_context_goes_on(limited):
    """Four nodes are one slice: the run has one block, whose waits end at the first read."""
    import torch

    L, beta = limited, [0.0, 0.0, 1e-9]
    u = _dev(_random(5000)[0])
    C = np.stack([S.op_c_vector(o, 2) for o in ("dx", "dy", "lap")])
    L.step(beta, u, 1e-9, 2)
    _gives_up(L, lambda: L.build_weights(C, uniform_order=2, node_status=torch.zeros(5000, dtype=torch.int32, device="cuda")))
    L.build_weights(C, uniform_order=2, node_status=torch.zeros(5000, dtype=torch.int32, device="cuda"))
    L.step(beta, u, 1e-9, 2)
    xy, h = np.array([[0.3, 0.3], [0.6, 0.35], [0.32, 0.62], [0.7, 0.65]]), np.full(4, 0.4)
    _gives_up(L, lambda: L.build_neighbours(_dev(xy), _dev(h), False))
    L.build_neighbours(_dev(xy), _dev(h), False)
    C = np.stack([S.op_c_vector(o, 1) for o in ("dx", "dy")])
    L.build_weights(C, uniform_order=1, node_status=torch.zeros(4, dtype=torch.int32, device="cuda"))
    rp, col = (t.cpu().numpy() for t in L.get_neighbours())
    wc = L.get_weights().cpu().numpy() @ np.array([0.3, -0.2])
    f = _random(4)[0]
    row = np.repeat(np.arange(4), np.diff(rp))
    dt = 0.1 / _row_sums(rp, np.abs(wc)).max()
    x = _dev(f)
    L.step([0.3, -0.2], x, dt, 1)
    ref = _rk4(lambda s: _row_sums(rp, wc * (s[col] - s[row])), f, dt, 1)
    assert np.abs(x.cpu().numpy() - ref).max() <= 4 * (3 + 8) * EPS * 0.4 < np.abs(ref - f).max()


def test_a_solve_tells_its_own_wait_from_an_earlier_run(limited):
    L = limited
    f, phi = _dev(_random(5000)[0]), _dev(np.zeros(5000))
    assert "solver" in _gives_up(L, lambda: L.solve(2, f, phi))
    L.step([0.0, 0.0, 1e-9], f.clone(), 1e-9, 2)
    assert "earlier run" in _gives_up(L, lambda: L.solve(2, f, phi))
    assert "solver" in _gives_up(L, lambda: L.solve(2, f, phi))


def test_a_run_of_several_launches():
    """1e9 / (entries + 1e5) steps go into one launch: as many and some more against the same in two calls, bit for bit."""
    L, rp, _, _, f = _context(40, False, "f64")
    per = int(1000000000 // (rp[-1] + 100000))
    beta, dt = [0.1, -0.2, 1e-3], 1e-9
    one, two = _dev(f[0]), _dev(f[0])
    L.step(beta, one, dt, per + 50)
    L.step(beta, two, dt, per // 2)
    L.step(beta, two, dt, per + 50 - per // 2)
    assert np.array_equal(one.cpu().numpy(), two.cpu().numpy())
    one, two = (_dev(f[0]), _dev(f[1])), (_dev(f[0]), _dev(f[1]))
    L.step_burgers([0.0, 0.0, 1e-3], *one, dt, per + 50)
    L.step_burgers([0.0, 0.0, 1e-3], *two, dt, per // 2)
    L.step_burgers([0.0, 0.0, 1e-3], *two, dt, per + 50 - per // 2)
    assert all(np.array_equal(a.cpu().numpy(), b.cpu().numpy()) for a, b in zip(one, two))
    L.close()
