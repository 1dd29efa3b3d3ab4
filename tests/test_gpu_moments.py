"""FP64 weights of the orders built from moments, in both forms of the ABFs, against the oracle: stencils just above the
order's need, of about one staged chunk, and of several, and a node set of a few listed nodes per group."""
import numpy as np
import pytest

import labfm_synth as S

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["chain", "dw0"])
@pytest.mark.parametrize("k", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("wide", [1.0, 1.1, 1.5])
def test_moment_weights(k, form, wide):
    ns = S.jittered_lattice(29, G.HS[k] * wide, k, seed=60 + k, jitter=0.2)
    ops = G.OPS[k]
    rbf = "wendland_c6" if wide > 1.2 else "wendland_c2"
    _, rp, col, w, status, _ = G.gpu_run(ns, k, ops, rbf=rbf, abf_form=form)
    q = np.arange(1, ns.n, 7)
    rp_q, col_q, idx = G.rows_of(rp, col, q)
    r64, rld = G.oracle_refs(ns, k, ops, q, rp_q, col_q, rbf=rbf, abf_form=form)
    assert np.array_equal(status[q], r64["status"])
    G.assert_weights_parity(w[idx], r64, rld, rp_q, label=f"{form} k={k} x{wide}")
