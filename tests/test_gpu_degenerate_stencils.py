"""Node sets whose stencils have |dy| = 2^e |dx| throughout: two rows of X are equal up to a power of two, every M is
singular, and every node is flagged, without weights, at the orders built from moments as at the others."""
import numpy as np
import pytest

import labfm_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["dw0", "chain"])
@pytest.mark.parametrize("k", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("slope", [1.0, -1.0, 2.0, 0.5])
def test_nodes_on_a_line(slope, k, form):
    import torch

    from paper_1912_06441_gb300 import Labfm

    rng = np.random.default_rng(5)
    t = rng.choice(1 << 19, 300, replace=False) / 2.0 ** 20 + 0.25  # dyadic: every offset is exact
    xy = np.stack([t, 0.5 + slope * (t - 0.5)], 1)
    dev = torch.device("cuda", 0)
    L = Labfm(0)
    L.build_neighbours(torch.from_numpy(xy).to(dev), torch.full((300,), 0.1, dtype=torch.float64, device=dev), False)
    status = torch.zeros(300, dtype=torch.int32, device=dev)
    bad = L.build_weights(S.op_c_vector("dx", k)[None], uniform_order=k, node_status=status, abf_form=form, rbf="quadratic")
    assert bad == 300 and bool((status != 0).all())
    assert bool((L.get_weights() == 0).all())
    L.close()
