"""The FP32 observables and their gradients at the edges of the kernel's tiles (32 x 8 columns marched in
chunks of at least 8 planes; in 2D 256 columns), against the oracle on the same values: a site's value is
a few float roundings of terms of order one (J: within 1e-5, as the adjoint tests; the gradient likewise
relative to its largest entry)."""
import numpy as np
import pytest

import oracle
import paper_1710_10420_gb300 as prs
import prs_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("obs", [prs.PRS_OBS_GRAD_ENERGY, prs.PRS_OBS_SMOOTH_AREA])
@pytest.mark.parametrize("shape", [(3, 3), (255, 9), (256, 8), (257, 17), (3, 3, 3), (31, 7, 9), (32, 8, 8), (33, 9, 17),
                                   (64, 17, 5)])
def test_observable_at_tile_edges(shape, obs):
    import torch

    prs.load(build=True)
    phi = (0.8 * inp.random_field(shape, seed=41)).astype(np.float32)
    sim = prs.Sim(shape, precision=prs.PRS_FP32)
    sim.init(phi)
    g = torch.empty(tuple(reversed(shape)), dtype=torch.float32, device="cuda")
    J, dA = prs.prs_adjoint(sim.handle, 0, obs, 0.3, 0, g, None)
    J2 = prs.prs_observable(sim.handle, obs, 0.3)
    sim.close()
    p, ref = oracle.Params(shape), phi.astype(np.float64)
    want, grad = oracle.observable(p, obs, ref, 0.3), oracle.observable_grad(p, obs, ref, 0.3)
    assert J == pytest.approx(want, rel=1e-5) and J2 == J and dA == 0.0
    assert np.max(np.abs(g.cpu().numpy() - grad)) <= 1e-5 * np.max(np.abs(grad))
