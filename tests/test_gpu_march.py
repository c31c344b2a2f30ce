"""The register marches (FP32 steps of any box, several a pass) at the edges of their strips and chunks.

A strip keeps 52 to 60 (2D also 112 and 120) of its 64 (128) columns, a warp takes four rows in 3D, and
a call's steps are planned into passes of up to six (2D) or three (3D).  Every pass evaluates a site as
one step a pass does, so the fields are those of tblock = 1 bit for bit, whatever the sides, the number of
steps and the owner of the buffers; one step a pass follows the oracle to 1e-5 (as in the parity tests).
The reverse steps of the same boxes follow the oracle's gradient to 1e-5.
"""
import numpy as np
import pytest

import oracle
import paper_1710_10420_gb300 as prs
import prs_inputs as inp

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3), (51, 7), (52, 9), (53, 40), (57, 3), (111, 5), (113, 64), (121, 33), (250, 61), (384, 20), (128, 4),
          (3, 3, 3), (55, 4, 5), (56, 5, 9), (57, 17, 6), (60, 16, 7), (61, 15, 20), (121, 6, 4), (128, 16, 12),
          (130, 9, 33)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available()
    prs.load(build=True)


def _owned(shape, phi, v, calls, **kw):
    h = prs.prs_create(prs.make_params(shape, **kw))
    prs.prs_init(h, phi, v)
    for k in calls:
        prs.prs_step(h, k)
    a, b = np.empty_like(phi), np.empty_like(v)
    assert prs.prs_get_state(h, a, b) == sum(calls)
    prs.prs_destroy(h)
    return a, b


@pytest.mark.parametrize("shape", SHAPES)
def test_planned_passes_equal_single_steps(shape):
    phi = inp.random_field(shape, seed=51, dtype=np.float32)
    v = (0.1 * inp.random_field(shape, seed=52)).astype(np.float32)
    calls = (1, 2, 3, 4, 5, 7, 11)
    one = _owned(shape, phi, v, calls, tblock=1)
    many = _owned(shape, phi, v, calls)
    assert np.array_equal(one[0], many[0]) and np.array_equal(one[1], many[1])
    sim = prs.Sim(shape)
    sim.init(phi, v)
    home = sim._bufs[2].data_ptr()
    for k in calls:
        sim.step(k)
        assert prs.prs_device_state(sim.handle)[1] == home
    a, b, n = sim.get_state()
    sim.close()
    assert n == sum(calls) and np.array_equal(a, one[0]) and np.array_equal(b, one[1])
    p = oracle.Params(shape)
    oa, ob = oracle.step(p, phi.astype(np.float64), v.astype(np.float64), 6)
    a, b = _owned(shape, phi, v, (6,))
    assert np.max(np.abs(a - oa)) <= 1e-5 * np.max(np.abs(oa)) and np.max(np.abs(b - ob)) <= 1e-5 * np.max(np.abs(ob))


@pytest.mark.parametrize("shape", [(3, 3, 3), (59, 4, 5), (60, 17, 6), (61, 15, 9), (128, 24, 5), (130, 9, 12)])
def test_reverse_steps_at_strip_edges(shape):
    import torch

    phi = (0.8 * inp.random_field(shape, seed=53)).astype(np.float32)
    v = (0.05 * inp.random_field(shape, seed=54)).astype(np.float32)
    sim = prs.Sim(shape, W0=6.0, eta0=2.0)
    sim.init(phi, v)
    gp, gv = (torch.empty(tuple(reversed(shape)), dtype=torch.float32, device="cuda") for _ in range(2))
    J, dA = prs.prs_adjoint(sim.handle, 7, prs.PRS_OBS_SMOOTH_AREA, 0.3, 3, gp, gv)
    sim.close()
    ref = oracle.adjoint(oracle.Params(shape, W0=6.0, eta0=2.0), phi.astype(np.float64), v.astype(np.float64), 7,
                         prs.PRS_OBS_SMOOTH_AREA, 0.3)
    assert J == pytest.approx(ref["J"], rel=1e-5)
    assert abs(dA - ref["dJ_dalpha"]) <= 1e-5 * max(abs(ref["dJ_dalpha"]), 1e-3 * abs(ref["J"]))
    for got, want in ((gp, ref["dJ_dphi"]), (gv, ref["dJ_dv"])):
        assert np.max(np.abs(got.cpu().numpy() - want)) <= 1e-5 * np.max(np.abs(want))
