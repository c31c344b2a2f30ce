"""The FP64 step whose force runs in 64-bit fixed point, at the edges of what it takes.

A warp owns 30 output columns and four rows (2D: one), so sides on both sides of 30, 60 and 16, and
boxes smaller than a warp; amplitudes at which every warp takes the integers, none does (values below
1/16 or at 2 phi0 and beyond), or some do; phi0 away from a power of two.  One step against the oracle:
each double operation of either side rounds terms of at most c1 |v|, 12 g |phi| and c2 |f| by 2^-53, so
the kick may differ by 2^-53 (2 |v'| + 8 times the largest term), the drift by deta times that and an ulp.
"""
import math

import numpy as np
import pytest

import oracle
import paper_1710_10420_gb300 as prs

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3), (29, 5), (30, 7), (31, 40), (61, 33), (128, 130), (4030, 66), (4031, 66), (4097, 64), (5, 52429),
          (3, 3, 3), (30, 16, 4), (31, 17, 5), (59, 15, 9), (90, 33, 3), (64, 20, 21)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available()
    prs.load(build=True)


def _field(shape, kind, phi0):
    rng = np.random.Generator(np.random.PCG64(len(shape) * 1000 + sum(shape)))
    fshape = tuple(reversed(shape))
    phi = phi0 * rng.uniform(-1.0, 1.0, fshape)
    if kind == "small":
        phi *= 1e-3
    elif kind == "large":
        phi *= 7.0
    elif kind == "mixed":  # warps of both forms, and values across the whole exponent range
        phi *= np.where(rng.random(fshape) < 0.5, 1.0, 10.0 ** rng.uniform(-300, 0, fshape))
        phi.reshape(-1)[:: max(7, phi.size // 5)] = 0.0
        phi[fshape[0] // 2:] *= 1e-4
    return phi, 0.1 * phi0 * rng.standard_normal(fshape)


def _step(shape, phi, v, phi0, dx):
    sim = prs.Sim(shape, precision=prs.PRS_FP64, phi0=phi0, dx=dx, W0=7.0)
    sim.init(phi, v)
    sim.step(1)
    a, b, _ = sim.get_state()
    sim.close()
    return a, b


@pytest.mark.parametrize("kind", ["full", "small", "large", "mixed"])
@pytest.mark.parametrize("phi0,dx", [(1.0, 1.0), (1.3, 0.7)])
@pytest.mark.parametrize("shape", SHAPES)
def test_one_step_against_the_oracle(shape, phi0, dx, kind):
    phi, v = _field(shape, kind, phi0)
    a, b = _step(shape, phi, v, phi0, dx)
    p = oracle.Params(shape, phi0=phi0, dx=dx, W0=7.0)
    oa, ob = oracle.step(p, phi, v, 1)
    c = oracle.coeffs(p, 0)
    top = np.max(np.abs(phi))
    term = max(12.0 * c["c2"] / dx ** 2 * top, c["c2"] * c["cV"] * top * (1.0 + (top / phi0) ** 2))
    tol_v = 2.0 ** -53 * (2.0 * np.abs(ob) + np.abs(v) + 8.0 * term)
    assert np.all(np.abs(b - ob) <= tol_v)
    assert np.all(np.abs(a - oa) <= 0.1 * tol_v + 2.0 ** -52 * np.abs(oa))
    na, nb = _step(shape, -phi, -v, phi0, dx)  # odd in phi, bit for bit
    assert np.array_equal(na, -a) and np.array_equal(nb, -b)


@pytest.mark.parametrize("shape", [(61, 33), (517, 509), (31, 17, 5)])
def test_a_non_finite_value_reaches_its_neighbours_only(shape):
    phi, v = _field(shape, "full", 1.0)
    phi.reshape(-1)[phi.size // 2] = math.inf
    a, b = _step(shape, phi, v, 1.0, 1.0)
    bad = ~np.isfinite(b)
    want = np.isinf(phi)
    for axis in range(phi.ndim):
        want = want | np.isinf(np.roll(phi, 1, axis)) | np.isinf(np.roll(phi, -1, axis))
    assert np.array_equal(bad, want) and np.array_equal(~np.isfinite(a), want)
