"""The FP64 fixed-point step where the size of the field changes: every site to the precision of its own
terms, not of the largest value of the box.

One step against the oracle.  With u = 2^-53, A = c2 (sum of |neighbours| + 2D |phi|)/dx^2 and
B = c2 cV |phi| (1 + phi^2/phi0^2), the oracle's operations round the force by at most 9 u A + 11 u B (the
neighbour sum 3, the centre term, the difference and 1/dx^2 6, the force 8, their difference and c2 3), the
folded double form by 6 u A + 6 u B, and the kick and its constants add 2 u (|v'| + c1 |v|) a side.
"""
import numpy as np
import pytest

import oracle
import paper_1710_10420_gb300 as prs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available()
    prs.load(build=True)


def _step(shape, phi, v, **kw):
    sim = prs.Sim(shape, precision=prs.PRS_FP64, **kw)
    sim.init(phi, v)
    sim.step(1)
    a, b, _ = sim.get_state()
    sim.close()
    return a, b


def _check(shape, phi, v, **kw):
    a, b = _step(shape, phi, v, **kw)
    p = oracle.Params(shape, **kw)
    oa, ob = oracle.step(p, phi, v, 1)
    c = oracle.coeffs(p, 0)
    near = sum(np.abs(np.roll(phi, s, axis)) for axis in range(phi.ndim) for s in (1, -1))
    A = c["c2"] / kw.get("dx", 1.0) ** 2 * (near + 2 * phi.ndim * np.abs(phi))
    B = c["c2"] * c["cV"] * np.abs(phi) * (1.0 + (phi / kw.get("phi0", 1.0)) ** 2)
    tol = U * (15.0 * A + 17.0 * B + 4.0 * (np.abs(ob) + np.abs(v)))
    assert np.all(np.abs(b - ob) <= tol), float(np.max(np.abs(b - ob) / np.maximum(tol, 1e-300)))
    assert np.all(np.abs(a - oa) <= 0.1 * tol + 2 * U * np.abs(oa))
    na, nb = _step(shape, -phi, -v, **kw)  # odd in phi, bit for bit
    assert np.array_equal(na, -a) and np.array_equal(nb, -b)


# values just below a power of two round up to it in fewer bits
DROPS = [np.nextafter(2.0 ** -10, 0.0), 2.0 ** -40 * (1.0 - 2.0 ** -30), 3e-7, 1e-30, 1e-290]


@pytest.mark.parametrize("drop", DROPS)
@pytest.mark.parametrize("shape", [(64, 60), (700, 400), (64, 20, 24)])
def test_planes_behind_a_drop_in_size(shape, drop):
    """Along the march axis two planes of order one, then small ones, and back."""
    phi = np.full(tuple(reversed(shape)), drop)
    n = phi.shape[0]
    for at in (0, n // 3, n // 2):
        phi[at:at + 2] = 0.9
    sign = np.where(np.arange(n) % 5 == 0, -1.0, 1.0)
    phi *= sign.reshape([-1] + [1] * (phi.ndim - 1))
    _check(shape, phi, np.zeros_like(phi))


def _smooth_noise(rng, fshape, amplitude):
    phi = rng.uniform(-1.0, 1.0, fshape)
    for axis in range(phi.ndim):
        phi = phi + np.roll(phi, 1, axis) + np.roll(phi, -1, axis)
    return amplitude * phi / np.max(np.abs(phi))


def _varied(kind, fshape):
    rng = np.random.Generator(np.random.PCG64(sum(fshape) * 10 + len(fshape)))
    at = np.meshgrid(*[np.arange(n) - n // 3 for n in fshape], indexing="ij")
    r2 = sum(x.astype(np.float64) ** 2 for x in at)
    if kind == "bump":  # a localised perturbation of the symmetric state
        return 0.7 * np.exp(-r2 / 8.0) + _smooth_noise(rng, fshape, 1e-9)
    if kind == "bump on zeros":
        return 0.7 * np.exp(-r2 / 8.0) * (r2 < 60.0)
    if kind == "columns":  # every power of two in the columns of one warp
        return 1.2 * 2.0 ** -(np.abs(at[-1]) % 50).astype(np.float64) * rng.choice([-1.0, 1.0], fshape)
    if kind == "blocks":  # sizes that change from block to block, along every axis
        exps = rng.uniform(-14.0, 0.0, [n // 7 + 1 for n in fshape])
        for axis, n in enumerate(fshape):
            exps = np.repeat(exps, 7, axis).take(range(n), axis)
        return 10.0 ** exps * rng.uniform(-1.0, 1.0, fshape)
    walls = np.tanh(np.sin(2.0 * np.pi * at[0] / fshape[0]) + 0.7 * np.sin(2.0 * np.pi * at[-1] / fshape[-1]))
    return walls * 1e-6 if kind == "linear growth" else walls


@pytest.mark.parametrize("kind", ["bump", "bump on zeros", "columns", "blocks", "walls", "linear growth"])
@pytest.mark.parametrize("phi0,dx", [(1.0, 1.0), (1.3, 0.7), (1.0, 6.0)])
@pytest.mark.parametrize("shape", [(64, 60), (700, 400), (31, 17, 20), (64, 33, 40)])
def test_small_values_beside_large_ones(shape, phi0, dx, kind):
    fshape = tuple(reversed(shape))
    rng = np.random.Generator(np.random.PCG64(7))
    phi = phi0 * _varied(kind, fshape)
    _check(shape, phi, 1e-3 * phi * rng.standard_normal(fshape), phi0=phi0, dx=dx, W0=7.0)
