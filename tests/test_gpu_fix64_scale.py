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
DROPS = [np.nextafter(2.0 ** -10, 0.0), 2.0 ** -40 * (1.0 - 2.0 ** -30), 3e-7, 1e-30]


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
