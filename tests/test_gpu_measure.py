"""The wall diagnostics at the edges of their tiles.

A tile is 128 columns by up to 64 rows (2D) or 8 x 8 rows (3D), fewer on small boxes; its sites
are reduced to 32-bit sign words and its links and wall sites to lists of at most 16 entries per
word and pass.  So: sides on both sides of the tile's, of a word's and of the 16-byte staging's
edges, fields whose every link crosses (checkerboard: 96 links a word) and fields without walls,
zeros of both signs.  Counts must equal the FP64 oracle's on the same values; FP64 sums within
1e-13 (the order of the FP64 sums differs), FP32 within 1e-5 (a few roundings per term).
"""
import numpy as np
import pytest

import oracle
import paper_1710_10420_gb300 as prs
import prs_inputs as inp

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3), (31, 5), (32, 4), (33, 66), (127, 65), (128, 64), (129, 63), (130, 7), (260, 131), (3, 3, 3),
          (4, 9, 8), (126, 8, 9), (127, 7, 10), (128, 16, 16), (129, 17, 5), (132, 9, 4), (255, 3, 19), (384, 32, 8)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available()
    prs.load(build=True)


def _field(shape, kind, dtype):
    rng = np.random.Generator(np.random.PCG64(sum(shape)))
    phi = inp.random_field(shape, seed=7, dtype=dtype)
    if kind == "checkerboard":
        parity = sum(np.meshgrid(*[np.arange(n) for n in phi.shape], indexing="ij")) % 2
        phi = (np.abs(phi) * np.where(parity, -1, 1)).astype(dtype)
    elif kind == "one domain":
        phi = np.abs(phi)
    elif kind == "zeros":
        at = rng.random(phi.shape)
        phi[at < 0.2] = 0.0
        phi[at < 0.1] = -0.0
    return phi, rng.standard_normal(phi.shape).astype(dtype)


@pytest.mark.parametrize("kind", ["noise", "checkerboard", "one domain", "zeros"])
@pytest.mark.parametrize("precision,flags", [(prs.PRS_FP32, 0), (prs.PRS_FP32, prs.PRS_FP32_CR), (prs.PRS_FP64, 0)])
@pytest.mark.parametrize("shape", SHAPES)
def test_diagnostics_at_tile_edges(shape, precision, flags, kind):
    dtype = np.float32 if precision == prs.PRS_FP32 else np.float64
    phi, v = _field(shape, kind, dtype)
    sim = prs.Sim(shape, precision=precision, flags=flags)
    sim.init(phi, v)
    d = prs.prs_measure_ex(sim.handle)
    ref = oracle.measure(oracle.Params(shape), phi.astype(np.float64), v.astype(np.float64))
    sim.close()
    assert (d.n_links, d.n_wall, d.n_vzero, d.n_nonfinite) == (ref.n_links, ref.n_wall, ref.n_vzero, 0)
    tol = 1e-5 if precision == prs.PRS_FP32 else 1e-13
    assert d.sum_w == pytest.approx(ref.sum_w, rel=tol)
    assert d.sum_ratio == pytest.approx(ref.sum_ratio, rel=tol)


@pytest.mark.parametrize("precision", [prs.PRS_FP32, prs.PRS_FP64])
@pytest.mark.parametrize("shape", [(130, 70), (128, 9, 8)])
def test_non_finite_sites_are_counted_once(shape, precision):
    dtype = np.float32 if precision == prs.PRS_FP32 else np.float64
    phi, v = _field(shape, "one domain", dtype)
    flat_p, flat_v = phi.reshape(-1), v.reshape(-1)
    flat_p[0], flat_p[-1], flat_v[0], flat_v[shape[0]] = np.nan, np.inf, np.inf, -np.inf
    sim = prs.Sim(shape, precision=precision)
    sim.init(phi, v)
    d = prs.prs_measure_ex(sim.handle)
    sim.close()
    assert d.n_nonfinite == 3 and d.n_links == 0
