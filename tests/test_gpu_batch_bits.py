"""An ensemble's fields are those of its runs stepped alone, bit for bit: runs that share launches, leave their
group early, ask for a tblock of their own or are the only one of their box."""
import numpy as np
import pytest

import paper_1710_10420_gb300 as prs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available()
    prs.load(build=True)


@pytest.mark.parametrize("every", [0, 7])
def test_fields_are_those_of_the_runs_stepped_alone(every):
    boxes = [((256, 64), 18), ((128, 32, 16), 3), ((1024, 8, 6), 2), ((4096, 8), 1), ((512, 512), 2)]
    runs = [(shape, 1.0 + (i & 1), 100 * k + i, (0, 0, 1, 3, 2)[i % 5], 23 - 3 * (i % 4))
            for k, (shape, count) in enumerate(boxes) for i in range(count)]
    params = [prs.make_params(shape, era_m=era, seed=seed, tblock=tb) for shape, era, seed, tb, _ in runs]
    b = prs.prs_batch_create(params)
    try:
        ns = [n for *_, n in runs]
        prs.prs_batch_run(b, ns, every, 4)
        prs.prs_batch_run(b, [n // 2 for n in ns], every, 4)
        for r, (shape, era, seed, tb, n) in enumerate(runs):
            phi, v = (np.empty(tuple(reversed(shape)), np.float32) for _ in range(2))
            assert prs.prs_batch_get_state(b, r, phi, v) == n + n // 2
            sim = prs.Sim(shape, era_m=era, seed=seed, tblock=tb)
            sim.init()
            sim.step(n + n // 2)
            a, c, _ = sim.get_state()
            sim.close()
            assert np.array_equal(phi, a) and np.array_equal(v, c), (r, shape)
    finally:
        prs.prs_batch_destroy(b)
