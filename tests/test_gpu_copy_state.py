"""prs_set_state_device from sources of every kind of memory and alignment: what the copy kernel takes
and what goes through the driver's copies instead gives the same state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(128, 96), (7, 5), (64, 33, 20)])
@pytest.mark.parametrize("source", ["aligned", "offset", "pinned host"])
def test_sources_of_a_device_state(shape, source):
    import torch

    import paper_1710_10420_gb300 as prs

    rng = np.random.default_rng(5)
    n = int(np.prod(shape))
    host = torch.from_numpy(rng.uniform(-1.0, 1.0, (2, n + 1)).astype(np.float32))
    rows = host.pin_memory() if source == "pinned host" else host.cuda()
    off = 1 if source == "offset" else 0
    dims = tuple(reversed(shape))
    phi, v = (rows[k].contiguous().clone() if source == "aligned" else rows[k] for k in (0, 1))
    sim = prs.Sim(shape)
    try:
        prs.prs_set_state_device(sim.handle, phi[off:off + n], v[off:off + n], 3)
    except prs.PRSError:
        assert source == "pinned host"  # an error of the driver's copy, not of a kernel
        sim.set_state(rng.uniform(-1, 1, dims).astype(np.float32), np.zeros(dims, np.float32), 0)
        sim.step(1)
        sim.close()
        return
    p, w, step = sim.get_state()
    sim.close()
    assert step == 3
    assert np.array_equal(p.ravel(), host[0].numpy()[off:off + n])
    assert np.array_equal(w.ravel(), host[1].numpy()[off:off + n])
