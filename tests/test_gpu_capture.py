"""A run's first state and its steps captured into a CUDA graph: what the run allocates for itself on the way
is not part of the graph, and every replay gives the state stepped eagerly."""
import numpy as np
import pytest

import paper_1710_10420_gb300 as prs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available()
    prs.load(build=True)


@pytest.mark.parametrize("bound", [True, False])
@pytest.mark.parametrize("shape,precision", [((128, 128, 64), prs.PRS_FP32), ((130, 71), prs.PRS_FP32),
                                             ((61, 45, 40), prs.PRS_FP64)])
def test_first_state_and_steps_in_a_graph(shape, precision, bound):
    import torch

    dtype = torch.float32 if precision == prs.PRS_FP32 else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(5)
    phi = torch.rand(tuple(reversed(shape)), generator=gen, device="cuda", dtype=dtype) * 2 - 1
    v = 0.1 * phi.flip(0).contiguous()
    stream = torch.cuda.Stream()
    other = prs.Sim((64, 64))  # so that the captured run is not the only one
    h = prs.prs_create(prs.make_params(shape, precision=precision), stream.cuda_stream)
    bufs = [torch.empty_like(phi) for _ in range(3)]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        if bound:
            prs.prs_bind(h, *bufs)
        prs.prs_set_state_device(h, phi, v, 0)
        prs.prs_step(h, 7)
    ref = prs.Sim(shape, precision=precision)
    prs.prs_set_state_device(ref.handle, phi, v, 0)
    ref.step(7)
    a, b, n = ref.get_state()
    out = [np.empty(tuple(reversed(shape)), a.dtype) for _ in range(2)]
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert prs.prs_get_state(h, *out) == n
        assert np.array_equal(out[0], a) and np.array_equal(out[1], b)
    d = prs.prs_measure_ex(h)
    assert d.n_links == prs.prs_measure_ex(ref.handle).n_links
    prs.prs_destroy(h)
    ref.close()
    other.close()
