"""Numbers of steps below graph_steps, replayed when a call asks for the same
number again, and steps captured by the caller or moved to another stream."""
import pytest

from gpu_helpers import random_field, representable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,variant", [("f64", "A"), ("f32", "B"), ("f16", "C"), ("f32", "lbgk")])
def test_repeated_short_runs_give_the_bits_of_single_launches(dtype, variant):
    import torch

    from paper_1507_02509_gb300 import Lattice

    nx, ny = 96, 33
    g = representable(random_field(nx, ny, 6, amp=1e-3), dtype)
    a, b = (Lattice(nx, ny, variant=variant, beta=0.97, dtype=dtype) for _ in range(2))
    b.set_graph_steps(0)
    for lat in (a, b):
        lat.set_populations(g)
    for n in (10, 10, 10, 7, 7, 5, 5, 2, 12, 40, 40, 33, 10, 10):
        a.step(n)
        b.step(n)
    assert torch.equal(a.populations(), b.populations())
    if variant != "lbgk":  # a setting that the captured kernels carry
        for lat in (a, b):
            lat.set_gamma(1.0 / 0.97)
            lat.step(10)
            lat.step(10)
        assert torch.equal(a.populations(), b.populations())
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        a.step(6)
        a.step(6)
    torch.cuda.current_stream().wait_stream(s)
    b.step(12)
    assert torch.equal(a.populations(), b.populations())
    # captured by the caller: the replay goes on from the captured buffers
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.step(4)
    graph.replay()
    graph.replay()
    b.step(8)
    assert torch.equal(a.populations(), b.populations())
    a.close()
    b.close()
