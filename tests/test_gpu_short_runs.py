"""Short runs of several lengths: replays of the lengths asked for last, whose
exchange neither waits for the stream nor disturbs a capture."""
import pytest

from gpu_helpers import random_field, representable

pytestmark = pytest.mark.gpu

NX, NY, BETA = 96, 33, 0.97


def pair(dtype, variant):
    from paper_1507_02509_gb300 import Lattice

    g = representable(random_field(NX, NY, 6, amp=1e-3), dtype)
    a, b = (Lattice(NX, NY, variant=variant, beta=BETA, dtype=dtype) for _ in range(2))
    b.set_graph_steps(0)
    for lat in (a, b):
        lat.set_populations(g)
    return a, b


def busy(seconds=0.25):
    import torch

    torch.cuda._sleep(int(seconds * 2.07e9))  # at most: the clock's highest rate


@pytest.mark.parametrize("dtype,variant", [("f64", "B"), ("f32", "A"), ("f16", "D")])
def test_alternating_and_evicted_lengths_give_the_bits_of_single_launches(dtype, variant):
    import torch

    a, b = pair(dtype, variant)
    # a pattern of two lengths with a change of parity, then more lengths than are kept
    lengths = [10, 10, 7] * 6 + [n for n in (4, 6, 8, 12, 14, 16) for _ in range(7)] + [10, 7, 44, 42] * 4
    for n in lengths:
        a.step(n)
        b.step(n)
    assert torch.equal(a.populations(), b.populations())
    a.close()
    b.close()


def test_a_changed_length_does_not_wait_for_the_stream():
    import torch

    a, b = pair("f32", "B")
    lengths = [n for n in (4, 6, 8, 10, 12, 14) for _ in range(7)]
    for n in lengths:  # graphs of every kept length
        a.step(n)
        b.step(n)
    torch.cuda.synchronize()
    busy()
    a.step(14)  # replays of what is dropped below wait behind the sleep
    for n in lengths:
        a.step(n)
    a.set_graph_steps(16)
    a.step(6)
    waited = torch.cuda.current_stream().query()
    b.step(14)
    for n in lengths:
        b.step(n)
    b.step(6)
    assert not waited
    assert torch.equal(a.populations(), b.populations())
    a.close()
    b.close()


def test_graphs_dropped_while_the_stream_is_captured():
    import torch

    a, b = pair("f32", "C")
    for _ in range(4):
        a.step(10)
        b.step(10)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.set_graph_steps(64)
        a.step(4)
    graph.replay()
    graph.replay()
    b.step(8)
    assert torch.equal(a.populations(), b.populations())
    a.close()
    b.close()


@pytest.mark.parametrize("thread", [False, True])
def test_short_runs_beside_a_capture(thread):
    """A handle on a stream of its own takes, repeats and exchanges short runs
    while another handle's steps are captured in the global mode."""
    import threading

    import torch

    from paper_1507_02509_gb300 import Lattice

    a, b = pair("f32", "B")
    s = torch.cuda.Stream()
    g = a.populations()
    lat = Lattice(NX, NY, variant="B", beta=BETA, dtype="f32", stream=s)
    lat.set_populations(g)
    torch.cuda.synchronize()
    lengths = [n for n in (10, 4, 6, 8, 12) for _ in range(7)]
    failed = []

    def run():
        try:
            for n in lengths:
                lat.step(n)
            lat.set_graph_steps(16)
            lat.step(40)
        except Exception as e:
            failed.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        a.step(4)
        if thread:
            t = threading.Thread(target=run)
            t.start()
            t.join()
        else:
            run()
        a.step(4)
    assert not failed, failed
    graph.replay()
    b.step(8)
    assert torch.equal(a.populations(), b.populations())
    b.set_populations(g)
    for n in lengths + [40]:
        b.step(n)
    s.synchronize()
    assert torch.equal(lat.populations(), b.populations())
    for x in (a, b, lat):
        x.close()


@pytest.mark.parametrize("slabs", [False, True])
def test_destroying_a_handle_waits_for_replays_of_its_captured_steps(slabs):
    """A replay copies into the handle's status word, on whatever stream it is
    launched: the word is not given to another handle before it has ended."""
    import torch

    from paper_1507_02509_gb300 import Lattice
    from paper_1507_02509_gb300.slabs import SlabGroup

    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    kw = dict(variant="B", beta=BETA, dtype="f32", stream=s)
    x = SlabGroup(NX, NY, 2, **kw) if slabs else Lattice(NX, NY, **kw)
    with torch.cuda.stream(s):
        x.set_populations(torch.as_tensor(random_field(NX, NY, 6, amp=1e-3)).cuda())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        x.step(2)
    with torch.cuda.stream(t):
        busy()
        graph.replay()
    x.close()
    assert t.query()
