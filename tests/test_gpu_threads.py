"""Handles beside other threads' work: particles are loaded into a handle while another
thread captures a graph (its own capture, thread-local mode), and after the handle's
stream has changed."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1601_03801_gb300 import sedi  # noqa: E402
from paper_1601_03801_gb300.workloads import small_case  # noqa: E402


def load(h, parts, n):
    h.set_particles(*(parts[k][:n] for k in ("x", "v", "w", "d", "rho")))
    return h.neighbors()


@pytest.mark.parametrize("n", [1000, 999, 400])  # the buffers' block kept, kept, allocated anew
def test_load_while_another_thread_captures(n):
    prm, parts = small_case(parity_addon=True)
    h = sedi.Sedi(dict(prm, precision_form="split"))
    load(h, parts, 1000)
    want = load(sedi.Sedi(dict(prm, precision_form="split")), parts, n)
    got, err = [], []

    def other():
        try:
            got.append(load(h, parts, n))
        except sedi.SediError as e:
            err.append(e)

    a = torch.zeros(1000, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="thread_local"):
        a.add_(1.0)
        t = threading.Thread(target=other)
        t.start()
        t.join()
        a.add_(1.0)
    graph.replay()
    torch.cuda.synchronize()
    assert not err, err
    assert torch.all(a == 2.0)
    for x, y in zip(got[0], want):
        np.testing.assert_array_equal(x, y)


def test_reload_after_a_change_of_stream():
    """Steps queued on a stream, then another stream and new particles at once: the load waits
    for the steps, which still use the buffers that it fills."""
    prm, parts = small_case(parity_addon=True)
    h = sedi.Sedi(dict(prm, precision_form="split"))
    streams = [torch.cuda.Stream() for _ in range(2)]
    want = None
    for k in range(6):
        h.set_stream(streams[k % 2])
        load(h, parts, 1000)
        h.step(5)
        x = h.get_particles()[0]
        want = x if want is None else want
        np.testing.assert_array_equal(x, want)
        h.step(40)  # in flight when the stream changes
