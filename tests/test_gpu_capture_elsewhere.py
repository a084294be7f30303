"""A thread sets up and uses a context while another thread of the program has a
stream capture open (thread-local capture mode)."""
import threading

import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_set_up_beside_a_capture(precision):
    import torch
    n = 3000
    y = inputs.spread_embedding(np.arange(n) % 7, 3, rho_hi=8.0)
    own = torch.cuda.Stream()
    done = []

    def context():
        t = HyperbolicTSNE(precision=precision, stream=own.cuda_stream)
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(y)
        return t

    def work():
        try:
            t = context()
            done.extend([t, t.grad(0.5)[0]])
        except Exception as e:  # (looked at below: not inside the capture)
            done.append(e)

    with context() as t:
        g = t.grad(0.5)[0]
    x = torch.zeros(1000, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        x += 1.0
        other = threading.Thread(target=work)
        other.start()
        other.join()
        x += 1.0
    graph.replay()
    torch.cuda.synchronize()
    assert len(done) == 2, done
    done[0].close()
    assert np.array_equal(done[1], g) and bool((x == 2.0).all())
