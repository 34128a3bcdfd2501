"""Staging copies of the server, shared by its copy threads: several clients at
once, matrices around the size of one part (256 KiB) and of many, padded rows."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1001_4108_gb300 import binding, inputs

pytestmark = pytest.mark.gpu

SIZES = [1, 64, 255, 256, 257, 362, 363, 700, 1025, 2048]


def test_concurrent_clients():
    graphs = [inputs.int_graph(n, 0.05, 0, 900, seed=n, ld=n + 3, potential_max=50) for n in SIZES]
    want = []
    for g in graphs:
        n = g.shape[0]
        d = torch.from_numpy(np.ascontiguousarray(g[:, :n])).cuda()
        want.append(binding.apsp_fw(d).cpu().numpy())
    errors = []
    with binding.Server(max_inflight=16, hbm_budget_bytes=1 << 30, max_n=2048) as server:
        lock = threading.Lock()  # the Python wrapper keeps its tickets in a plain dict

        def client(k):
            try:
                order = [(i + k) % len(SIZES) for i in range(len(SIZES))]
                tickets = []
                for i in order:
                    n = SIZES[i]
                    t = server.submit(graphs[i][:, :n])
                    tickets.append((i, t))
                for i, t in tickets:
                    np.testing.assert_array_equal(server.wait(t), want[i])
            except BaseException as e:  # reported by the main thread
                with lock:
                    errors.append(e)

        threads = [threading.Thread(target=client, args=(k,)) for k in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert not errors, errors
