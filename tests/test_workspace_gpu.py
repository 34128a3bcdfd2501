"""Lifetime and sharing of the library's own workspaces: solves from many
threads and streams at once, each compared with its plain result."""
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_1001_4108_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def graph(dt, n, seed):
    w = inputs.dense_f32(n, seed=seed) if dt == "f32" else inputs.int_graph(n, 0.1, 1, 1000, seed=seed)
    return torch.from_numpy(w).cuda()


def solved(src):
    """The result of the kernels that need no workspace."""
    d = src.clone()
    binding.apsp_fw(d, flags=binding.FLAG_NO_WORKSPACE | binding.FLAG_NO_GRAPH)
    torch.cuda.synchronize()
    return d


def in_threads(workers):
    errors = []

    def call(f):
        try:
            f()
        except BaseException as e:  # reported by the main thread
            errors.append(e)

    th = [threading.Thread(target=call, args=(f,)) for f in workers]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("dt", ["i32", "f32"])
def test_more_streams_than_workspaces(dt):
    # 20 threads, a stream each, sizes that grow
    sizes = [200, 333, 512, 700]
    srcs = [graph(dt, n, n) for n in sizes]
    refs = [solved(s) for s in srcs]

    def worker(k):
        s = torch.cuda.Stream()
        ds = [torch.empty_like(x) for x in srcs]
        for r in range(6):
            i = (r + k) % len(sizes)
            with torch.cuda.stream(s):
                ds[i].copy_(srcs[i])
                binding.apsp_fw(ds[i], flags=binding.FLAG_NO_GRAPH if r % 2 else 0, stream=s)
            s.synchronize()
            assert torch.equal(ds[i], refs[i]), (k, r)

    in_threads([lambda k=k: worker(k) for k in range(20)])
    assert binding.device_error() == 0


def test_threads_on_one_stream():
    # the launches of one solve are enqueued together: the solves of a stream share its workspace
    sizes = [1000, 640, 1100, 321]
    srcs = [graph("i32" if k % 2 else "f32", n, n) for k, n in enumerate(sizes)]
    refs = [solved(s) for s in srcs]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def worker(k):
        d = torch.empty_like(srcs[k])
        for _ in range(8):
            with torch.cuda.stream(s):
                d.copy_(srcs[k])
                binding.apsp_fw(d, flags=binding.FLAG_NO_GRAPH, stream=s)
            s.synchronize()
            assert torch.equal(d, refs[k]), k

    in_threads([lambda k=k: worker(k) for k in range(len(sizes))])
    assert binding.device_error() == 0
