"""Lifetime and sharing of the library's own workspaces: solves from many
threads and streams at once, each compared with its plain result."""
import ctypes
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


def captured(d, s, flags=0):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        binding.apsp_fw(d, flags=flags, stream=s)
    return g


# aligned, unaligned, and int32 narrowed to int16 (sizes on both sides of the small-matrix schedule)
@pytest.mark.parametrize("dt,n,ld,flags", [("i32", 512, 512, 0), ("f32", 512, 512, 0), ("i32", 2624, 2624, 0),
                                           ("i32", 700, 701, 0), ("f32", 700, 701, 0),
                                           ("i32", 512, 512, binding.FLAG_NARROW)])
def test_capture_outlives_the_streams_workspace(dt, n, ld, flags):
    # an ordinary call, a capture, then larger solves and other streams; the graph still solves
    src = torch.zeros((n, ld), dtype=torch.int32 if dt == "i32" else torch.float32, device="cuda")
    w = graph(dt, n, n)
    if flags:  # (n - 1) Wmax < 16383
        w = torch.where(w < inputs.INF_I32, w.clamp(max=30), w)
    src[:, :n] = w
    d = src.clone()
    ref = src.clone()
    binding.apsp_fw(ref, n, flags=binding.FLAG_NO_WORKSPACE | binding.FLAG_NO_GRAPH)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        binding.apsp_fw(d, n, flags=flags, stream=s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        binding.apsp_fw(d, n, flags=flags, stream=s)
    big = graph(dt, n + 1500, 1)
    others = [s] + [torch.cuda.Stream() for _ in range(18)]
    for t in others:
        with torch.cuda.stream(t):
            x = big.clone()
            x.record_stream(t)
            binding.apsp_fw(x, stream=t)
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()
    junk = torch.full((1 << 27,), 123456789, dtype=torch.int32, device="cuda")  # over what was freed
    for _ in range(2):
        d.copy_(src)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(d, ref)
    assert bool((junk == 123456789).all())
    assert binding.device_error() == 0


@pytest.mark.parametrize("dt,n", [("i32", 900), ("f32", 900), ("i32", 2624)])
def test_two_graphs_of_one_stream_side_by_side(dt, n):
    srcs = [graph(dt, n, n + k) for k in range(2)]
    refs = [solved(x) for x in srcs]
    ds = [torch.empty_like(x) for x in srcs]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ds[0].copy_(srcs[0])
        binding.apsp_fw(ds[0], stream=s)
    s.synchronize()
    gs = [captured(d, s) for d in ds]
    ts = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(10):
        for k in range(2):
            with torch.cuda.stream(ts[k]):
                ds[k].copy_(srcs[k])
                gs[k].replay()
        torch.cuda.synchronize()
        for k in range(2):
            assert torch.equal(ds[k], refs[k])


def test_first_call_of_a_stream_in_a_capture():
    for dt, n in (("i32", 1000), ("f32", 3500), ("i32", 2624)):
        src = graph(dt, n, n)
        ref = solved(src)
        d = src.clone()
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        g = captured(d, s)
        d.copy_(src)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(d, ref)


def test_graphs_give_their_workspaces_back():
    n = 3300  # 52 stages: 3.4 MB each
    d = graph("f32", n, 3)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def cycle(count):
        for _ in range(count):
            captured(d, s).reset()
        binding.apsp_fw(d, stream=s)
        torch.cuda.synchronize()

    cycle(5)
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    cycle(100)
    torch.cuda.empty_cache()
    assert torch.cuda.mem_get_info()[0] > free0 - (150 << 20)


def test_per_thread_default_streams():
    # the handle cudaStreamPerThread (2) from four threads at once: four streams
    # (each waits for its solves before it ends)
    per_thread = 2
    rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    n = 1100
    srcs = [graph("i32" if k % 2 else "f32", n, n + k) for k in range(4)]
    refs = [solved(x) for x in srcs]
    ds = [[x.clone() for _ in range(6)] for x in srcs]
    torch.cuda.synchronize()
    code = [binding.APSP_F32, binding.APSP_I32]

    def worker(k):
        opt = binding.Options(0, binding.FLAG_NO_GRAPH, None, 0, None, 0)
        try:
            for d in ds[k]:
                assert binding.apsp_fw_raw(d.data_ptr(), n, n, code[k % 2], per_thread, opt) == binding.APSP_OK
        finally:
            assert rt.cudaStreamSynchronize(ctypes.c_void_p(per_thread)) == 0

    in_threads([lambda k=k: worker(k) for k in range(4)])
    torch.cuda.synchronize()
    for k in range(4):
        for d in ds[k]:
            assert torch.equal(d, refs[k]), k


def test_server_requests_on_both_sides_of_the_schedules():
    # 31, 32, 39 and 41 stages (int32 panel copies beyond 39), whatever the largest size of the server
    sizes = [1984, 1985, 2496, 2560]
    for max_n in (2560, 4096):
        with binding.Server(max_inflight=8, hbm_budget_bytes=1 << 30, max_n=max_n) as server:
            srcs = [graph(dt, n, n) for n in sizes for dt in ("i32", "f32")]
            tickets = [server.submit(x) for x in srcs]
            for x, t in zip(srcs, tickets):
                assert torch.equal(torch.from_numpy(server.wait(t)), solved(x).cpu()), x.shape
    assert binding.device_error() == 0


@pytest.mark.parametrize("n,ld,offset", [(700, 704, 0), (700, 701, 0), (2624, 2624, 0), (1500, 1501, 1)])
def test_int32_leaves_a_callers_workspace_alone(n, ld, offset):
    # apsp_workspace_bytes asks for none: neither written nor refused, aligned or not
    assert binding.workspace_bytes(n, binding.APSP_I32) == 0
    src = torch.zeros((n, ld), dtype=torch.int32, device="cuda")
    src[:, :n] = graph("i32", n, n)
    ref = src.clone()
    binding.apsp_fw(ref, n, flags=binding.FLAG_NO_WORKSPACE)
    ws = torch.full((6 << 20,), 77, dtype=torch.int32, device="cuda")
    for flags in (0, binding.FLAG_NO_GRAPH, binding.FLAG_NO_LOOKAHEAD):
        d = src.clone()
        opt = binding.Options(0, flags, None, 0, ws[offset:].data_ptr(), 4 * (ws.numel() - offset))
        assert binding.apsp_fw_raw(d.data_ptr(), n, ld, binding.APSP_I32, torch.cuda.current_stream().cuda_stream,
                                   opt) == binding.APSP_OK
        torch.cuda.synchronize()
        assert torch.equal(d, ref)
        assert bool((ws == 77).all()), flags


def test_unaligned_noalloc_calls_may_overlap():
    # rows that are not 16-byte aligned use none of the entry point's shared array
    n, ld = 1000, 1001
    srcs = []
    for k in range(2):
        srcs.append(torch.zeros((n, ld), device="cuda"))
        srcs[k][:, :n] = graph("f32", n, k)
    refs = []
    for x in srcs:
        d = x.clone()
        binding.apsp_fw(d, n, flags=binding.FLAG_NO_WORKSPACE | binding.FLAG_NO_GRAPH)
        refs.append(d)
    ss = [torch.cuda.Stream() for _ in range(2)]
    ds = [x.clone() for x in srcs]
    torch.cuda.synchronize()
    for _ in range(5):
        for k in range(2):
            with torch.cuda.stream(ss[k]):
                ds[k].copy_(srcs[k])
                assert binding.lib().apsp_fw_f32_noalloc(ds[k].data_ptr(), n, ld, ss[k].cuda_stream) == binding.APSP_OK
        torch.cuda.synchronize()
        for k in range(2):
            assert torch.equal(ds[k], refs[k])
