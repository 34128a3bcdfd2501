"""The s = 64 schedule of one head and one rest per stage (csrc/stage.cuh):
bit-identical to the plain schedule for any leading dimension and alignment,
and to the oracle for the integers.

The stage counts are the edges of its ranges: one stage (fw_phase1); head and rest in one
launch up to 5 stages; panel strips 16 wide up to 9 stages, 32 wide up to 30
(int16: 33), then 64; the lookahead schedule beyond 52 (fp32), 39 (int32) and 36 (int16) stages, with
the stage record beyond 80, 64 and 64.  Whole and ragged last stages.  Rows that are not 16-byte aligned
go through an aligned copy from 22 stages on."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1001_4108_gb300 import binding

pytestmark = pytest.mark.gpu


def graph(dt, n, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    if dt == "f32":  # sums are rounded: full 24-bit mantissas
        w = (1.0 - g.random((n, n))).astype(np.float32)
        w[g.random((n, n)) < 0.5] = np.inf
    elif dt == "i16":  # (n - 1) * 7 < 16383 up to n = 2341
        w = g.integers(0, 8, (n, n)).astype(np.int16)
        w[g.random((n, n)) > 0.05] = 16383
    else:
        p = g.integers(0, 51, n)
        w = (g.integers(0, 951, (n, n)) + p[:, None] - p[None, :]).astype(np.int32)
        w[g.random((n, n)) > 0.1] = 1 << 29
    np.fill_diagonal(w, 0)
    return w


def on_device(w, ld, offset=0):
    """The matrix in a larger buffer, `offset` elements in, -7 around it."""
    n = w.shape[0]
    t = torch.from_numpy(w)
    buf = torch.full((n * ld + offset,), -7, dtype=t.dtype, device="cuda")
    d = buf[offset:].view(n, ld)
    d[:, :n] = t.cuda()
    return d


@pytest.mark.parametrize("dt", ["f32", "i32", "i16"])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 128, 129, 320, 321, 576, 577, 640, 1536, 1537, 1921, 2047, 2048, 2049, 2113, 2305])
def test_stage_schedule_equals_plain(dt, n):
    w = graph(dt, n, n)
    ref = on_device(w, (n + 7) // 8 * 8)
    binding.apsp_fw(ref, n, flags=binding.FLAG_NO_LOOKAHEAD | binding.FLAG_NO_GRAPH)
    if dt == "i32" and n <= 1537:
        np.testing.assert_array_equal(ref[:, :n].cpu().numpy(), oracle.fw_int32_conv(w))
    if dt == "i16" and n <= 1537:
        np.testing.assert_array_equal(ref[:, :n].cpu().numpy(), oracle.fw_int16_conv(w))
    for ld, offset in ((n, 0), ((n + 7) // 8 * 8, 0), (n + 1, 0), (n + 37, 3)):
        d = on_device(w, ld, offset)
        binding.apsp_fw(d, n)
        torch.cuda.synchronize()
        assert torch.equal(d[:, :n], ref[:, :n]), (ld, offset)
        assert bool((d[:, n:] == -7).all())
    assert binding.device_error() == 0


@pytest.mark.parametrize("dt", ["f32", "i32", "i16"])
@pytest.mark.parametrize("n", [64, 65, 200, 321, 577, 1000, 1537])
def test_stage_schedule_paths(dt, n):
    # the stage record and the distances, against the plain schedule's
    w = graph(dt, n, n + 1)
    a, b = on_device(w, n), on_device(w, n)
    va, vb = (torch.empty((n, n), dtype=torch.int16, device="cuda") for _ in range(2))
    binding.apsp_fw_paths(a, va)
    binding.apsp_fw_paths(b, vb, flags=binding.FLAG_NO_LOOKAHEAD | binding.FLAG_NO_GRAPH)
    torch.cuda.synchronize()
    assert torch.equal(a, b) and torch.equal(va, vb)


@pytest.mark.parametrize("n", [321, 1600])
def test_stage_schedule_capture_and_replay(n):
    # direct, the library's graph, its replay, and a user's capture
    w = graph("i32", n, n + 2)
    src = on_device(w, n)
    ref = src.clone()
    binding.apsp_fw(ref, flags=binding.FLAG_NO_LOOKAHEAD | binding.FLAG_NO_GRAPH)
    s = torch.cuda.Stream()
    d = torch.empty_like(src)
    with torch.cuda.stream(s):
        for _ in range(3):
            d.copy_(src)
            binding.apsp_fw(d, stream=s)
            s.synchronize()
            assert torch.equal(d, ref)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        binding.apsp_fw(d, stream=s)
    d.copy_(src)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(d, ref)


@pytest.mark.parametrize("dt,n,paths", [
    ("f32", 3265, False), ("f32", 3328, False), ("f32", 3329, False), ("i32", 2433, False), ("i32", 2496, False),
    ("i32", 2497, False), ("i16", 2304, False), ("f32", 5120, True), ("f32", 5121, True), ("i32", 4096, True),
    ("i32", 4097, True), ("i16", 4033, True), ("i16", 4097, True)])
def test_stage_schedule_last_rounds(dt, n, paths):
    w = graph(dt, n, n + 3)
    a, b = on_device(w, (n + 7) // 8 * 8), on_device(w, (n + 7) // 8 * 8)
    plain = binding.FLAG_NO_LOOKAHEAD | binding.FLAG_NO_GRAPH
    if paths:
        va, vb = (torch.empty((n, n), dtype=torch.int16, device="cuda") for _ in range(2))
        binding.apsp_fw_paths(a, va, n, kblock=64)
        binding.apsp_fw_paths(b, vb, n, kblock=64, flags=plain)
        assert torch.equal(va, vb)
    else:
        binding.apsp_fw(a, n)
        binding.apsp_fw(b, n, flags=plain)
    assert torch.equal(a, b)
    assert binding.device_error() == 0


@pytest.mark.parametrize("dt", ["f32", "i32", "i16"])
@pytest.mark.parametrize("n", [1344, 1345, 2047])
def test_stage_schedule_unaligned_copy(dt, n):
    # in place below 22 stages, an aligned copy from there on, in place again under capture
    w = graph(dt, n, n + 4)
    ref = on_device(w, (n + 7) // 8 * 8)
    vr, v = (torch.empty((n, n), dtype=torch.int16, device="cuda") for _ in range(2))
    binding.apsp_fw_paths(ref, vr, n)
    s = torch.cuda.Stream()
    d = on_device(w, n + 9, 1)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        binding.apsp_fw_paths(d, v, n, stream=s)
    torch.cuda.synchronize()
    assert torch.equal(d[:, :n], ref[:, :n]) and torch.equal(v, vr)
    assert bool((d[:, n:] == -7).all())
    g = torch.cuda.CUDAGraph()
    d[:, :n] = torch.from_numpy(w).cuda()
    v.fill_(7)
    with torch.cuda.graph(g, stream=s):
        binding.apsp_fw_paths(d, v, n, stream=s)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(d[:, :n], ref[:, :n]) and torch.equal(v, vr)
    assert bool((d[:, n:] == -7).all())
