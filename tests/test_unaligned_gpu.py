"""Matrices whose rows are not 16-byte aligned: the staged kernels run on an
aligned copy.  Bit-identical to the aligned solve; nothing outside the n x n
block is touched."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1001_4108_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def graph(dt, n, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    if dt == "f32":
        w = (1.0 - g.random((n, n))).astype(np.float32)
        np.fill_diagonal(w, 0)
        return w
    if dt == "i16":
        return inputs.to_int16(inputs.int_graph(n, 0.05, 1, max(1, min(7, 16382 // max(1, n - 1))), seed))
    return inputs.int_graph(n, 0.05, 0, 950, seed, potential_max=50)


def matrix(w, ld, offset):
    n = w.shape[0]
    t = torch.from_numpy(w)
    buf = torch.full((n * ld + offset,), -7, dtype=t.dtype, device="cuda")
    d = buf[offset:].view(n, ld)
    d[:, :n] = t.cuda()
    return d


@pytest.mark.parametrize("dt,n", [("i16", 65), ("i16", 129), ("i16", 1001), ("i16", 2048), ("f32", 2049), ("i32", 2113),
                                  ("f32", 4607), ("i32", 4225), ("i16", 5121), ("f32", 4609)])
def test_unaligned_equals_aligned(dt, n):
    w = graph(dt, n, n)
    ref = matrix(w, (n + 7) // 8 * 8, 0)
    binding.apsp_fw(ref, n)
    if dt == "i16" and n <= 1001:
        np.testing.assert_array_equal(ref[:, :n].cpu().numpy(), oracle.fw_int16_conv(w))
    for ld, offset in ((n + 1 if n % 2 == 0 else n, 0), ((n + 7) // 8 * 8, 1)):
        d = matrix(w, ld, offset)
        for _ in range(2):  # the second call may replay a graph
            d[:, :n] = torch.from_numpy(w).cuda()
            binding.apsp_fw(d, n)
            torch.cuda.synchronize()
            assert torch.equal(d[:, :n], ref[:, :n]), (ld, offset)
            assert bool((d[:, n:] == -7).all())
    # the stage record too, and a user's capture (no allocation: the kernels for any layout)
    d = matrix(w, n + 1, 0)
    va, vb = (torch.empty((n, n), dtype=torch.int16, device="cuda") for _ in range(2))
    binding.apsp_fw_paths(d, va, n)
    r2 = matrix(w, (n + 7) // 8 * 8, 0)
    binding.apsp_fw_paths(r2, vb, n)
    torch.cuda.synchronize()
    assert torch.equal(d[:, :n], ref[:, :n]) and torch.equal(va, vb)
    s = torch.cuda.Stream()
    d = matrix(w, n + 1, 0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        binding.apsp_fw(d, n, stream=s)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(d[:, :n], ref[:, :n])
    assert binding.device_error() == 0
