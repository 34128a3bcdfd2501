"""The partial k-block of a ragged matrix's last stage on the staged kernels
(lookahead and plain schedules): k-blocks of 1 to 127 vertices, at the edges
of the 32-k slices, against the generic kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1001_4108_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def graph(dt, n, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    if dt == "f32":
        w = (1.0 - g.random((n, n))).astype(np.float32)
        np.fill_diagonal(w, 0)
        return w
    if dt == "i16":
        return inputs.to_int16(inputs.int_graph(n, 0.02, 1, max(1, min(7, 16382 // n)), seed))
    return inputs.int_graph(n, 0.02, 0, 950, seed, potential_max=50)  # unreachable pairs too


@pytest.mark.parametrize("dt", ["f32", "i32", "i16"])
@pytest.mark.parametrize("kb,r", [(64, 1), (64, 31), (64, 33), (64, 63), (128, 1), (128, 4), (128, 32), (128, 65),
                                  (128, 100), (128, 127)])
def test_ragged_last_stage(dt, kb, r):
    n = 3 * kb + r
    ld = (n + 7) // 8 * 8
    w = graph(dt, n, n)
    src = torch.zeros((n, ld), dtype=torch.from_numpy(w).dtype, device="cuda")
    src[:, :n] = torch.from_numpy(w).cuda()
    ref = src.clone()
    binding.apsp_fw(ref, n, kblock=kb, flags=binding.FLAG_GENERIC)
    for flags in (binding.FLAG_NO_LOOKAHEAD, binding.FLAG_REVERSE_K, binding.FLAG_NO_WORKSPACE, 0):
        d = src.clone()
        binding.apsp_fw(d, n, kblock=kb, flags=flags | binding.FLAG_NO_GRAPH)
        torch.cuda.synchronize()
        assert torch.equal(d, ref), flags
    va, vb = (torch.empty((n, n), dtype=torch.int16, device="cuda") for _ in range(2))
    a, b = src.clone(), src.clone()
    binding.apsp_fw_paths(a, va, n, kblock=kb, flags=binding.FLAG_NO_LOOKAHEAD)
    binding.apsp_fw_paths(b, vb, n, kblock=kb, flags=binding.FLAG_GENERIC)
    torch.cuda.synchronize()
    assert torch.equal(a, ref) and torch.equal(b, ref) and torch.equal(va, vb)
    assert binding.device_error() == 0
