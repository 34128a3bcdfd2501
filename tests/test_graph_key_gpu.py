"""Replays of the library's graph cache: a call whose workspace, matrix or rows
differ from the captured one's gets its own launches."""
import pytest

torch = pytest.importorskip("torch")

from paper_1001_4108_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["f32", "i32"])
def test_shrinking_caller_workspace(dt):
    # large, large (captured), then the same pointer with fewer bytes: nothing past them is written
    n = 1024
    code = binding.APSP_F32 if dt == "f32" else binding.APSP_I32
    w = inputs.dense_f32(n, seed=1) if dt == "f32" else inputs.int_graph(n, 0.1, 1, 1000, seed=1)
    src = torch.from_numpy(w).cuda()
    ref = src.clone()
    binding.apsp_fw(ref, flags=binding.FLAG_NO_WORKSPACE)
    large = (4 * 16 + 2) << 14
    small = binding.workspace_bytes(n, code) // 2
    ws = torch.empty(large // 4, dtype=torch.int32, device="cuda")
    d = torch.empty_like(src)
    for size in (large, large, large, small, small, 0 if dt == "i32" else small):
        d.copy_(src)
        ws.fill_(77)
        opt = binding.Options(0, 0, None, 0, ws.data_ptr(), size)
        assert binding.apsp_fw_raw(d.data_ptr(), n, n, code, torch.cuda.current_stream().cuda_stream,
                                   opt) == binding.APSP_OK
        torch.cuda.synchronize()
        assert torch.equal(d, ref), size
        assert bool((ws[size // 4:] == 77).all()), size


@pytest.mark.parametrize("dt,n", [("f32", 512), ("i32", 512), ("f32", 4608)])
def test_host_matrix_of_another_leading_dimension(dt, n):
    # one pinned buffer: rows of n, n (captured), n, then of n + 64 elements
    w = inputs.dense_f32(n, seed=2) if dt == "f32" else inputs.int_graph(n, 0.1, 1, 1000, seed=2)
    code = binding.APSP_F32 if dt == "f32" else binding.APSP_I32
    ref = torch.from_numpy(w).cuda()
    binding.apsp_fw(ref)
    ref = ref.cpu()
    buf = torch.empty(n * (n + 64), dtype=ref.dtype).pin_memory()
    stream = torch.cuda.current_stream().cuda_stream
    for ld in (n, n, n, n + 64, n + 64, n):
        buf.fill_(-7)
        h = buf[:n * ld].view(n, ld)
        h[:, :n] = torch.from_numpy(w)
        assert binding.lib().apsp_fw_host(buf.data_ptr(), n, ld, code, stream) == binding.APSP_OK
        assert torch.equal(h[:, :n], ref), ld
        assert bool((h[:, n:] == -7).all()) and bool((buf[n * ld:] == -7).all()), ld
