"""The stage record of int16 matrices with weights of both signs (outside the
stated input range, solved all the same as long as no sum leaves int16): the
packed kernels compare as signed values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1001_4108_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [129, 200, 1000])
def test_signed_int16_record(n):
    g = np.random.default_rng(n)
    p = g.integers(0, 60, n)
    w = (g.integers(0, 90, (n, n)) + p[:, None] - p[None, :]).astype(np.int16)
    np.fill_diagonal(w, 0)
    a = torch.from_numpy(w).cuda()
    b = a.clone()
    va, vb = (torch.empty((n, n), dtype=torch.int16, device="cuda") for _ in range(2))
    binding.apsp_fw_paths(a, va)
    binding.apsp_fw_paths(b, vb, flags=binding.FLAG_NO_LOOKAHEAD | binding.FLAG_NO_GRAPH)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a.cpu().numpy(), oracle.fw_int32_conv(w.astype(np.int32)))
    assert torch.equal(a, b) and torch.equal(va, vb)
