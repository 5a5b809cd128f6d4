"""The weight-streaming linear (one or two rows) takes weight rows in pairs and
activation sums in 16-byte chunks: sizes around a warp's pair, a CTA's pairs
and a lane's chunks, every code at its extremes, against the oracle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2])
@pytest.mark.parametrize("N,K", [(8, 128), (16, 1024), (24, 4096), (3640, 4224), (7304, 128), (14600, 384), (256, 16384)])
def test_gemv_pairs_bit_exact(p4q, dev, M, N, K):
    rng = np.random.default_rng(M + N + K)
    a = rng.integers(0, 256, size=(M, K // 2), dtype=np.uint8)
    w = rng.integers(0, 256, size=(N, K // 2), dtype=np.uint8)
    a[-1], w[0], w[-1] = 0x88, 0x88, 0x77
    acc = p4q.w4a4_gemm_s32(torch.from_numpy(a).to(dev), torch.from_numpy(w).to(dev))
    torch.cuda.synchronize()
    assert p4q.p4q_device_status() == 0
    assert np.array_equal(acc.cpu().numpy(), oracle.gemm_s32(oracle.unpack_codes(a), oracle.unpack_codes(w)))
