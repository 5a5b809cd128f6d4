"""The weight-streaming linear (one or two rows, more on small weights) takes weight rows in pairs and
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


@pytest.mark.parametrize("M,N,K", [(3, 8, 128), (4, 1216, 1024), (5, 1224, 1024), (6, 8, 8192), (7, 2048, 2048),
                                   (8, 4096, 2048), (8, 264, 6784), (3, 2728, 16384), (8, 6912, 256), (5, 2448, 512),
                                   (3, 2736, 16384), (8, 264, 6912), (4, 4096, 5120), (4, 4096, 5248)])
def test_few_rows_on_small_weights_bit_exact(p4q, dev, M, N, K):
    """Three to eight rows: the lines to the tensor-core kernel (either side), one
    and two weight rows per warp, rows that fill the warps unevenly; int32
    accumulators and fp16 outputs."""
    rng = np.random.default_rng(M + N + K)
    a = rng.integers(0, 256, size=(M, K // 2), dtype=np.uint8)
    w = rng.integers(0, 256, size=(N, K // 2), dtype=np.uint8)
    a[-1], w[0], w[-1] = 0x88, 0x88, 0x77
    sa = (rng.random(M) * 0.5 + 0.01).astype(np.float32)
    sw = (rng.random(N) * 0.002 + 1e-4).astype(np.float32)
    xa, xw = torch.from_numpy(a).to(dev), torch.from_numpy(w).to(dev)
    acc = p4q.w4a4_gemm_s32(xa, xw)
    Y = p4q.w4a4_linear(xa, torch.from_numpy(sa).to(dev), xw, torch.from_numpy(sw).to(dev))
    torch.cuda.synchronize()
    assert p4q.p4q_device_status() == 0
    ref = oracle.gemm_s32(oracle.unpack_codes(a), oracle.unpack_codes(w))
    assert np.array_equal(acc.cpu().numpy(), ref)
    y = (ref.astype(np.float32) * sa[:, None]) * sw[None]
    assert np.array_equal(Y.cpu().numpy(), y.astype(np.float16))
