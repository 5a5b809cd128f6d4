"""The W4A4 linear for few rows (3 .. 128: weights on the tensor cores' row
side, k split over a cluster) against the oracle, at the edges of its tiles:
int32 accumulators and fp16 outputs bit-exact."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

# rows around the 16-column steps with the row of ones (15 | 16, 31 | 32, 63 |
# 64) and the two row tiles from 128 on; weight rows around a 128-row tile;
# one, an odd number of and many k-blocks; every split of k
SHAPES = [(3, 8, 128), (15, 128, 384), (16, 136, 128), (31, 120, 640), (32, 4096, 512), (63, 264, 1152),
          (64, 3000, 1024), (127, 256, 2176), (128, 4096, 1408), (128, 136, 16384), (17, 16384, 256), (24, 5120, 13824),
          (3, 22016, 4096), (96, 4096, 4096)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_fewrows_bit_exact(p4q, dev, M, N, K):
    rng = np.random.default_rng(M + N * 3 + K)
    a = rng.integers(0, 256, size=(M, K // 2), dtype=np.uint8)
    w = rng.integers(0, 256, size=(N, K // 2), dtype=np.uint8)
    a[0], w[-1] = 0x88, 0x88  # the largest products
    sa = (rng.random(M) * 0.5 + 0.01).astype(np.float32)
    sw = (rng.random(N + 1) * 0.002 + 1e-4).astype(np.float32)
    xa, xw = torch.from_numpy(a).to(dev), torch.from_numpy(w).to(dev)
    xs = torch.from_numpy(sw).to(dev)[1:]  # the weight scales need no 16-byte alignment
    acc = p4q.w4a4_gemm_s32(xa, xw)
    Y = p4q.w4a4_linear(xa, torch.from_numpy(sa).to(dev), xw, xs)
    torch.cuda.synchronize()
    assert p4q.p4q_device_status() == 0
    ref = oracle.gemm_s32(oracle.unpack_codes(a), oracle.unpack_codes(w))
    assert np.array_equal(acc.cpu().numpy(), ref)
    y = (ref.astype(np.float32) * sa[:, None]) * sw[None, 1:]
    assert np.array_equal(Y.cpu().numpy(), y.astype(np.float16))


@pytest.mark.parametrize("M,N,K", [(128, 8448, 128), (65, 16384, 256), (65, 19712, 128), (64, 16640, 128),
                                   (129, 1016, 384), (129, 1024, 384), (255, 1032, 640), (160, 4096, 11008),
                                   (109, 1032, 13824), (112, 1032, 13824), (128, 1032, 11008), (128, 264, 8320),
                                   (95, 1024, 16384), (96, 1024, 16384)])
def test_dispatch_edges(p4q, dev, M, N, K):
    """Around the lines between the few-rows kernel, the CTA pairs and the single CTAs."""
    test_fewrows_bit_exact(p4q, dev, M, N, K)


@pytest.mark.parametrize("M,N,K", [(24, 256, 128), (25, 256, 128), (56, 1024, 128), (57, 1024, 128), (64, 1024, 256),
                                   (65, 1024, 256), (127, 1032, 512), (128, 1032, 512), (96, 264, 768), (97, 264, 768),
                                   (48, 16384, 384), (49, 16384, 384), (128, 3640, 8320), (128, 3656, 8320),
                                   (192, 1024, 1920), (192, 1024, 2048)])
def test_dispatch_edges_of_short_rows(p4q, dev, M, N, K):
    """Around the lines that Kin moves, for fp16 and int32 outputs."""
    test_fewrows_bit_exact(p4q, dev, M, N, K)
