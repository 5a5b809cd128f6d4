"""The quantizers' rounding of fp16 rows (one multiplier per row; ties to even
where the scale is exact) against round_half_even(fl32(x / s)), s = fl32(a / 7):
on the CPU for every row maximum, on the GPU through the kernels."""
import numpy as np
import pytest
import torch

import oracle

TIES = 2 * np.arange(7) + 1  # quotients x / a of (2k + 1) / 14


def _near_ties(a):
    """[len(a), 7 * 5]: the fp16 values within two steps of a (2k + 1) / 14, at most a."""
    t = (a.astype(np.float64)[:, None] * TIES[None] / 14).astype(np.float16).view(np.uint16).astype(np.int32)
    x = (t[..., None] + np.arange(-2, 3)).reshape(len(a), -1)
    return np.clip(x, 0, a.view(np.uint16)[:, None]).astype(np.uint16).view(np.float16)


def test_multiplier_rounds_as_the_quotient():
    """Every finite positive fp16 maximum, the values next to each rounding
    boundary (the codes are monotone in between). float64 holds a product of an
    fp16 and an fp32 value exactly, so np.rint is the fused operation's rounding."""
    a = np.arange(1, 0x7C00, dtype=np.uint16).view(np.float16)
    x = _near_ties(a).astype(np.float32)
    s = a.astype(np.float32) / np.float32(7)
    ref = np.rint(x / s[:, None])
    inv = np.float32(1) / s
    tie = s.astype(np.float64) * 7 == a.astype(np.float64)
    up = (np.float32(0.5) * a.astype(np.float32)) / s >= np.float32(3.5)
    m = inv * np.where(up, np.float32(1 + 2.0 ** -20), np.float32(1 - 2.0 ** -20))
    one = np.rint(x.astype(np.float64) * m[:, None])
    hi = np.rint(x.astype(np.float64) * (inv * np.float32(1 + 2.0 ** -21))[:, None])
    lo = np.rint(x.astype(np.float64) * (inv * np.float32(1 - 2.0 ** -21))[:, None])
    two = np.where(hi % 2 == 1, lo, hi)
    assert tie.any() and not tie.all()
    assert np.array_equal(np.where(tie[:, None], two, one), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("M", [31, 4096])  # the streaming and the register-resident kernel
def test_codes_next_to_ties(p4q, dev, M):
    rng = np.random.default_rng(M)
    a = rng.integers(1, 0x7C00, size=M).astype(np.uint16)
    a[::3] = (a[::3] & 0x7C00) | (np.uint16(7) * rng.integers(147, 292, size=len(a[::3])).astype(np.uint16) & 0x3FF)
    a[:4] = [1, 2, 14, 0x7BFF]
    a = a.view(np.float16)
    x = np.zeros((M, 256), dtype=np.float16)
    near = _near_ties(a)
    x[:, :35], x[:, 64:99] = near, -near
    x[:, 128:] = (rng.random((M, 128), dtype=np.float32) * 2 - 1).astype(np.float16) * a[:, None]
    x[:, 40] = a
    q, s = p4q.quant_act(torch.from_numpy(x).to(dev))
    torch.cuda.synchronize()
    assert p4q.p4q_device_status() == 0
    c, sr = oracle.quantize_rows(x)
    assert np.array_equal(s.cpu().numpy().view(np.uint32), sr.view(np.uint32))
    assert np.array_equal(oracle.unpack_codes(q.cpu().numpy()), c)


@pytest.mark.gpu
@pytest.mark.parametrize("B,N,d,J", [(1, 5, 256, 1), (3, 33, 1024, 4), (2, 70, 1280, 5), (1, 300, 4096, 16),
                                     (2, 65, 5120, 3), (1, 130, 4864, 0), (40, 9, 2048, 2)])
def test_token_pass_rows(p4q, dev, B, N, d, J):
    """The selector's token pass (two warps per row, every number of chunks per
    lane, few and many concepts) through the kept tokens of rows near ties."""
    from paper_2609_34867_gb300 import workloads as wl
    K = max(1, N // 2)
    w = wl.Workload("t", B=B, N=N, d=d, K=K, T=0, J=max(J, 1), seed=d + N, heavy_tail=True, linears=())
    x = wl.selector_inputs(w)
    V = x.V.copy()
    V[:, ::2, : d // 2] = np.float16(0.5) * np.abs(V[:, ::2]).max(axis=2, keepdims=True)
    Q = x.Q if J else np.zeros((B, 0, d), dtype=np.float16)
    idx = p4q.select(torch.from_numpy(V).to(dev), torch.from_numpy(Q).to(dev), torch.from_numpy(x.A).to(dev), K)
    torch.cuda.synchronize()
    assert p4q.p4q_device_status() == 0
    assert np.array_equal(idx.cpu().numpy(), oracle.select_batch(V, K, Q, x.A))
