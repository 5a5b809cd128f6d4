"""Kernels of one stream overlap: the next may start before the one two ahead of
it has read a buffer that the one in between rewrites. Chains of quantizers and
linears on reused buffers, back to back and as a CUDA graph, must give bit for
bit what the same calls give when each is waited for."""
import glob
import os
import re

import pytest
import torch

from paper_2609_34867_gb300 import build as B


def _code(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def test_stream_data_is_not_read_as_read_only():
    """The read-only path (ld.global.nc, __ldg, const __restrict__) requires data
    that nothing writes while the kernel is resident. Only ldg_readonly16 takes
    it, in the selector's row gather, two launches after the codes that it reads."""
    uses = []
    for path in sorted(glob.glob(os.path.join(B.CSRC, "*.cu*"))):
        code = _code(path)
        assert not re.search(r"__ldg|const[^,()]*\*\s*__restrict__", code), path
        assert len(re.findall(r"ld\.global\.nc", code)) == (1 if path.endswith("p4q_device.cuh") else 0), path
        uses += [os.path.basename(path)] * len(re.findall(r"(?<!uint4 )ldg_readonly16\(", code))
    assert uses == ["p4q_select.cu"]


D, F, LAYERS = 1024, 2048, 6


@pytest.mark.gpu
@pytest.mark.parametrize("M", [1, 2, 5, 24, 130, 600])
def test_chain_on_reused_buffers(p4q, dev, M):
    g = torch.Generator(device=dev).manual_seed(M)
    half = lambda *s: torch.randn(s, generator=g, device=dev).half()
    W = [[p4q.quant_weight(half(n, k) * 0.03) for n, k in ((2 * F, D), (D, F), (F, D), (D, F))] for _ in range(LAYERS)]
    w = [(1 + 0.1 * half(D)).contiguous() for _ in range(LAYERS)]
    X0 = half(M, D)
    X, Y = torch.empty_like(X0), torch.empty((M, 2 * F), dtype=torch.float16, device=dev)
    Z = torch.empty((M, F), dtype=torch.float16, device=dev)
    q, s = torch.empty((M * F // 2,), dtype=torch.uint8, device=dev), torch.empty((M,), device=dev)
    u, su = torch.empty((M, F), dtype=torch.uint8, device=dev), torch.empty((M,), dtype=torch.int32, device=dev)
    ws = p4q.linear_workspace(M, 2 * F, F, dev)
    qd, qf = q[:M * D // 2].view(M, D // 2), q.view(M, F // 2)
    kept = torch.empty((LAYERS, M, D + F), dtype=torch.float16, device=dev)

    def chain(after):
        X.copy_(X0)
        for i in range(LAYERS):
            calls = [
                # one code buffer, one scale buffer; X is rewritten by the linears that its own quantizers feed
                lambda: p4q.p4q_rmsnorm_quant_expanded(X, w[i], 1e-5, qd, s),
                lambda: p4q.p4q_w4a4_linear_ws(qd, s, *W[i][0], Y, ws),
                lambda: p4q.p4q_swiglu_quant_expanded(Y[:, :F], Y[:, F:], qf, s, u, su),
                lambda: p4q.p4q_w4a4_linear(qf, s, *W[i][1], X),
                lambda: p4q.p4q_quant_act(X, qd, s),
                lambda: p4q.p4q_w4a4_linear(qd, s, *W[i][2], Z),
                lambda: p4q.p4q_quant_act(Z, qf, s),
                lambda: p4q.p4q_w4a4_linear_ws(qf, s, *W[i][3], X, ws),
            ]
            for c in calls:
                c()
                after()
            kept[i, :, :D].copy_(X)
            kept[i, :, D:].copy_(Z)
        return kept

    ref = chain(torch.cuda.synchronize).clone()
    assert torch.isfinite(ref).all() and ref[-1].abs().max() > 0
    for _ in range(10):
        kept.zero_()
        assert torch.equal(chain(lambda: None), ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(lambda: None)
    for _ in range(30):
        kept.zero_()
        graph.replay()
        assert torch.equal(kept, ref)
    assert p4q.p4q_device_status() == 0
