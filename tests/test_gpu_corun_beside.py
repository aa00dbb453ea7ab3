"""A co-run's add beside its GEMM on one stream: each co-run of a chain reads
what the one before wrote (its C as A, its Z as X), enqueued back to back
without a wait, alone and captured in a CUDA graph, against the same chain one
kernel after another, byte for byte.  A GEMM that needs no kernel (K = 0, no
rows) leaves the add in stream order."""
import pytest
import torch

from paper_2409_02227_gb300 import goldy as G

pytestmark = pytest.mark.gpu

BF16, F32 = G.GOLDY_BF16, G.GOLDY_F32


def _chain(policy, M, K, capture, steps=6):
    lut = G.goldy_lut_load()
    n = 1 << 20
    c = G.goldy_corun_plan(G.desc(M, K, K, BF16, lda=max(8, K), ldb=max(8, K), ldc=max(1, K)), n, F32, lut, policy)
    conc, _, _, ws_bytes = G.goldy_corun_query(c)
    gen = torch.Generator(device="cuda").manual_seed(9)
    A = [torch.randn((M, max(8, K)), generator=gen, device="cuda").bfloat16() for _ in range(steps + 1)]
    B = (torch.randn((max(8, K), max(8, K)), generator=gen, device="cuda") / max(1, K) ** 0.5).bfloat16()
    Z = [torch.randn(n, generator=gen, device="cuda") for _ in range(steps + 1)]
    Y = torch.randn(n, generator=gen, device="cuda")
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    s0, s1 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()

    def enqueue(stream):
        for i in range(steps):
            G.goldy_corun_run(c, A[i].data_ptr(), B.data_ptr(), A[i + 1].data_ptr(), ws.data_ptr(), ws_bytes,
                              Z[i].data_ptr(), Y.data_ptr(), Z[i + 1].data_ptr(), [stream, s1.cuda_stream])

    if capture:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s0):
            enqueue(torch.cuda.current_stream().cuda_stream)
        for _ in range(3):
            g.replay()
    else:
        for _ in range(3):
            enqueue(s0.cuda_stream)
    torch.cuda.synchronize()
    assert G.goldy_device_error(clear=True) == 0
    return A, Z, conc


@pytest.mark.parametrize("M,K", [(256, 512), (1000, 1024), (24, 2048), (0, 64), (64, 0)])
@pytest.mark.parametrize("capture", [False, True])
def test_chained_coruns_see_each_others_results(cuda_ok, M, K, capture):
    a0, z0, conc0 = _chain(G.GOLDY_PLAN_SEQUENTIAL, M, K, False)
    for policy in (G.GOLDY_PLAN_DEFAULT, G.GOLDY_PLAN_GO):
        a1, z1, conc1 = _chain(policy, M, K, capture)
        assert conc0 == 0 and conc1 == 1
        for x, y in zip(z0, z1):
            assert torch.equal(x, y)
        if policy == G.GOLDY_PLAN_DEFAULT:           # the same GEMM kernel as the sequential policy
            for x, y in zip(a0, a1):
                assert torch.equal(x.view(torch.int16), y.view(torch.int16))
