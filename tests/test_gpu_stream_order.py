"""What a caller enqueues on a run's other streams keeps its place in their
order.  Inputs are written there behind a delay of about a millisecond, and the
results are read there, with no event between the caller's work and the run."""
import pytest
import torch

from paper_2409_02227_gb300 import goldy as G

pytestmark = pytest.mark.gpu

F32, BF16 = G.GOLDY_F32, G.GOLDY_BF16


def _late(stream, dst, src):
    """On `stream`: about a millisecond of nothing, then dst <- src."""
    with torch.cuda.stream(stream):
        torch.cuda._sleep(2_000_000)
        dst.copy_(src)


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("policy", [G.GOLDY_PLAN_DEFAULT, G.GOLDY_PLAN_GO])
def test_coruns_add_keeps_the_order_of_its_stream(cuda_ok, policy, prepared):
    M, N, K, n = 300, 512, 256, 1 << 18
    c = G.goldy_corun_plan(G.desc(M, N, K, BF16), n, F32, G.goldy_lut_load(), policy)
    concurrent, _, _, ws_bytes = G.goldy_corun_query(c)
    assert concurrent == 1
    gen = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randint(-3, 4, (M, K), generator=gen, device="cuda").bfloat16()
    B = torch.randint(-3, 4, (K, N), generator=gen, device="cuda").bfloat16()
    C = torch.zeros((M, N), device="cuda").bfloat16()
    src = [torch.randn(n, generator=gen, device="cuda") for _ in range(3)]
    Y = torch.randn(n, generator=gen, device="cuda")
    X, Z = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    out = [torch.zeros(n, device="cuda") for _ in src]
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    s0, s1 = torch.cuda.Stream(), torch.cuda.Stream()
    args = (c, A.data_ptr(), B.data_ptr(), C.data_ptr(), ws.data_ptr(), ws_bytes, X.data_ptr(), Y.data_ptr(),
            Z.data_ptr(), [s0.cuda_stream, s1.cuda_stream])
    torch.cuda.synchronize()
    ex = G.goldy_corun_exec_create(*args) if prepared else None
    for x, o in zip(src, out):
        _late(s1, X, x)                       # the add's input, on the add's stream
        G.goldy_exec_launch(ex) if prepared else G.goldy_corun_run(*args)
        with torch.cuda.stream(s1):           # and its result, there too
            o.copy_(Z)
    torch.cuda.synchronize()
    assert G.goldy_device_error(clear=True) == 0
    for x, o in zip(src, out):
        assert torch.equal(o, x + Y)
    assert torch.equal(C.float(), (A.double() @ B.double()).bfloat16().float())
    del ex
