"""What a caller enqueues on a run's other streams keeps its place in their
order.  Inputs are written there behind a delay of about a millisecond, and the
results are read there, with no event between the caller's work and the run."""
import pytest
import torch

from paper_2409_02227_gb300 import goldy as G
from paper_2409_02227_gb300 import profile_lut as P

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


# (M, N, K, kind): one launch each of a fused wave, so one stream each; the
# first set's three kinds join into two launches, the second's into one, the
# third's run side by side
WAVES = [[(100, 320, 1496, 2), (40, 1500, 1200, 8), (2500, 2600, 1096, 10)],
         [(200, 320, 456, 2), (40, 300, 520, 8), (20, 600, 1000, 6)],
         [(100, 320, 1496, 2), (40, 1500, 1200, 8), (700, 600, 1096, 10)]]


@pytest.mark.parametrize("how", ["run", "exec", "captured run", "captured exec"])
@pytest.mark.parametrize("wave", [0, 1, 2])
def test_joined_run_keeps_the_order_of_its_streams(cuda_ok, wave, how):
    specs = WAVES[wave]
    entries, descs = [], []
    for M, N, K, kind in specs:
        d = G.desc(M, N, K, F32, lda=K, ldb=(N + 7) // 8 * 8, ldc=N)
        key = G.goldy_bucket_key(d)
        entries.append((((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255), 4,
                        [G.variant_id(kind, 1, 1)] * 5))
        descs.append(d)
    lut = G.goldy_lut_from_memory(P.write_lut(entries, G.goldy_variant_count(), 152))
    plan = G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | G.GOLDY_PLAN_FUSED)
    slots = [G.goldy_schedule_entry(plan, i)[2] for i in range(len(specs))]
    assert sorted(slots) == [0, 1, 2]
    _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
    gen = torch.Generator(device="cuda").manual_seed(4)
    new = lambda r, c: torch.randint(-3, 4, (r, c), generator=gen, device="cuda").bfloat16()
    src = [[new(M, K) for M, N, K, _ in specs] for _ in range(3)]
    A = [torch.zeros_like(a) for a in src[0]]
    B = [new(K, (N + 7) // 8 * 8) for M, N, K, _ in specs]
    C = [torch.zeros((M, N), device="cuda") for M, N, K, _ in specs]
    out = [[torch.zeros_like(c) for c in C] for _ in src]
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    handles = [s.cuda_stream for s in streams]
    args = (plan, [a.data_ptr() for a in A], [b.data_ptr() for b in B], [c.data_ptr() for c in C], ws.data_ptr(),
            ws_bytes, handles)
    ex = G.goldy_exec_create(*args) if "exec" in how else None
    launch = (lambda: G.goldy_exec_launch(ex)) if ex else (lambda: G.goldy_run(*args))

    def step(a, o):
        # each GEMM's A is written, and its C read, on the stream of its slot
        for i, k in enumerate(slots):
            _late(streams[k], A[i], a[i])
        launch()
        for i, k in enumerate(slots):
            with torch.cuda.stream(streams[k]):
                o[i].copy_(C[i])

    torch.cuda.synchronize()
    if "captured" in how:
        launch()                              # loads the kernels
        torch.cuda.synchronize()
        for a, o in zip(src, out):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=streams[0]):
                for s in streams[1:]:
                    s.wait_stream(streams[0])
                step(a, o)
                for s in streams[1:]:
                    streams[0].wait_stream(s)
            g.replay()
            torch.cuda.synchronize()
        # a capture that uses streams[0] alone: the run leaves no stream unjoined
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[0]):
            launch()
        g.replay()
    else:
        for a, o in zip(src, out):
            step(a, o)
    torch.cuda.synchronize()
    assert G.goldy_device_error(clear=True) == 0
    for a, o in zip(src, out):
        for i, (M, N, K, _) in enumerate(specs):
            assert torch.equal(o[i].double(), a[i].double() @ B[i][:, :N].double()), (specs[i], how)
    del ex


@pytest.mark.parametrize("how", ["run", "exec", "captured run"])
def test_joined_run_reads_what_the_kernel_before_it_wrote(cuda_ok, how):
    """The later launches of a joined run start while its first is still going on; their operands, written by
    the kernel right before the run, have to be there all the same."""
    specs = [(2500, 2600, 1096, 10), (100, 1320, 4096, 2), (40, 1500, 2200, 8), (20, 600, 4000, 6)]
    entries, descs = [], []
    for M, N, K, kind in specs:
        d = G.desc(M, N, K, F32, lda=K, ldb=(N + 7) // 8 * 8, ldc=N)
        key = G.goldy_bucket_key(d)
        entries.append((((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255), 4,
                        [G.variant_id(kind, 1, 1)] * 5))
        descs.append(d)
    lut = G.goldy_lut_from_memory(P.write_lut(entries, G.goldy_variant_count(), 152))
    plan = G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | G.GOLDY_PLAN_FUSED)
    kinds = [G.goldy_variant_info_get(G.goldy_schedule_entry(plan, i)[1])["kind"] for i in range(len(specs))]
    assert kinds == [s[3] for s in specs]    # one launch of the pair kernel, one of the others
    _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
    gen = torch.Generator(device="cuda").manual_seed(6)
    new = lambda r, c: torch.randint(-3, 4, (r, c), generator=gen, device="cuda").bfloat16()
    rounds = 8
    # all A and all B in one buffer each round, so that one kernel writes them right before the run
    sizes = [M * K + K * ((N + 7) // 8 * 8) for M, N, K, _ in specs]
    src = [torch.cat([new(1, n)[0] for n in sizes]) for _ in range(rounds)]
    buf = torch.zeros(sum(sizes), dtype=torch.bfloat16, device="cuda")

    def views(t):
        A, B, at = [], [], 0
        for M, N, K, _ in specs:
            ld = (N + 7) // 8 * 8
            A.append(t[at:at + M * K].view(M, K))
            B.append(t[at + M * K:at + M * K + K * ld].view(K, ld))
            at += M * K + K * ld
        return A, B

    A, B = views(buf)
    C = [torch.zeros((M, N), device="cuda") for M, N, K, _ in specs]
    out = [[torch.zeros_like(c) for c in C] for _ in range(rounds)]
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    args = (plan, [a.data_ptr() for a in A], [b.data_ptr() for b in B], [c.data_ptr() for c in C], ws.data_ptr(),
            ws_bytes, [s.cuda_stream for s in streams])
    assert all(t.data_ptr() % 16 == 0 for t in A + B)
    ex = G.goldy_exec_create(*args) if how == "exec" else None
    launch = (lambda: G.goldy_exec_launch(ex)) if ex else (lambda: G.goldy_run(*args))
    torch.cuda.synchronize()

    def steps():
        for r in range(rounds):
            buf.copy_(src[r])
            launch()
            for c, o in zip(C, out[r]):
                o.copy_(c)

    if how == "captured run":
        launch()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[0]):
            steps()
        g.replay()
    else:
        with torch.cuda.stream(streams[0]):
            steps()
    torch.cuda.synchronize()
    assert G.goldy_device_error(clear=True) == 0
    for r in range(rounds):
        a, b = views(src[r])
        for i, (M, N, K, _) in enumerate(specs):
            assert torch.equal(out[r][i].double(), a[i].double() @ b[i][:, :N].double()), (r, specs[i], how)
    del ex
