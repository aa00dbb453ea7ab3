"""With inputs_ready a launch of at most two CTAs' worth of units per SM runs as
the two-per-SM kind of its tile shape: the bytes of the plain run, alone and
fused, at unit counts on both sides of the rule's lines (152 SMs: half, one and
two units per SM), with and without K splits, replayed back to back."""
import pytest
import torch

from paper_2409_02227_gb300 import goldy as G
from paper_2409_02227_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

F32, BF16 = G.GOLDY_F32, G.GOLDY_BF16
TORCH = {F32: torch.float32, BF16: torch.bfloat16}


@pytest.mark.parametrize("out", [F32, BF16])
@pytest.mark.parametrize("kind,split,rc", [(0, 1, 1), (0, 4, 1), (2, 1, 2), (2, 4, 1), (2, 8, 4), (4, 1, 1), (6, 1, 1),
                                           (6, 8, 1), (8, 1, 4), (8, 2, 1)])
def test_inputs_ready_runs_match_plain_ones(cuda_ok, kind, split, rc, out):
    # 1, 10, 40, 80 and 400 units' worth of columns per GEMM (tiles x splits), ragged edges
    cols = 128 if kind >= 6 else {0: 64, 2: 128, 4: 256}[kind]
    rows = {6: 32, 8: 64}.get(kind, 128)
    v = G.variant_id(kind, split, rc)
    for i, (tiles, gemms) in enumerate([(1, 1), (10, 2), (40, 2), (80, 3), (400 // split, 1)]):
        M, N, K = rows - 5, cols * tiles - 8, 64 * 9 + 24
        A = [wl.integer_matrix(M, K, 7000 + 10 * i + j).cuda() for j in range(gemms)]
        B = [wl.integer_matrix(K, N, 7100 + 10 * i + j).cuda() for j in range(gemms)]
        C = [torch.empty((M, N), dtype=TORCH[out], device="cuda") for _ in range(gemms)]
        want = [(a.double() @ b.double()).float().to(TORCH[out]) for a, b in zip(A, B)]
        s = G.goldy_schedule_build([G.desc(M, N, K, out)] * gemms, [0] * gemms, [v] * gemms, list(range(gemms)),
                                   G.GOLDY_PLAN_FUSED)
        _, _, ns, ws_bytes = G.goldy_schedule_query(s)
        ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
        streams = [torch.cuda.Stream() for _ in range(ns)]
        ptrs = [[t.data_ptr() for t in ts] for ts in (A, B, C)]
        for ready in (True, False):
            ex = G.goldy_exec_create(s, *ptrs, ws.data_ptr(), ws_bytes, [x.cuda_stream for x in streams],
                                     inputs_ready=ready)
            for c in C:
                c.fill_(float("nan"))
            torch.cuda.synchronize()
            for _ in range(4):
                G.goldy_exec_launch(ex)
            torch.cuda.synchronize()
            assert G.goldy_device_error(clear=True) == 0
            for c, w in zip(C, want):
                assert torch.equal(c, w), (kind, split, rc, out, tiles, gemms, ready)
            del ex
