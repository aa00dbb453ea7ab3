"""An explicit schedule runs the kinds that its variants name: the grid of each
launch, read from the phase trace, is that of the named kind (one CTA per SM for
the full kinds), also where a planned run would take the two-per-SM or the
transposed kind of the tile."""
import pytest
import torch

from gpu_util import Launch
from paper_2409_02227_gb300 import goldy as G
from paper_2409_02227_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

F32 = G.GOLDY_F32


def _grids(launch, **opts):
    """Grid sizes of the launches of one traced run, and its results."""
    ctas = 1024
    trace = torch.zeros(ctas * 16, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    G.goldy_run_ex(launch.sched, *launch.ptrs(), launch.ws.data_ptr(), launch.ws_bytes,
                   [s.cuda_stream for s in launch.streams], trace=trace.data_ptr(), trace_ctas=ctas, **opts)
    got = launch.results()
    rows = trace.view(ctas, 16).cpu()
    grids, at = [], 0
    while at < ctas and int(rows[at, 0]) != 0:
        grids.append(int(rows[at, 12]))
        at += grids[-1]
    return grids, got


@pytest.mark.parametrize("ready", [False, True])
@pytest.mark.parametrize("gemms,flags", [(1, 0), (1, G.GOLDY_PLAN_FUSED), (2, G.GOLDY_PLAN_FUSED)])
@pytest.mark.parametrize("kind,M,tile_cols", [(0, 100, 64), (2, 100, 128), (2, 20, 128), (2, 50, 128), (6, 30, 128),
                                              (8, 60, 128)])
def test_explicit_schedules_run_the_named_kind(cuda_ok, kind, M, tile_cols, gemms, flags, ready):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles, K = sms + sms // 4, 200                     # between one and two units per SM
    per = [tiles // gemms] * (gemms - 1)
    per.append(tiles - sum(per))
    A = [wl.integer_matrix(M, K, 8000 + i) for i in range(gemms)]
    B = [wl.integer_matrix(K, t * tile_cols, 8010 + i) for i, t in enumerate(per)]
    s = G.goldy_schedule_build([G.desc(M, t * tile_cols, K, F32) for t in per], [0] * gemms,
                               [G.variant_id(kind, 1, 1)] * gemms, list(range(gemms)), flags)
    grids, got = _grids(Launch(s, A, B, [F32] * gemms), inputs_ready=ready)
    assert grids == [sms]
    for a, b, c in zip(A, B, got):
        assert torch.equal(c.double(), a.double() @ b.double())
