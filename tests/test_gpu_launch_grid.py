"""Grids of planned launches, read from the phase trace: a GEMM planned for a
share of the GPU (half or a quarter of the SMs) keeps to it, whatever kind its
launch takes."""
import pytest
import torch

from gpu_util import Launch
from paper_2409_02227_gb300 import goldy as G
from paper_2409_02227_gb300 import profile_lut as P
from paper_2409_02227_gb300 import workloads as wl
from test_gpu_named_kinds import _grids

pytestmark = pytest.mark.gpu

F32, BF16 = G.GOLDY_F32, G.GOLDY_BF16


def _plan(shapes, kinds, rc, flags, out=F32, split=1):
    """AUTO plan of GEMMs (M, N, K), a table entry each: kind, split and share as given, at every CD."""
    entries, descs = {}, []
    for (M, N, K), kind in zip(shapes, kinds):
        d = G.desc(M, N, K, out)
        key = G.goldy_bucket_key(d)
        key = ((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255)
        entries[key] = (key, min(16, len(shapes)), [G.variant_id(kind, split, rc)] * 5)
        descs.append(d)
    lut = G.goldy_lut_from_memory(P.write_lut(entries.values(), G.goldy_variant_count(), 152))
    return G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | flags)


def _run(plan, shapes, out=F32, **opts):
    A = [wl.integer_matrix(M, K, 8100 + i) for i, (M, N, K) in enumerate(shapes)]
    B = [wl.integer_matrix(K, N, 8120 + i) for i, (M, N, K) in enumerate(shapes)]
    grids, got = _grids(Launch(plan, A, B, [out] * len(shapes)), **opts)
    for a, b, c in zip(A, B, got):
        assert torch.equal(c.double(), (a.double() @ b.double()).to(c.dtype).double())
    return grids


@pytest.mark.parametrize("ready", [False, True])
@pytest.mark.parametrize("rc", [1, 2, 4])
@pytest.mark.parametrize("kind,tile_cols", [(0, 64), (2, 128)])
def test_planned_launch_keeps_its_share(cuda_ok, kind, tile_cols, rc, ready):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cap = sms // rc
    for units in (cap // 2, cap, cap + 1, 2 * cap, 2 * cap + 1, sms + 1, 2 * sms, 2 * sms + 1):
        shapes = [(100, units * tile_cols, 136)]
        for flags in (0, G.GOLDY_PLAN_FUSED):
            # the whole GPU: up to two units per SM all at once on the two-per-SM kind
            want = units if rc == 1 and units <= 2 * sms else min(units, cap)
            assert _run(_plan(shapes, [kind], rc, flags), shapes, inputs_ready=ready) == [want], (units, flags)


@pytest.mark.parametrize("ready", [False, True])
def test_fused_launch_keeps_the_sum_of_its_shares(cuda_ok, ready):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for rc, tiles in ((4, sms // 2), (4, sms // 4 - 2), (2, sms // 2 + 10)):
        cap = 2 * (sms // rc)
        shapes = [(100, tiles * 128, 136), (100, tiles * 128, 136)]
        units = 2 * tiles
        want = units if cap >= sms and units <= 2 * sms else min(units, cap)
        assert _run(_plan(shapes, [2, 2], rc, G.GOLDY_PLAN_FUSED), shapes, inputs_ready=ready) == [want]
