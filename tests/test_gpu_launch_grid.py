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
    for rc, tiles in ((4, sms // 4 - 2), (4, sms // 4), (4, sms // 4 + 1), (4, sms // 2), (4, sms // 2 + 1),
                      (2, sms // 2 + 10), (2, sms), (2, sms + 1)):
        cap = 2 * (sms // rc)
        shapes = [(100, tiles * 128, 136), (100, tiles * 128, 136)]
        units = 2 * tiles
        # the run's only launch: twice as many half-size CTAs are the same share
        half = units <= 2 * sms if ready else cap < units <= 2 * cap
        want = min(units, 2 * cap if half else cap)
        assert _run(_plan(shapes, [2, 2], rc, G.GOLDY_PLAN_FUSED), shapes, inputs_ready=ready) == [want]


def _all_at_once(plan, shapes, out, grid, **opts):
    """Whether one launch of `grid` CTAs has all of them running at one time (operands of zeros)."""
    _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
    dt = torch.bfloat16 if out == BF16 else torch.float32
    A = [torch.zeros((M, K), dtype=torch.bfloat16, device="cuda") for M, N, K in shapes]
    B = [torch.zeros((K, N), dtype=torch.bfloat16, device="cuda") for M, N, K in shapes]
    C = [torch.empty((M, N), dtype=dt, device="cuda") for M, N, K in shapes]
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    trace = torch.zeros(1024 * 16, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(2):                       # the first run loads the kernel
        G.goldy_run_ex(plan, [t.data_ptr() for t in A], [t.data_ptr() for t in B], [t.data_ptr() for t in C],
                       ws.data_ptr(), ws_bytes, [s.cuda_stream for s in streams], trace=trace.data_ptr(),
                       trace_ctas=1024, **opts)
        torch.cuda.synchronize()
    assert G.goldy_device_error(clear=True) == 0
    rows = trace.view(1024, 16).cpu()
    rows = rows[rows[:, 0] != 0]
    assert rows.shape[0] == grid and set(rows[:, 12].tolist()) == {grid}
    return int(rows[:, 0].max()) < int(rows[:, 9].min())


@pytest.mark.parametrize("out", [F32, BF16])
@pytest.mark.parametrize("kind,M,tile_cols", [(0, 100, 64), (2, 100, 128), (6, 30, 128), (8, 60, 128)])
def test_two_ctas_per_sm_are_resident(cuda_ok, kind, M, tile_cols, out):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shapes = [(M, 2 * sms * tile_cols, 4096)]
    for flags in (0, G.GOLDY_PLAN_FUSED):
        assert _all_at_once(_plan(shapes, [kind], 1, flags, out), shapes, out, 2 * sms)


@pytest.mark.parametrize("out", [F32, BF16])
@pytest.mark.parametrize("wide", [False, True])
def test_mixed_launch_has_two_ctas_per_sm(cuda_ok, wide, out):
    # two kinds in one launch of two units per SM; one CTA per SM where 256-column tiles write f32
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    kind, cols = (4, 256) if wide else (2, 128)
    shapes = [(200, sms // 2 * cols, 4096), (60, sms * 128, 8192)]
    plan = _plan(shapes, [kind, 8], 1, G.GOLDY_PLAN_FUSED, out)
    kinds = [G.goldy_variant_info_get(G.goldy_schedule_entry(plan, i)[1])["kind"] for i in range(2)]
    assert kinds == [kind, 8]
    one = wide and out == F32
    assert _all_at_once(plan, shapes, out, sms if one else 2 * sms, inputs_ready=True)


@pytest.mark.parametrize("out", [F32, BF16])
@pytest.mark.parametrize("ready", [False, True])
def test_cluster_reduced_launches_stay_apart(cuda_ok, ready, out):
    """Two launches of which K splits that clusters reduce are two thirds stay two; with less they join, if with
    inputs_ready."""
    # (M, N, K, kind, split): 48 of 59 units split 4; 32 of 43; two splits of one kind; 16 of 43; split 2
    for specs, want in (([(122, 1536, 2624, 2, 4), (38, 704, 256, 0, 1)], [48, 11]),
                        ([(122, 1024, 2624, 2, 4), (38, 704, 256, 0, 1)], [32, 11]),
                        ([(60, 1024, 1472, 8, 8), (41, 512, 1600, 8, 4)], [64, 16] if ready else [80]),
                        ([(122, 512, 2624, 2, 4), (38, 1728, 256, 0, 1)], [43] if ready else [16, 27]),
                        ([(122, 1536, 2624, 2, 2), (38, 704, 256, 0, 1)], [35] if ready else [24, 11])):
        shapes = [s[:3] for s in specs]
        entries, descs = [], []
        for M, N, K, kind, split in specs:
            d = G.desc(M, N, K, out)
            key = G.goldy_bucket_key(d)
            entries.append((((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255), 2,
                            [G.variant_id(kind, split, 1)] * 5))
            descs.append(d)
        lut = G.goldy_lut_from_memory(P.write_lut(entries, G.goldy_variant_count(), 152))
        plan = G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | G.GOLDY_PLAN_FUSED)
        got = [G.goldy_variant_info_get(G.goldy_schedule_entry(plan, i)[1]) for i in range(2)]
        assert [(v["kind"], v["split_k"]) for v in got] == [s[3:] for s in specs]
        assert sorted(_run(plan, shapes, out, inputs_ready=ready), reverse=True) == sorted(want, reverse=True)


def _table_plan(specs, out):
    """Fused AUTO plan of (M, N, K, kind, split), each its own table entry, all at once."""
    entries, descs = {}, []
    for M, N, K, kind, split in specs:
        d = G.desc(M, N, K, out)
        key = G.goldy_bucket_key(d)
        key = ((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255)
        entries[key] = (key, 8, [G.variant_id(kind, split, 1)] * 5)
        descs.append(d)
    lut = G.goldy_lut_from_memory(P.write_lut(entries.values(), G.goldy_variant_count(), 152))
    plan = G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | G.GOLDY_PLAN_FUSED)
    got = [G.goldy_variant_info_get(G.goldy_schedule_entry(plan, i)[1]) for i in range(len(specs))]
    assert [(v["kind"], v["split_k"]) for v in got] == [s[3:] for s in specs]
    return plan


def _units(specs, out, **opts):
    """Units of every CTA, launch by launch, of one traced run; its results are checked."""
    plan = _table_plan(specs, out)
    A = [wl.integer_matrix(s[0], s[2], 8200 + i) for i, s in enumerate(specs)]
    B = [wl.integer_matrix(s[2], s[1], 8220 + i) for i, s in enumerate(specs)]
    launch = Launch(plan, A, B, [out] * len(specs))
    trace = torch.zeros(1024 * 16, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    G.goldy_run_ex(plan, *launch.ptrs(), launch.ws.data_ptr(), launch.ws_bytes,
                   [s.cuda_stream for s in launch.streams], trace=trace.data_ptr(), trace_ctas=1024, **opts)
    for a, b, c in zip(A, B, launch.results()):
        want = torch.matmul(a.cuda().double(), b.cuda().double()).to(c.dtype).cpu()
        assert torch.equal(c, want)
    rows = trace.view(1024, 16).cpu()
    counts, at = [], 0
    while at < 1024 and int(rows[at, 0]) != 0:
        grid = int(rows[at, 12])
        counts.append(rows[at:at + grid, 14].tolist())
        at += grid
    return counts


def test_short_units_of_a_last_round_are_spread(cuda_ok):
    """150 pair tiles of 34 K blocks, 6 of 15 and 2 of 4 on 76 pairs: round-robin, at most three to a pair."""
    specs = [(1289, 6208, 2176, 10, 1), (150, 1472, 960, 10, 1), (216, 448, 256, 10, 1), (66, 1280, 2240, 0, 1)]
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the numbers are those of 152 SMs")
    pair, single = sorted(_units(specs, F32, inputs_ready=True), key=len, reverse=True)
    assert len(pair) == 152 and sum(pair) == 2 * 158 and max(pair) == 3 and min(pair) == 2
    assert len(single) == 20


@pytest.mark.parametrize("ready", [False, True])
def test_pair_launch_leaves_room_beside_it(cuda_ok, ready):
    """77 pair tiles take two rounds on 76 pairs and on 58: next to 36 CTAs they take 58.  With one tile more
    than two rounds of 58, or with one tile to a pair of 76, they take all."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the numbers are those of 152 SMs")
    small = (79, 384, 2816, 6, 4)            # 36 units
    for tiles_n, tiles_m, want in ((11, 7, 2 * 58), (29, 4, 2 * 58), (39, 3, 2 * 76), (25, 3, 2 * 75)):
        specs = [(256 * tiles_m - 6, 256 * tiles_n - 64, 896, 10, 1), small]
        grids = sorted((len(u) for u in _units(specs, F32, inputs_ready=ready)), reverse=True)
        # without inputs_ready the launches with room for each other are not joined: resident together
        if ready or want > 2 * 58:
            assert grids == [want, 36], (tiles_n, tiles_m)
        else:
            assert grids[1] == 36 and grids[0] % 2 == 0 and grids[0] + 36 <= 152, (tiles_n, tiles_m)


@pytest.mark.parametrize("stride,per_sm", [(200 * 1024, 2), (200 * 1024 + 1, 1)])
def test_mixed_launch_with_unaligned_batch_entries(cuda_ok, stride, per_sm):
    """Two CTAs per SM want C's rows 16-byte aligned in every entry of a strided batch."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M, N, K, batch = 200, 1024, 136, 12       # 192 units of 128 x 128
    descs = [G.desc(M, N, K, F32, batch=batch, stride_c=stride), G.desc(60, 2048, 200, F32)]
    entries = []
    for d, kind in zip(descs, (2, 8)):
        key = G.goldy_bucket_key(d)
        entries.append((((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255), 2,
                        [G.variant_id(kind, 1, 1)] * 5))
    lut = G.goldy_lut_from_memory(P.write_lut(entries, G.goldy_variant_count(), 152))
    plan = G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | G.GOLDY_PLAN_FUSED)
    gen = torch.Generator(device="cuda").manual_seed(5)
    new = lambda *s: torch.randint(-3, 4, s, generator=gen, device="cuda").bfloat16()
    A, B = [new(batch, M, K), new(60, 200)], [new(batch, K, N), new(200, 2048)]
    C0 = torch.full((batch * stride,), -7.0, device="cuda")
    C = [torch.as_strided(C0, (batch, M, N), (stride, N, 1)), torch.empty((60, 2048), device="cuda")]
    _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    trace = torch.zeros(1024 * 16, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    G.goldy_run_ex(plan, [a.data_ptr() for a in A], [b.data_ptr() for b in B], [c.data_ptr() for c in C],
                   ws.data_ptr(), ws_bytes, [s.cuda_stream for s in streams], trace=trace.data_ptr(), trace_ctas=1024,
                   inputs_ready=True)
    torch.cuda.synchronize()
    assert G.goldy_device_error(clear=True) == 0
    for a, b, c in zip(A, B, C):
        assert torch.equal(c.double(), a.double() @ b.double())
    for e in range(batch - 1):                # nothing written between the entries
        assert bool((C0[e * stride + M * N:(e + 1) * stride] == -7.0).all())
    assert int(trace[12]) == min(192 + 16, per_sm * sms)


@pytest.mark.parametrize("ready", [False, True])
def test_launches_that_run_side_by_side_stay_apart(cuda_ok, ready):
    """Pair tiles next to single-CTA kinds that all fit on the GPU at once: a launch each without inputs_ready,
    one of the pair kernel and one of the others with it; with more tiles than fit, joined either way."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small = [(100, 640, 1400, 2, 1), (40, 1280, 1200, 8, 1)]              # 5 and 10 units
    for tiles_n, fits in (((sms - 15) // 4, True), ((sms - 15) // 4 + 2, False)):
        specs = [(500, 256 * tiles_n - 64, 1096, 10, 1)] + small          # two rows of tiles
        grids = sorted(len(u) for u in _units(specs, F32, inputs_ready=ready))
        pair = min(4 * tiles_n, sms // 2 * 2)
        if fits and not ready:
            assert grids == sorted([pair, 5, 10])
        else:
            assert len(grids) == 2 and grids[0] == 15


def test_long_pair_launch_takes_the_whole_gpu(cuda_ok):
    """Next to 4 CTAs a pair launch ends within 4% on the SMs that they leave, but one of over a millisecond
    does not leave them (the other launch would wait for it, loaded, for as long)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small = (60, 512, 9216, 8, 1)             # 4 units
    for M, want in ((4096, sms - 4), (20480, sms)):
        specs = [(M, 8192, 8192, 10, 1), small]
        plan = _table_plan(specs, BF16)
        _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
        A = [torch.zeros((s[0], s[2]), dtype=torch.bfloat16, device="cuda") for s in specs]
        B = [torch.zeros((s[2], s[1]), dtype=torch.bfloat16, device="cuda") for s in specs]
        C = [torch.ones((s[0], s[1]), dtype=torch.bfloat16, device="cuda") for s in specs]
        ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
        streams = [torch.cuda.Stream() for _ in range(n_streams)]
        trace = torch.zeros(1024 * 16, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        G.goldy_run_ex(plan, [t.data_ptr() for t in A], [t.data_ptr() for t in B], [t.data_ptr() for t in C],
                       ws.data_ptr(), ws_bytes, [x.cuda_stream for x in streams], trace=trace.data_ptr(),
                       trace_ctas=1024)
        torch.cuda.synchronize()
        assert G.goldy_device_error(clear=True) == 0
        rows = trace.view(1024, 16).cpu()
        rows = rows[rows[:, 0] != 0]
        assert sorted(set(rows[:, 12].tolist())) == [4, want]
        assert not any(bool(c.any()) for c in C)
