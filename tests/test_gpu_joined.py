"""Fused plans of the dynamic logic join their launches: all single-CTA kinds
of a run in one launch that reads the tile shape per GEMM, all CTA-pair GEMMs
in one launch of the pair kernel, the units dealt out in equal shares.  Integer
inputs make every fp32 result exact; a table written here gives each GEMM the
kernel under test.  The joined run must also give the bytes of the same plan in
streams mode (one launch per GEMM)."""
import pytest
import torch

from paper_2409_02227_gb300 import goldy as G
from paper_2409_02227_gb300 import profile_lut as P
from paper_2409_02227_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

F32, BF16 = G.GOLDY_F32, G.GOLDY_BF16
TORCH = {F32: torch.float32, BF16: torch.bfloat16}
PAIR = 10


def _plan(specs, out, flags, pref=1):
    """Plan specs (M, N, K, batch, kind, split): one bucket each (their floor
    log2 sizes differ), its kernel at every CD."""
    entries = {}
    descs = []
    for M, N, K, batch, kind, split in specs:
        d = G.desc(M, N, K, out, lda=(K + 7) // 8 * 8, ldb=(N + 7) // 8 * 8, ldc=N, batch=batch)
        key = G.goldy_bucket_key(d)
        key = ((key >> 24) & 255, (key >> 16) & 255, (key >> 8) & 255, key & 255)
        assert key not in entries, "specs of one test lie in different buckets"
        entries[key] = (key, pref, [G.variant_id(kind, split, 1)] * 5)
        descs.append(d)
    lut = G.goldy_lut_from_memory(P.write_lut(entries.values(), G.goldy_variant_count(), 152))
    return descs, G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | flags)


def _pad8(t):
    out = torch.full((*t.shape[:-1], (t.shape[-1] + 7) // 8 * 8), 5.0, dtype=t.dtype)
    out[..., :t.shape[-1]] = t
    return out


def _check(specs, out, seed):
    A, B, want = [], [], []
    for i, (M, N, K, batch, _, _) in enumerate(specs):
        a = torch.stack([wl.integer_matrix(M, K, seed + 40 * i + j) for j in range(batch)])
        b = torch.stack([wl.integer_matrix(K, N, seed + 40 * i + 20 + j) for j in range(batch)])
        A.append(_pad8(a).cuda())
        B.append(_pad8(b).cuda())
        want.append(torch.bmm(a.cuda().double(), b.cuda().double()).float().to(TORCH[out]))
    C = [torch.empty((s[3], s[0], s[1]), dtype=TORCH[out], device="cuda") for s in specs]
    ptrs = [[t.data_ptr() for t in ts] for ts in (A, B, C)]
    streams = [torch.cuda.Stream() for _ in range(G.GOLDY_MAX_STREAMS)]
    handles = [s.cuda_stream for s in streams]
    for fused in (G.GOLDY_PLAN_FUSED, 0):
        _, plan = _plan(specs, out, fused)
        _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
        ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        ex = G.goldy_exec_create(plan, *ptrs, ws.data_ptr(), ws_bytes, handles[:n_streams])
        gr = G.goldy_graph_create(plan, *ptrs, ws.data_ptr(), ws_bytes, handles[:n_streams])

        def run(**kw):
            G.goldy_run_ex(plan, *ptrs, ws.data_ptr(), ws_bytes, handles[:n_streams], **kw)

        for how in (run, lambda: run(inputs_ready=True), lambda: run(serial_launch=True),
                    lambda: G.goldy_exec_launch(ex), lambda: G.goldy_graph_launch(gr, handles[0])):
            for c in C:
                c.fill_(float("nan"))
            torch.cuda.synchronize()
            for _ in range(3):               # back to back: each run's launches overlap the one before
                how()
            torch.cuda.synchronize()
            assert G.goldy_device_error(clear=True) == 0
            for i, c in enumerate(C):
                assert torch.equal(c, want[i]), (specs[i], out, fused)
        del ex, gr


# (M, N, K, batch, kind, split); kinds 0-5: 128 x 64 / 128 / 256 (full, half), 6-9: 32 / 64 x 128 transposed
SETS = {
    # every single-CTA kind, ragged sizes
    "kinds": [(200, 320, 456, 1, 0, 1), (130, 700, 72, 1, 1, 1), (97, 1100, 200, 1, 2, 1), (300, 150, 1000, 1, 3, 1),
              (520, 130, 136, 1, 4, 1), (70, 257, 2056, 1, 5, 1), (16, 600, 520, 1, 6, 1), (33, 2100, 264, 1, 7, 1),
              (65, 129, 328, 1, 8, 1), (40, 64, 64, 1, 9, 1)],
    # K splits of several tile shapes in one launch, next to unsplit GEMMs
    "splits": [(130, 320, 1160, 1, 0, 4), (200, 136, 2056, 1, 2, 8), (257, 520, 600, 1, 4, 2), (20, 1030, 4104, 1, 6, 8),
               (50, 260, 520, 1, 8, 4), (140, 72, 264, 1, 2, 1)],
    # rows that are not 16-byte aligned, split and unsplit
    "odd_rows": [(33, 65, 129, 1, 0, 1), (129, 257, 515, 1, 4, 2), (17, 1025, 259, 1, 6, 1), (260, 131, 1031, 1, 2, 4)],
    # pair GEMMs (one split, one with a narrow last tile) and single-CTA ones: two launches
    "pair": [(700, 600, 1096, 1, PAIR, 1), (300, 128, 200, 1, PAIR, 1), (1030, 300, 2056, 1, PAIR, 4),
             (40, 1500, 520, 1, 8, 1), (130, 200, 72, 1, 2, 2), (20, 70, 264, 1, 6, 1)],
    # strided batches next to plain GEMMs; many more units than CTAs; K shorter than a block
    "batched": [(130, 136, 200, 6, 2, 1), (40, 72, 64, 9, 8, 1), (1500, 1100, 136, 1, 0, 1), (300, 300, 8, 1, 3, 1)],
    # more units than SMs and aligned rows: with inputs_ready two CTAs per SM, with one 256-column accumulator ...
    "two_per_sm_wide": [(520, 4096, 456, 1, 4, 1), (200, 2048, 2056, 1, 2, 4), (33, 2048, 520, 1, 8, 2),
                        (20, 1032, 4104, 1, 6, 8), (300, 72, 72, 1, 0, 1), (600, 520, 1032, 1, 4, 2)],
    # ... and with two of 128
    "two_per_sm": [(200, 2048, 2056, 1, 2, 4), (33, 4096, 520, 1, 8, 2), (20, 1032, 4104, 1, 6, 8),
                   (300, 72, 72, 1, 0, 1), (1100, 1048, 200, 1, 2, 1), (64, 2048, 64, 1, 9, 1)],
    # one unit per GEMM: fewer units than CTAs
    "tiny": [(1, 1, 8, 1, 0, 1), (16, 64, 64, 1, 8, 1), (5, 130, 16, 1, 2, 1)],
}


@pytest.mark.parametrize("out", [F32, BF16])
@pytest.mark.parametrize("name", sorted(SETS))
def test_joined_launches(cuda_ok, name, out):
    _check(SETS[name], out, 5000)


def test_more_gemms_than_one_launch_holds(cuda_ok):
    # 20 single-CTA GEMMs of two kinds: two joined launches
    specs = []
    for i, lm in enumerate((4, 5, 6, 7, 8)):
        for j, ln in enumerate((6, 7, 8, 9)):
            specs.append(((1 << lm) + 3, (1 << ln) + 8 * j, 264, 1, 2 if (i + j) % 2 else 8, 1))
    _check(specs, F32, 6000)
