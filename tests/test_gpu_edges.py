"""Tile edges of the output paths, exactly: integer inputs (every partial sum
an integer below 2^24, so fp32 results are exact and bf16 ones the rounding of
an exact value), C inside a larger sentinel-filled buffer at row strides and
offsets that are and are not 16-byte aligned.  Every element of C must be
exact and nothing outside it may change."""
import pytest
import torch

from paper_2409_02227_gb300 import goldy as G
from paper_2409_02227_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

F32, BF16 = G.GOLDY_F32, G.GOLDY_BF16
TORCH = {F32: torch.float32, BF16: torch.bfloat16}
PAIR = 10
SENTINEL = -777.0


def _pad8(t):
    r, c = t.shape
    out = torch.full((r, (c + 7) // 8 * 8), 3.0, dtype=t.dtype)   # the padding is never part of the product
    out[:, :c] = t
    return out


def _check(kind, split, out, M, N, K, ldc, offset, seed):
    a, b = wl.integer_matrix(M, K, seed), wl.integer_matrix(K, N, seed + 1)
    exact = (a.to(torch.int64) @ b.to(torch.int64)).to(torch.float32).to(TORCH[out])
    dA, dB = _pad8(a).cuda(), _pad8(b).cuda()
    d = G.desc(M, N, K, out, lda=dA.shape[1], ldb=dB.shape[1], ldc=ldc)
    s = G.goldy_schedule_build([d], [0], [G.variant_id(kind, split, 1)], [0])
    ws_bytes = G.goldy_schedule_query(s)[3]
    ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
    buf = torch.full((offset + M * ldc + 64,), SENTINEL, dtype=TORCH[out], device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for ready in (False, True):
        buf.fill_(SENTINEL)
        torch.cuda.synchronize()
        for _ in range(2):
            G.goldy_run_ex(s, [dA.data_ptr()], [dB.data_ptr()], [buf.data_ptr() + offset * buf.element_size()],
                           ws.data_ptr(), ws_bytes, [st.cuda_stream], inputs_ready=ready)
        torch.cuda.synchronize()
        assert G.goldy_device_error(clear=True) == 0
        want = torch.full((offset + M * ldc + 64,), SENTINEL, dtype=TORCH[out])
        want[offset:offset + M * ldc].view(M, ldc)[:, :N] = exact
        assert torch.equal(buf.cpu(), want), (kind, split, out, M, N, K, ldc, offset, ready)


@pytest.mark.parametrize("kind", [0, 2, 3, 4, 5, PAIR])
@pytest.mark.parametrize("out", [F32, BF16])
def test_output_rows_at_any_alignment(cuda_ok, kind, out):
    # (M, N, ldc, offset): one row or column; whole and ragged chunks of 32 / 64
    # columns; odd row strides (every other bf16 row 2 bytes off); an aligned
    # stride from a base that is not
    for i, (M, N, ldc, offset) in enumerate([(1, 1, 1, 0), (33, 65, 65, 0), (129, 127, 127, 1), (200, 320, 320, 0),
                                             (200, 320, 320, 1), (31, 191, 193, 3), (300, 257, 264, 0),
                                             (97, 64, 64, 0)]):
        _check(kind, 1, out, M, N, 136, ldc, offset, 3000 + 10 * i)


@pytest.mark.parametrize("kind,split", [(0, 2), (2, 4), (4, 2), (PAIR, 2), (PAIR, 4)])
@pytest.mark.parametrize("out", [F32, BF16])
def test_split_k_output_rows_at_any_alignment(cuda_ok, kind, split, out):
    for i, (M, N, ldc, offset) in enumerate([(33, 65, 65, 0), (129, 159, 159, 1), (300, 320, 320, 0),
                                             (160, 257, 264, 2)]):
        _check(kind, split, out, M, N, 520, ldc, offset, 3100 + 10 * i)


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("N", [64, 127, 128, 129, 256, 257, 384, 385])
def test_pair_kernel_last_column_tile(cuda_ok, N, split):
    # a last column tile of at most 128 columns is computed with the narrow MMA
    _check(PAIR, split, F32, 300, N, 448, N, 0, 3200 + N)


def test_pair_kernel_batched_narrow_tiles(cuda_ok):
    # entries of 128 columns and of 256 + 128, several units per CTA pair
    for N in (128, 384):
        M, K, batch = 520, 192, 40
        a = torch.stack([wl.integer_matrix(M, K, 3300 + i) for i in range(batch)])
        b = torch.stack([wl.integer_matrix(K, N, 3400 + i) for i in range(batch)])
        dA, dB = a.cuda(), b.cuda()
        C = torch.full((batch, M, N), float("nan"), device="cuda")
        s = G.goldy_schedule_build([G.desc(M, N, K, F32, batch=batch)], [0], [G.variant_id(PAIR, 1, 4)], [0])
        torch.cuda.synchronize()
        st = torch.cuda.Stream()
        G.goldy_run(s, [dA.data_ptr()], [dB.data_ptr()], [C.data_ptr()], 0, 0, [st.cuda_stream])
        torch.cuda.synchronize()
        assert G.goldy_device_error(clear=True) == 0
        assert torch.equal(C, torch.bmm(dA.double(), dB.double()).float())
