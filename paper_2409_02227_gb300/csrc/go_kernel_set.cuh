// GO-Kernel over GEMMs of different tile shapes: one persistent launch for all
// the single-CTA kinds of a run.
//
// What it is for: a heterogeneous set plans a kernel kind per GEMM (tile
// shape, transposed or not, K split), and one launch per kind leaves most of
// the GPU idle most of the time: each launch has tens of short units, pays its
// own start (about 2 us to the first data) and its stores wait for the launch
// before.  Here the tile shape is a property of the GEMM, read per unit, so
// the run's units of every shape share one launch and are dealt out in equal
// shares (UnitShares).  Nine GEMMs of M = 18 .. 364 in five kinds ran as five
// launches of 4 to 12 us each.
//
// The arithmetic of a unit is that of go_gemm_kernel with the same tile shape
// and K split, so the bytes are those of the GEMM run alone.  Split-K partials
// go through the workspace, the last split to arrive sums them in split order.
//
// CTAS = 1, one CTA per SM: tensor memory holds two accumulators of 256 columns
// whatever the tile's width; the operand ring is cut into stages of the
// launch's widest tile (192 KB: 4 stages of 48 KB up to 8 of 24 KB or less).
// CTAS = 2, two per SM, for runs with inputs_ready and launches behind the first
// of a run: half the ring and half the tensor memory (two accumulators of 128
// columns, or one of 256 when a bf16 launch has tiles that wide; an fp32 launch
// with such tiles runs one CTA per SM), no staging buffers (tiles other than a CTA's last are
// stored from registers), so that the next run's CTAs load and multiply while
// this run's finish.  The units, sorted longest first, go to the CTAs back and
// forth (0 .. n-1, n-1 .. 0, ...), which balances the few units a CTA gets.
#pragma once

#include "go_kernel.cuh"

namespace goldy {

constexpr int kSetStages = 8;              // barriers for the most stages a launch may use
template <int CTAS>
constexpr int kSetRingBytes = 4 * 49152 / CTAS;

template <bool OUT_BF16, int MAXG, int CTAS>
__global__ void __launch_bounds__(192, CTAS) go_gemm_set_kernel(const __grid_constant__ LaunchParams<MAXG> p) {
  constexpr int ACC = 2;                             // accumulators at most (p.acc_stages of them in use)
  const int acc_stages = CTAS == 1 ? ACC : p.acc_stages;
  const uint32_t acc_cols = CTAS == 1 ? 256u : 256u / uint32_t(p.acc_stages);
  constexpr uint32_t X_BYTES = 128 * 64 * 2;         // MMA operand A: 128 rows x 64 K
  constexpr uint32_t TMEM_COLS = 512 / CTAS;
  constexpr uint32_t KMAJ_STEP = 32;                 // bytes per 16 K elements, K-major
  constexpr uint32_t MNMAJ_STEP = 2048;              // bytes per 16 K rows, N-major
  constexpr uint32_t MNMAJ_LBO = 64 * 128;           // bytes between 64-wide N chunks
  constexpr int STAGING_BYTES = CTAS == 1 ? 2 * 16384 : 0;
  constexpr int RING_BYTES = kSetRingBytes<CTAS>;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RING_BYTES + STAGING_BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + kSetStages;
  uint64_t* tfull = bars + 2 * kSetStages;
  uint64_t* tempty = bars + 2 * kSetStages + ACC;
  uint64_t* drain = bars + 2 * kSetStages + 2 * ACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* last_flag = reinterpret_cast<volatile int*>(tmem_slot + 2);
  UnitTable* utab = reinterpret_cast<UnitTable*>(tmem_slot + 4);   // MAXG entries, inside the 1 KB barrier area
  static_assert((2 * kSetStages + 2 * ACC + 1) * 8 + 16 + MAXG * int(sizeof(UnitTable)) <= 1024, "barrier area");
  const int n_gemms = p.n_gemms;
  const uint32_t stage_bytes = uint32_t(p.stage_bytes);
  const int stages = p.stages;

  const uint32_t tiles_base = ptx::smem_u32(smem);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  unsigned long long* const trace = p.trace;
  if (!p.late_trigger) ptx::griddep_launch_dependents();   // see go_gemm_kernel

  if (threadIdx.x == 0) {
    trace_stamp(trace, kTrStart);
    for (int g = 0; g < p.n_gemms; ++g) {
      ptx::prefetch_tensormap(&p.tmap_a[g]);
      ptx::prefetch_tensormap(&p.tmap_b[g]);
    }
    if (trace) {
      uint32_t sm;
      asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
      trace[blockIdx.x * kTracePerCta + kTrSm] = sm;
      trace[blockIdx.x * kTracePerCta + kTrGrid] = gridDim.x;
      trace[blockIdx.x * kTracePerCta + kTrCta] = blockIdx.x;
    }
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(ptx::smem_u32(&full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&empty[s]), 1);
    }
    for (int a = 0; a < ACC; ++a) {
      ptx::mbar_init(ptx::smem_u32(&tfull[a]), 1);
      ptx::mbar_init(ptx::smem_u32(&tempty[a]), 128);
    }
    ptx::mbar_init(ptx::smem_u32(drain), 1);
    *abort_flag = 0;
    *last_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(tmem_slot), TMEM_COLS);
    ptx::tmem_relinquish();
  } else if (warp == 2) {
    fill_unit_table(utab, p, int(blockIdx.x), lane);
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = ptx::uniform(*tmem_slot);
  const uint64_t wlim = p.wait_ns ? p.wait_ns : ptx::kWaitLimitNs;
  // a wait of a whole role (warp); whichever lane gives up first raises the error
  auto role_wait = [&](uint64_t* bar, uint32_t parity, int code) {
    const bool done = ptx::mbar_wait(ptx::smem_u32(bar), parity, abort_flag, wlim);
    if (!done) raise_error(p.err, abort_flag, code);
    return ptx::warp_all(done);
  };
  UnitWalk walk(utab, n_gemms, p.shares.on, p.total_units, int(blockIdx.x), int(gridDim.x));
  if (threadIdx.x == 0) trace_stamp(trace, kTrPreWait);
  // where each role waits for the previous grid: see go_gemm_kernel
  const bool early = p.early_loads != 0 && warp < 2;
  const bool epi_defer = p.early_loads != 0 && warp >= 2;
  if (!early && !epi_defer) ptx::griddep_wait();
  if (p.late_trigger) ptx::griddep_launch_dependents();
  if (threadIdx.x == 64 && !epi_defer) trace_stamp(trace, kTrSetup);

  // load and MMA roles as whole warps, one elected thread issuing: see
  // go_gemm_kernel
  if (warp == 0) {
    {
      // ------------------------------------------------------------ producer
      const bool leader = ptx::elect_one();
      int stage = 0;
      uint32_t phase = 0, issued = 0, last_phase = 0;
      bool ok = true, stalled = false;
      while (ok && !stalled && ptx::warp_all(walk.next())) {
        if (issued == 0 && lane == 0) trace_stamp(trace, kTrProducerGo);
        const UnitCoord c = walk.coord().uniform();
        const void* ta = &p.tmap_a[c.g];
        const void* tb = &p.tmap_b[c.g];
        const int mma_n = ptx::uniform(utab[c.g].mma_n);
        const bool swap = ptx::uniform(utab[c.g].swap) != 0;
        const uint32_t bytes = X_BYTES + uint32_t(mma_n) * 128u;
        const int m0 = c.tm * (swap ? mma_n : 128);
        const int n0 = c.tn * (swap ? 128 : mma_n);
        // 64-column boxes of B go to MMA operand A when transposed, else to B
        const int boxes = swap ? 2 : mma_n / 64;
        const uint32_t a_off = swap ? X_BYTES : 0u, b_off = swap ? 0u : X_BYTES;
        for (int kb = c.kb0; kb < c.kb1; ++kb) {
          // only a slot filled before is waited for (see go_gemm_kernel)
          if ((issued >> stage & 1) &&
              !role_wait(&empty[stage], phase ^ 1, kErrProducerWait)) {
            ok = false;
            break;
          }
          if (p.stall_test && blockIdx.x == 0 && issued == 0) {
            // test hook: the first stage is never filled (see go_gemm_kernel)
            const uint64_t t0 = ptx::global_timer();
            while (!*abort_flag && ptx::global_timer() - t0 < 4 * wlim) {
            }
            stalled = true;
            break;
          }
          const uint32_t fb = ptx::smem_u32(&full[stage]);
          const uint32_t base = tiles_base + uint32_t(stage) * stage_bytes;
          const int k0 = kb * 64;
          if (leader) {
            ptx::mbar_arrive_expect_tx(fb, bytes);
            ptx::tma_load_3d(base + a_off, ta, fb, k0, m0, c.b);
            for (int j = 0; j < boxes; ++j)
              ptx::tma_load_3d(base + b_off + uint32_t(j) * 8192u, tb, fb, n0 + 64 * j, k0, c.b);
          }
          __syncwarp();
          if (issued == 0 && lane == 0) trace_stamp(trace, kTrFirstLoad);
          issued |= 1u << stage;
          last_phase = (last_phase & ~(1u << stage)) | (phase << stage);
          if (++stage == stages) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
      if (!ok && leader) {
        // let every copy this thread started land before the CTA can exit
        for (int s = 0; s < stages; ++s)
          if (issued >> s & 1) ptx::mbar_wait(ptx::smem_u32(&full[s]), (last_phase >> s) & 1, nullptr);
      }
    }
  } else if (warp == 1) {
    {
      // ---------------------------------------------------------- MMA issuer
      const bool leader = ptx::elect_one();
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0, acc_used = 0;
      bool ok = true, any = false, first = true;
      while (ok && ptx::warp_all(walk.next())) {
        const UnitCoord c = walk.coord().uniform();
        const int mma_n = ptx::uniform(utab[c.g].mma_n);
        const bool swap = ptx::uniform(utab[c.g].swap) != 0;
        // untransposed: MMA-A = A tile (K-major), MMA-B = B tile (N-major);
        // transposed: MMA-A = B tile (N-major), MMA-B = A tile (K-major)
        const uint32_t idesc = ptx::make_idesc_bf16(128, mma_n, swap ? 1 : 0, swap ? 0 : 1);
        const uint32_t a_step = swap ? MNMAJ_STEP : KMAJ_STEP, b_step = swap ? KMAJ_STEP : MNMAJ_STEP;
        const uint32_t a_lbo = swap ? MNMAJ_LBO : 16u, b_lbo = swap ? 16u : MNMAJ_LBO;
        if ((acc_used >> acc & 1) &&
            !role_wait(&tempty[acc], acc_phase ^ 1, kErrMmaWait)) {
          ok = false;
          break;
        }
        acc_used |= 1u << acc;
        ptx::tc_fence_after();
        const uint32_t d_tmem = tmem_base + uint32_t(acc) * acc_cols;
        for (int kb = c.kb0; kb < c.kb1; ++kb) {
          if (!role_wait(&full[stage], phase, kErrMmaWait)) {
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          if (!any && lane == 0) trace_stamp(trace, kTrFirstFull);
          const uint32_t xs = tiles_base + uint32_t(stage) * stage_bytes;
          const uint32_t ys = xs + X_BYTES;
          if (leader) {
#pragma unroll
            for (uint32_t kk = 0; kk < 4; ++kk) {
              const uint64_t adesc = ptx::make_sdesc_sw128(xs + kk * a_step, a_lbo, 1024);
              const uint64_t bdesc = ptx::make_sdesc_sw128(ys + kk * b_step, b_lbo, 1024);
              ptx::mma_bf16(d_tmem, adesc, bdesc, idesc, (kb > c.kb0 || kk > 0) ? 1u : 0u);
            }
            ptx::mma_commit(ptx::smem_u32(&empty[stage]));   // frees the slot when these MMAs finish
          }
          __syncwarp();
          any = true;
          if (++stage == stages) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (!ok) break;
        if (leader) ptx::mma_commit(ptx::smem_u32(&tfull[acc]));   // accumulator complete
        __syncwarp();
        if (first && lane == 0) trace_stamp(trace, kTrFirstMmaDone);
        first = false;
        if (++acc == acc_stages) {
          acc = 0;
          acc_phase ^= 1;
        }
      }
      if (!ok && leader) {
        if (any) {
          ptx::mma_commit(ptx::smem_u32(drain));
          ptx::mbar_wait(ptx::smem_u32(drain), 0, nullptr);
        }
      }
    }
  } else {
    // -------------------------------------------------------------- epilogue
    const int q = warp & 3;                 // tensor-memory lane quarter of this warp
    const int r = q * 32 + lane;            // accumulator row handled by this thread
    const int et = threadIdx.x - 64;        // 0 .. 127
    int acc = 0;
    uint32_t acc_phase = 0;
    uint32_t stg = 0;                       // staging buffers used
    const uint32_t staging = tiles_base + RING_BYTES;
    bool waited = !epi_defer;               // past the wait for the previous grid
    auto wait_prev = [&]() {
      if (waited) return;
      ptx::griddep_wait();
      waited = true;
      if (et == 0) trace_stamp(trace, kTrSetup);
    };
    bool first_unit = true;
    for (; walk.next(); first_unit = false) {
      const UnitCoord c = walk.coord();
      const GemmWork w = p.g[c.g];          // read while the accumulator is computed
      const CView cv = c_view<OUT_BF16>(w, c.b);
      // (a little longer than the other roles wait: what they wait for is what
      // this wait hangs on, so the role that is stuck reports)
      bool ok = ptx::mbar_wait(ptx::smem_u32(&tfull[acc]), acc_phase, abort_flag, wlim + wlim / 8);
      ok = ptx::named_bar_and(1, 128, ok);
      if (!ok) {
        if (et == 0) raise_error(p.err, abort_flag, kErrEpilogueWait);
        break;
      }
      ptx::tc_fence_after();
      if (first_unit && et == 0) trace_stamp(trace, kTrFirstAcc);
      const bool swap = w.swap != 0;
      const int m0 = c.tm * (swap ? w.mma_n : 128);
      const int n0 = c.tn * (swap ? 128 : w.mma_n);
      const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16) + uint32_t(acc) * acc_cols;
      // accumulator columns that lie in C (columns of C, or its rows when
      // transposed), and whether any of this warp's accumulator rows do
      const int ncols = swap ? min(w.mma_n, w.m - m0) : min(w.mma_n, w.n - n0);
      const bool live = swap ? n0 + 32 * q < w.n : m0 + 32 * q < w.m;
      // see go_gemm_kernel; a launch of two CTAs per SM has fp32 tiles of at most
      // 128 columns (the host sees to it), which its half ring holds
      static_assert(128 * (OUT_BF16 ? 256 * 2 : CTAS == 1 ? 256 * 4 : 128 * 4) <= RING_BYTES, "the ring holds a tile");
      const bool wide = !swap && w.split == 1 && walk.last();
      if (wide) {
        stage_tile_wide<OUT_BF16>(cv, tiles_base, taddr, et, q, m0, ncols);
        wait_prev();
        send_tile_wide<OUT_BF16>(cv, &p.tmap_c[c.g], w.c_tma != 0, tiles_base, et, q, m0, n0, ncols, c.b);
      } else if (CTAS == 1 && w.split == 1 && !swap) {
        wait_prev();
        store_tile<256, OUT_BF16>(cv, &p.tmap_c[c.g], w.c_tma != 0, staging, stg, taddr, et, q, m0, n0, ncols,
                                       c.b);
      } else {
        wait_prev();
        const int nc = live ? ncols : 0;
        const int tile_f4 = 32 * w.mma_n;      // float4 of a 128-row partial tile
        float4* tile_parts = reinterpret_cast<float4*>(w.ws_part) + size_t(c.tile) * w.split * tile_f4 + r;
        bool mine = true;                      // this CTA stores the tile
        if (w.split > 1) {
          // publish the partial (layout [column / 4][row]) and count it in
          float4* part = tile_parts + size_t(c.s) * tile_f4;
#pragma unroll 1
          for (int c0 = 0; c0 < nc; c0 += 32) {
            uint32_t raw[32];
            __syncwarp();
            ptx::tmem_ld_32x32b_x32(taddr + c0, raw);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j4 = 0; j4 < 8; ++j4)
              part[((c0 / 4) + j4) * 128] =
                  make_float4(__uint_as_float(raw[4 * j4]), __uint_as_float(raw[4 * j4 + 1]),
                              __uint_as_float(raw[4 * j4 + 2]), __uint_as_float(raw[4 * j4 + 3]));
          }
          __threadfence();
          ptx::named_bar_sync(1, 128);
          if (et == 0) {
            if (first_unit) trace_stamp(trace, kTrPartials);
            const uint32_t old = atomicAdd(&w.ws_cnt[c.tile], 1u);
            *last_flag = (old == uint32_t(w.split - 1)) ? 1 : 0;
            if (first_unit) trace_stamp(trace, kTrArrived);
          }
          ptx::named_bar_sync(1, 128);
          mine = *last_flag != 0;
          if (mine) __threadfence();
        }
        if (CTAS == 1 && mine && w.split > 1 && !swap && w.c_tma == 0) {
          sum_and_store_tile<OUT_BF16>(cv, tile_parts, tile_f4, w.split, c.s, staging, stg, taddr, et, q, m0, n0,
                                       ncols);
        } else if (mine) {
#pragma unroll 1
          for (int c0 = 0; c0 < nc; c0 += 32) {
            float v[32];
            if (w.split == 1) {
              uint32_t raw[32];
              __syncwarp();
              ptx::tmem_ld_32x32b_x32(taddr + c0, raw);
              ptx::tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(raw[j]);
            } else {
              sum_partials(tile_parts, tile_f4, w.split, c.s, taddr, c0, v);
            }
            if (swap)
              store_chunk<true, OUT_BF16>(cv, m0, n0, r, c0, v);
            else
              store_chunk<false, OUT_BF16>(cv, m0, n0, r, c0, v);
          }
        }
        if (w.split > 1 && mine && et == 0) w.ws_cnt[c.tile] = 0u;   // leave the counter zeroed for the next run
      }
      if (first_unit && et == 0) trace_stamp(trace, kTrFirstStore);
      ptx::tc_fence_before();
      ptx::mbar_arrive(ptx::smem_u32(&tempty[acc]));
      if (++acc == acc_stages) {
        acc = 0;
        acc_phase ^= 1;
      }
    }
    // tensor stores must have read the staging buffers before the CTA leaves
    // (their writes to C complete with the grid)
    if (et == 0) ptx::bulk_wait_group_read<0>();
  }

  __syncthreads();
  if (threadIdx.x == 0) {
    trace_stamp(trace, kTrEnd);
    if (trace) {
      int n = 0;
      for (UnitWalk all(utab, n_gemms, p.shares.on, p.total_units, int(blockIdx.x), int(gridDim.x)); all.next();) ++n;
      trace[blockIdx.x * kTracePerCta + kTrUnits] = n;
    }
  }
  if (warp == 1) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

}  // namespace goldy
