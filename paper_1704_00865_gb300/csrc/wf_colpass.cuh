// wf_colpass.cuh -- the column pass of the messenger iteration (Huffenberger
// 2017, Sec. 2 and Appendix A): the forward column DFT that completes the 2D
// transform of the data-side messenger, the 2D-Fourier updates (the 1/f part
// and the signal prior are both diagonal there), and the inverse column DFT.
// One CTA owns W adjacent complex columns.
// PREC selects the radix-16 stages: FP32 (0) or the tensor-core DFT-as-GEMM
// stages of wf_device.cuh (1: split TF32, 2: TF32).
// Bound by the chain of one CTA (load, transform, update, transform, store): 4.5
// us at 1024^2, 15.0 at 2048^2, 60 at 4096^2 (3.4 TB/s of 12 bytes per pixel);
// 6.4, 17.4 and 95.6 with twiddles read from the table exp(-2 pi i k / L), two
// barriers an exchange and, at 4096^2, one CTA per SM.
#pragma once

#include "wf_cols_common.cuh"

namespace wf {


// Column pass geometry: W columns per CTA, TPC = L/E threads per column.  W is a
// whole number of column tiles, half a tile at 4096.

// Values per thread of the two shapes the autotuner chooses between (one
// where both coincide): 16 measured fastest for columns of 1024 and more,
// 8 for 512; 3 * 2^k columns take 12 or 24.
template <int L>
struct ColPassE {
  static constexpr int v0 = (L % 3 == 0) ? ((L >= 1536) ? 24 : 12) : ((L >= 512) ? 16 : 8);
  static constexpr int v1 = (L % 3 == 0) ? 24 : (L > 2048) ? v0 : ((L >= 512) ? 8 : (L >= 128 ? 16 : v0));
};

template <int L, int MODE, int EV, int PREC = 0>
struct ColPassCfg {
  static constexpr bool T0 = (MODE == COL_PASS_2DF);
  static constexpr bool SRC = (MODE == COL_PASS_MERGE_SRC);
  static constexpr bool EXTRA = T0 || SRC;  // a third field
  static constexpr int E = EV;
  static constexpr int TPC = L / E;
  static constexpr int W_MIN = (TPC >= 32) ? 1 : 32 / TPC;  // at least one warp
  static constexpr int W_FIT = L >= 4096 ? 2 : WF_TW;
  static constexpr int W_WANT = (W_MIN > W_FIT) ? ((W_MIN + WF_TW - 1) / WF_TW) * WF_TW : W_FIT;
  static constexpr int W_CAP = 1024 / TPC;  // at most 1024 threads per CTA
  static constexpr int W = (W_WANT <= W_CAP) ? W_WANT
                           : (W_CAP >= WF_TW ? (W_CAP / WF_TW) * WF_TW : (W_CAP >= 2 ? 2 : 1));
  static constexpr bool TILED = (W % WF_TW == 0);
  static constexpr int THREADS = W * TPC;
  static constexpr int SP = SPad<L>::size;
  static constexpr int WANT = (W >= 32) ? 1 : (16 / W) % 16;
  static constexpr int STRIDE = SP + ((WANT - SP % 16) + 16) % 16;
  // STAGED (columns up to 2048): the tiles arrive in shared memory by TMA, (C,
  // P1f) and the twiddles while the previous kernel drains; from 1536 on the
  // messenger lands in the transform's own buffer.  At 4096 (70 KB of
  // transform buffers for two columns) nothing is staged and the registers
  // are held to 64 a thread, so two CTAs of an SM cover one another's loads:
  // 60 us a pass against 96 us with staged tiles and one CTA of 198 KB.
  static constexpr bool STAGED = L <= 2048;
  static constexpr bool LAND = L >= 1536;
  static constexpr size_t al(size_t n) { return (n + 15) / 16 * 16; }
  static constexpr size_t tile = STAGED ? (size_t)L * W * 8 : 0;
  static constexpr size_t fft_off = 16;
  // PP: the messenger's tile, once read, is the second exchange buffer
  static constexpr bool PP = STAGED && !LAND && PREC == 0;
  static constexpr size_t fft_bytes = al((size_t)W * STRIDE * 8);
  static constexpr size_t y_off = LAND ? fft_off : fft_off + fft_bytes;
  static constexpr size_t eig_off = LAND ? fft_off + fft_bytes : y_off + (PP ? fft_bytes : tile);
  static constexpr size_t t0_off = eig_off + tile;
  static constexpr size_t tw_off = t0_off + (EXTRA ? tile : 0);
  // the twiddle table too where it costs no CTA per SM
  // (the stage table; the tensor-core stages read exp(-2 pi i k / L))
  static constexpr uint32_t tw_bytes = (PREC ? L : StageTable<L, EV>::size) * 8;
  static constexpr bool TWS = STAGED && tw_off + tw_bytes <= kMaxDynSmem &&
                              kSmSmem / (tw_off + tw_bytes + kCtaSmem) == kSmSmem / (tw_off + kCtaSmem);
  static constexpr size_t bytes = tw_off + (TWS ? tw_bytes : 0);
  static constexpr int min_ctas = STAGED ? 1 : 1024 / THREADS;
  static_assert(bytes <= kMaxDynSmem, "column pass staging exceeds shared memory");
  // position of (ky, column c of the CTA) in the staged tiles
  static __device__ __forceinline__ int sidx(int ky, int c) {
    if constexpr (TILED) return (c / WF_TW) * L * WF_TW + ky * WF_TW + (c % WF_TW);
    else return ky * W + c;
  }
};

// Extra shared memory of the tcgen05 stages (PREC 3, 4) after the column
// pass's own: 1 KB of alignment slack, the A tiles (16 KB per 128 threads,
// twice for the split), the four 4 KB DFT matrices, the mbarrier.
template <int L, int MODE, int EV, int PREC>
struct Tc5Smem {
  static constexpr int tiles = ColPassCfg<L, MODE, EV, PREC>::THREADS / 128;
  static constexpr size_t bytes = PREC >= 3 ? 1024 + (size_t)tiles * 16384 * (PREC == 3 ? 2 : 1) + 16384 + 16 : 0;
};
template <int L, int MODE, int EV, int PREC>
__device__ __forceinline__ uint64_t* tc5_mbar(unsigned char* smem) {
  return reinterpret_cast<uint64_t*>(smem + ColPassCfg<L, MODE, EV, PREC>::bytes + Tc5Smem<L, MODE, EV, PREC>::bytes - 16);
}

// The column pass (Sec. 2 / Appendix A: the 2D-Fourier updates between the
// forward and inverse column DFTs).  d_2DF goes straight from the registers of
// the last stage to global memory (a warp covers 8 rows of a tile, 256
// contiguous bytes), at 4096 the messenger and the tables come the same way.
// ONE: compiled for one CTA per SM (the plain sweep's unstaged columns on a grid
// that gives an SM no second one).
template <int L, int MODE, int EV, int PREC = 0, bool ONE = false>
__global__ void __launch_bounds__(ColPassCfg<L, MODE, EV, PREC>::THREADS,
                                  PREC || ONE ? 1 : ColPassCfg<L, MODE, EV, PREC>::min_ctas)
col_pass_kernel(ColArgs a) {
  using Cfg = ColPassCfg<L, MODE, EV, PREC>;
  constexpr int E = Cfg::E, TPC = Cfg::TPC, W = Cfg::W;
  constexpr bool STAGED = Cfg::STAGED, MERGED = (MODE == COL_PASS_MERGE || MODE == COL_PASS_MERGE_SRC);
  static_assert(!STAGED || Cfg::TILED, "whole tiles are staged");
  static_assert(!Cfg::PP || Cfg::fft_bytes >= Cfg::tile, "the second exchange buffer holds the tile");
  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
  float2* s_fft = reinterpret_cast<float2*>(smem + Cfg::fft_off);
  float2* s_y = reinterpret_cast<float2*>(smem + Cfg::y_off);
  float2* s_eig = reinterpret_cast<float2*>(smem + Cfg::eig_off);
  float2* s_t0 = reinterpret_cast<float2*>(smem + Cfg::t0_off);  // plain sweep: t_2DF; source: j^
  float2* s_tw = reinterpret_cast<float2*>(smem + Cfg::tw_off);

  const int c = threadIdx.x % W;
  const int t = threadIdx.x / W;
  const int col0 = blockIdx.x * W;
  const int col = col0 + c;
  float2* sb = s_fft + c * Cfg::STRIDE;
  float2* sb2 = s_y + c * Cfg::STRIDE;  // PP
  const size_t at0 = tidx(0, col, a.ny);  // (ky, this column) in the tiled fields: at0 + 4 ky
  const size_t tile0 = tidx(0, col0, a.ny);
  const bool packed = (blockIdx.x == 0 && c == 0);

  // before the previous kernel has finished: what is fixed during a solve,
  // (C, P1f), the twiddle table and the source, on barrier 1
  if constexpr (STAGED) {
    if (threadIdx.x == 0) {
      mbar_init(&bar[0], 1);
      mbar_init(&bar[1], 1);
      mbar_fence_init();
      mbar_expect_tx(&bar[1], (uint32_t)(Cfg::tile * (Cfg::SRC ? 2 : 1) + (Cfg::TWS ? Cfg::tw_bytes : 0)));
      bulk_g2s(s_eig, a.eig + tile0, (uint32_t)Cfg::tile, &bar[1]);
      if constexpr (Cfg::TWS) bulk_g2s(s_tw, PREC ? a.twy : a.tws, Cfg::tw_bytes, &bar[1]);
      if constexpr (Cfg::SRC) bulk_g2s(s_t0, a.src + tile0, (uint32_t)Cfg::tile, &bar[1]);
    }
  } else {
    // the tables are read in mid-kernel: into L2 until then
    if (threadIdx.x == 0 && col0 % WF_TW == 0) {
      prefetch_l2_range(a.eig + tile0, (size_t)L * WF_TW * 8);
      if constexpr (Cfg::SRC) prefetch_l2_range(a.src + tile0, (size_t)L * WF_TW * 8);
    }
  }
  // (C, P1f) at kx = nx/2 for the packed column: CTA 0 is the last to finish
  // of a grid that fits on the device at once, so it reads them early too
  float2 eq[STAGED ? E : 1];
  if (STAGED && packed) {
#pragma unroll
    for (int m = 0; m < E; ++m) eq[STAGED ? m : 0] = __ldg(&a.eig_nyq[t + m * TPC]);
  }
  // the row pass's CTAs may start beside this one: their prologue (the pixel
  // table) then costs nothing (when this came in: 256^2 sweep 6.5 -> 5.5 us,
  // 2048^2 40.8 -> 39.7)
  pdl_trigger();
  // Maps above L2: the CTA that will run on this SM one wave later (pf CTAs
  // on) finds its tiles in L2 -- (C, P1f) now, the messenger once the
  // previous kernel is done.  Half-tile CTAs hint the whole tile from the
  // first CTA of the tile.
  const int nb = blockIdx.x + a.pf;
  const bool pf = a.pf > 0 && nb < (int)gridDim.x && threadIdx.x == 0 && (Cfg::TILED || (nb * W) % WF_TW == 0);
  constexpr size_t pf_bytes = (size_t)L * (Cfg::TILED ? W : WF_TW) * 8;
  if (pf) prefetch_l2_range(a.eig + tidx(0, nb * W, a.ny), pf_bytes);
  pdl_wait();
  const bool done = a.check_done && a.st->done;  // uniform: set only between launches
  float2 v[E];
  if constexpr (STAGED) {
    if (threadIdx.x == 0 && !done) {
      mbar_expect_tx(&bar[0], (uint32_t)Cfg::tile * (Cfg::T0 ? 2 : 1));
      bulk_g2s(s_y, a.f_y + tile0, (uint32_t)Cfg::tile, &bar[0]);
      if constexpr (Cfg::T0) bulk_g2s(s_t0, a.f_t0 + tile0, (uint32_t)Cfg::tile, &bar[0]);
    }
  } else if (!done) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = a.f_y[at0 + (size_t)(t + m * TPC) * WF_TW];
  }
  if (pf) {
    prefetch_l2_range(a.f_y + tidx(0, nb * W, a.ny), pf_bytes);
    if constexpr (Cfg::SRC) prefetch_l2_range(a.src + tidx(0, nb * W, a.ny), pf_bytes);
  }
  // link covariances of this lambda level (written by the controller)
  const float Tl = a.has_rf ? a.st->Tf[1] : a.st->Tf[2];  // link to the RF/PX messenger
  const float off0 = (float)a.st->off[0];
  const float T0 = Cfg::T0 ? a.st->Tf[0] : 0.f;
  const float T0s = Cfg::T0 ? a.st->T0s[a.parity] : 0.f;

  if constexpr (STAGED) {
    __syncthreads();  // the barriers are initialised
    // the copies land before the block exits on every path
    bool ok = mbar_wait(&bar[1], 0, WF_WAIT_TRIES);
    if (!done) ok = mbar_wait(&bar[0], 0, WF_WAIT_TRIES) && ok;
    const bool bad = __syncthreads_or(!ok);
    if (bad && threadIdx.x == 0) atomicOr(&a.st->err, WF_ERR_TIMEOUT);
    if (bad || done) return;
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = s_y[Cfg::sidx(t + m * TPC, c)];
    if constexpr (Cfg::LAND) __syncthreads();  // the messenger is read
  } else {
    if (done) return;
  }
  // radix-16 stages on tcgen05: operand tiles, DFT matrices, TMEM (after the
  // early return, so every path that allocates also releases)
  if constexpr (PREC >= 3)
    tc5_setup<L, PREC>(smem + Cfg::bytes, tc5_mbar<L, MODE, EV, PREC>(smem), Cfg::TWS ? s_tw : a.twy, 1);

  if constexpr (PREC) fft_block<L, E, false, false, Cfg::TWS, PREC>(v, sb, t, Cfg::TWS ? s_tw : a.twy, 1);
  else if constexpr (Cfg::PP) fft_pingpong<L, E, false, false, Cfg::TWS>(v, sb, sb2, t, Cfg::TWS ? s_tw : a.tws);
  else fft_staged<L, E, false, false, Cfg::TWS>(v, sb, t, Cfg::TWS ? s_tw : a.tws);

  // partner values Z[-k] for the packed column 0, read below from shared
  // memory (CTA 0 only; uniform).  Unstaged, t_2DF's partners too, since the
  // update overwrites the field: column 1's buffer is free for them (held in
  // registers they spilled 344 bytes a thread: 22.3 us a sweep at 4096 x 32)
  constexpr bool T0_DIRECT = Cfg::T0 && !STAGED;
  static_assert(!T0_DIRECT || W > 1, "a second buffer for the partners of t_2DF");
  if (blockIdx.x == 0) {
    if constexpr (!Cfg::PP) __syncthreads();
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + m * TPC;
      if constexpr (T0_DIRECT) sb[spad(k)] = c == 0 ? v[m] : a.f_t0[tile0 + (size_t)k * WF_TW];
      else sb[spad(k)] = v[m];
    }
    __syncthreads();
  }

  // value ky of this column of the third field (t_2DF or the source)
  auto third = [&](int k) -> float2 {
    if constexpr (STAGED) return s_t0[Cfg::sidx(k, c)];
    else if constexpr (Cfg::SRC) return __ldg(&a.src[at0 + (size_t)k * WF_TW]);
    else return a.f_t0[at0 + (size_t)k * WF_TW];
  };
  auto eig_of = [&](int k) -> float2 {
    return STAGED ? s_eig[Cfg::sidx(k, c)] : __ldg(&a.eig[at0 + (size_t)k * WF_TW]);
  };
  if (blockIdx.x != 0) {
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + m * TPC;
      const float2 e = eig_of(k);
      if constexpr (MERGED) {
        const float2 jv = Cfg::SRC ? third(k) : make_float2(0.f, 0.f);
        v[m] = merged_mode<Cfg::SRC>(v[m], v[m], e, e, off0, Tl, false, jv, jv);
      } else {
        float2 t0n;
        v[m] = mode_2df(v[m], third(k), e.x, e.y, off0, Tl, T0, T0s, t0n);
        a.f_t0[at0 + (size_t)k * WF_TW] = t0n;
      }
    }
  } else {
    // the CTA of the packed column
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + m * TPC;
      const float2 e = eig_of(k);
      // (C, P1f) at kx = nx/2 for the packed column
      const float2 egn = packed ? (STAGED ? eq[STAGED ? m : 0] : __ldg(&a.eig_nyq[k])) : e;
      const float2 zp = sb[spad(neg_mod<L>(k))];
      const float2 vp = make_float2(packed ? zp.x : v[m].x, packed ? zp.y : v[m].y);
      if constexpr (MERGED) {
        constexpr bool SRC = Cfg::SRC;
        const float2 jv = SRC ? third(k) : make_float2(0.f, 0.f);
        const float2 jn = SRC ? third(neg_mod<L>(k)) : jv;
        const float2 jp = make_float2(packed ? jn.x : jv.x, packed ? jn.y : jv.y);
        v[m] = merged_pair<SRC>(v[m], vp, e, egn, off0, Tl, jv, jp);
      } else {
        const float2 t0o = third(k);
        const float2 t0p = STAGED ? third(neg_mod<L>(k)) : s_fft[Cfg::STRIDE + spad(neg_mod<L>(k))];
        // (the pair is formed by every lane and kept by the packed column's)
        float2 yA, yB, tA, tB, tnA, tnB;
        unpack_pair(v[m], vp, yA, yB);
        unpack_pair(t0o, t0p, tA, tB);
        const float2 dB = mode_2df(yB, tB, egn.x, egn.y, off0, Tl, T0, T0s, tnB);
        yA = make_float2(packed ? yA.x : v[m].x, packed ? yA.y : v[m].y);
        tA = make_float2(packed ? tA.x : t0o.x, packed ? tA.y : t0o.y);
        const float2 dA = mode_2df(yA, tA, e.x, e.y, off0, Tl, T0, T0s, tnA);
        const float2 dp = repack_pair(dA, dB), tq = repack_pair(tnA, tnB);
        const float2 d0 = make_float2(packed ? dp.x : dA.x, packed ? dp.y : dA.y);
        const float2 t0n = make_float2(packed ? tq.x : tnA.x, packed ? tq.y : tnA.y);
        v[m] = d0;
        a.f_t0[at0 + (size_t)k * WF_TW] = t0n;
      }
    }
  }
  if constexpr (Cfg::T0) {
    // publish the T_0 that the new t_2DF was made with (implicit s)
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->T0s[a.parity ^ 1] = T0;
  }
  if (blockIdx.x == 0) {
    if constexpr (Cfg::PP) {  // its partners are still being read: the other buffer
      float2* x = sb;
      sb = sb2;
      sb2 = x;
    } else {
      __syncthreads();  // the partners are read
    }
  }
  if constexpr (PREC) fft_block<L, E, true, false, Cfg::TWS, PREC>(v, sb, t, Cfg::TWS ? s_tw : a.twy, 1);
  else if constexpr (Cfg::PP) fft_pingpong<L, E, true, false, Cfg::TWS>(v, sb, sb2, t, Cfg::TWS ? s_tw : a.tws);
  else fft_staged<L, E, true, false, Cfg::TWS>(v, sb, t, Cfg::TWS ? s_tw : a.tws);
  if constexpr (PREC >= 3) {
    tc5_teardown();
    if (threadIdx.x == 0 && !tc5_ctx().ok) atomicOr(&a.st->err, WF_ERR_TIMEOUT);
  }
  const float sc = 1.0f / (float)L;
#pragma unroll
  for (int m = 0; m < E; ++m) a.f_x[at0 + (size_t)(t + m * TPC) * WF_TW] = cscale(v[m], sc);
}

template <int L, int MODE, int EV, int PREC, bool ONE>
static int launch_col_pass_one(const ColArgs& a, cudaStream_t s) {
  using Cfg = ColPassCfg<L, MODE, EV, PREC>;
  constexpr size_t kBytes = Cfg::bytes + Tc5Smem<L, MODE, EV, PREC>::bytes;
  static_assert(kBytes <= kMaxDynSmem, "column pass staging exceeds shared memory");
  static_assert(PREC < 3 || Cfg::THREADS % 128 == 0, "tcgen05 tiles are 128 threads");
  constexpr auto kernel = col_pass_kernel<L, MODE, EV, PREC, ONE>;
  static DeviceOnce once;
  int dist = 0;  // CTAs one wave ahead
  const cudaError_t cfg_err = once.run(
      [](int* ahead) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(kBytes > kSpreadSmem ? kBytes : kSpreadSmem));
        if (e == cudaSuccess) *ahead = resident_ctas(kernel, Cfg::THREADS, kBytes);
        return e;
      },
      &dist);
  if (cfg_err != cudaSuccess) return (int)cfg_err;
  const dim3 grid(a.nx / 2 / Cfg::W), block(Cfg::THREADS);
  ColArgs b = a;
  b.pf = a.prefetch ? dist : 0;
  return launch_pdl(kernel, grid, block, spread_cols_smem(grid.x, kBytes, a.sms, a.row_ctas), s, b);
}

template <int L, int MODE, int EV, int PREC = 0>
static int launch_col_pass_e(const ColArgs& a, cudaStream_t s) {
  using Cfg = ColPassCfg<L, MODE, EV, PREC>;
  const int ncols = a.nx / 2;
  if (ncols % Cfg::W != 0) return (int)cudaErrorInvalidValue;
  // t_2DF, (C, P1f) and the values of an unstaged column do not fit in the 64
  // registers that two CTAs per SM leave (56 bytes spilled, the loads in
  // several batches): with no more CTAs than SMs there is nothing to trade
  if constexpr (Cfg::T0 && !Cfg::STAGED)
    if (ncols / Cfg::W <= kSms) return launch_col_pass_one<L, MODE, EV, PREC, true>(a, s);
  return launch_col_pass_one<L, MODE, EV, PREC, false>(a, s);
}

}  // namespace wf
