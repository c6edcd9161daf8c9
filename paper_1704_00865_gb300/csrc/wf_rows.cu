// wf_rows.cu -- the row pass of the messenger iteration and the row steps of
// the residual (Huffenberger 2017, Sec. 2).
//
// One CTA owns ROWS map rows; each row is a real length-nx signal handled by
// TPF = (nx/2)/E threads through a complex length-nx/2 Stockham FFT in
// shared memory.  The pixel-space messenger update (eq. 2mess_t1 analogue:
// white noise and mask, diagonal in pixels) sits between the inverse and the
// forward row transform, and the stripe-basis updates (eqs. 2mess_d0 and
// 2mess_t0 analogues: stripe noise, diagonal in the row-wise DFT) follow the
// forward transform, so a row is read and written once per iteration.
#include "wf_device.cuh"
#include "wf_internal.h"
#include "wf_rows_common.cuh"

namespace wf {

template <int M>
struct RowCfg {
  static constexpr int E = row_kernel_e(M);
  static constexpr int TPF = M / E;
  // one row per CTA, or as many as a warp holds: a 512 x 384 map gives 256 CTAs
  // (with 256 threads each it gave 32 and the residual's row steps took 27
  // and 15 us there)
  static constexpr int ROWS = TPF >= 32 ? 1 : 32 / TPF;
  static constexpr int THREADS = ROWS * TPF;
};

// deterministic block sum of one double per thread (fixed tree)
template <int THREADS>
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  constexpr int NW = (THREADS + 31) / 32;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < NW; ++i) s += red[i];
  }
  return s;
}

template <int M, int MODE>
__global__ void __launch_bounds__(RowCfg<M>::THREADS)
row_kernel(RowArgs a) {
  using Cfg = RowCfg<M>;
  constexpr int E = Cfg::E, TPF = Cfg::TPF, ROWS = Cfg::ROWS;
  __shared__ float2 sbuf[ROWS][SPad<M>::size];
  __shared__ double red[(Cfg::THREADS + 31) / 32];

  const int g = threadIdx.x / TPF;
  const int t = threadIdx.x - g * TPF;
  const int y = blockIdx.x * ROWS + g;
  const bool valid = y < a.ny;
  const size_t row0 = (size_t)(valid ? y : 0) * M;
  float2* sb = sbuf[g];
  pdl_trigger();
  // the pixel table, fixed during a solve, while the previous kernel drains
  constexpr bool PX = (MODE == ROW_RESID_B || MODE == ROW_RESID_D);
  float4 px[PX ? E : 1];
  if constexpr (PX) {
#pragma unroll
    for (int m = 0; m < E; ++m) px[m] = valid ? __ldg(&a.dn[row0 + t + m * TPF]) : make_float4(0.f, -1.f, 0.f, -1.f);
  }
  pdl_wait();

  // uniform: both flags are set only between launches
  if ((a.check_done && a.st->done) || (a.skip_ok && a.st->skip_resid)) return;

  float2 v[E];

  if constexpr (MODE == ROW_RESID_B) {
    // g = S^-1 s and s arrive in RF; go to pixels.
    float2 w[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
      v[m] = valid ? a.r_g[row0 + t + m * TPF] : make_float2(0.f, 0.f);
      w[m] = valid ? a.r_q[row0 + t + m * TPF] : make_float2(0.f, 0.f);
    }
    c2r_pre<M, E>(v, sb, t, a.twx);
    fft_staged<M, E, true>(v, sb, t, a.twk);
    c2r_pre<M, E>(w, sb, t, a.twx);
    fft_staged<M, E, true>(w, sb, t, a.twk);
    const float vshift = (float)a.st->var_shift;
    double gm2 = 0.0, g2 = 0.0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const float4 q = px[m];
      const float2 jm = (valid && a.src_px != nullptr) ? a.src_px[row0 + t + m * TPF] : make_float2(0.f, 0.f);
      float gp[2], qp[2], go[2];
      const float gv[2] = {v[m].x, v[m].y}, sv[2] = {w[m].x, w[m].y};
      const float dv[2] = {q.x, q.z}, nv[2] = {q.y, q.w}, jv[2] = {jm.x, jm.y};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double gd = (double)gv[h];
        const bool masked = nv[h] < 0.f;  // the residual there is S^-1 s (minus a source)
        const double rm = masked ? gd - (double)jv[h] : 0.0;
        if (valid) {
          g2 += gd * gd;
          gm2 += rm * rm;
        }
        // N_PX g' + s - d with the full pixel variance
        const float qu = fmaf(nv[h] + vshift, gv[h], sv[h] - dv[h]);
        gp[h] = masked ? 0.f : gv[h];
        qp[h] = masked ? 0.f : qu;
        go[h] = masked ? gv[h] : 0.f;
      }
      if (valid && a.gm_out != nullptr) a.gm_out[row0 + t + m * TPF] = make_float2(go[0], go[1]);
      v[m] = make_float2(gp[0], gp[1]);
      w[m] = make_float2(qp[0], qp[1]);
    }
    fft_staged<M, E, false>(v, sb, t, a.twk);
    r2c_post<M, E>(v, sb, t, a.twx);
    fft_staged<M, E, false>(w, sb, t, a.twk);
    r2c_post<M, E>(w, sb, t, a.twx);
    if (valid) {
      const float a2y = (a.a2 != nullptr) ? a.a2[y] : 1.f;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int k = t + m * TPF;
        float2 q = w[m];
        if (a.has_rf) {  // + N_RF g' with the given stripe eigenvalues
          if (k == 0) {
            q.x = fmaf(a2y * a.pst[0], v[m].x, q.x);
            q.y = fmaf(a2y * a.pst[M], v[m].y, q.y);
          } else {
            const float n1 = a2y * a.pst[k];
            q = make_float2(fmaf(n1, v[m].x, q.x), fmaf(n1, v[m].y, q.y));
          }
        }
        a.r_g[row0 + k] = v[m];
        a.r_q[row0 + k] = q;
      }
    }
    double s0 = block_sum<Cfg::THREADS>(gm2, red);
    double s1 = block_sum<Cfg::THREADS>(g2, red);
    if (threadIdx.x == 0) {
      a.part0[blockIdx.x] = s0;
      a.part1[blockIdx.x] = s1;
    }
  } else if constexpr (MODE == ROW_RESID_D) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = valid ? a.r_q[row0 + t + m * TPF] : make_float2(0.f, 0.f);
    c2r_pre<M, E>(v, sb, t, a.twx);
    fft_staged<M, E, true>(v, sb, t, a.twk);
    double r2 = 0.0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const float4 q = px[m];
      if (valid) {
        const double r0 = q.y >= 0.f ? (double)v[m].x : 0.0, r1 = q.w >= 0.f ? (double)v[m].y : 0.0;
        r2 += r0 * r0;
        r2 += r1 * r1;
        // optional map of Delta d on unmasked pixels (defect correction)
        if (a.out_px != nullptr)
          a.out_px[row0 + t + m * TPF] = make_float2(q.y >= 0.f ? v[m].x : 0.f, q.w >= 0.f ? v[m].y : 0.f);
      }
    }
    double s0 = block_sum<Cfg::THREADS>(r2, red);
    if (threadIdx.x == 0) a.part0[blockIdx.x] = s0;
  } else if constexpr (MODE == ROW_C2R) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = valid ? a.in_rf[row0 + t + m * TPF] : make_float2(0.f, 0.f);
    c2r_pre<M, E>(v, sb, t, a.twx);
    fft_staged<M, E, true>(v, sb, t, a.twk);
    if (valid) {
#pragma unroll
      for (int m = 0; m < E; ++m) a.out_px[row0 + t + m * TPF] = v[m];
    }
  } else if constexpr (MODE == ROW_R2C) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = valid ? a.in_px[row0 + t + m * TPF] : make_float2(0.f, 0.f);
    fft_staged<M, E, false>(v, sb, t, a.twk);
    r2c_post<M, E>(v, sb, t, a.twx);
    if (valid) {
#pragma unroll
      for (int m = 0; m < E; ++m) a.out_rf[row0 + t + m * TPF] = v[m];
    }
  }
}


// Row pass geometry: each row is one real length-2M transform done by TPF
// threads with E values each -- a single warp per row up to M = 256 with 8
// values per thread (then the exchange steps need only warp barriers), two
// warps at M = 512.  Short rows are packed several to a warp.  One CTA = ROWS rows; the grid is ny / ROWS CTAs, small enough
// units that the SMs finish within one row of each other.
// Values per thread of the two shapes the autotuner chooses between (one
// where both coincide): 8 (two warps per 1024-point row) measured fastest at
// 1024^2 and above (16 values: 20.1 against 19.0 us at 2048^2, 97 against 90 at
// 4096^2), 4 at 512^2 and below; 3 * 2^k rows take 24 (13.0 against 17.0 us at 1536^2)
// or 12 (faster from 768^2 down).
template <int M>
struct RowPassE {
  static constexpr int v0 = (M % 3 == 0) ? 12 : 8;
  static constexpr int v1 = (M % 3 == 0) ? 24 : 4;
};
template <int M, int EV>
struct RowPassCfg {
  static constexpr int E = EV;
  static constexpr int TPF = M / E;
  static constexpr int ROWS = (TPF >= 32) ? 1 : 32 / TPF;
  static constexpr int THREADS = ROWS * TPF;
  static constexpr bool WARP = (THREADS == 32);
};

// Shared memory of the row pass.  The tiles of the column-tiled fields keep
// their order, [tile][row][4 columns].  EARLY (rows up to 512 values, whose
// CTAs all fit at once): every input has its own buffer and is requested at the
// start, and the first transform's field's, once read, is the second exchange
// buffer (one barrier per exchange instead of two).  Longer rows: the field of the first transform lands in the
// transform's own buffer (its values and their partners -k are read from there
// before the first exchange overwrites them), and t_RF and the signal-side
// field take the pixel table's place once the pixel update has read it -- 50
// instead of 99 KB at 2048 values, so four CTAs of an SM overlap one
// another's loads and transforms.
template <int M, int MODE, int EV>
struct RowPassSmem {
  static constexpr int ROWS = RowPassCfg<M, EV>::ROWS;
  static constexpr int NT = RowPassCfg<M, EV>::THREADS;
  static constexpr bool RF = (MODE == ROW_PASS_RF);
  static constexpr bool EARLY = M <= 512;
  static constexpr size_t al(size_t n) { return (n + 127) / 128 * 128; }
  static constexpr size_t field = (size_t)ROWS * M * 8;
  static constexpr size_t fft_off = 128;
  static constexpr size_t fft_bytes = al((size_t)ROWS * SPad<M>::size * 8);
  static constexpr size_t dn_off = fft_off + fft_bytes;
  static constexpr size_t in_off = EARLY ? dn_off + 2 * field : fft_off;  // the first transform's field
  static constexpr size_t t_off = !RF ? dn_off : (EARLY ? in_off + fft_bytes : dn_off);  // t_RF, then the signal side
  static constexpr size_t tw_off = EARLY ? in_off + fft_bytes + (RF ? 2 * field : 0) : dn_off + 2 * field;
  // the transform twiddles are staged too for short rows
  static constexpr bool TWS = M <= 512;
  static constexpr uint32_t tw_bytes = StageTable<M, EV>::size * 8;  // a multiple of 16
  static constexpr size_t bytes = tw_off + (TWS ? tw_bytes : 0);
  // resident CTAs the registers are held to: 64 a thread for long rows, 102
  // and 170 for 12 and 24 values
  static constexpr int min_ctas =
      EV == 12 ? 640 / NT : (EV == 24 ? 384 / NT : (M >= 768 ? 1024 / NT : 1));
  // position of value k of row r in a tiled buffer
  static __device__ __forceinline__ int tpos(int r, int k) {
    return (k / WF_TW) * (ROWS * WF_TW) + r * WF_TW + (k % WF_TW);
  }
};

constexpr int kBoxTiles = 256;  // column tiles of one tensor copy

// The row pass (Sec. 2: eq. 2mess_t1 analogue in pixels between the inverse
// and forward row DFTs, then the stripe-basis updates).  Every copy is the
// TMA's: row-major inputs (d_RF, the pixel table) by bulk copies, the
// column-tiled ones (t_RF, the signal-side field) and the new t_RF by 2D tensor
// copies of all the row's 32-byte pieces.  (Gathered by 16-byte asynchronous
// copies and stored by 8-byte stores, those pieces took a shared-memory
// wavefront each: 66 % of the load-store pipe at 4096^2, the pass's bound.)
// 5.5 us at 1024^2, 19.0 at 2048^2, 88 at 4096^2 (7.3, 29 and 141 so): memory
// bound at 2048^2 (6.2 TB/s of 28 bytes per pixel) and beyond, below by the chain
// of one CTA.
// Waits are bounded; on a timeout the CTA records WF_ERR_TIMEOUT, drains its
// copies (bounded) and returns.
template <int M, int MODE, int EV>
__global__ void __launch_bounds__(RowPassCfg<M, EV>::THREADS, RowPassSmem<M, MODE, EV>::min_ctas)
row_pass_kernel(const __grid_constant__ RowArgs a) {
  using Cfg = RowPassCfg<M, EV>;
  using SM = RowPassSmem<M, MODE, EV>;
  constexpr int E = Cfg::E, TPF = Cfg::TPF, ROWS = Cfg::ROWS;
  constexpr bool W = Cfg::WARP;
  constexpr bool RF = SM::RF, EARLY = SM::EARLY;
  constexpr uint32_t kField = (uint32_t)SM::field;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
  float2* s_fft = reinterpret_cast<float2*>(smem + SM::fft_off);
  float4* s_dn = reinterpret_cast<float4*>(smem + SM::dn_off);
  float2* s_in = reinterpret_cast<float2*>(smem + SM::in_off);
  float2* s_t1 = reinterpret_cast<float2*>(smem + SM::t_off);
  float2* s_x = s_t1 + ROWS * M;
  float2* s_tw = reinterpret_cast<float2*>(smem + SM::tw_off);

  const int g = threadIdx.x / TPF;
  const int t = threadIdx.x - g * TPF;
  const int y0 = blockIdx.x * ROWS;  // ny is a multiple of ROWS
  const int y = y0 + g;
  float2* sb = s_fft + g * SPad<M>::size;

  // one row group of a column-tiled field into (or out of) a tiled buffer
  auto load_tiled = [&](float2* dst, const CUtensorMap* map, uint64_t* b) {
#pragma unroll
    for (int j = 0; j < M / WF_TW; j += kBoxTiles)
      tma2d_g2s(dst + j * ROWS * WF_TW, map, y0 * 2 * WF_TW, j, b);
  };

  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&bar[2], 1);
    mbar_fence_init();
    // before the previous kernel has finished: the pixel table (fixed during
    // a solve) and the transform twiddles
    mbar_expect_tx(&bar[1], 2 * kField + (SM::TWS ? SM::tw_bytes : 0));
    if constexpr (SM::TWS) bulk_g2s(s_tw, a.tws, SM::tw_bytes, &bar[1]);
    bulk_g2s(s_dn, a.dn + (size_t)y0 * M, 2 * kField, &bar[1]);
    tma_prefetch_map(&a.tm_t);
    tma_prefetch_map(&a.tm_x);
  }
  float2 wk[EARLY ? E : 1];
  if constexpr (EARLY) load_rtw<M, E>(wk, t, a.twx);
  // stripe spectrum a(y)^2 Pst(k) of this thread's modes (fixed during a solve)
  float pk[RF && EARLY ? E : 1];
  float a2y = 1.f, pkn = 0.f;  // pkn: Pst at kx = M, packed with kx = 0
  if constexpr (RF) {
    if (a.a2 != nullptr) a2y = __ldg(&a.a2[y]);
    if constexpr (EARLY) {
#pragma unroll
      for (int m = 0; m < E; ++m) pk[m] = __ldg(&a.pst[t + m * TPF]);
    }
    if (t == 0) pkn = __ldg(&a.pst[M]);
  }
  pdl_wait();
  // the fields the previous kernels wrote
  if (threadIdx.x == 0) {
    mbar_expect_tx(&bar[0], kField);
    if constexpr (RF) {
      if constexpr (EARLY) {
        bulk_g2s(s_in, a.f_d1 + (size_t)y0 * M, kField, &bar[0]);
        mbar_expect_tx(&bar[2], 2 * kField);
        load_tiled(s_t1, &a.tm_t, &bar[2]);
        load_tiled(s_x, &a.tm_x, &bar[2]);
      } else {
#pragma unroll
        for (int r = 0; r < ROWS; ++r) bulk_g2s(s_in + r * M, a.f_d1 + (size_t)(y0 + r) * M, M * 8, &bar[0]);
      }
    } else {
      load_tiled(s_in, &a.tm_x, &bar[0]);
    }
  }
  // link covariances of this lambda level (written by the controller)
  const float T2 = a.st->Tf[2];
  const float T1 = RF ? a.st->Tf[1] : 0.f;
  const float off1 = RF ? (float)a.st->off[1] : 0.f;
  const bool done = a.check_done && a.st->done;  // uniform: set only between launches
  __syncthreads();  // the barriers are initialised

  // the copies requested so far, for a CTA that leaves early
  auto drain = [&]() {
    const bool ok0 = mbar_wait(&bar[0], 0, WF_WAIT_TRIES);
    const bool ok1 = mbar_wait(&bar[1], 0, WF_WAIT_TRIES);
    const bool ok2 = !(RF && EARLY) || mbar_wait(&bar[2], 0, WF_WAIT_TRIES);
    if (!(ok0 && ok1 && ok2)) atomicOr(&a.st->err, WF_ERR_TIMEOUT);
  };
  if (done) {
    drain();
    return;
  }
  const bool ok = mbar_wait(&bar[0], 0, WF_WAIT_TRIES) && mbar_wait(&bar[1], 0, WF_WAIT_TRIES);
  if (__syncthreads_or(!ok)) {
    drain();
    return;
  }

  float2 v[E];
  c2r_pre_at<M, E>(v, t, [&](int k) { return RF ? s_in[g * M + k] : s_in[SM::tpos(g, k)]; },
                   [&](int m, int k) { return EARLY ? wk[EARLY ? m : 0] : __ldg(&a.twx[k]); });
  if constexpr (!EARLY) fft_sync<W>();  // read before the first exchange overwrites it
  float2* sb2 = s_in + g * SPad<M>::size;  // EARLY: the second exchange buffer
  if constexpr (EARLY) fft_pingpong<M, E, true, W, SM::TWS>(v, sb, sb2, t, s_tw);
  else fft_staged<M, E, true, W, SM::TWS>(v, sb, t, a.tws);
  // eq. (2mess_t1) analogue in pixel space, two pixels per complex value
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const float4 q = s_dn[g * M + t + m * TPF];
    v[m] = make_float2(tpx_update(q.x, q.y, v[m].x, T2), tpx_update(q.z, q.w, v[m].y, T2));
  }
  if constexpr (RF && !EARLY) {
    __syncthreads();  // the pixel table is read
    if (threadIdx.x == 0) {
      mbar_expect_tx(&bar[2], 2 * kField);
      load_tiled(s_t1, &a.tm_t, &bar[2]);
      load_tiled(s_x, &a.tm_x, &bar[2]);
    }
  }
  if constexpr (EARLY) fft_pingpong<M, E, false, W, SM::TWS>(v, sb, sb2, t, s_tw);
  else fft_staged<M, E, false, W, SM::TWS>(v, sb, t, a.tws);
  if constexpr (EARLY) r2c_post_w<M, E, W, true>(v, sb, t, wk);
  else r2c_post<M, E, W, true>(v, sb, t, a.twx);
  pdl_trigger();
  if constexpr (RF) {
    if (__syncthreads_or(!mbar_wait(&bar[2], 0, WF_WAIT_TRIES))) {
      drain();
      if (!mbar_wait(&bar[2], 0, WF_WAIT_TRIES) || threadIdx.x == 0) atomicOr(&a.st->err, WF_ERR_TIMEOUT);
      return;
    }
    // eqs. (2mess_d0), (2mess_t0) analogues in the stripe basis
    const size_t row0 = (size_t)y * M;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + m * TPF, i = SM::tpos(g, k);
      const float2 t1o = s_t1[i];
      const float2 xo = s_x[i];
      const float2 t2 = v[m];
      const float pv = EARLY ? pk[EARLY ? m : 0] : __ldg(&a.pst[k]);
      float2 d1, t1;
      stripe_mode(t2, t1o, xo, fmaf(a2y, pv, off1), T2, T1, d1, t1);
      if (m == 0 && t == 0) stripe_update(0, t2, t1o, xo, a2y, pv, pkn, off1, T2, T1, d1, t1);
      a.f_d1[row0 + k] = d1;
      s_t1[i] = t1;
    }
  } else {
    if constexpr (!EARLY) __syncthreads();
    else fft_sync<W>();
#pragma unroll
    for (int m = 0; m < E; ++m) s_t1[SM::tpos(g, t + m * TPF)] = v[m];
  }
  // the new messenger leaves by tensor copies
  fence_async_smem();
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < M / WF_TW; j += kBoxTiles) tma2d_s2g(&a.tm_t, y0 * 2 * WF_TW, j, s_t1 + j * ROWS * WF_TW);
    bulk_store_wait();
  }
}

template <int M, int MODE, int EV>
static int launch_row_pass_e(const RowArgs& a, cudaStream_t s) {
  using Cfg = RowPassCfg<M, EV>;
  constexpr size_t bytes = RowPassSmem<M, MODE, EV>::bytes;
  static DeviceOnce once;
  const cudaError_t cfg_err = once.run([](int*) {
    return cudaFuncSetAttribute(row_pass_kernel<M, MODE, EV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(bytes > kSpreadSmem ? bytes : kSpreadSmem));
  });
  if (cfg_err != cudaSuccess) return (int)cfg_err;
  const dim3 grid(a.ny / Cfg::ROWS), block(Cfg::THREADS);
  return launch_pdl(row_pass_kernel<M, MODE, EV>, grid, block, spread_smem(grid.x, bytes, a.sms), s, a);
}

// a.variant selects the shape (0 or 1, RowPassE)
template <int M, int MODE>
static int launch_row_pass(const RowArgs& a, cudaStream_t s) {
  if constexpr (RowPassE<M>::v1 != RowPassE<M>::v0) {
    if (a.variant == 1) return launch_row_pass_e<M, MODE, RowPassE<M>::v1>(a, s);
  }
  return launch_row_pass_e<M, MODE, RowPassE<M>::v0>(a, s);
}

template <int M>
static int launch_row_M(int mode, const RowArgs& a, cudaStream_t s) {
  using Cfg = RowCfg<M>;
  const dim3 grid((a.ny + Cfg::ROWS - 1) / Cfg::ROWS), block(Cfg::THREADS);
  const bool whole = whole_split(a.ny, a.nx, a.sms);
  switch (mode) {
    case ROW_PASS_RF: return launch_row_pass<M, ROW_PASS_RF>(a, s);
    case ROW_PASS_NORF: return launch_row_pass<M, ROW_PASS_NORF>(a, s);
    case ROW_RESID_B: return launch_pdl_split(whole, row_kernel<M, ROW_RESID_B>, grid, block, 0, s, a);
    case ROW_RESID_D: return launch_pdl_split(whole, row_kernel<M, ROW_RESID_D>, grid, block, 0, s, a);
    case ROW_C2R: return launch_pdl(row_kernel<M, ROW_C2R>, grid, block, 0, s, a);
    case ROW_R2C: return launch_pdl(row_kernel<M, ROW_R2C>, grid, block, 0, s, a);
    default: return (int)cudaErrorInvalidValue;
  }
  return (int)cudaGetLastError();
}

int launch_row(int mode, const RowArgs& a, cudaStream_t s) {
  switch (a.nx / 2) {
    case 16: return launch_row_M<16>(mode, a, s);
    case 32: return launch_row_M<32>(mode, a, s);
    case 64: return launch_row_M<64>(mode, a, s);
    case 128: return launch_row_M<128>(mode, a, s);
    case 256: return launch_row_M<256>(mode, a, s);
    case 192: return launch_row_M<192>(mode, a, s);
    case 384: return launch_row_M<384>(mode, a, s);
    case 512: return launch_row_M<512>(mode, a, s);
    case 768: return launch_row_M<768>(mode, a, s);
    case 1024: return launch_row_M<1024>(mode, a, s);
    case 2048: return launch_row_M<2048>(mode, a, s);
    default: return (int)cudaErrorInvalidValue;
  }
}

template <int M>
static int rows_per_cta() { return RowCfg<M>::ROWS; }

int row_grid(int nx, int ny) {
  int r = 1;
  switch (nx / 2) {
    case 16: r = rows_per_cta<16>(); break;
    case 32: r = rows_per_cta<32>(); break;
    case 64: r = rows_per_cta<64>(); break;
    case 128: r = rows_per_cta<128>(); break;
    case 256: r = rows_per_cta<256>(); break;
    case 192: r = rows_per_cta<192>(); break;
    case 384: r = rows_per_cta<384>(); break;
    case 512: r = rows_per_cta<512>(); break;
    case 768: r = rows_per_cta<768>(); break;
    case 1024: r = rows_per_cta<1024>(); break;
    case 2048: r = rows_per_cta<2048>(); break;
    default: r = 1;
  }
  return (ny + r - 1) / r;
}

template <int M>
static int row_rows(int v) {
  return v == 1 ? RowPassCfg<M, RowPassE<M>::v1>::ROWS : RowPassCfg<M, RowPassE<M>::v0>::ROWS;
}

// rows per CTA of the row pass
int row_pass_rows(int M, int v) {
  switch (M) {
    case 16: return row_rows<16>(v);
    case 32: return row_rows<32>(v);
    case 64: return row_rows<64>(v);
    case 128: return row_rows<128>(v);
    case 192: return row_rows<192>(v);
    case 256: return row_rows<256>(v);
    case 384: return row_rows<384>(v);
    case 512: return row_rows<512>(v);
    case 768: return row_rows<768>(v);
    case 1024: return row_rows<1024>(v);
    case 2048: return row_rows<2048>(v);
    default: return 0;
  }
}

template <int M>
static int row_e(int v) { return v == 1 ? RowPassE<M>::v1 : RowPassE<M>::v0; }

int row_pass_e(int M, int v) {
  switch (M) {
    case 16: return row_e<16>(v);
    case 32: return row_e<32>(v);
    case 64: return row_e<64>(v);
    case 128: return row_e<128>(v);
    case 192: return row_e<192>(v);
    case 256: return row_e<256>(v);
    case 384: return row_e<384>(v);
    case 512: return row_e<512>(v);
    case 768: return row_e<768>(v);
    case 1024: return row_e<1024>(v);
    case 2048: return row_e<2048>(v);
    default: return 0;
  }
}

bool size_supported(int n) {
  // powers of two from 32 to 4096, and 384, 768, 1536 (3 * 2^k, one radix-3 stage)
  return (n >= 32 && n <= 4096 && (n & (n - 1)) == 0) || n == 384 || n == 768 || n == 1536;
}

}  // namespace wf
