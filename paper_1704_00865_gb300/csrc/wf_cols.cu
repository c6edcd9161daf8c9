// wf_cols.cu -- the column steps of the residual (Huffenberger 2017, Sec. 2)
// and the column transforms, plus the dispatch of every column kernel by
// column length (the column pass itself is in wf_colpass.cu).
//
// One CTA owns W adjacent complex columns (kx) of a row-transformed field;
// TPC = ny/E threads per column run a complex length-ny Stockham FFT in shared
// memory, which completes the 2D DFT.  s is never stored: it is
// C t0 / (C + T_0) (eq. 2mess_s), recomputed with the T_0 in force when t0
// was made, or C d0 / (C + N0) with the merged 2DF block.
//
// Column 0 packs the two real-signal columns kx = 0 and kx = nx/2 as
// Z = A + i B (see wf_cols_common.cuh), treated as separate modes with their
// own eigenvalues.
#include "wf_cols_common.cuh"

namespace wf {

// NARROW (long columns): at most 256 threads, one or two columns per CTA.
template <int L, bool NARROW = false>
struct ColCfg {
  static constexpr int E = col_kernel_e(L);
  static constexpr int TPC = L / E;
  // whole tiles, 32-byte pieces of the row-major fields (half of that at 4096,
  // where four columns would not fit)
  static constexpr int W = NARROW ? 256 / TPC : TPC < 16 ? 64 / TPC : (L >= 4096 ? 2 : WF_TW);
  static_assert(!NARROW || (TPC >= 128 && TPC <= 256), "one or two long columns");
  static constexpr int THREADS = W * TPC;
  // Stride between the per-column FFT buffers (complex values): a half-warp
  // covers W columns x 16/W consecutive indices, which are bank-conflict free
  // when the stride is congruent to 16/W modulo 16 (odd for W = 32).
  static constexpr int SP = SPad<L>::size;
  static constexpr int WANT = (W >= 32) ? 1 : (16 / W) % 16;
  static constexpr int STRIDE = SP + ((WANT - SP % 16) + 16) % 16;
  static constexpr size_t bytes = (size_t)W * STRIDE * 8;
};

// the plain transforms are held to 64 registers a thread, so that two CTAs of
// long columns share an SM
template <int L, int MODE, bool NARROW>
constexpr int col_min_ctas() {
  return (MODE == COL_FWD || MODE == COL_INV || MODE == COL_FWD_TILED || MODE == COL_INV_TILED) && L >= 1024 && !NARROW
             ? 1024 / ColCfg<L>::THREADS
             : 1;
}

template <int L, int MODE, bool NARROW = false>
__global__ void __launch_bounds__(ColCfg<L, NARROW>::THREADS, col_min_ctas<L, MODE, NARROW>())
col_kernel(ColArgs a) {
  using Cfg = ColCfg<L, NARROW>;
  constexpr int E = Cfg::E, TPC = Cfg::TPC, W = Cfg::W;
  extern __shared__ __align__(16) float2 sbuf[];  // [W][STRIDE]

  const int c = threadIdx.x % W;
  const int t = threadIdx.x / W;
  const int ncols = a.nx / 2;
  const int col = blockIdx.x * W + c;  // ncols is a multiple of W
  float2* sb = sbuf + c * Cfg::STRIDE;

  pdl_trigger();
  // the eigenvalues, fixed during a solve, while the previous kernel drains
  constexpr bool EIG = (MODE == COL_RESID_A || MODE == COL_RESID_C || MODE == COL_G_FROM_S), PRE = EIG && E <= 12;
  float2 eg0[PRE ? E : 1];
  if constexpr (PRE) {
#pragma unroll
    for (int m = 0; m < E; ++m) eg0[m] = __ldg(&a.eig[tidx(t + m * TPC, col, a.ny)]);
  }
  pdl_wait();
  // uniform: both flags are set only between launches
  if ((a.check_done && a.st->done) || (a.skip_ok && a.st->skip_resid)) return;

  auto eig_at = [&](int m) -> float2 {
    return PRE ? eg0[PRE ? m : 0] : a.eig[tidx(t + m * TPC, col, a.ny)];
  };
  auto at = [&](int k) -> size_t { return (size_t)k * ncols + col; };       // row-major
  auto att = [&](int k) -> size_t { return tidx(k, col, a.ny); };           // column-tiled
  float2 v[E];

  // Partner value Z[-k] of column 0 (only meaningful where col == 0).  Every
  // thread of CTA 0 takes part in the exchange; CTA 0 is uniform.
  auto exchange0 = [&](float2 (&u)[E], float2 (&up)[E]) {
#pragma unroll
    for (int m = 0; m < E; ++m) sb[spad(t + m * TPC)] = u[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + m * TPC;
      up[m] = sb[spad(neg_mod<L>(k))];
    }
    __syncthreads();
  };

  // Every mode through f(m, whether it belongs to the packed column): CTA 0
  // has a loop of its own, so that the others' loads overlap.
  auto each_mode = [&](auto&& f) {
    if (blockIdx.x != 0) {
#pragma unroll
      for (int m = 0; m < E; ++m) f(m, false);
    } else {
#pragma unroll
      for (int m = 0; m < E; ++m) f(m, c == 0);
    }
  };

  if constexpr (MODE == COL_RESID_A) {
    // g = S^-1 s and s = C g in RF, for the residual and the export of s:
    // from the data-side messenger (merged 2DF block, or no 1/f part), or
    // g = t0 / (C + T0) from the stored t_2DF (plain sweep)
    float2 vp[E];
    const float sc = 1.0f / (float)L;
    if (!a.has_f || a.merge) {
      // From the data-side messenger y that the last column pass used:
      // s = C/(C + N0 + T) y and g = S^-1 s = y/(C + N0 + T), with N0 = 0
      // without a 1/f part.  Forming g from y (not from the stored, high-k
      // suppressed d_2DF or s) keeps FP32 rounding out of the 1/C factor.
      const float Tl = a.has_rf ? a.st->Tf[1] : a.st->Tf[2];
      const float off0 = (float)a.st->off[0];
      float2 w[E];
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = a.f_y[att(t + m * TPC)];
      fft_staged<L, E, false>(v, sb, t, a.twk);
      if (blockIdx.x == 0) exchange0(v, vp);
      each_mode([&](int m, bool pk) {
        const int k = t + m * TPC;
        const float2 eg = eig_at(m);
        // with a source j: g = (y + (N0 + T) j^) / (C + N0 + T)
        const float2 jv = (a.src != nullptr) ? a.src[att(k)] : make_float2(0.f, 0.f);
        if (pk) {
          const float2 egb = a.eig_nyq[k];
          const float2 jp = (a.src != nullptr) ? a.src[att(neg_mod<L>(k))] : make_float2(0.f, 0.f);
          float2 A, B, JA, JB;
          unpack_pair(v[m], vp[m], A, B);
          unpack_pair(jv, jp, JA, JB);
          const float na = eg.y + off0 + Tl, nb = egb.y + off0 + Tl;
          const float2 gA = cscale(make_float2(fmaf(na, JA.x, A.x), fmaf(na, JA.y, A.y)), __fdividef(1.f, eg.x + na));
          const float2 gB = cscale(make_float2(fmaf(nb, JB.x, B.x), fmaf(nb, JB.y, B.y)), __fdividef(1.f, egb.x + nb));
          v[m] = repack_pair(gA, gB);
          w[m] = repack_pair(cscale(gA, eg.x), cscale(gB, egb.x));
        } else {
          const float na = eg.y + off0 + Tl;
          const float2 g = cscale(make_float2(fmaf(na, jv.x, v[m].x), fmaf(na, jv.y, v[m].y)),
                                  __fdividef(1.f, eg.x + na));
          v[m] = g;
          w[m] = cscale(g, eg.x);
        }
      });
      fft_staged<L, E, true>(v, sb, t, a.twk);
      fft_staged<L, E, true>(w, sb, t, a.twk);
#pragma unroll
      for (int m = 0; m < E; ++m) {
        a.r_g[at(t + m * TPC)] = cscale(v[m], sc);
        a.r_q[at(t + m * TPC)] = cscale(w[m], sc);
      }
    } else if (a.has_f) {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = a.f_t0[att(t + m * TPC)];
      const float T0s = a.st->T0s[a.parity];
      float2 w[E];
      each_mode([&](int m, bool pk) {
        const int k = t + m * TPC;
        const float2 eg = eig_at(m);
        if (pk) {
          const int kp = neg_mod<L>(k);
          const float2 egb = a.eig_nyq[k];
          float2 A, B;
          unpack_pair(v[m], a.f_t0[att(kp)], A, B);
          const float ia = __fdividef(1.f, eg.x + T0s), ib = __fdividef(1.f, egb.x + T0s);
          const float2 gA = cscale(A, ia), gB = cscale(B, ib);
          v[m] = repack_pair(gA, gB);
          w[m] = repack_pair(cscale(gA, eg.x), cscale(gB, egb.x));
        } else {
          const float2 g = cscale(v[m], __fdividef(1.f, eg.x + T0s));
          v[m] = g;
          w[m] = cscale(g, eg.x);
        }
      });
      fft_staged<L, E, true>(v, sb, t, a.twk);
      fft_staged<L, E, true>(w, sb, t, a.twk);
#pragma unroll
      for (int m = 0; m < E; ++m) {
        a.r_g[at(t + m * TPC)] = cscale(v[m], sc);
        a.r_q[at(t + m * TPC)] = cscale(w[m], sc);
      }
    }
  } else if constexpr (MODE == COL_RESID_C) {
    // q += N_2DF g'  (the given 1/f eigenvalues)
    float2 vp[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = a.r_g[at(t + m * TPC)];
    fft_staged<L, E, false>(v, sb, t, a.twk);
    if (blockIdx.x == 0) exchange0(v, vp);
    each_mode([&](int m, bool pk) {
      const int k = t + m * TPC;
      const float2 eg = eig_at(m);
      if (pk) {
        float2 A, B;
        unpack_pair(v[m], vp[m], A, B);
        v[m] = repack_pair(cscale(A, eg.y), cscale(B, a.eig_nyq[k].y));
      } else {
        v[m] = cscale(v[m], eg.y);
      }
    });
    fft_staged<L, E, true>(v, sb, t, a.twk);
    const float sc = 1.0f / (float)L;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const size_t i = at(t + m * TPC);
      const float2 q = a.r_q[i];
      a.r_q[i] = make_float2(fmaf(v[m].x, sc, q.x), fmaf(v[m].y, sc, q.y));
    }
  } else if constexpr (MODE == COL_G_FROM_S) {
    // residual of a given s: r_q holds s in RF (kept); r_g <- S^-1 s in RF
    float2 vp[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = a.r_q[at(t + m * TPC)];
    fft_staged<L, E, false>(v, sb, t, a.twk);
    if (blockIdx.x == 0) exchange0(v, vp);
    each_mode([&](int m, bool pk) {
      const int k = t + m * TPC;
      const float2 eg = eig_at(m);
      if (pk) {
        float2 A, B;
        unpack_pair(v[m], vp[m], A, B);
        v[m] = repack_pair(cscale(A, __fdividef(1.f, eg.x)), cscale(B, __fdividef(1.f, a.eig_nyq[k].x)));
      } else {
        v[m] = cscale(v[m], __fdividef(1.f, eg.x));
      }
    });
    fft_staged<L, E, true>(v, sb, t, a.twk);
    const float sc = 1.0f / (float)L;
#pragma unroll
    for (int m = 0; m < E; ++m) a.r_g[at(t + m * TPC)] = cscale(v[m], sc);
  } else if constexpr (MODE == COL_WARM) {
    // warm start from s (in RF, row-major in a.in): the data-side messenger
    // gets s itself (tiled copy), the signal-side field d_2DF = (C + N_0)/C s
    // with the merged 2DF block (s = C/(C + N_0) d_2DF), or s itself
    float2 vp[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
      v[m] = a.in[at(t + m * TPC)];
      a.warm_copy[att(t + m * TPC)] = v[m];
    }
    if (a.has_f) {
      const float off0 = (float)a.st->off[0];
      fft_staged<L, E, false>(v, sb, t, a.twk);
      if (blockIdx.x == 0) exchange0(v, vp);
      each_mode([&](int m, bool pk) {
        const int k = t + m * TPC;
        const float2 eg = a.eig[att(k)];
        const float fa = __fdividef(eg.x + eg.y + off0, eg.x);
        if (pk) {
          const float2 egb = a.eig_nyq[k];
          float2 A, B;
          unpack_pair(v[m], vp[m], A, B);
          v[m] = repack_pair(cscale(A, fa), cscale(B, __fdividef(egb.x + egb.y + off0, egb.x)));
        } else {
          v[m] = cscale(v[m], fa);
        }
      });
      fft_staged<L, E, true>(v, sb, t, a.twk);
      const float sc = 1.0f / (float)L;
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = cscale(v[m], sc);
    }
#pragma unroll
    for (int m = 0; m < E; ++m) a.out[att(t + m * TPC)] = v[m];
  } else if constexpr (MODE == COL_UNTILE) {
#pragma unroll
    for (int m = 0; m < E; ++m) a.out[at(t + m * TPC)] = a.in[att(t + m * TPC)];
  } else if constexpr (MODE == COL_FWD || MODE == COL_INV || MODE == COL_FWD_TILED || MODE == COL_INV_TILED) {
    constexpr bool INV = (MODE == COL_INV || MODE == COL_INV_TILED), TILED_IN = (MODE == COL_INV_TILED);
#pragma unroll
    for (int m = 0; m < E; ++m)
      v[m] = a.in[TILED_IN ? att(t + m * TPC) : at(t + m * TPC)];
    fft_staged<L, E, INV>(v, sb, t, a.twk);
    const float sc = INV ? 1.0f / (float)L : 1.0f;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      if constexpr (MODE == COL_FWD_TILED) a.out[att(t + m * TPC)] = cscale(v[m], sc);
      else a.out[at(t + m * TPC)] = cscale(v[m], sc);
    }
  }
}

template <int L, int MODE, bool NARROW>
static int launch_col_kernel_w(const ColArgs& a, cudaStream_t s) {
  using Cfg = ColCfg<L, NARROW>;
  constexpr auto kernel = col_kernel<L, MODE, NARROW>;
  static DeviceOnce once;
  const cudaError_t cfg_err = once.run(
      [](int*) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::bytes); });
  if (cfg_err != cudaSuccess) return (int)cfg_err;
  if (a.nx / 2 % Cfg::W != 0) return (int)cudaErrorInvalidValue;
  const dim3 grid(a.nx / 2 / Cfg::W), block(Cfg::THREADS);
  const bool whole = (MODE == COL_RESID_A || MODE == COL_RESID_C) && whole_split(a.ny, a.nx, a.sms);
  return launch_pdl_split(whole, kernel, grid, block, Cfg::bytes, s, a);
}

template <int L, int MODE>
static int launch_col_kernel(const ColArgs& a, cudaStream_t s) {
  // Narrow CTAs while there are no more of them than SMs: with wider ones half
  // the SMs stay idle (a forward and an inverse transform of 2048 x 512 59.6 us,
  // 51.7 narrow; of 4096 x 256 69.3 and 58.2).  Beyond, whole 32-byte pieces count
  // (4096 x 1024: 87.8 us, 107 narrow).  1024-long columns take 10 us either way.
  if constexpr (L >= 1536)
    if (a.nx / 2 / ColCfg<L, true>::W <= kSms) return launch_col_kernel_w<L, MODE, true>(a, s);
  return launch_col_kernel_w<L, MODE, false>(a, s);
}

template <int L>
static int launch_col_L(int mode, const ColArgs& a, cudaStream_t s) {
  switch (mode) {
    case COL_PASS_2DF:
    case COL_PASS_NO2DF:
    case COL_PASS_MERGE:
    case COL_PASS_MERGE_SRC: return launch_col_pass_any<L>(mode, a, s);
    case COL_RESID_A: return launch_col_kernel<L, COL_RESID_A>(a, s);
    case COL_RESID_C: return launch_col_kernel<L, COL_RESID_C>(a, s);
    case COL_FWD: return launch_col_kernel<L, COL_FWD>(a, s);
    case COL_INV: return launch_col_kernel<L, COL_INV>(a, s);
    case COL_G_FROM_S: return launch_col_kernel<L, COL_G_FROM_S>(a, s);
    case COL_UNTILE: return launch_col_kernel<L, COL_UNTILE>(a, s);
    case COL_FWD_TILED: return launch_col_kernel<L, COL_FWD_TILED>(a, s);
    case COL_WARM: return launch_col_kernel<L, COL_WARM>(a, s);
    case COL_INV_TILED: return launch_col_kernel<L, COL_INV_TILED>(a, s);
    default: return (int)cudaErrorInvalidValue;
  }
  return (int)cudaGetLastError();
}

int launch_col(int mode, const ColArgs& a, cudaStream_t s) {
  switch (a.ny) {
    case 32: return launch_col_L<32>(mode, a, s);
    case 64: return launch_col_L<64>(mode, a, s);
    case 128: return launch_col_L<128>(mode, a, s);
    case 256: return launch_col_L<256>(mode, a, s);
    case 384: return launch_col_L<384>(mode, a, s);
    case 512: return launch_col_L<512>(mode, a, s);
    case 768: return launch_col_L<768>(mode, a, s);
    case 1024: return launch_col_L<1024>(mode, a, s);
    case 1536: return launch_col_L<1536>(mode, a, s);
    case 2048: return launch_col_L<2048>(mode, a, s);
    case 4096: return launch_col_L<4096>(mode, a, s);
    default: return (int)cudaErrorInvalidValue;
  }
}

}  // namespace wf
