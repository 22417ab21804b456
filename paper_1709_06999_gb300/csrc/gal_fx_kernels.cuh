// Row and column passes of the double-precision path on 64-bit integers
// (gal_fx.cuh): the passes of gal_kernels.cuh with each sequence brought to a
// common power of two before its transform.  Images, F1 and the window are
// doubles.  Measured against the same passes in FP64 arithmetic (which kept the
// FP64 pipe 83 % busy): row pass of 4096^2 pixels, 61 columns kept, 481 -> 113
// us; of 2048^2 pixels, 413 columns kept, 161 -> 38 us; column pass of 4096 x 61
// 41 -> 12 us, of 2048 x 413 66 -> 19 us.
#pragma once

#include <climits>

#include "gal_fx.cuh"
#include "gal_kernels.cuh"

namespace gal {

// Rows of 2^(LG+1) pixels as complex sequences of M = 2^LG points.
template <int LG> struct FxRowShape {
  static constexpr int M = 1 << LG, N = 2 * M;
  using SH = Shape3<double, M, N, 128, 8>;
  static constexpr int ntab = FxPlan<M>::ntab;
  // header (barriers, reduction scratch, row scales), factor table, row buffers
  static constexpr int kHead = 512;
  static constexpr size_t smem(bool tma) {
    return kHead + (size_t)ntab * sizeof(fxtw) + (size_t)(tma ? 3 : 2) * SH::G * SH::RS * sizeof(fx2);
  }
};

// Row pass (see row_fft3_kernel).  Persistent blocks own row groups; TMA: the
// image rows come through a two-slot ring of bulk copies, SWEEP: they are
// generated from the profile.
template <int LG, bool SWEEP, int K, bool BEAM = false>
__global__ void __launch_bounds__(FxRowShape<LG>::SH::threads,
                                  min_blocks_128regs<FxRowShape<LG>::SH::threads>())
row_fx_kernel(const __grid_constant__ Jobs<RowJob<double>, K> jobs, const double2* __restrict__ twd,
              int* __restrict__ err) {
  grid_dep_launch();  // the column pass may be scheduled as our blocks retire
  using S = FxRowShape<LG>;
  using SH = typename S::SH;
  using P = typename SH::P;
  constexpr int M = S::M, N = S::N, TT = P::T, G = SH::G, RS = SH::RS;
  const RowJob<double>& jb = jobs.j[K == 1 ? 0 : blockIdx.y];
  const double* __restrict__ image = jb.image;
  const double* __restrict__ beam = BEAM ? jb.beam : nullptr;
  double2* __restrict__ F1 = jb.F1;
  const fxtw* __restrict__ tw = reinterpret_cast<const fxtw*>(twd + N);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw);
  unsigned* red_max = reinterpret_cast<unsigned*>(smem_raw + 32);   // one per warp, <= 16
  unsigned* red_sum = reinterpret_cast<unsigned*>(smem_raw + 96);
  int* row_q = reinterpret_cast<int*>(smem_raw + 192);              // per row of the group, <= 64
  fxtw* tab = reinterpret_cast<fxtw*>(smem_raw + S::kHead);
  fx2* base = reinterpret_cast<fx2*>(smem_raw + S::kHead + (size_t)S::ntab * sizeof(fxtw));
  static_assert(G <= 64 && SH::threads <= 512, "header");
  const int g = threadIdx.x / TT, t = threadIdx.x - g * TT;
  const int ngroups = N / G;
  fx2* slot0 = base;
  fx2* work = base + (size_t)(SWEEP ? 1 : 2) * G * RS;
  const uint32_t half_bytes = (uint32_t)(M * sizeof(double));
  if constexpr (!SWEEP) {
    if (threadIdx.x == 0) {
      mbar_init(&bars[0], 1);
      mbar_init(&bars[1], 1);
      mbar_init_fence();
    }
    __syncthreads();
  }
  auto issue = [&](int it) {  // thread 0 only
    const int grp = blockIdx.x + it * gridDim.x;
    if (grp >= ngroups) return;
    const int sl = it & 1;
    mbar_arrive_expect_tx(&bars[sl], 2u * half_bytes * (uint32_t)G);
    for (int rl = 0; rl < G; ++rl) {
      const double* src = image + (size_t)(((grp * G + rl) + M) & (N - 1)) * N;
      double* dst = reinterpret_cast<double*>(slot0 + (size_t)(sl * G + rl) * RS);
      bulk_load(dst, src + M, half_bytes, &bars[sl]);
      bulk_load(dst + M, src, half_bytes, &bars[sl]);
    }
  };
  if constexpr (!SWEEP) {
    if (threadIdx.x == 0) {
      issue(0);
      issue(1);
    }
  }
  fx_fill_tab<M, 2>(tab, tw);
  const Bounds bd = block_bounds(jb.rho2, jb.S, N);  // synchronises
  const bool pruned = P::nstage >= 2 && bd.Kc <= P::Nsl;
  if constexpr (BEAM) grid_dep_wait();  // the beam tables
  for (int it = 0;; ++it) {
    const int grp = blockIdx.x + it * gridDim.x;
    if (grp >= ngroups) break;
    const int sl = SWEEP ? 0 : it & 1;
    const int row = grp * G + g;
    fx2* slot = slot0 + (size_t)(sl * G + g) * RS;
    double2 z[8];
    if constexpr (SWEEP) {
      const int irow = (row + M) & (N - 1);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int j = (2 * (t + r * TT) + M) & (N - 1);
        z[r] = make_double2(sweep_pixel(jb.I, jb.sp, N, irow, j), sweep_pixel(jb.I, jb.sp, N, irow, j + 1));
      }
    } else {
      const bool ok = mbar_wait(&bars[sl], (uint32_t)((it >> 1) & 1));
      if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
          atomicOr(err, 2);
          for (int k = it; k < it + 2; ++k)
            if (blockIdx.x + k * gridDim.x < ngroups) mbar_wait(&bars[k & 1], (uint32_t)((k >> 1) & 1));
        }
        return;
      }
#pragma unroll
      for (int r = 0; r < 8; ++r) z[r] = reinterpret_cast<const double2*>(slot)[t + r * TT];
    }
    if constexpr (BEAM) {
#pragma unroll
      for (int r = 0; r < 8; ++r) z[r] = beam_pair(z[r], beam, N, row, t + r * TT);
    }
    fx2 v[8];
    const FxScale sc = fx_load<TT>(z, v, red_max, red_sum);
    // the slot is written from stage 1 on, after the barrier that ends stage 0
    fx2* A = work + (size_t)g * RS;
    fx2* B = slot;
    FxHead<M, 0>::run(v, A, B, t, tab);
    fx2* in = last_input<M, 8>(A, B);
    double2* out = F1 + row;  // column-major: bin j of this row at out[j N]
    auto emit = [&](double2* o, fx2 x2, int q, bool bad) {
      *o = bad ? make_double2(fx_nan(), fx_nan()) : make_double2(fx_to(x2.x, q - 1), fx_to(x2.y, q - 1));
    };
    if (pruned) {
      for (int j = t; j < bd.Kc; j += TT) {
        fx2 zj, zmj;
        fx_pruned_pair<M, 2>(in, j, tw, zj, zmj);
        emit(out + (size_t)j * N, fx_r2c_unpack2(zj, zmj, ldg_tw(tw + j)), sc.q, sc.bad);
      }
    } else {
      fx_last_full<M, 2>(v, in, t, tw);
      fx2* o = in == A ? B : A;
      store_full<M, 8>(v, o, t);
      if (t == 0) row_q[g] = sc.bad ? INT_MAX : sc.q;
      __syncthreads();
      // bin by bin, the G rows of the group side by side (row_fft3_kernel)
      const fx2* o0 = o - (size_t)g * RS;
      double2* out0 = out - g;
      for (int q = threadIdx.x; q < bd.Kc * G; q += G * TT) {
        const int k = q / G, gg = q - k * G;
        const fx2* og = o0 + (size_t)gg * RS;
        emit(out0 + (size_t)k * N + gg,
             fx_r2c_unpack2(og[pad3<8>(k & (M - 1))], og[pad3<8>((M - k) & (M - 1))], ldg_tw(tw + k)),
             row_q[gg], row_q[gg] == INT_MAX);
      }
    }
    __syncthreads();  // every read of this slot and of the work buffer is done
    if constexpr (!SWEEP) {
      if (threadIdx.x == 0) {
        fence_proxy_async_smem();
        issue(it + 2);
      }
    }
  }
}

template <int LG> struct FxColShape {
  static constexpr int N = 1 << LG;
  using SH = ColShape3<double, N, 8>;
  static constexpr int ntab = FxPlan<N>::ntab;
  static constexpr int kHead = 128 + 1024;  // reduction scratch, a scale per column
  static constexpr size_t smem =
      kHead + (size_t)ntab * sizeof(fxtw) + (size_t)2 * SH::G * SH::RS * sizeof(fx2);
};

// Column pass (see col_fft3_kernel).
template <int LG, int K>
__global__ void __launch_bounds__(FxColShape<LG>::SH::threads)
col_fx_kernel(const __grid_constant__ Jobs<ColJob<double>, K> jobs, const double2* __restrict__ twd) {
  using S = FxColShape<LG>;
  using SH = typename S::SH;
  using P = typename SH::P;
  constexpr int N = S::N, TT = P::T, G = SH::G, RS = SH::RS;
  const ColJob<double>& jb = jobs.j[K == 1 ? 0 : blockIdx.y];
  const double2* __restrict__ F1 = jb.F1;
  double2* __restrict__ Gw = jb.Gw;
  const fxtw* __restrict__ tw = reinterpret_cast<const fxtw*>(twd + N);
  grid_dep_launch();  // the gather may start its prologue on the SMs we leave idle
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned* red_max = reinterpret_cast<unsigned*>(smem_raw);
  unsigned* red_sum = reinterpret_cast<unsigned*>(smem_raw + 64);
  int* col_q = reinterpret_cast<int*>(smem_raw + 128);
  fxtw* tab = reinterpret_cast<fxtw*>(smem_raw + S::kHead);
  fx2* base = reinterpret_cast<fx2*>(smem_raw + S::kHead + (size_t)S::ntab * sizeof(fxtw));
  static_assert(G <= 256 && SH::threads <= 512, "header");
  const int g = threadIdx.x / TT, t = threadIdx.x - g * TT;
  fx_fill_tab<N, 1>(tab, tw);
  const Bounds bd = block_bounds(jb.rho2, jb.S, N);  // synchronises
  const int ncol = jb.full ? full_cols(bd, N).W : bd.Kc;
  const int kmax = N / 2 - bd.r0;
  const bool pruned = P::nstage >= 2 && bd.r0 > 0 && kmax < P::Nsl;
  fx2* A = base + (size_t)g * RS;
  fx2* B = base + (size_t)(G + g) * RS;
  grid_dep_wait();  // F1 is the row pass's output
  for (int c0 = blockIdx.x * G; c0 < ncol; c0 += gridDim.x * G) {
    const int c = c0 + g;
    const bool act = c < ncol;
    double2 z[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) z[r] = act ? F1[(size_t)c * N + t + r * TT] : make_double2(0.0, 0.0);
    fx2 v[8];
    const FxScale sc = fx_load<TT>(z, v, red_max, red_sum);
    FxHead<N, 0>::run(v, A, B, t, tab);
    fx2* in = last_input<N, 8>(A, B);
    auto value = [&](fx2 x, int q, bool bad) {
      return bad ? make_double2(fx_nan(), fx_nan()) : make_double2(fx_to(x.x, q), fx_to(x.y, q));
    };
    if (pruned) {
      for (int j = t; j <= kmax; j += TT) {
        fx2 xj, xmj;
        fx_pruned_pair<N, 1>(in, j, tw, xj, xmj);
        if (act) {
          Gw[(size_t)(kmax + j) * ncol + c] = value(xj, sc.q, sc.bad);
          if (j > 0) Gw[(size_t)(kmax - j) * ncol + c] = value(xmj, sc.q, sc.bad);
        }
      }
    } else {
      fx_last_full<N, 1>(v, in, t, tw);
      fx2* o = in == A ? B : A;
      store_full<N, 8>(v, o, t);
      if (t == 0) col_q[g] = sc.bad ? INT_MAX : sc.q;
      __syncthreads();
      const fx2* o0 = o - (size_t)g * RS;
      for (int q = threadIdx.x; q < bd.nrw * G; q += G * TT) {
        const int rr = q / G, gg = q - rr * G;
        if (c0 + gg < ncol)
          Gw[(size_t)rr * ncol + c0 + gg] =
              value(o0[(size_t)gg * RS + pad3<8>((bd.r0 + rr + N / 2) & (N - 1))], col_q[gg],
                    col_q[gg] == INT_MAX);
      }
    }
    __syncthreads();
  }
}

// Launches over n jobs (grid row y = job y); scale: the share of the GPU's
// resident blocks a launch asks for; dep: a programmatic dependent (the beam
// tables were launched just before).
template <int LG, bool SWEEP, int K, bool BEAM>
cudaError_t launch_row_fx(const Jobs<RowJob<double>, K>& jb, int n, int scale, bool dep,
                          const double2* tw, int* err, cudaStream_t st) {
  using S = FxRowShape<LG>;
  constexpr auto kern = row_fx_kernel<LG, SWEEP, K, BEAM>;
  constexpr size_t smem = S::smem(!SWEEP);
  cudaError_t e = ensure_smem_attr<kern>(smem);
  if (e) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, S::SH::threads, smem);
  if (e) return e;
  if (per_sm < 1) per_sm = 1;
  int x = (per_sm * current_device_sms() * (scale < 1 ? 1 : scale) + n - 1) / n;
  if (x > S::N / S::SH::G) x = S::N / S::SH::G;
  if (x < 1) x = 1;
  if (dep) return launch_dependent(kern, dim3(x, n), dim3(S::SH::threads), smem, st, jb, tw, err);
  kern<<<dim3(x, n), S::SH::threads, smem, st>>>(jb, tw, err);
  return cudaGetLastError();
}

// cols: the widest job's window; dep as above (after the row pass)
template <int LG, int K>
cudaError_t launch_col_fx(const Jobs<ColJob<double>, K>& jb, int n, int cols, bool dep,
                          const double2* tw, cudaStream_t st) {
  using S = FxColShape<LG>;
  constexpr auto kern = col_fx_kernel<LG, K>;
  const cudaError_t e = ensure_smem_attr<kern>(S::smem);
  if (e) return e;
  int x = (cols + S::SH::G - 1) / S::SH::G;
  const int cap = 2 * current_device_sms();
  if (x > cap) x = cap;
  if (dep) return launch_dependent(kern, dim3(x, n), dim3(S::SH::threads), S::smem, st, jb, tw);
  kern<<<dim3(x, n), S::SH::threads, S::smem, st>>>(jb, tw);
  return cudaGetLastError();
}

}  // namespace gal
