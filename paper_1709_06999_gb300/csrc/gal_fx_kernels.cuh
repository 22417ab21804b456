// Row and column passes of the double-precision path on 64-bit integers
// (gal_fx.cuh): the passes of gal_kernels.cuh with each sequence brought to a
// common power of two before its transform.  Images, F1 and the window are
// doubles.  Measured against the same passes in FP64 arithmetic (which kept the
// FP64 pipe 83 % busy): row pass of 4096^2 pixels, 61 columns kept, 481 -> 102
// us; of 2048^2 pixels, 413 columns kept, 161 -> 39 us; column pass of 4096 x 61
// 41 -> 12 us, of 2048 x 413 66 -> 19 us.  (With one scale for all stages, which
// lost precision, the row passes took 100 and 38 us.)
#pragma once

#include "gal_fx.cuh"
#include "gal_kernels.cuh"

namespace gal {

// Rows of 2^(LG+1) pixels as complex sequences of M = 2^LG points, G rows to a
// block of at least 128 threads.  One buffer of arriving rows beside the two
// work buffers, not a ring of two that double as work buffers, lets two blocks
// of 4096-pixel rows share an SM (116 KB each): 113 -> 100 us.  (Two rows of
// 2048 pixels to a block of 256 threads: 1 % slower than one to 128.)
template <int LG> struct FxRowShape {
  static constexpr int M = 1 << LG, N = 2 * M;
  using SH = Shape3<double, M, N, 128, 8>;
  static constexpr int G = SH::G, RS = SH::RS;
  static constexpr int ntab = fx_ntab<M, 1024>();
  // header (barrier, reduction scratch, row scales), factors, two work buffers, the
  // image rows as they arrive
  static constexpr int kHead = 512;
  static constexpr size_t work = (size_t)G * RS * sizeof(fx2);
  static constexpr size_t smem(bool image) {
    return kHead + (size_t)ntab * sizeof(fxtw) + 2 * work + (image ? (size_t)G * N * sizeof(double) : 0);
  }
};

// Row pass (see row_fft3_kernel).  Persistent blocks own row groups.  Image
// rows come by bulk copy into a buffer of their own, which is free again as
// soon as the rows are in registers, so the next group is in flight during the
// whole transform; SWEEP: the rows are generated from the profile.
template <int LG, bool SWEEP, int K, bool BEAM = false>
__global__ void __launch_bounds__(FxRowShape<LG>::SH::threads,
                                  min_blocks_128regs<FxRowShape<LG>::SH::threads>())
row_fx_kernel(const __grid_constant__ Jobs<RowJob<double>, K> jobs, const double2* __restrict__ twd,
              int* __restrict__ err) {
  // The column pass may be scheduled as our blocks retire.  No wait comes first, and
  // the image is read before one: this kernel is launched normally or after a kernel
  // that is (see launch_dependent).
  grid_dep_launch();
  using S = FxRowShape<LG>;
  using SH = typename S::SH;
  using P = typename SH::P;
  constexpr int M = S::M, N = S::N, TT = P::T, G = S::G, RS = S::RS;
  const RowJob<double>& jb = jobs.j[K == 1 ? 0 : blockIdx.y];
  const double* __restrict__ image = jb.image;
  const double* __restrict__ beam = BEAM ? jb.beam : nullptr;
  double2* __restrict__ F1 = jb.F1;
  const fxtw* __restrict__ tw = reinterpret_cast<const fxtw*>(twd + TwTab<double, 8>::fx(N));
  const fxtw* __restrict__ tws = reinterpret_cast<const fxtw*>(twd + TwTab<double, 8>::fx_row(N));
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  unsigned* red_max = reinterpret_cast<unsigned*>(smem_raw + 32);   // one per warp, <= 16
  unsigned* red_sum = reinterpret_cast<unsigned*>(smem_raw + 96);
  int* row_q = reinterpret_cast<int*>(smem_raw + 192);              // scale per row of the group, <= 64
  fxtw* tab = reinterpret_cast<fxtw*>(smem_raw + S::kHead);
  fx2* A0 = reinterpret_cast<fx2*>(tab + S::ntab);
  fx2* B0 = A0 + G * RS;
  double* slot = reinterpret_cast<double*>(B0 + G * RS);
  static_assert(G <= 64 && SH::threads <= 512, "header");
  const int g = threadIdx.x / TT, t = threadIdx.x - g * TT;
  constexpr bool EVEN = even_rows<double, SWEEP, BEAM>(N);  // rows 0 .. N/2 only
  constexpr int LD = EVEN ? kEvenRows(N) : N;
  constexpr int ngroups = EVEN ? (M + 1 + G - 1) / G : N / G;
  const uint32_t half_bytes = (uint32_t)(M * sizeof(double));
  auto issue = [&](int grp) {  // thread 0 only
    if (grp >= ngroups) return;
    mbar_arrive_expect_tx(bar, 2u * half_bytes * (uint32_t)G);
    for (int rl = 0; rl < G; ++rl) {
      const double* src = image + (size_t)(((grp * G + rl) + M) & (N - 1)) * N;
      double* dst = slot + (size_t)rl * N;
      bulk_load(dst, src + M, half_bytes, bar);
      bulk_load(dst + M, src, half_bytes, bar);
    }
  };
  if constexpr (!SWEEP) {
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      mbar_init_fence();
      issue(blockIdx.x);
    }
  }
  for (int i = threadIdx.x; i < S::ntab; i += blockDim.x) tab[i] = ldg_tw(tws + i);
  const Bounds bd = block_bounds(jb.rho2, jb.S, N);  // synchronises
  const bool pruned = P::nstage >= 2 && bd.Kc <= P::Nsl;
  if constexpr (BEAM) grid_dep_wait();  // the beam tables
  uint32_t phase = 0;
  for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x, phase ^= 1u) {
    const int row = grp * G + g;
    double2 z[8];
    if constexpr (SWEEP) {
      sweep_row<double, M, 8>(z, jb.I, jb.sp, row, t, reinterpret_cast<double*>(B0 + g * RS),
                              !EVEN || row <= M);
    } else {
      // a wait that gives up (never expected) is reported, and the block ends:
      // its one copy in flight is the one it has waited for
      const bool ok = mbar_wait(bar, phase);
      if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
          atomicOr(err, 2);
          mbar_wait(bar, phase);
        }
        return;
      }
#pragma unroll
      for (int r = 0; r < 8; ++r) z[r] = reinterpret_cast<const double2*>(slot + (size_t)g * N)[t + r * TT];
      __syncthreads();  // the rows are in registers: the next group may land
      if (threadIdx.x == 0) {
        fence_proxy_async_smem();
        issue(grp + gridDim.x);
      }
    }
    if constexpr (BEAM) {
#pragma unroll
      for (int r = 0; r < 8; ++r) z[r] = beam_pair(z[r], beam, N, row, t + r * TT);
    }
    fx2 v[8];
    FxScale sc = fx_load<TT>(z, v, red_max, red_sum);
    fx2* A = A0 + g * RS;
    fx2* B = B0 + g * RS;
    if (t == 0) {  // of the last stage: shift, growth, exponent of its outputs
      FxScale end = sc;
#pragma unroll
      for (int i = 1; i < P::nstage - 1; ++i) end.stage();
      const FxLast l = fx_last<M>(end);
      row_q[g] = sc.bad ? (kFxBad + 1) * 16 : end.q * 16 + l.g * 4 + l.r;
    }
    if constexpr (S::ntab > 0) FxHead<M, 0, true>::run(v, A, B, t, tab, sc);
    else FxHead<M, 0, false>::run(v, A, B, t, tws, sc);
    fx2* in = last_input<M, 8>(A, B);
    if (!pruned) {
      fx_last_full<M>(v, in, t, tws, fx_last<M>(sc).g);
      in = in == A ? B : A;
      store_full<M, 8>(v, in, t);
      __syncthreads();
    }
    // Bin by bin with the G rows of the group side by side, so that neighbouring
    // lanes fill the sectors of a column of F1 (column-major: bin k of row i at
    // F1[k LD + i]); row gg's buffer lies (gg - g) RS from ours.
    const fx2* in0 = in - g * RS;
    for (int o = threadIdx.x; o < bd.Kc * G; o += G * TT) {
      const int k = o / G, gg = o - k * G;
      if (EVEN && grp * G + gg > M) continue;
      const fx2* x = in0 + gg * RS;
      const int rq = row_q[gg], r = rq & 3, q = (rq >> 4) + r;
      fx2 zk, zmk;
      if (pruned) {
        fx_pruned_pair<M>(x, k, tws, (rq >> 2) & 3, zk, zmk);
      } else {
        zk = x[pad3<8>(k & (M - 1))];
        zmk = x[pad3<8>((M - k) & (M - 1))];
      }
      const fx2 X2 = fx_r2c_unpack2(fx_shr(zk, r), fx_shr(zmk, r), ldg_tw(tw + k));
      F1[(size_t)k * LD + grp * G + gg] = fx_to(X2, q - 1);
    }
    __syncthreads();  // every read of the work buffers and scales is done
  }
}

template <int LG> struct FxColShape {
  static constexpr int N = 1 << LG;
  using SH = ColShape3<double, N, 8>;
  static constexpr int ntab = fx_ntab<N, 2048>();
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
  const fxtw* __restrict__ tws = reinterpret_cast<const fxtw*>(twd + TwTab<double, 8>::fx_col(N));
  grid_dep_launch();  // the gather may start its prologue on the SMs we leave idle
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned* red_max = reinterpret_cast<unsigned*>(smem_raw);
  unsigned* red_sum = reinterpret_cast<unsigned*>(smem_raw + 64);
  int* col_q = reinterpret_cast<int*>(smem_raw + 128);
  fxtw* tab = reinterpret_cast<fxtw*>(smem_raw + S::kHead);
  fx2* base = reinterpret_cast<fx2*>(tab + S::ntab);
  static_assert(G <= 256 && SH::threads <= 512, "header");
  const int g = threadIdx.x / TT, t = threadIdx.x - g * TT;
  for (int i = threadIdx.x; i < S::ntab; i += blockDim.x) tab[i] = ldg_tw(tws + i);
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
    for (int r = 0; r < 8; ++r) z[r] = act ? F1[f1_index(jb.even, N, c, t + r * TT)] : make_double2(0.0, 0.0);
    fx2 v[8];
    FxScale sc = fx_load<TT>(z, v, red_max, red_sum);
    if constexpr (S::ntab > 0) FxHead<N, 0, true>::run(v, A, B, t, tab, sc);
    else FxHead<N, 0, false>::run(v, A, B, t, tws, sc);
    const int lg = fx_last<N>(sc).g, cq = sc.bad ? kFxBad : sc.q;
    fx2* in = last_input<N, 8>(A, B);
    if (pruned) {
      for (int j = t; j <= kmax; j += TT) {
        fx2 xj, xmj;
        fx_pruned_pair<N>(in, j, tws, lg, xj, xmj);
        if (act) {
          Gw[(size_t)(kmax + j) * ncol + c] = fx_to(xj, cq);
          if (j > 0) Gw[(size_t)(kmax - j) * ncol + c] = fx_to(xmj, cq);
        }
      }
    } else {
      fx_last_full<N>(v, in, t, tws, lg);
      fx2* o = in == A ? B : A;
      store_full<N, 8>(v, o, t);
      if (t == 0) col_q[g] = cq;
      __syncthreads();
      const fx2* o0 = o - (size_t)g * RS;
      for (int q = threadIdx.x; q < bd.nrw * G; q += G * TT) {
        const int rr = q / G, gg = q - rr * G;
        if (c0 + gg < ncol)
          Gw[(size_t)rr * ncol + c0 + gg] =
              fx_to(o0[(size_t)gg * RS + pad3<8>((bd.r0 + rr + N / 2) & (N - 1))], col_q[gg]);
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
  const int per_sm = resident_blocks<kern>(S::SH::threads, smem);
  int x = (per_sm * current_device_sms() * (scale < 1 ? 1 : scale) + n - 1) / n;
  constexpr int rows = even_rows<double, SWEEP, BEAM>(S::N) ? S::M + 1 : S::N;
  if (x > (rows + S::G - 1) / S::G) x = (rows + S::G - 1) / S::G;
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
