// CTA-wide complex GEMM on CUDA cores with arbitrary operand strides.
//
//   C(i, j) = sum_k A(i, k) B(k, j)
//
// A(i, k) = a.p[i * a.si + k * a.sk] (conjugated if a.conj), B likewise, so
// every contraction of the effective-Hamiltonian networks is one call with no
// explicit transposes.  Products of small bonds, and all in FP64, read their
// operands where they are (gemm_direct); the others run in 64 x 64 output tiles
// (gemm_core), 16-deep K slices staged in shared memory, each thread owning 16
// complex FP32 accumulators.
#pragma once
#include "tjm_common.cuh"
#include "tjm_tc.cuh"

namespace tjm {

template <class T> struct MatA { const cx<T>* p; long long si, sk; int conj; };
template <class T> struct MatB { const cx<T>* p; long long sk, sj; int conj; };

template <class T> __host__ __device__ inline MatA<T> matA(const cx<T>* p, long long si, long long sk, int cj = 0) {
  MatA<T> m; m.p = p; m.si = si; m.sk = sk; m.conj = cj; return m;
}
template <class T> __host__ __device__ inline MatB<T> matB(const cx<T>* p, long long sk, long long sj, int cj = 0) {
  MatB<T> m; m.p = p; m.sk = sk; m.sj = sj; m.conj = cj; return m;
}

constexpr int GB_K = 16;
// bytes of shared memory reserved for GEMM staging (and, between GEMMs, for the factorizations)
constexpr int kSmemGemm = 32768;
// Rows of a staged slice are 2 elements longer than the tile: a k-contiguous operand
// is stored transposed, 16 lanes in 16 rows, and an unpadded row puts all of them in
// one bank.  Rows stay 16-byte aligned for the paired loads.
constexpr int GB_PAD = 2;
static_assert(GB_K * 2 * (64 + GB_PAD) * 8 <= kSmemGemm, "two slices fit");

// -x if neg, by its sign bit (a negation is an FP64 instruction otherwise)
__device__ __forceinline__ float flip(float x, int neg) { return __uint_as_float(__float_as_uint(x) ^ ((unsigned)neg << 31)); }
__device__ __forceinline__ double flip(double x, int neg) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)neg << 63));
}

// One 16-deep slice on a thread's FP32 accumulators: rows and columns come in
// pairs (one 16-byte load each), 32 apart; HR / HC pairs of them are in range.
// (Packed FP32 multiply-adds with A stored as (x, x, -y, y) ran 18 % faster on
// resident slices with two CTAs per SM, 10 % slower with one, and 20 % slower in
// whole runs, where the other CTA is mostly in a factorization.)
template <int TM, int HR, int HC>
__device__ __forceinline__ void slice_f32(int kn, const cx<float>* As, const cx<float>* Bs,
                                          cx<float> (&acc)[TM / 16][TM / 16]) {
  constexpr int LD = TM + GB_PAD;
#pragma unroll 4
  for (int kk = 0; kk < kn; ++kk) {
    float4 av[HR], bv[HC];
#pragma unroll
    for (int r = 0; r < HR; ++r) av[r] = *reinterpret_cast<const float4*>(As + kk * LD + 32 * r);
#pragma unroll
    for (int c = 0; c < HC; ++c) bv[c] = *reinterpret_cast<const float4*>(Bs + kk * LD + 32 * c);
#pragma unroll
    for (int r = 0; r < HR; ++r)
#pragma unroll
      for (int c = 0; c < HC; ++c) {
        cfma(acc[2 * r][2 * c], mk(av[r].x, av[r].y), mk(bv[c].x, bv[c].y));
        cfma(acc[2 * r][2 * c + 1], mk(av[r].x, av[r].y), mk(bv[c].z, bv[c].w));
        cfma(acc[2 * r + 1][2 * c], mk(av[r].z, av[r].w), mk(bv[c].x, bv[c].y));
        cfma(acc[2 * r + 1][2 * c + 1], mk(av[r].z, av[r].w), mk(bv[c].z, bv[c].w));
      }
  }
}

// One layout variant: AK = A's k index is contiguous (else its i index),
// BJ = B's j index is contiguous (else its k index); TM x TM output tiles
// (TM = 64 or 32).  Each thread loads TM/16 elements of A and of B per 16-deep
// slice; their tile coordinates are fixed per thread, so the loads need no
// per-element index arithmetic.  A tile at the edge of C computes only the part of
// it that exists, and the last slice only the k that are left.
//
// A warp covers 16 x 32 outputs of the tile (4 x 8 threads), (TM/16) x (TM/16)
// per thread, in halves of 32 rows and columns; a k costs 4 wavefronts of 16-byte
// loads per 64 FMA instructions.  The next slice (after the last, the next tile's) is
// in flight while a slice is multiplied, and nothing touches it before it is stored (a
// conjugation right after the load would wait for it there).  Bound by issue and by
// the barriers around the store of a slice: 160 to 170 of 256 flop per clock and SM
// with two CTAs at 320 x 128 x 64 and 128 x 64 x 320, 138 at 64 x 32 x 160, against 197 on
// slices that are already there (106 to 130 and 70 with whole 64 x 64 tiles, unpadded
// rows and a bounds check per load).  Copied
// element by element into two buffers (cp.async) in 128 x 64 tiles: 149 to 163, and 98
// instead of 138 at 64 x 32 x 160.  Strides between batches are 32-bit like the others (registers are short here).
template <bool AK, bool BJ, int TM>
__device__ __noinline__ void gemm_core(int batch, int M, int N, int K, const cx<float>* __restrict__ A, int sai, int sak,
                                       int ca, int sa, const cx<float>* __restrict__ B, int sbk, int sbj, int cb,
                                       int sb, cx<float>* C, int sci, int scj, int sc, char* smem) {
  constexpr int NQ = TM / 16;              // loads and accumulator rows / columns per thread
  constexpr int KS = TJM_THREADS / TM;     // k rows covered per load round in the i- / j-contiguous layouts
  constexpr int LD = TM + GB_PAD;
  cx<float>* As = reinterpret_cast<cx<float>*>(smem);            // [GB_K][LD]
  cx<float>* Bs = As + GB_K * LD;                            // [GB_K][LD]
  const int tid = threadIdx.x;
  // thread (ty, tx) owns rows 2 ty, 2 ty + 1 (+ 32 r) and columns likewise
  const int ty = ((tid >> 6) << 2) + ((tid >> 3) & 3), tx = ((tid >> 5) & 1) * 8 + (tid & 7);
  const int a_i = AK ? (tid >> 4) : (tid % TM);          // + 16 q   (AK)
  const int a_k = AK ? (tid & 15) : (tid / TM);          // + KS q   (!AK)
  const int b_j = BJ ? (tid % TM) : (tid >> 4);          // + 16 q   (!BJ)
  const int b_k = BJ ? (tid / TM) : (tid & 15);          // + KS q   (BJ)
  const int tm = (M + TM - 1) / TM, tn = (N + TM - 1) / TM;
  const int ntile = batch * tm * tn;
  const int nk = (K + GB_K - 1) / GB_K;
  cx<float> ra[NQ], rb[NQ];
  // Rows, columns and k beyond the operands are read from the last one that exists: what comes of them is
  // not stored (or, k, not reached), and a load costs one addition instead of a bounds check of its own.
  int oa[NQ], ob[NQ];
  const cx<float>* Ap = A;
  const cx<float>* Bp = B;
  auto tile = [&](int t) {
    const int bt = t / (tm * tn), r0 = t - bt * (tm * tn);
    const int i0 = (r0 / tn) * TM, j0 = (r0 % tn) * TM;
    Ap = A + bt * sa;
    Bp = B + bt * sb;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      oa[q] = min(i0 + a_i + (AK ? 16 * q : 0), M - 1) * sai;
      ob[q] = min(j0 + b_j + (BJ ? 0 : 16 * q), N - 1) * sbj;
    }
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      ra[q] = Ap[oa[q] + min(k0 + a_k + (AK ? 0 : KS * q), K - 1) * sak];
      rb[q] = Bp[ob[q] + min(k0 + b_k + (BJ ? KS * q : 0), K - 1) * sbk];
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      ra[q].y = flip(ra[q].y, ca);
      rb[q].y = flip(rb[q].y, cb);
      As[(a_k + (AK ? 0 : KS * q)) * LD + a_i + (AK ? 16 * q : 0)] = ra[q];
      Bs[(b_k + (BJ ? KS * q : 0)) * LD + b_j + (BJ ? 0 : 16 * q)] = rb[q];
    }
  };
  tile(0);
  load(0);
  for (int t = 0; t < ntile; ++t) {
    const int bt = t / (tm * tn), r0 = t - bt * (tm * tn);
    const int i0 = (r0 / tn) * TM, j0 = (r0 % tn) * TM;
    cx<float>* Cp = C + bt * sc;
    const int mr = M - i0 < TM ? M - i0 : TM, nc = N - j0 < TM ? N - j0 : TM;
    cx<float> acc[NQ][NQ];
#pragma unroll
    for (int r = 0; r < NQ; ++r)
#pragma unroll
      for (int c = 0; c < NQ; ++c) acc[r][c] = czero<float>();
    for (int ks = 0; ks < nk; ++ks) {
      __syncthreads();
      store();
      __syncthreads();
      const int kn = K - ks * GB_K < GB_K ? K - ks * GB_K : GB_K;
      if (ks + 1 < nk) {
        load((ks + 1) * GB_K);
      } else if (t + 1 < ntile) {
        tile(t + 1);
        load(0);
      }
      const cx<float>* Aw = As + 2 * ty;
      const cx<float>* Bw = Bs + 2 * tx;
      if (TM == 32 || (mr <= 32 && nc <= 32)) slice_f32<TM, 1, 1>(kn, Aw, Bw, acc);
      else if (mr <= 32) slice_f32<TM, 1, TM / 32>(kn, Aw, Bw, acc);
      else if (nc <= 32) slice_f32<TM, TM / 32, 1>(kn, Aw, Bw, acc);
      else slice_f32<TM, TM / 32, TM / 32>(kn, Aw, Bw, acc);
    }
#pragma unroll
    for (int r = 0; r < NQ; ++r) {
      const int i = i0 + 32 * (r >> 1) + 2 * ty + (r & 1);
      if (i >= M) continue;
#pragma unroll
      for (int c = 0; c < NQ; ++c) {
        const int j = j0 + 32 * (c >> 1) + 2 * tx + (c & 1);
        if (j >= N) continue;
        Cp[i * sci + j * scj] = acc[r][c];
      }
    }
  }
  __syncthreads();
}

// Small products: every thread forms whole outputs, reading its operands where
// they are (the working set of a small bond sits in L1 and L2), so there is no
// staging, no barrier before the last and no padding; consecutive threads own
// consecutive j of as many rows as fit the CTA, one index division per thread; rows
// longer than the CTA are dealt by flat index (taken one row at a time, the last pass over
// 320 columns has 64 of the 256 threads: FP64 64 x 320 x 128 7.28 M cycles with one CTA per SM
// instead of 5.66 M, 11.8 instead of 10.8 M with two).
// Bound by instruction issue (an output's index arithmetic used to cost as much as
// eight of its multiply-adds; two or four outputs of a thread along together, for
// more loads in flight, were 10 % slower).
template <class T, bool CONJ>
__device__ __forceinline__ void direct_rows(int batch, int M, int N, int K, const cx<T>* __restrict__ A, int sai, int sak,
                                            int ca, long long sa, const cx<T>* __restrict__ B, int sbk, int sbj, int cb,
                                            long long sb, cx<T>* C, int sci, int scj, long long sc) {
  const int MB = batch * M;
  auto one = [&](int ib, int j) {
    const int bt = batch == 1 ? 0 : ib / M, i = ib - bt * M;
    const cx<T>* a = A + bt * sa + i * sai;
    const cx<T>* b = B + bt * sb + j * sbj;
    cx<T> acc = czero<T>();
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      cx<T> x = *a, y = *b;
      a += sak;
      b += sbk;
      if (CONJ) { x.y = flip(x.y, ca); y.y = flip(y.y, cb); }
      cfma(acc, x, y);
    }
    C[bt * sc + i * sci + j * scj] = acc;
  };
  if (N > TJM_THREADS) {
    for (int e = threadIdx.x; e < MB * N; e += TJM_THREADS) one(e / N, e % N);
    return;
  }
  const int rows = TJM_THREADS / N, ti = threadIdx.x / N, j = threadIdx.x - ti * N;
  if (ti >= rows) return;
  for (int ib = ti; ib < MB; ib += rows) one(ib, j);
}
template <class T>
__device__ __noinline__ void gemm_direct(int batch, int M, int N, int K, const cx<T>* __restrict__ A, int sai, int sak,
                                         int ca, long long sa, const cx<T>* __restrict__ B, int sbk, int sbj, int cb,
                                         long long sb, cx<T>* C, int sci, int scj, long long sc) {
  if (ca | cb) direct_rows<T, true>(batch, M, N, K, A, sai, sak, ca, sa, B, sbk, sbj, cb, sb, C, sci, scj, sc);
  else direct_rows<T, false>(batch, M, N, K, A, sai, sak, ca, sa, B, sbk, sbj, cb, sb, C, sci, scj, sc);
  __syncthreads();
}

// Which FP32 products are small: up to 8192 multiply-adds.  Two CTAs per SM, direct
// against tiled, in cycles: 40 x 16 x 8 2.7 k / 3.5 k, 32 x 16 x 16 3.1 / 3.6, 40 x 32 x 8
// 4.4 / 3.5, 64 x 16 x 16 5.4 / 4.9, 32 x 32 x 32 9.0 / 6.1, 128 x 32 x 16 19.6 / 9.9.  The
// one-pass form of the MPO block stands against two steps and goes to twice that.
// FP64 is bound by its unit, 2 multiply-adds per clock and SM, in which a lane without
// an output costs as much as one with: the direct form has none but in its last warp
// (40 x 16 x 8 19.7 k against 22.9 k cycles in tiles without padding and 213 k with, 80 x 32 x 16
// 145 / 153 / 424 k, 160 x 64 x 32 1178 / 1180 / 1257 k, means over two CTAs per SM).  At the largest
// products both are at the unit (bond 64, two CTAs per SM, the later one: 320 x 128 x 64 10.7 M cycles against
// 10.8 M in whole tiles, 128 x 64 x 320 10.7 / 10.7, 64 x 320 x 128 10.8 / 10.7; least possible 10.5), and with
// one CTA per SM the direct form waits a little on operands that L1 does not hold (5.67 / 5.44, 5.55 / 5.44, 5.66 / 5.39;
// least possible 5.24).  Whole FP64 runs at bond 64, one step of L = 16: 1.53 against 1.96 s with one
// trajectory per SM, 2.77 against 3.56 with two.  So every FP64 product takes it.
constexpr long long kDirectF32 = 8192, kOnePassF32 = 16384;

// Tile choice of the tiled form.  gemm_tile_rule == 0: always 64 x 64 tiles.
// == 1: 32 x 32 tiles when either output dimension is at most 32.
// The rule is a per-launch setting (see the kernel), picked by the host-side
// autotuner from timed launches.
__shared__ int gemm_tile_rule;

// Tensor-core state of the CTA (tjm_tc.cuh).  When enabled, every FP32 GEMM of
// at least tc_ctl.min_work complex multiply-adds runs on the tensor cores;
// smaller ones (chain ends, tiny bonds) stay on the CUDA cores, where one
// 128-row MMA tile would be mostly padding.
__shared__ tc::Ctl tc_ctl;

// TJM_TENSOR_CORES (per translation unit) decides whether the kernels built
// there carry the tcgen05 path at all.  A kernel image that holds any tcgen05
// instruction is granted a single resident CTA per SM (measured on GB300 with
// the occupancy API: the same 128-register, 256-thread trajectory kernel
// reports two without them), so the CUDA-core instantiations are compiled
// without it and the tensor-core ones live in translation units of their own.
#ifndef TJM_TENSOR_CORES
#define TJM_TENSOR_CORES 0
#endif

__device__ __forceinline__ bool use_tc(long long work) {
#if TJM_TENSOR_CORES
  return tc_ctl.enabled && work >= tc_ctl.min_work;
#else
  (void)work;
  return false;
#endif
}

template <bool AK, bool BJ>
__device__ __forceinline__ void gemm_layout(int batch, int M, int N, int K, MatA<float> A, long long sa, MatB<float> B,
                                            long long sb, cx<float>* C, int sci, int scj, long long sc, char* smem) {
  if (gemm_tile_rule == 1 && (M <= 32 || N <= 32))
    gemm_core<AK, BJ, 32>(batch, M, N, K, A.p, (int)A.si, (int)A.sk, A.conj, (int)sa, B.p, (int)B.sk, (int)B.sj, B.conj,
                          (int)sb, C, sci, scj, (int)sc, smem);
  else
    gemm_core<AK, BJ, 64>(batch, M, N, K, A.p, (int)A.si, (int)A.sk, A.conj, (int)sa, B.p, (int)B.sk, (int)B.sj, B.conj,
                          (int)sb, C, sci, scj, (int)sc, smem);
}

// Batched: for b < batch, operands offset by (sa, sb, sc) elements.
template <class T>
__device__ __forceinline__ void blk_gemm_batched(int batch, int M, int N, int K, MatA<T> A, long long sa, MatB<T> B,
                                                 long long sb, cx<T>* C, int sci, int scj, long long sc, char* smem) {
  if (M <= 0 || N <= 0) return;
  if constexpr (sizeof(T) == 4) {
    if (K > 0 && use_tc((long long)M * N * K)) {
      tc::TcA ta = {};
      ta.si = A.si; ta.sk = A.sk; ta.conj = A.conj;
      tc::TcB tb = {};
      tb.sk = B.sk; tb.sj = B.sj; tb.conj = B.conj;
      for (int b = 0; b < batch; ++b) {
        ta.p = A.p + b * sa;
        tb.p = B.p + b * sb;
        tc::cgemm(&tc_ctl, M, N, K, mk(1.f, 0.f), ta, tb, C + b * sc, sci, scj, false, smem);
      }
      return;
    }
    if ((long long)batch * M * N * K > kDirectF32) {
      const bool ak = A.sk == 1;
      const bool bj = (B.sj == 1) || (B.sk != 1);
      if (ak && bj) gemm_layout<true, true>(batch, M, N, K, A, sa, B, sb, C, sci, scj, sc, smem);
      else if (ak) gemm_layout<true, false>(batch, M, N, K, A, sa, B, sb, C, sci, scj, sc, smem);
      else if (bj) gemm_layout<false, true>(batch, M, N, K, A, sa, B, sb, C, sci, scj, sc, smem);
      else gemm_layout<false, false>(batch, M, N, K, A, sa, B, sb, C, sci, scj, sc, smem);
      return;
    }
  }
  gemm_direct<T>(batch, M, N, K, A.p, (int)A.si, (int)A.sk, A.conj, sa, B.p, (int)B.sk, (int)B.sj, B.conj, sb, C, sci, scj,
                 sc);
}

template <class T>
__device__ __forceinline__ void blk_gemm(int M, int N, int K, MatA<T> A, MatB<T> B, cx<T>* C, int sci, int scj,
                                         char* smem) {
  blk_gemm_batched<T>(1, M, N, K, A, 0, B, 0, C, sci, scj, 0, smem);
}

// out[p][o][q] = sum_i Wm[o][i] in[p][i][q] -- the small MPO contraction
// between the two big GEMMs of an effective-Hamiltonian application.
// Wm (O x I <= 32 x 32, complex double, row-major) is compressed into a
// row-sparse list in shared memory (the MPO is mostly zeros), then every thread
// handles (p, q) pairs reading only the inputs that matter.
//
// A scalar `shift` can be added on nsh diagonal entries (o, i) =
// (so0 + t * so_step, si0 + t * si_step), t < nsh: this is how a constant
// times the identity rides on an MPO's on-site channel.
// Row-sparse form of Wm (+ the shift entries) in shared memory at csr: row o's
// entries are val / col [o * I .. re[o]), with val [O * I], col [O * I], re [O].
// One warp per row, one lane per column (O, I <= 32); zeros are recognised by
// their bits, off the FP64 unit.  One thread per row, walking its columns twice,
// was several thousand cycles in front of every effective-Hamiltonian
// application.  Ends with a barrier.
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
template <class T>
__device__ __forceinline__ void wcsr_build(int O, int I, const cx<double>* Wm, char* csr, double shift, int nsh,
                                           int so0, int so_step, int si0, int si_step) {
  cx<T>* val = reinterpret_cast<cx<T>*>(csr);
  int* col = reinterpret_cast<int*>(val + O * I);
  int* re = col + O * I;
  __syncthreads();
  const int i = threadIdx.x & 31;
  for (int o = threadIdx.x >> 5; o < O; o += TJM_WARPS) {
    cx<double> w = czero<double>();
    if (i < I) w = Wm[o * I + i];
    if (o >= so0 && !is_zero(shift)) {   // this row's shift entry, if any
      const int t = (o - so0) / so_step;
      if (o - so0 == t * so_step && t < nsh && i == si0 + t * si_step) w.x += shift;
    }
    const bool nz = !is_zero(w.x) || !is_zero(w.y);
    const unsigned m = __ballot_sync(0xffffffffu, nz);
    if (nz) {
      const int pos = o * I + __popc(m & ((1u << i) - 1));
      val[pos] = cvt<T>(w);
      col[pos] = i;
    }
    if (i == 0) re[o] = o * I + __popc(m);
  }
  __syncthreads();
}

template <class T>
__device__ __noinline__ void blk_wapply(int P, int O, int I, int Q, const cx<double>* Wm, const cx<T>* __restrict__ in,
                                        long long sip, long long sii, cx<T>* __restrict__ out, long long sop, long long soo,
                                        char* smem, double shift = 0.0, int nsh = 0, int so0 = 0, int so_step = 1,
                                        int si0 = 0, int si_step = 1) {
  const cx<T>* val = reinterpret_cast<const cx<T>*>(smem);
  const int* col = reinterpret_cast<const int*>(val + O * I);
  const int* re = col + O * I;
  wcsr_build<T>(O, I, Wm, smem, shift, nsh, so0, so_step, si0, si_step);
  if (P * Q < 2 * TJM_THREADS) {       // fewer (p, q) pairs than keep the CTA busy: one output per thread
    for (int e = threadIdx.x; e < P * O * Q; e += TJM_THREADS) {
      const int r = e / Q, q = e - r * Q, p = r / O, o = r - p * O;
      const cx<T>* src = in + p * sip + q;
      cx<T> acc = czero<T>();
      const int e1 = re[o];
      for (int z = o * I; z < e1; ++z) cfma(acc, val[z], src[col[z] * sii]);
      out[p * sop + o * soo + q] = acc;
    }
    __syncthreads();
    return;
  }
  // four (p, q) pairs at a time: the row-sparse loops cannot be unrolled, so the loads in flight are those of
  // the pairs (one pair at a time: 65k cycles per block at bond 64, all latency)
  const int tot = P * Q;
  for (int e0 = threadIdx.x; e0 < tot; e0 += 4 * TJM_THREADS) {
    const cx<T>* src[4];
    cx<T>* dst[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * TJM_THREADS < tot ? e0 + u * TJM_THREADS : e0;
      const int p = e / Q, q = e - p * Q;
      src[u] = in + p * sip + q;
      dst[u] = out + p * sop + q;
    }
    const int nu = (tot - e0 + TJM_THREADS - 1) / TJM_THREADS;
    for (int o = 0; o < O; ++o) {
      cx<T> acc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = czero<T>();
      const int e1 = re[o];
      for (int z = o * I; z < e1; ++z) {
        const cx<T> w = val[z];
        const long long off = col[z] * sii;
#pragma unroll
        for (int u = 0; u < 4; ++u) cfma(acc[u], w, src[u][off]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) dst[u][o * soo] = acc[u];
    }
  }
  __syncthreads();
}

// y[(x t)][j] = sum_(v b) [sum_(w s) Wm[(t v)][(w s)] t1[x][(w s)][b]] R[(v b)][j]
// for x < P, t < dd, j < chr: the MPO contraction and the second GEMM of an
// effective-Hamiltonian application of a small bond in one pass (kOnePassF32),
// as sum_z val[z] (t1 R): the entries of the block that meet output row t, each
// times one row of t1 R_v, with no intermediate and no barrier between.
template <class T>
__device__ __noinline__ void blk_wgemm_small(int P, int dd, int Dr, int I, int chr, const cx<double>* Wm,
                                             const cx<T>* __restrict__ t1, const cx<T>* __restrict__ R,
                                             cx<T>* __restrict__ y, char* smem, double shift, int nsh, int so0,
                                             int so_step, int si0, int si_step) {
  const int O = dd * Dr, M = P * dd, N = chr;
  const cx<T>* val = reinterpret_cast<const cx<T>*>(smem);
  const int* col = reinterpret_cast<const int*>(val + O * I);
  const int* re = col + O * I;
  wcsr_build<T>(O, I, Wm, smem, shift, nsh, so0, so_step, si0, si_step);
  const int rows = N < TJM_THREADS ? TJM_THREADS / N : 1;
  const int ti = threadIdx.x / N, j = threadIdx.x - ti * N;
  if (ti < rows && j < N) {
    for (int i = ti; i < M; i += rows) {
      const int x = i / dd, t = i - x * dd;
      const cx<T>* tx = t1 + x * I * chr;
      cx<T> acc = czero<T>();
      for (int v = 0; v < Dr; ++v) {
        const int o = t * Dr + v, z1 = re[o];
        const cx<T>* rv = R + v * chr * chr + j;
        for (int z = o * I; z < z1; ++z) {
          const cx<T>* src = tx + col[z] * chr;
          const cx<T>* r = rv;
          cx<T> s = czero<T>();
#pragma unroll 4
          for (int b = 0; b < chr; ++b) {
            cfma(s, src[b], *r);
            r += chr;
          }
          cfma(acc, val[z], s);
        }
      }
      y[i * N + j] = acc;
    }
  }
  __syncthreads();
}

}  // namespace tjm
