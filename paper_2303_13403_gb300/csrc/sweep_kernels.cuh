#pragma once
// PQMC sweep kernels for GB300 (sm_103a).
//
// This header holds the device code and the launch templates; each
// sweep_*.cu translation unit instantiates the kernels of one path (FP64,
// reduced precision, reduced precision with dense chain packing) so the three
// compile in parallel, and sweep.cu holds the precision dispatch.
//
// One CTA owns one Markov chain for the whole launch and runs complete
// sweeps: Metropolis flips of the Ising fields with delayed (blocked)
// updates, slice wrapping, QR stabilisation of the B_L / B_R stacks, and the
// measurement at the middle slice.  Chains are independent, so a batch of
// chains of uneven size is one launch with one CTA per chain.
//
// Paper: Method section (PQMC estimator, Eq. (1) HS of the Gutzwiller
// factor) and honeycomb Hubbard section (Eq. (2), trial state of Eq. (3)).
//
// Conventions (shared with the header):
//   slices tau = 0..Ltau+1; 0 and Ltau+1 carry the Gutzwiller fields;
//   B_tau = e^{-dtau K} e^{V(s_tau)} (interaction), e^{V(s_tau)} (Gutzwiller);
//   G(tau) = 1 - B_R(tau) (B_L(tau) B_R(tau))^{-1} B_L(tau),
//   B_R(tau) = B_tau ... B_0 P,  B_L(tau) = P^T B_{Ltau+1} ... B_{tau+1}.
//   A flip of s_{tau,i} is proposed on G(tau-1): R_sigma = 1 + Delta_sigma (1 - G_ii).
//
// Precision: T (double or float) is the path precision of G, the ratios,
// the wrap, the delayed updates, the products that advance the stack blocks
// and the assembly of G from them.  The QR of the stack blocks (Householder on
// the FP64 path; Cholesky on the reduced paths, Householder where that breaks
// down), the product Q_L^T Q_R, its inverse and the log-determinant / sign are
// FP64 in every path.  FP64 products run as exact digit products on the tensor
// cores where that is faster (digit_gemm.cuh).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/pqmc.h"
#include "chain.h"
#include "model.h"
#include "philox.cuh"
#include "tc_gemm.cuh"
#include "digit_gemm.cuh"

namespace pqmc {


// --------------------------------------------------------------------------
// small CTA helpers

static __device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
static __device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Loop over a 2D index range with warps along rows and lanes along columns
// (no runtime integer division in the element loops).
#define PQMC_FOR_2D(i, i0, i1, j, j0, j1)                                          \
  for (int i = (i0) + (int)(threadIdx.x >> 5); i < (i1); i += (int)(blockDim.x >> 5)) \
    for (int j = (j0) + (int)(threadIdx.x & 31); j < (j1); j += 32)

// Sum / max over the CTA; every thread gets the result.  red holds >= 32 doubles.
static __device__ double cta_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = lane < nw ? red[lane] : 0.0;
  return warp_sum(t);
}
static __device__ double cta_max(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_max(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = lane < nw ? red[lane] : 0.0;
  return warp_max(t);
}

// --------------------------------------------------------------------------
// CTA-wide register-tiled GEMM: C = A B, A(i,k) = A[i*sai + k*sak],
// B(k,j) = B[k*sbk + j*sbj]; inputs are converted to the accumulation type T
// on load; the epilogue receives (i, j, value).  Every thread owns 4x4
// outputs.  When A is contiguous in i and B in j (sai = sbj = 1, strides and
// pointers 16-byte aligned, same type as T) the operands are read with
// 16-byte vector loads.

struct EpiStore {
  static constexpr bool kRow4 = true;   // supports 4 contiguous outputs of a row at once
  template <typename T, typename TC> __device__ void operator()(TC* C, int sci, int scj, int i, int j, T v) const {
    C[(long)i * sci + (long)j * scj] = (TC)v;
  }
  template <typename T> __device__ void row4(T* c, const T v[4]) const { c[0] = v[0]; c[1] = v[1]; c[2] = v[2]; c[3] = v[3]; }
};
struct EpiSub {
  static constexpr bool kRow4 = true;
  template <typename T, typename TC> __device__ void operator()(TC* C, int sci, int scj, int i, int j, T v) const {
    C[(long)i * sci + (long)j * scj] -= (TC)v;
  }
  template <typename T> __device__ void row4(T* c, const T v[4]) const {
    c[0] -= v[0]; c[1] -= v[1]; c[2] -= v[2]; c[3] -= v[3];
  }
};
template <typename E, typename = void> struct HasRow4 { static constexpr bool value = false; };
template <typename E> struct HasRow4<E, std::void_t<decltype(E::kRow4)>> { static constexpr bool value = E::kRow4; };

template <typename T> struct Vec4;
template <> struct Vec4<float> {
  __device__ static void load(const float* p, float v[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  }
  static constexpr int kAlign = 4;
};
template <> struct Vec4<double> {
  __device__ static void load(const double* p, double v[4]) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    const double2 y = *reinterpret_cast<const double2*>(p + 2);
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
  }
  static constexpr int kAlign = 2;
};

template <typename T>
__device__ __forceinline__ bool vec_ok(const T* p, long stride) {
  return ((reinterpret_cast<uintptr_t>(p) & 15) == 0) && (stride % Vec4<T>::kAlign == 0);
}

template <typename T, typename TA, typename TB, typename TC, typename Epi>
__device__ void cta_gemm(int M, int Nn, int K, const TA* A, int sai, int sak, const TB* B, int sbk, int sbj,
                         TC* C, int sci, int scj, Epi epi) {
  const int tm = (M + 3) >> 2, tn = (Nn + 3) >> 2;
  bool vec = false, vec_row = false, st_row = false;
  if constexpr (std::is_same<T, TA>::value && std::is_same<T, TB>::value) {
    vec = sai == 1 && sbj == 1 && vec_ok<T>((const T*)A, sak) && vec_ok<T>((const T*)B, sbk) &&
          (M % 4 == 0) && (Nn % 4 == 0);
    // A contiguous along k (row-major): 4 x 4 blocks of A per four k-steps
    vec_row = !vec && sak == 1 && sbj == 1 && vec_ok<T>((const T*)A, sai) && vec_ok<T>((const T*)B, sbk) &&
              (M % 4 == 0) && (Nn % 4 == 0) && (K % 4 == 0);
  }
  if constexpr (std::is_same<T, TC>::value && HasRow4<Epi>::value) {
    st_row = scj == 1 && vec_ok<T>((const T*)C, sci) && (Nn % 4 == 0);
  }
  for (int t = threadIdx.x; t < tm * tn; t += blockDim.x) {
    const int i0 = (t / tn) << 2, j0 = (t % tn) << 2;
    T acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[r][q] = T(0);
    if constexpr (std::is_same<T, TA>::value && std::is_same<T, TB>::value) {
      if (vec) {
        const T* pa = (const T*)A + i0;
        const T* pb = (const T*)B + j0;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
          T a[4], b[4];
          Vec4<T>::load(pa + (long)k * sak, a);
          Vec4<T>::load(pb + (long)k * sbk, b);
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r], b[q], acc[r][q]);
        }
      }
    }
    if constexpr (std::is_same<T, TA>::value && std::is_same<T, TB>::value) {
      if (vec_row) {
        const T* pa = (const T*)A + (long)i0 * sai;
        const T* pb = (const T*)B + j0;
        for (int k = 0; k < K; k += 4) {
          T a[4][4], b[4][4];
#pragma unroll
          for (int r = 0; r < 4; ++r) Vec4<T>::load(pa + (long)r * sai + k, a[r]);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) Vec4<T>::load(pb + (long)(k + kk) * sbk, b[kk]);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r][kk], b[kk][q], acc[r][q]);
        }
      }
    }
    if (!vec && !vec_row) {
      for (int k = 0; k < K; ++k) {
        T a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) a[r] = (i0 + r < M) ? (T)A[(long)(i0 + r) * sai + (long)k * sak] : T(0);
#pragma unroll
        for (int q = 0; q < 4; ++q) b[q] = (j0 + q < Nn) ? (T)B[(long)k * sbk + (long)(j0 + q) * sbj] : T(0);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r], b[q], acc[r][q]);
      }
    }
    if constexpr (std::is_same<T, TC>::value && HasRow4<Epi>::value) {
      if (st_row) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (i0 + r < M) epi.row4((T*)C + (long)(i0 + r) * sci + j0, acc[r]);
        continue;
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i0 + r < M && j0 + q < Nn) epi(C, sci, scj, i0 + r, j0 + q, acc[r][q]);
  }
}

// The same in FP32 for operands laid out in whole vectors, which is how the
// reduced paths keep theirs: A(i,k) = A[i + k lda], or with kRowA A[i lda + k];
// B(k,j) = B[k ldb + j], C row-major; lda, ldb, ldc multiples of four, bases
// 16-byte aligned, and rows of A and B readable up to the next multiple of
// four elements (whatever they hold there).  One layout per instantiation:
// no fallback to scalar loads inside, so the loop keeps its registers and the
// phase its code small.  (162 sites: rank-21 update, stack products and
// assembly took 29 + 22 + 24 Mcycles per 42 slices with scalar loads and a
// bounds check per element)
template <bool kRowA, typename Epi>
__device__ __forceinline__ void cta_gemm_f32(int M, int Nn, int K, const float* A, int lda, const float* B, int ldb,
                                             float* C, int ldc, Epi epi) {
  const int tm = (M + 3) >> 2, tn = (Nn + 3) >> 2;
  for (int t = threadIdx.x; t < tm * tn; t += blockDim.x) {
    const int i0 = (t / tn) << 2, j0 = (t % tn) << 2;
    float acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[r][q] = 0.f;
    const float* pb = B + j0;
    if constexpr (!kRowA) {
      const float* pa = A + i0;
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        float a[4], b[4];
        Vec4<float>::load(pa + (long)k * lda, a);
        Vec4<float>::load(pb + (long)k * ldb, b);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r], b[q], acc[r][q]);
      }
    } else {
      // 4 x 4 blocks of A per four k-steps (the last rows of a ragged M are read again)
      const int l1 = min(1, M - 1 - i0) * lda, l2 = min(2, M - 1 - i0) * lda, l3 = min(3, M - 1 - i0) * lda;
      const float* pa = A + (long)i0 * lda;
      int k = 0;
      for (; k + 4 <= K; k += 4) {
        float a[4][4], b[4][4];
        Vec4<float>::load(pa + k, a[0]);
        Vec4<float>::load(pa + l1 + k, a[1]);
        Vec4<float>::load(pa + l2 + k, a[2]);
        Vec4<float>::load(pa + l3 + k, a[3]);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) Vec4<float>::load(pb + (long)(k + kk) * ldb, b[kk]);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r][kk], b[kk][q], acc[r][q]);
      }
#pragma unroll 1
      for (; k < K; ++k) {
        float a[4], b[4];
        a[0] = pa[k];
        a[1] = pa[l1 + k];
        a[2] = pa[l2 + k];
        a[3] = pa[l3 + k];
        Vec4<float>::load(pb + (long)k * ldb, b);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r], b[q], acc[r][q]);
      }
    }
    if constexpr (HasRow4<Epi>::value) {
      if (j0 + 4 <= Nn) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (i0 + r < M) epi.row4(C + (long)(i0 + r) * ldc + j0, acc[r]);
        continue;
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i0 + r < M && j0 + q < Nn) epi(C, ldc, 1, i0 + r, j0 + q, acc[r][q]);
  }
}

// --------------------------------------------------------------------------
// Split-precision tensor-core GEMM (the BF16X3 path): C = A B for FP32 A, B
// with every operand split as x = hi + lo, hi = bf16(x), lo = bf16(x - hi),
// and C = A_hi B_hi + A_hi B_lo + A_lo B_hi accumulated in FP32 by
// mma.sync.m16n8k16 (Henry, Tang & Heinecke 2019 use the same split).  Each
// warp owns 16 x 32 output tiles; operands are read with arbitrary strides
// (zero outside the matrix) and split on the fly.

static __device__ __forceinline__ void split_bf16(float v, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(v);
  l = __float2bfloat16_rn(v - __bfloat162float(h));
}

static __device__ __forceinline__ uint32_t pack2(__nv_bfloat16 first, __nv_bfloat16 second) {
  return (uint32_t)__bfloat16_as_ushort(first) | ((uint32_t)__bfloat16_as_ushort(second) << 16);
}

static __device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <typename Epi>
__device__ void cta_gemm_bf16x3(int M, int Nn, int K, const float* A, int sai, int sak, const float* B, int sbk,
                                int sbj, float* C, int sci, int scj, Epi epi) {
  // each warp owns a 16 x 32 output tile: the A fragment of a k-step is
  // loaded and split once and used by the four 16 x 8 products of the tile
  constexpr int kNs = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int tm = (M + 15) >> 4, tn = (Nn + 8 * kNs - 1) / (8 * kNs);
  auto a_at = [&](int r, int k) -> float { return (r < M && k < K) ? A[(long)r * sai + (long)k * sak] : 0.0f; };
  auto b_at = [&](int k, int n) -> float { return (k < K && n < Nn) ? B[(long)k * sbk + (long)n * sbj] : 0.0f; };
  for (int t = warp; t < tm * tn; t += nw) {
    const int m0 = (t / tn) << 4, n0 = (t % tn) * 8 * kNs;
    const int r0 = m0 + g, r1 = m0 + g + 8;
    const int nsub = min(kNs, (Nn - n0 + 7) >> 3);          // sub-tiles holding columns (warp-uniform)
    float c[kNs][4];
#pragma unroll
    for (int q = 0; q < kNs; ++q) c[q][0] = c[q][1] = c[q][2] = c[q][3] = 0.f;
    for (int k0 = 0; k0 < K; k0 += 16) {
      const int k = k0 + 2 * tg;
      const float av[8] = {a_at(r0, k), a_at(r0, k + 1), a_at(r1, k), a_at(r1, k + 1),
                           a_at(r0, k + 8), a_at(r0, k + 9), a_at(r1, k + 8), a_at(r1, k + 9)};
      __nv_bfloat16 ah[8], al[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) split_bf16(av[q], ah[q], al[q]);
      const uint32_t AH[4] = {pack2(ah[0], ah[1]), pack2(ah[2], ah[3]), pack2(ah[4], ah[5]), pack2(ah[6], ah[7])};
      const uint32_t AL[4] = {pack2(al[0], al[1]), pack2(al[2], al[3]), pack2(al[4], al[5]), pack2(al[6], al[7])};
#pragma unroll
      for (int q = 0; q < kNs; ++q) {
        if (q < nsub) {
          const int nn = n0 + 8 * q + g;
          const float bv[4] = {b_at(k, nn), b_at(k + 1, nn), b_at(k + 8, nn), b_at(k + 9, nn)};
          __nv_bfloat16 bh[4], bl[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) split_bf16(bv[u], bh[u], bl[u]);
          const uint32_t BH[2] = {pack2(bh[0], bh[1]), pack2(bh[2], bh[3])};
          const uint32_t BL[2] = {pack2(bl[0], bl[1]), pack2(bl[2], bl[3])};
          mma_bf16(c[q], AH, BL);
          mma_bf16(c[q], AL, BH);
          mma_bf16(c[q], AH, BH);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kNs; ++q) {
      if (q < nsub) {
        const int cc = n0 + 8 * q + 2 * tg;
        if (r0 < M) {
          if (cc < Nn) epi(C, sci, scj, r0, cc, c[q][0]);
          if (cc + 1 < Nn) epi(C, sci, scj, r0, cc + 1, c[q][1]);
        }
        if (r1 < M) {
          if (cc < Nn) epi(C, sci, scj, r1, cc, c[q][2]);
          if (cc + 1 < Nn) epi(C, sci, scj, r1, cc + 1, c[q][3]);
        }
      }
    }
  }
}

// --------------------------------------------------------------------------
// shared memory of one chain CTA

// Buffers of one flip block (lives in shared memory, see make_cta).
template <typename T>
struct FlipBuf {
  union {
    T Tu[2][kBlock][kBlock + 1];    // t-V: 1 + (1 - G_SS) Gamma, inverted in place, then M
    alignas(16) T sv[2][kBlock][kBlock];  // Hubbard: the update vectors at the accepted sites (sm_vectors)
  };
  T rs[2][kBlock];                  // ratio R_sigma of each proposal of the decision sub-block
  T cl[2][kMaxDelay];               // Delta of each accepted flip of the delayed block (diagonal of Gamma)
  T fr[2][kMaxDelay];               // Delta / R_sigma of each accepted flip
  int gsite[kMaxDelay];             // site of each accepted flip
};
static_assert(sizeof(FlipBuf<double>) <= flipbuf_bytes(8) && sizeof(FlipBuf<float>) <= flipbuf_bytes(4),
              "flip buffer layout");

template <typename T>
struct Smem {
  ChainDesc desc;                   // this chain's descriptor, copied in at launch
  double red[32];                   // reduction scratch
  // e^{V_sigma} of one site as a function of m = the staged value fr[i]
  // (a site field +-1, or for t-V the signed sum of the site's bond fields,
  // -3..3): [Gutzwiller?][spin][m + 3]; unused entries are 1
  double vtab[2][2][7];
  T vt[2][2][7];                    // the same in the path precision
  T vti[2][2][7];                   // and its inverse
  long long cyc[kPhases];           // per-phase clock cycles (thread 0)
  long long t_mark;
  signed char fr[kMaxN];            // fields of the staged slice
  int na;                           // accepted flips in the block
  int nswap[2];
  int chol_bad[2];                  // the spin's Cholesky factor broke down
  int fperm[kBlock];                // row interchanges of the flush inverse (t-V)
  int staged;                       // slice held in fr, or -1
  double sign_running;
  double sign_spin[2];
  double logw_spin[2];
  double dGmax;
  long long n_prop, n_acc, acc_pos;
  int err;
  int res;                          // G and the scratch live in shared memory
  uint64_t seed;
  ScratchLayout L;                  // offsets of the phase buffers in the scratch
  uint32_t scr_off;                 // RES: the scratch's offset from the shared-memory base
  uint32_t tcs_off;                 // tensor-core staging area (BF16X3, chains in global memory), or 0
  uint32_t tmem;                    // its TMEM accumulator
  int src;                          // where phase_stack left the block: Mt (0; FP64 path also Mt2, 1), e^V P (2)
  double gj_ip[2];                  // reciprocal of the Gauss-Jordan pivot
  double gj_logabs[2], gj_sign[2];  // log|det O| and sign of the last Gauss-Jordan inverse
};

// One chain CTA: its descriptor, shared memory, and where G and the phase
// scratch live (RES: shared memory, when they fit; else the chain's global
// buffers).  Each phase of the sweep is a function of its own (not inlined), so
// that ptxas gives it the whole register budget, and builds its Cta from the
// shared-memory base, so that with RES every access is a shared-memory
// instruction on a 32-bit address.  At 128 registers the FP32 kernels still spill
// 156 bytes around the calls and up to 104 in a phase (the digit products and
// the assembly); the FP64 kernels (206 registers) and spread mode's do not.
template <typename T, bool RES>
struct Cta {
  static constexpr bool resident = RES;
  const ChainDesc& c;
  Smem<T>& sh;
  T* Gp;
  unsigned char* scr;
  const ScratchLayout& L;
  FlipBuf<T>* fb;
  __device__ T* G(int s) const { return Gp + (long)s * c.N * c.ld; }
  __device__ T* Gt() const { return reinterpret_cast<T*>(scr + L.gt); }
  __device__ T* Ub() const { return reinterpret_cast<T*>(scr + L.u); }
  // update vectors of spin s: U (column m at m ldu()), V (row m at m ld)
  __device__ int ldu() const { return std::is_same<T, double>::value ? c.N : c.ld; }
  __device__ T* Uv(int s) const { return reinterpret_cast<T*>(scr + (s == 0 ? L.u : L.u2)); }
  __device__ T* Vv(int s) const { return reinterpret_cast<T*>(scr + (s == 0 ? L.w : L.mw)); }
  __device__ T* Wb() const { return reinterpret_cast<T*>(scr + L.w); }
  __device__ double* M64() const { return reinterpret_cast<double*>(scr + L.m64); }
  __device__ double* Q64() const { return reinterpret_cast<double*>(scr + L.q64); }
  // row length of the stack products' buffers (FP32: whole vectors)
  __device__ int ldn(int s) const { return std::is_same<T, double>::value ? nsig(s) : pad4(nsig(s)); }
  __device__ T* Mt(int s) const { return reinterpret_cast<T*>(scr + L.mtq + s * L.mts); }
  __device__ T* Mt2() const { return reinterpret_cast<T*>(scr + L.mt2); }
  __device__ double* qbeta() const { return reinterpret_cast<double*>(scr + L.qaux); }
  __device__ double* qalpha() const { return qbeta() + c.nmax; }
  __device__ double* qw() const { return qbeta() + 2 * c.nmax; }
  __device__ double* qpart() const { return qbeta() + 3 * c.nmax; }
  __device__ double* chol(int s) const { return reinterpret_cast<double*>(scr + L.chol + s * L.chs); }
  __device__ double* Ob(int s) const {
    return reinterpret_cast<double*>(scr + L.o + s * al16((size_t)c.nmax * c.nmax * 8));
  }
  __device__ T* Yb() const { return reinterpret_cast<T*>(scr + L.y); }
  __device__ T* QRt() const { return reinterpret_cast<T*>(scr + L.qrt); }
  __device__ T* QLt() const { return reinterpret_cast<T*>(scr + L.qlt); }
  __device__ T* Ot() const { return reinterpret_cast<T*>(scr + L.ot); }
  // staging area of the tensor-core products (when sh.tcs_off != 0)
  __device__ unsigned char* tcs() const {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return smem_raw + sh.tcs_off;
  }
  // Gauss-Jordan of spin s: pivots, column in hand (two), pivot row, row of each step (and two work arrays)
  __device__ double* pval(int s) const { return reinterpret_cast<double*>(scr + L.laux) + s * 6 * c.nmax; }
  __device__ double* gj_col(int s) const { return pval(s) + c.nmax; }
  __device__ double* gj_row(int s) const { return pval(s) + 3 * c.nmax; }
  __device__ int* gj_rows(int s) const { return reinterpret_cast<int*>(pval(s) + 4 * c.nmax); }
  __device__ const T* Em() const { return reinterpret_cast<const T*>(c.expKm); }
  __device__ const T* Ep() const { return reinterpret_cast<const T*>(c.expKp); }
  __device__ int nsig(int s) const { return s == 0 ? c.nup : c.ndn; }
  __device__ bool gutz(int tau) const { return tau == 0 || tau == c.Ltau + 1; }
  // fermion species carried by the chain: both spins, or one (t-V)
  __device__ int nspec() const { return c.tv ? 1 : 2; }
  // stage slice tau into shared memory (collective): the site fields, or for
  // t-V the sum m_i of the site's three bond fields (+ at A ends, - at B ends)
  __device__ void stage(int tau) {
    __syncthreads();
    const int8_t* f = c.fields + (long)tau * c.nfld;
    if (c.tv) {
      for (int i = threadIdx.x; i < c.N; i += blockDim.x) {
        const int* sb = c.site_bonds + 3 * i;
        const int m = (int)f[sb[0]] + (int)f[sb[1]] + (int)f[sb[2]];
        sh.fr[i] = (signed char)((i & 1) ? -m : m);
      }
    } else {
      for (int i = threadIdx.x; i < c.N; i += blockDim.x) sh.fr[i] = f[i];
    }
    if (threadIdx.x == 0) sh.staged = tau;
    __syncthreads();
  }
  // diagonal of e^{V_sigma(s_tau)} at site i for the staged slice tau
  __device__ double vexp(int tau, int s, int i) const { return sh.vtab[gutz(tau) ? 1 : 0][s][sh.fr[i] + 3]; }
  __device__ T vexpT(int tau, int s, int i) const { return sh.vt[gutz(tau) ? 1 : 0][s][sh.fr[i] + 3]; }
  __device__ T vinvT(int tau, int s, int i) const { return sh.vti[gutz(tau) ? 1 : 0][s][sh.fr[i] + 3]; }
  // charge the cycles since the last mark to phase ph (thread 0 only)
  __device__ void mark(int ph) {
    if (threadIdx.x == 0) {
      const long long t = clock64();
      sh.cyc[ph] += t - sh.t_mark;
      sh.t_mark = t;
    }
  }
};

// The Cta of this block, from the shared-memory base (setup_cta has run).
template <typename T, bool RES>
__device__ __forceinline__ Cta<T, RES> this_cta() {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<T>& sh = *reinterpret_cast<Smem<T>*>(smem_raw);
  unsigned char* dyn = smem_raw + al16(sizeof(Smem<T>));
  if constexpr (RES) {
    unsigned char* scr = smem_raw + sh.scr_off;
    return Cta<T, RES>{sh.desc, sh, reinterpret_cast<T*>(dyn), scr, sh.L, reinterpret_cast<FlipBuf<T>*>(scr + sh.L.fb)};
  } else {
    return Cta<T, RES>{sh.desc, sh, reinterpret_cast<T*>(sh.desc.G), reinterpret_cast<unsigned char*>(sh.desc.scratch),
                       sh.L, reinterpret_cast<FlipBuf<T>*>(dyn)};
  }
}

// Product of the reduced paths' wrap.  On the BF16X3 path it runs
// as split-precision tensor-core products: tcgen05 MMAs into tensor memory
// when the CTA holds a staging area for them (kTc: 512-thread CTAs, a chain
// kept in global memory; a kernel that holds tcgen05 code runs one CTA per
// SM, so the smaller CTAs are built without it), mma.sync otherwise.  The
// delayed update is a rank-a correction (a <= 64) whose cost is reading and
// writing G: it runs in FP32 on the CUDA cores on the BF16X3 path too
// (measured faster than either tensor-core form at 162-648 sites, and exact
// to FP32).  FP32 path: CUDA-core FMA.
// kRowA: A is row-major (ld ld), else A(i, k) = A[i + k ld].
template <bool kTc, bool kRowA, bool RES, typename Epi>
__device__ __forceinline__ void wrap_gemm(Cta<float, RES>& x, int n, const float* A, const float* B, float* C, int ld, Epi epi) {
  const int sai = kRowA ? ld : 1, sak = kRowA ? 1 : ld;
  if (x.c.tc) {
    if constexpr (kTc && !RES) {
      if (x.sh.tcs_off) {
        cta_gemm_tc(n, n, n, A, sai, sak, B, ld, 1, C, ld, 1, epi, x.tcs(), x.sh.tmem, &x.sh.err, kErrTimeout);
        __syncthreads();
        return;
      }
    }
    cta_gemm_bf16x3(n, n, n, A, sai, sak, B, ld, 1, C, ld, 1, epi);
    return;
  }
  cta_gemm_f32<kRowA>(n, n, n, A, ld, B, ld, C, ld, epi);
}

// --------------------------------------------------------------------------
// Metropolis updates of one slice with delayed updates in blocks of kBlock
// sites.  Inside a block one warp (lane = column of the block) proposes the
// flips in order on the kBlock x kBlock diagonal block of G.  Later proposals
// read only rows and columns of later sites, so an accepted flip at j updates
// just that future part: G_rq += c G_rj G_jq (r, q > j), c = Delta/R_sigma.
// After the block the whole CTA applies the accepted set S at once:
//     G <- G - (E_S - G_{:,S}) M G_{S,:},  M = Gamma (1 + (1 - G_SS) Gamma)^{-1},
// G the G of the block start, Gamma = diag(Delta) of the accepted flips.  This
// equals the sequence of Sherman-Morrison updates because the new G depends
// only on the new fields; the pivots of the a x a inverse are the accepted
// ratios, so Gauss-Jordan without pivoting follows the sequential process.

// The Metropolis uniform u = m 2^-53 of the 53-bit Philox mantissa m, in the
// decision precision: exact in FP64; in FP32 rounded down to 24 bits, so
// u < |R| is decided in FP32 on both sides of a comparison with the oracle.
template <typename T>
__device__ __forceinline__ T uniform_of(uint64_t m53) {
  if constexpr (std::is_same<T, double>::value) return (double)m53 * 0x1.0p-53;
  else return (float)(uint32_t)(m53 >> 29) * 0x1.0p-24f;
}

// Applies the a accepted flips of a block, recorded in fb (global sites
// gsite, Delta per species cl), to the whole G of every species:
//     G <- G - (E_S - G_{:,S}) Gamma (1 + (1 - G_SS) Gamma)^{-1} G_{S,:}
// with G the G of the block start (flush_block, t-V blocks; a Hubbard chain
// swept by the whole GPU takes the middle factor from block_inverse).
// X = 1 + (1 - G_SS) Gamma is inverted in place; Hubbard blocks need no
// pivoting (its pivots are the accepted ratios), the bond blocks of the t-V
// model pivot on rows (a single end of an accepted bond may have a vanishing
// ratio).

// M = Gamma (1 + (1 - G_SS) Gamma)^{-1} of the a accepted flips of a block
// into fb.Tu[s] for every species s (collective; G is the G of the block
// start).  Per pivot the species' first warp finds it, exchanges the rows and
// hands on the pivot row and reciprocal; then every warp takes its rows (lane:
// column), two barriers in all.  (One warp doing it alone, a row at a time
// through shared memory, took 35 kcycles for 21 Hubbard flips and 49 for the
// 32 ends of a t-V block.)
template <typename T, bool RES>
__device__ __forceinline__ void block_inverse(Cta<T, RES>& x, int a, bool pivot) {
  FlipBuf<T>& fb = *x.fb;
  const int ld = x.c.ld, ns = x.nspec();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  // the warps of a species: every ns-th one
  const int s = warp % ns, w = warp / ns, ws = nw / ns;
  const unsigned full = 0xffffffffu;
  PQMC_FOR_2D(sl, 0, ns * a, m, 0, a) {
    const int sp = sl >= a ? 1 : 0, l = sl - sp * a;
    const T g = x.G(sp)[(long)fb.gsite[l] * ld + fb.gsite[m]];
    fb.Tu[sp][l][m] = ((l == m) ? T(1) : T(0)) + ((l == m ? T(1) : T(0)) - g) * fb.cl[sp][m];
  }
  __syncthreads();
  T (*X)[kBlock + 1] = fb.Tu[s];
  T* prow = fb.rs[s];                    // pivot row of the step
  int* perm = x.sh.fperm;
  for (int p = 0; p < a; ++p) {
    if (w == 0) {
      if (pivot) {
        // largest |X_rp|, r >= p, ties to the lower row; swap rows r and p
        T best = T(-1);
        int bi = p;
        if (lane >= p && lane < a) { best = fabs(X[lane][p]); bi = lane; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const T ob = __shfl_xor_sync(full, best, o);
          const int oi = __shfl_xor_sync(full, bi, o);
          if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (lane == 0) perm[p] = bi;
        if (bi != p && lane < a) {
          const T t = X[p][lane];
          X[p][lane] = X[bi][lane];
          X[bi][lane] = t;
        }
        __syncwarp();
      }
      if (lane < a) prow[lane] = X[p][lane];
    }
    __syncthreads();
    const T xpl = lane < a ? prow[lane] : T(0);
    const T ip = T(1) / prow[p];
    // several rows of a warp in flight: eight without a branch where a warp has
    // up to eight rows (two FP32 species), four with the absent ones left out where
    // that would be idle work (one species) or FP64 instructions
    auto eliminate = [&](auto in_flight, auto skip) {
      constexpr int kU = decltype(in_flight)::value;
      for (int r0 = w; r0 < a; r0 += kU * ws) {
        T xrp[kU], xrl[kU];
#pragma unroll
        for (int q = 0; q < kU; ++q) {
          const int r = min(r0 + q * ws, a - 1);
          xrp[q] = X[r][p];
          xrl[q] = X[r][lane];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < kU; ++q) {
          const int r = r0 + q * ws;     // (the same in the whole warp)
          if (decltype(skip)::value && r >= a) continue;
          const T m = xrp[q] * ip;
          T v = fma(-m, xpl, xrl[q]);
          if (lane == p) v = -m;
          if (r == p) v = lane == p ? ip : xpl * ip;
          if (r < a && lane < a) X[r][lane] = v;
        }
        __syncwarp();
      }
    };
    if (std::is_same<T, double>::value || ns == 1) eliminate(std::integral_constant<int, 4>(), std::true_type());
    else eliminate(std::integral_constant<int, 8>(), std::false_type());
    __syncthreads();
  }
  if (w == 0 && pivot) {
    // the row interchanges of the factorisation become column
    // interchanges of the inverse, undone last step first
    for (int p = a - 1; p >= 0; --p) {
      const int q = perm[p];
      if (q != p && lane < a) {
        const T t = X[lane][p];
        X[lane][p] = X[lane][q];
        X[lane][q] = t;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int l = w; l < a; l += ws)
    if (lane < a) X[l][lane] *= fb.cl[s][l];
  __syncthreads();
}

template <typename T, bool RES>
__device__ __forceinline__ void flush_block(Cta<T, RES>& x, int a) {
  const ChainDesc& c = x.c;
  FlipBuf<T>& fb = *x.fb;
  const int N = c.N, ld = c.ld, ldu = x.ldu(), ns = x.nspec();
  T* Ubuf = x.Ub();                                    // kBlock x N  (U column-major, ld N)
  T* Wbuf = x.Wb();                                    // kBlock x ld (rows G_{S,:})
  block_inverse(x, a, true);
  // per species: A_S = E_S - G_{:,S} (N x a, column-major) and W = G_{S,:}
  // (a x N) gathered before G changes, then MW = M W and G -= A_S MW
  T* MW = reinterpret_cast<T*>(x.scr + x.L.mw);
  for (int s = 0; s < ns; ++s) {
    T* Gs = x.G(s);
    PQMC_FOR_2D(m, 0, a, i, 0, N) {
      const int col = fb.gsite[m];
      Ubuf[(long)m * ldu + i] = (i == col ? T(1) : T(0)) - Gs[(long)i * ld + col];
    }
    PQMC_FOR_2D(l, 0, a, q, 0, N) Wbuf[(long)l * ld + q] = Gs[(long)fb.gsite[l] * ld + q];
    __syncthreads();
    cta_gemm<T>(a, N, a, &fb.Tu[s][0][0], kBlock + 1, 1, Wbuf, ld, 1, MW, ld, 1, EpiStore());
    __syncthreads();
    if constexpr (std::is_same<T, double>::value) cta_gemm<T>(N, N, a, Ubuf, 1, ldu, MW, ld, 1, Gs, ld, 1, EpiSub());
    else cta_gemm_f32<false>(N, N, a, Ubuf, ldu, MW, ld, Gs, ld, EpiSub());
    __syncthreads();
  }
  x.mark(kPhFlush);
}

// The accepted flips of a Hubbard delayed block, applied to G as the chain of
// rank-1 updates they stand for, in acceptance order (the update of one
// flip at site i with G the G just before it):
//     G <- G - (e_i - G_{:,i}) (Delta_i / R_i) G_{i,:}.
// Written as G <- G - U V over the block: column m of U and row m of V are
// the vectors of flip m, obtained from the block-start G and the earlier
// vectors (c = G_{:,s_m} - U V_{:,s_m}, r = G_{s_m,:} - U_{s_m,:} V)
// (sm_vectors, for flips m0..m1-1 once their decisions are taken), then one
// rank-a product per spin (apply_vectors).  Same result as the block form of
// flush_block, without the a x a inverse.
//
// Step m of any row o or column j needs of the other flips only their
// vectors' elements at the accepted sites, V_m[s_p] and U_m[s_p] (p > m).  So
// the chain first runs on the accepted sites alone (sm_core) and leaves those
// elements in a table; then every row and column of G is an independent
// thread that keeps its own vector in registers and reads the table as
// 16-byte broadcasts (sm_vectors): one CTA barrier per block instead of one
// per flip.  Every element sees the same FMAs in the same order as flip by
// flip.
//
// The loops over the flips stay rolled and move the register window down
// instead (the element of flip m is always in register 0): unrolled over the
// 32 flips, one warp runs through 20-40 KB of code once per block and waits
// for instruction fetches.

// The table of a spin (FlipBuf::sv): V_m[s_p] at row m, column p; U_m[s_p] at
// row 31 - m, column 31 - p (p > m: above and below the diagonal).
template <typename T>
__device__ __forceinline__ T& sm_v(T (*tab)[kBlock], int m, int p) { return tab[m][p]; }
template <typename T>
__device__ __forceinline__ T& sm_u(T (*tab)[kBlock], int m, int p) { return tab[kBlock - 1 - m][kBlock - 1 - p]; }

// The chain on the accepted sites, one warp per spin and role: rows (lane q:
// row s_q, register p: column s_p; gives the U_m) or columns (transposed; the
// V_m).  The two roles form the same elements and need no word of each other.
template <typename T, bool RES>
__device__ __forceinline__ void sm_core(Cta<T, RES>& x, int i0, int m0, int cnt) {
  FlipBuf<T>& fb = *x.fb;
  const int lane = threadIdx.x & 31, nw = (int)blockDim.x >> 5;
  for (int w = threadIdx.x >> 5; w < max(4, nw); w += nw) {
    const int s = (w >> 1) & 1;
    const bool row = (w & 1) == 0;
    T (*tab)[kBlock] = fb.sv[s];
    const int sq = min(fb.gsite[m0 + lane] - i0, kBlock - 1);
    // element p of this line: block element (s_q, s_p) or (s_p, s_q), as staged
    // for the decisions
    T a[kBlock];
#pragma unroll
    for (int p = 0; p < kBlock; ++p) {
      const int sp = fb.gsite[m0 + p] - i0;
      a[p] = row ? fb.Tu[s][sq][sp] : fb.Tu[s][sp][sq];
    }
    __syncthreads();                     // the table takes the staged block's place
    if (w >= 4) continue;
#pragma unroll 1
    for (int m = 0; m < cnt; ++m) {
      const T f = fb.fr[s][m0 + m];
      const int rem = cnt - 1 - m;       // flips after this one
      if (row) {
        const T u = (T(0) - a[0]) * f;
        if (lane > m && lane < cnt) sm_u(tab, m, lane) = u;
#pragma unroll
        for (int p0 = 1; p0 < kBlock; p0 += 8)
          if (p0 <= rem) {
#pragma unroll
            for (int p = p0; p < (p0 + 8 < kBlock ? p0 + 8 : kBlock); ++p)
              a[p - 1] = fma(-u, __shfl_sync(0xffffffffu, a[p], m), a[p]);
          }
      } else {
        const T v = a[0];
        if (lane > m && lane < cnt) sm_v(tab, m, lane) = v;
#pragma unroll
        for (int p0 = 1; p0 < kBlock; p0 += 8)
          if (p0 <= rem) {
#pragma unroll
            for (int p = p0; p < (p0 + 8 < kBlock ? p0 + 8 : kBlock); ++p) {
              const T u = (T(0) - __shfl_sync(0xffffffffu, a[p], m)) * f;
              a[p - 1] = fma(-u, v, a[p]);
            }
          }
      }
    }
  }
}

// Where sm_four reads a spin's table (flat, four elements from there): for flip
// k + i the elements of the flips k + q .. k + q + 3, in the place of sm_v (rows)
// or sm_u (columns, the four in reverse).  A window that reaches past the last
// flip of the block reads the last four once more instead (its elements there
// stand for no flip), so that no read leaves the flip's row.
__host__ __device__ constexpr int sm_at(bool row, int k, int i, int q) {
  const int qc = q < kBlock - 4 - k ? q : kBlock - 4 - k;
  return row ? (k + i) * kBlock + k + qc : (kBlock - 1 - k - i) * kBlock + kBlock - 4 - k - qc;
}
constexpr bool sm_reads_in_row() {
  for (int k = 0; k < kBlock; k += 4)
    for (int i = 0; i < 4; ++i)
      for (int q = 0; q < kBlock; q += 4) {
        const int v = sm_at(true, k, i, q), u = sm_at(false, k, i, q);
        if (v / kBlock != k + i || (v + 3) / kBlock != k + i || u < 0 || u / kBlock != kBlock - 1 - k - i ||
            (u + 3) / kBlock != kBlock - 1 - k - i)
          return false;
        if (k + q < kBlock && (v % kBlock != k + q || u % kBlock != kBlock - 4 - k - q)) return false;
      }
  return true;
}
static_assert(kBlock % 4 == 0 && sm_reads_in_row(), "the update vectors' table reads");

// Four flips k .. k + 3 on a thread's window w of kW elements (register i:
// flip k + i): the flips' vector elements go out, the later elements take
// their updates.  No branch inside: the table rows are read ahead of the
// FMAs (flips beyond cnt work on leftovers that nothing reads).
template <bool kRow, int kW, typename T>
__device__ __forceinline__ void sm_four(T (&w)[kBlock], const T (*tab)[kBlock], int k, int cnt, int j, const int* site,
                                        const T* fr, T* out, long os) {
  const T* t0 = &tab[0][0];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    T cv = w[i];
    if (kRow) cv = (T(j == site[k + i] ? 1 : 0) - cv) * fr[k + i];
    if (k + i < cnt) out[(k + i) * os] = cv;
#pragma unroll
    for (int q = 0; q < kW; q += 4)
      if (q + 3 > i) {
        T t[4];
        Vec4<T>::load(t0 + sm_at(kRow, k, i, q), t);
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if (q + h > i) w[q + h] = fma(-cv, kRow ? t[h] : t[3 - h], w[q + h]);
      }
  }
#pragma unroll
  for (int p = 0; p + 4 < kW; ++p) w[p] = w[p + 4];
}

// kLater: flips of the delayed block's earlier sub-blocks come first (m0 > 0)
template <bool kRow, bool kLater, typename T, bool RES>
__device__ __forceinline__ void sm_line(Cta<T, RES>& x, int s, int j, int m0, int cnt) {
  const ChainDesc& c = x.c;
  FlipBuf<T>& fb = *x.fb;
  const int ld = c.ld;
  // element p of this line: G[j][s_p] (row) or G[s_p][j] (column)
  const T* g = kRow ? x.G(s) + (long)j * ld : x.G(s) + j;
  T* out = kRow ? x.Uv(s) + j : x.Vv(s) + j;
  const long os = ld;                    // (FP32: U and V share the row length)
  const int* site = fb.gsite + m0;
  T w[kBlock];
#pragma unroll
  for (int p = 0; p < kBlock; ++p) w[p] = g[kRow ? site[p] : site[p] * ld];
  if (kLater) {
    const T* other = kRow ? x.Vv(s) : x.Uv(s);
    for (int l = 0; l < m0; ++l) {
      const T a = out[l * os];
#pragma unroll
      for (int p = 0; p < kBlock; ++p) w[p] = fma(-a, other[l * os + site[p]], w[p]);
    }
  }
  out += m0 * os;
  int k = 0;
#pragma unroll 1
  for (; cnt - k > 16; k += 4) sm_four<kRow, 32>(w, fb.sv[s], k, cnt, j, site, fb.fr[s] + m0, out, os);
#pragma unroll 1
  for (; k < cnt; k += 4) sm_four<kRow, 16>(w, fb.sv[s], k, cnt, j, site, fb.fr[s] + m0, out, os);
}

// every row of U and every column of V, both spins: a warp takes 32 rows or
// 32 columns of one spin at a time
template <bool kLater, typename T, bool RES>
__device__ __forceinline__ void sm_vectors(Cta<T, RES>& x, int m0, int cnt) {
  const int N = x.c.N, lane = threadIdx.x & 31;
  const int groups = (N + 31) >> 5;
  for (int t = threadIdx.x >> 5; t < 4 * groups; t += blockDim.x >> 5) {
    const int s = t & 1, j = 32 * (t >> 2) + lane;
    if (j >= N) continue;
    if (t & 2) sm_line<true, kLater>(x, s, j, m0, cnt);
    else sm_line<false, kLater>(x, s, j, m0, cnt);
  }
}

// FP64: flip by flip, one step per flip for the two spins at once (half of
// the CTA each).  Here the FP64 pipe sets the time (16 cycles per warp
// instruction and SM): the form above, which repeats the accepted sites'
// part and works on padding, takes 1.9 times as long.
template <typename T, bool RES>
__device__ __forceinline__ void sm_vectors_by_flip(Cta<T, RES>& x, int m0, int m1) {
  const ChainDesc& c = x.c;
  FlipBuf<T>& fb = *x.fb;
  const int N = c.N, ld = c.ld, ldu = x.ldu();
  const int half = (int)blockDim.x >> 1;
  const int s = (int)threadIdx.x >= half ? 1 : 0;
  const int t = (int)threadIdx.x - s * half;
  const T* Gs = x.G(s);
  T* U = x.Uv(s);
  T* V = x.Vv(s);
  for (int m = m0; m < m1; ++m) {
    const int sm = fb.gsite[m];
    const T f = fb.fr[s][m];
    for (int o = t; o < 2 * N; o += half) {
      if (o < N) {
        T cv = Gs[(long)o * ld + sm];
        for (int l = 0; l < m; ++l) cv = fma(-U[(long)l * ldu + o], V[(long)l * ld + sm], cv);
        U[(long)m * ldu + o] = ((o == sm ? T(1) : T(0)) - cv) * f;
      } else {
        const int j = o - N;
        T rv = Gs[(long)sm * ld + j];
        for (int l = 0; l < m; ++l) rv = fma(-U[(long)l * ldu + sm], V[(long)l * ld + j], rv);
        V[(long)m * ld + j] = rv;
      }
    }
    // the two halves step independently: one named barrier per spin
    if (s == 0) asm volatile("bar.sync 2, %0;" ::"r"(half) : "memory");
    else asm volatile("bar.sync 3, %0;" ::"r"(half) : "memory");
  }
}

// FP64: the product on the tensor cores, U and V turned into digits in place.
template <typename T, bool RES>
__device__ __forceinline__ void apply_vectors(Cta<T, RES>& x, int a) {
  const ChainDesc& c = x.c;
  const int N = c.N, ld = c.ld;
  if constexpr (std::is_same<T, double>::value) {
    int* red = reinterpret_cast<int*>(x.sh.red);
    const int ldu = x.ldu();
    for (int sp = 0; sp < 2; ++sp) {
      double* U = x.Uv(sp);
      double* V = x.Vv(sp);
      double* G = x.G(sp);
      int eu = kDigitNone, ev = kDigitNone;
      PQMC_FOR_2D(m, 0, a, i, 0, N) {
        eu = max(eu, digit_exp(U[(long)m * ldu + i]));
        ev = max(ev, digit_exp(V[(long)m * ld + i]));
      }
      const int EU = digit_cta_max(eu, red), EV = digit_cta_max(ev, red);
      unsigned long long* DU = reinterpret_cast<unsigned long long*>(U);
      unsigned long long* DV = reinterpret_cast<unsigned long long*>(V);
      PQMC_FOR_2D(m, 0, a, i, 0, N) {
        DU[(long)m * ldu + i] = digit_pack(U[(long)m * ldu + i], EU);
        DV[(long)m * ld + i] = digit_pack(V[(long)m * ld + i], EV);
      }
      __syncthreads();
      digit_gemm<false, false>(N, N, a, DU, 1, ldu, DV, 1, ld, [EU](int) { return EU; }, [EV](int) { return EV; }, false,
                               false, [G, ld](int i, int j, double v) { G[(long)i * ld + j] -= v; });
    }
  } else {
    for (int sp = 0; sp < 2; ++sp) cta_gemm_f32<false>(N, N, a, x.Uv(sp), ld, x.Vv(sp), ld, x.G(sp), ld, EpiSub());
  }
  __syncthreads();
  x.mark(kPhFlush);
}

// The diagonal block of G at sites i0 .. i0 + nbk - 1, both spins, into
// fb.Tu (zero beyond nbk), brought up to date by the vectors of the a_done flips the
// delayed block has accepted so far: G_SS - U_S V_S (collective).
template <typename T, bool RES>
__device__ __forceinline__ void stage_block(Cta<T, RES>& x, int i0, int nbk, int a_done) {
  FlipBuf<T>& fb = *x.fb;
  const int ld = x.c.ld;
  for (int e = threadIdx.x; e < 2 * kBlock * kBlock; e += blockDim.x) {
    const int s = e / (kBlock * kBlock), r = e / kBlock % kBlock, q = e % kBlock;
    T v = T(0);
    if (r < nbk && q < nbk) {
      v = x.G(s)[(long)(i0 + r) * ld + i0 + q];
      for (int l = 0; l < a_done; ++l) v = fma(-x.Uv(s)[(long)l * x.ldu() + i0 + r], x.Vv(s)[(long)l * ld + i0 + q], v);
    }
    fb.Tu[s][r][q] = v;
  }
  __syncthreads();
}

// The proposals of one decision sub-block, sites i0 .. i0 + nbk - 1 of slice
// tau (nbk <= kBlock), after a_done flips of the delayed block were accepted
// (their update vectors in the scratch correct the diagonal block read from
// G): warps 0 and 1 decide; sh.na receives the accepted count of the delayed
// block, fb the accepted sites and their Delta, Delta / R.
template <typename T, bool RES>
__device__ __forceinline__ void decide_sub_block(Cta<T, RES>& x, int tau, uint32_t sweep, int i0, int nbk, int a_done) {
  const ChainDesc& c = x.c;
  Smem<T>& sh = x.sh;
  FlipBuf<T>& fb = *x.fb;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kap = x.gutz(tau) ? 1 : 0;
  int8_t* f = c.fields + (long)tau * c.nfld;
  const T dl[2][2] = {{(T)c.delta[kap][0][0], (T)c.delta[kap][0][1]}, {(T)c.delta[kap][1][0], (T)c.delta[kap][1][1]}};
  if (warp < 2) {
    // warp s (spin s): lane q holds column q of the spin's diagonal block in
    // registers; the two warps exchange the spin ratios through shared
    // memory once per proposal and take the same decision
    const int s = warp;
    T gs[kBlock];
    const bool colq = lane < nbk;
#pragma unroll
    for (int r = 0; r < kBlock; ++r) gs[r] = fb.Tu[s][r][lane];
    // lane j: uniform (in the decision precision) and field of site i0 + j
    T uj = T(2);
    int flj = 1;
    if (colq) {
      const U4 w = philox4x32_10((uint32_t)(i0 + lane), (uint32_t)tau, sweep, c.chain_index, (uint32_t)x.sh.seed,
                                 (uint32_t)(x.sh.seed >> 32));
      uj = uniform_of<T>(((uint64_t)w.x0 << 21) | (uint64_t)(w.x1 >> 11));
      flj = (int)f[i0 + lane];
    }
    int a = a_done, bad = 0, nneg = 0, last = i0;
    const long long pos0 = sh.acc_pos;
#pragma unroll
    for (int j = 0; j < kBlock; ++j) {
      if (j < nbk) {
        const int si = __shfl_sync(0xffffffffu, flj, j) > 0 ? 0 : 1;
        const T ds = dl[s][si];
        const T rs = T(1) + ds * (T(1) - __shfl_sync(0xffffffffu, gs[j], j));
        if (lane == 0) fb.rs[s][j] = rs;
        __syncwarp();
        asm volatile("bar.sync 1, 64;" ::: "memory");
        const T R = fb.rs[0][j] * fb.rs[1][j];
        const bool acc = __shfl_sync(0xffffffffu, (int)(uj < (R < T(0) ? -R : R)), j) != 0;
        if (s == 0 && lane == 0) {
          if (!isfinite(R)) bad = 1;
          if (pos0 + j < c.acc_cap) c.acc_log[pos0 + j] = acc ? 1 : 0;
        }
        if (acc) {
          // G_rq += c G_rj G_jq for future rows r > j and columns q > j
          const T y = lane > j ? (ds / rs) * gs[j] : T(0);
#pragma unroll
          for (int r = j + 1; r < kBlock; ++r) gs[r] = fma(__shfl_sync(0xffffffffu, gs[r], j), y, gs[r]);
          if (lane == j) {
            flj = -flj;
            if (s == 0) f[i0 + j] = (int8_t)flj;
          }
          if (lane == 0) fb.fr[s][a] = ds / rs;
          if (s == 0 && lane == 0) {
            fb.gsite[a] = i0 + j;
            fb.cl[0][a] = ds;
            fb.cl[1][a] = dl[1][si];
            nneg += R < T(0) ? 1 : 0;
          }
          last = i0 + j;
          ++a;
        }
      }
    }
    // (the site list goes on with the last accepted site: sm_vectors reads whole blocks of it)
    if (s == 0 && a > a_done && a + lane < a_done + kBlock) fb.gsite[a + lane] = last;
    if (s == 0 && lane == 0) {
      sh.na = a;
      sh.acc_pos = pos0 + nbk;
      sh.n_prop += nbk;
      sh.n_acc += a - a_done;
      if (nneg & 1) sh.sign_running = -sh.sign_running;
      if (bad) sh.err |= kErrNaN;
    }
  }
}

// The same in FP32 by one warp: half-warp s holds spin s's diagonal block,
// lane q of it the columns q and q + 16 in registers.  A proposal's chain is
// then two shuffles (the diagonal element, the other spin's ratio), the
// ratios' arithmetic and a compare, with no barrier; an accepted flip costs
// one shuffle per future row for both spins together.  Every value is formed
// by the operations of the two-warp form above, so the decisions and the
// factors are the same bits.  What a decision leaves behind (fields, logs,
// sites, Delta) is written after the loop, by all lanes at once.
// kRolled: the proposal loop stays rolled and the register window moves down
// one row per proposal, so row j is always register 0.  In the one-CTA sweep,
// whose phases evict one another from the instruction caches, the 40 KB of
// the unrolled loop cost more to fetch than the moves (5.3 against 3.8 Mcycles
// per sweep at 72 sites); in a kernel of its own (spread mode) the
// unrolled loop is the faster one (13 against 20 kcycles per block).
template <bool kRolled, bool RES>
__device__ __forceinline__ void decide_sub_block_pair(Cta<float, RES>& x, int tau, uint32_t sweep, int i0, int nbk,
                                                             int a_done) {
  if (threadIdx.x >= 32) return;
  const ChainDesc& c = x.c;
  Smem<float>& sh = x.sh;
  FlipBuf<float>& fb = *x.fb;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x, s = lane >> 4, q = lane & 15, half = lane & 16;
  const int kap = x.gutz(tau) ? 1 : 0;
  int8_t* f = c.fields + (long)tau * c.nfld;
  const float d0 = (float)c.delta[kap][s][0], d1 = (float)c.delta[kap][s][1];
  float ga[kBlock], gb[kBlock];
#pragma unroll
  for (int r = 0; r < kBlock; ++r) {
    ga[r] = fb.Tu[s][r][q];
    gb[r] = fb.Tu[s][r][q + 16];
  }
  // lane j: uniform (in the decision precision) and field of site i0 + j
  float uj = 2.f;
  int flj = 1;
  if (lane < nbk) {
    const U4 w = philox4x32_10((uint32_t)(i0 + lane), (uint32_t)tau, sweep, c.chain_index, (uint32_t)x.sh.seed,
                               (uint32_t)(x.sh.seed >> 32));
    uj = uniform_of<float>(((uint64_t)w.x0 << 21) | (uint64_t)(w.x1 >> 11));
    flj = (int)f[i0 + lane];
  }
  const unsigned up = __ballot_sync(full, flj > 0);
  unsigned accepted = 0;
  int a = a_done, bad = 0, nneg = 0;
  float* frs = &fb.fr[s][0];
  if constexpr (kRolled) {
    // sites 0..15 (their columns in ga), then 16..31 (in gb)
    const int n_lo = min(nbk, 16);
#pragma unroll 1
    for (int j = 0; j < n_lo; ++j) {
      const float u = __shfl_sync(full, uj, j);
      const float ds = ((up >> j) & 1u) ? d0 : d1;
      const float rs = 1.f + ds * (1.f - __shfl_sync(full, ga[0], half | j));
      const float R = rs * __shfl_xor_sync(full, rs, 16);
      const float fac = ds / rs;
      bad |= isfinite(R) ? 0 : 1;
      const bool acc = u < fabsf(R);     // the same value in every lane
      // G_rq += c G_rj G_jq for future rows r > j and columns q > j
      const float ya = acc && q > j ? fac * ga[0] : 0.f, yb = acc ? fac * gb[0] : 0.f;
      if (acc) {
        accepted |= 1u << j;
        nneg += R < 0.f ? 1 : 0;
        if (q == 0) frs[a] = fac;
        ++a;
#pragma unroll
        for (int r0 = 1; r0 < kBlock; r0 += 8)
          if (r0 < nbk - j) {
#pragma unroll
            for (int r = r0; r < (r0 + 8 < kBlock ? r0 + 8 : kBlock); ++r) {
              const float xr = __shfl_sync(full, ga[r], half | j);
              ga[r - 1] = fma(xr, ya, ga[r]);
              gb[r - 1] = fma(xr, yb, gb[r]);
            }
          }
      } else {
#pragma unroll
        for (int r = 1; r < kBlock; ++r) {
          ga[r - 1] = ga[r];
          gb[r - 1] = gb[r];
        }
      }
    }
#pragma unroll 1
    for (int j = 16; j < nbk; ++j) {
      const float u = __shfl_sync(full, uj, j);
      const float ds = ((up >> j) & 1u) ? d0 : d1;
      const float rs = 1.f + ds * (1.f - __shfl_sync(full, gb[0], half | (j - 16)));
      const float R = rs * __shfl_xor_sync(full, rs, 16);
      const float fac = ds / rs;
      bad |= isfinite(R) ? 0 : 1;
      const bool acc = u < fabsf(R);
      const float yb = acc && q + 16 > j ? fac * gb[0] : 0.f;
      if (acc) {
        accepted |= 1u << j;
        nneg += R < 0.f ? 1 : 0;
        if (q == 0) frs[a] = fac;
        ++a;
#pragma unroll
        for (int r0 = 1; r0 < 16; r0 += 8)
          if (r0 < nbk - j) {
#pragma unroll
            for (int r = r0; r < (r0 + 8 < 16 ? r0 + 8 : 16); ++r)
              gb[r - 1] = fma(__shfl_sync(full, gb[r], half | (j - 16)), yb, gb[r]);
          }
      } else {
#pragma unroll
        for (int r = 1; r < 16; ++r) gb[r - 1] = gb[r];
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < kBlock; ++j) {
      if (j < nbk) {
        const float u = __shfl_sync(full, uj, j);
        const float ds = ((up >> j) & 1u) ? d0 : d1;
        const float rs = 1.f + ds * (1.f - __shfl_sync(full, j < 16 ? ga[j] : gb[j], half | (j & 15)));
        const float R = rs * __shfl_xor_sync(full, rs, 16);
        const float fac = ds / rs;
        bad |= isfinite(R) ? 0 : 1;
        if (u < fabsf(R)) {            // the same value in every lane
          accepted |= 1u << j;
          nneg += R < 0.f ? 1 : 0;
          if (q == 0) frs[a] = fac;
          ++a;
          // G_rq += c G_rj G_jq for future rows r > j and columns q > j
          if (j < 16) {
            const float ya = q > j ? fac * ga[j] : 0.f, yb = fac * gb[j];
#pragma unroll
            for (int r = j + 1; r < kBlock; ++r) {
              const float xr = __shfl_sync(full, ga[r], half | j);
              ga[r] = fma(xr, ya, ga[r]);
              gb[r] = fma(xr, yb, gb[r]);
            }
          } else {
            const float yb = q + 16 > j ? fac * gb[j] : 0.f;
#pragma unroll
            for (int r = j + 1; r < kBlock; ++r) gb[r] = fma(__shfl_sync(full, gb[r], half | (j - 16)), yb, gb[r]);
          }
        }
      }
    }
  }
  const bool mine = (accepted >> lane) & 1u;
  if (mine) {
    const int at = a_done + __popc(accepted & ((1u << lane) - 1u));
    const int si = flj > 0 ? 0 : 1;
    fb.gsite[at] = i0 + lane;
    fb.cl[0][at] = (float)c.delta[kap][0][si];
    fb.cl[1][at] = (float)c.delta[kap][1][si];
    f[i0 + lane] = (int8_t)-flj;
  }
  // (the site list goes on with the last accepted site: sm_vectors reads whole blocks of it)
  if (accepted && a + lane < a_done + kBlock) fb.gsite[a + lane] = i0 + 31 - __clz((int)accepted);
  const long long pos0 = sh.acc_pos;
  if (lane < nbk && pos0 + lane < c.acc_cap) c.acc_log[pos0 + lane] = mine ? 1 : 0;
  __syncwarp();
  if (lane == 0) {
    sh.na = a;
    sh.acc_pos = pos0 + nbk;
    sh.n_prop += nbk;
    sh.n_acc += a - a_done;
    if (nneg & 1) sh.sign_running = -sh.sign_running;
    if (bad) sh.err |= kErrNaN;
  }
}

// kPair: the one-warp form (FP32 kernels with room for its 64 block registers)
template <bool kPair, bool kRolled, typename T, bool RES>
__device__ __forceinline__ void decide(Cta<T, RES>& x, int tau, uint32_t sweep, int i0, int nbk, int a_done) {
  stage_block(x, i0, nbk, a_done);
  if constexpr (kPair && std::is_same<T, float>::value) decide_sub_block_pair<kRolled>(x, tau, sweep, i0, nbk, a_done);
  else decide_sub_block(x, tau, sweep, i0, nbk, a_done);
}

template <typename T, bool RES, bool kPair>
__device__ __noinline__ void phase_decide(int tau, uint32_t sweep, int i0, int nbk, int a_done) {
  auto x = this_cta<T, RES>();
  decide<kPair, true>(x, tau, sweep, i0, nbk, a_done);
  __syncthreads();
  x.mark(kPhFlip);
}
template <typename T, bool RES, bool kLater>
__device__ __noinline__ void phase_vectors(int i0, int m0, int m1) {
  auto x = this_cta<T, RES>();
  if constexpr (std::is_same<T, double>::value) {
    sm_vectors_by_flip(x, m0, m1);
  } else {
    sm_core(x, i0, m0, m1 - m0);
    __syncthreads();
    sm_vectors<kLater>(x, m0, m1 - m0);
  }
  __syncthreads();
  x.mark(kPhFlushVec);
}
template <typename T, bool RES>
__device__ __noinline__ void phase_apply(int a) {
  auto x = this_cta<T, RES>();
  apply_vectors(x, a);
}

// Hubbard slice: delayed blocks of c.kb sites (8, 16, 32 or 64), each
// decided in sub-blocks of up to kBlock sites (FP32: by one warp, else one warp
// per spin) and then applied to G at once.  Within a delayed block a later
// sub-block reads its diagonal block of G corrected by the update vectors of the
// flips already accepted, G_SS - U_S V_S, so every decision sees the current G.
template <typename T, bool RES, bool kPair>
__device__ __forceinline__ void update_slice(int tau, uint32_t sweep) {
  auto x = this_cta<T, RES>();
  const int N = x.c.N;
  const int kd = x.c.kb;
  const int sub = kd < kBlock ? kd : kBlock;

  for (int d0 = 0; d0 < N; d0 += kd) {
    const int d1 = min(d0 + kd, N);
    int a_done = 0;                                  // flips of the delayed block already accepted
    for (int i0 = d0; i0 < d1; i0 += sub) {
      phase_decide<T, RES, kPair>(tau, sweep, i0, min(sub, d1 - i0), a_done);
      const int a = x.sh.na;
      if (a > a_done) {
        if (a_done == 0 || std::is_same<T, double>::value) phase_vectors<T, RES, false>(i0, a_done, a);
        else phase_vectors<T, RES, true>(i0, a_done, a);
      }
      a_done = a;
    }
    if (a_done > 0) phase_apply<T, RES>(a_done);
  }
}

// Metropolis updates of one slice of the spinless t-V model: the bonds in
// blocks of 16 of one class (a class is a perfect matching, so a block
// touches 32 distinct sites W).  Warp 0 holds G_WW in registers, lane q the
// column of site W[q] (pair p = bond p of the block: A end in lane 2p, B end
// in lane 2p+1); lane p draws the uniform of bond p.  Bond p's flip changes
// V at its two ends by Gamma = diag(Delta_A, Delta_B) and is accepted with
// R = det(1 + Gamma (1 - G_SS)); an accepted flip updates the rows and
// columns of the later pairs by the rank-2 form
//     G_rq <- G_rq + sum_{s in S} G_rs (M G_{S,q})_s,  M = Gamma (1 + (1 - G_SS) Gamma)^{-1}.
// The accepted ends then go to flush_block as one set.
template <typename T, bool RES>
__device__ __forceinline__ void update_slice_tv(Cta<T, RES>& x, int tau, uint32_t sweep) {
  const ChainDesc& c = x.c;
  Smem<T>& sh = x.sh;
  FlipBuf<T>& fb = *x.fb;
  const int ld = c.ld, nc = c.N / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kap = x.gutz(tau) ? 1 : 0;
  int8_t* f = c.fields + (long)tau * c.nfld;
  // Delta at the A end (coupled like spin up) and at the B end, field +1 / -1
  const T dA[2] = {(T)c.delta[kap][0][0], (T)c.delta[kap][0][1]};
  const T dB[2] = {(T)c.delta[kap][1][0], (T)c.delta[kap][1][1]};
  constexpr int kPairs = kBlock / 2;
  for (int k = 0; k < 3; ++k) {
    for (int c0 = 0; c0 < nc; c0 += kPairs) {
      const int np = min(kPairs, nc - c0);
      if (warp == 0) {
        const bool on = (lane >> 1) < np;
        const int wq = on ? c.bond_ends[2 * (3 * (c0 + (lane >> 1)) + k) + (lane & 1)] : 0;
        T g[kBlock];
        const T* G0 = x.G(0);
#pragma unroll
        for (int r = 0; r < kBlock; ++r) {
          const int wr = __shfl_sync(0xffffffffu, wq, r);
          g[r] = (on && (r >> 1) < np) ? G0[(long)wr * ld + wq] : T(0);
        }
        T up = T(2);
        int fp = 1;
        if (lane < np) {
          const int b = 3 * (c0 + lane) + k;
          const U4 w = philox4x32_10((uint32_t)b, (uint32_t)tau, sweep, c.chain_index, (uint32_t)x.sh.seed,
                                     (uint32_t)(x.sh.seed >> 32));
          up = uniform_of<T>(((uint64_t)w.x0 << 21) | (uint64_t)(w.x1 >> 11));
          fp = (int)f[b];
        }
        int a = 0, bad = 0, nneg = 0;
        const long long pos0 = sh.acc_pos;
#pragma unroll
        for (int p = 0; p < kPairs; ++p) {
          if (p < np) {
            const int si = __shfl_sync(0xffffffffu, fp, p) > 0 ? 0 : 1;
            const T di = dA[si], dj = dB[si];
            const T gii = __shfl_sync(0xffffffffu, g[2 * p], 2 * p);
            const T gjj = __shfl_sync(0xffffffffu, g[2 * p + 1], 2 * p + 1);
            const T gij = __shfl_sync(0xffffffffu, g[2 * p], 2 * p + 1);
            const T gji = __shfl_sync(0xffffffffu, g[2 * p + 1], 2 * p);
            // R = det(1 + Gamma (1 - G_SS))
            const T m00 = T(1) + di * (T(1) - gii), m01 = -di * gij;
            const T m10 = -dj * gji, m11 = T(1) + dj * (T(1) - gjj);
            const T R = m00 * m11 - m01 * m10;
            const bool acc = __shfl_sync(0xffffffffu, (int)(up < (R < T(0) ? -R : R)), p) != 0;
            if (lane == 0) {
              if (!isfinite(R)) bad = 1;
              if (pos0 + p < c.acc_cap) c.acc_log[pos0 + p] = acc ? 1 : 0;
            }
            if (acc) {
              // X = 1 + (1 - G_SS) Gamma, M = Gamma X^{-1}
              const T x00 = T(1) + (T(1) - gii) * di, x01 = -gij * dj;
              const T x10 = -gji * di, x11 = T(1) + (T(1) - gjj) * dj;
              const T inv = T(1) / (x00 * x11 - x01 * x10);
              const T M00 = di * (x11 * inv), M01 = di * (-x01 * inv);
              const T M10 = dj * (-x10 * inv), M11 = dj * (x00 * inv);
              const bool fut = lane >= 2 * p + 2;
              const T y0 = fut ? M00 * g[2 * p] + M01 * g[2 * p + 1] : T(0);
              const T y1 = fut ? M10 * g[2 * p] + M11 * g[2 * p + 1] : T(0);
#pragma unroll
              for (int r = 2 * p + 2; r < kBlock; ++r) {
                const T gri = __shfl_sync(0xffffffffu, g[r], 2 * p);
                const T grj = __shfl_sync(0xffffffffu, g[r], 2 * p + 1);
                g[r] = fma(gri, y0, fma(grj, y1, g[r]));
              }
              if (lane == p) {
                fp = -fp;
                f[3 * (c0 + p) + k] = (int8_t)fp;
              }
              const int wi = __shfl_sync(0xffffffffu, wq, 2 * p), wj = __shfl_sync(0xffffffffu, wq, 2 * p + 1);
              if (lane == 0) {
                fb.gsite[a] = wi;
                fb.cl[0][a] = di;
                fb.gsite[a + 1] = wj;
                fb.cl[0][a + 1] = dj;
                nneg += R < T(0) ? 1 : 0;
              }
              a += 2;
            }
          }
        }
        if (lane == 0) {
          sh.na = a;
          sh.acc_pos = pos0 + np;
          sh.n_prop += np;
          sh.n_acc += a / 2;
          if (nneg & 1) sh.sign_running = -sh.sign_running;
          if (bad) sh.err |= kErrNaN;
        }
      }
      __syncthreads();
      x.mark(kPhFlip);
      const int a = sh.na;
      if (a == 0) continue;
      flush_block(x, a);
    }
  }
}

// --------------------------------------------------------------------------
// Slice wrapping.  dir = +1: G(tau) = B_tau G(tau-1) B_tau^{-1};
// dir = -1: G(tau-1) = B_tau^{-1} G(tau) B_tau.

// The two products of an FP64 wrap on the tensor cores (digit_gemm.cuh): G_s
// <- E1 (f G_s) E2 with f the diagonal factors of pre (or 1), E1 and E2 the
// digit tables of the model; G_s is packed, receives the first product, is
// packed again and receives the second.  E1 is read transposed, as the other
// paths read it.
template <typename T, bool RES, typename F>
__device__ __forceinline__ void wrap_digits(Cta<T, RES>& x, int s, const unsigned long long* E1, int e1,
                                            const unsigned long long* E2, int e2, F pre) {
  const int N = x.c.N, ld = x.c.ld, ldd = digit_ld(N);
  T* G = x.G(s);
  unsigned long long* D = reinterpret_cast<unsigned long long*>(x.Gt());
  int* red = reinterpret_cast<int*>(x.sh.red);
  int e = kDigitNone;
  PQMC_FOR_2D(i, 0, N, j, 0, N) e = max(e, digit_exp(G[(long)i * ld + j] * pre(i, j)));
  const int EG = digit_cta_max(e, red);
  PQMC_FOR_2D(i, 0, N, j, 0, N) D[(long)j * ld + i] = digit_pack(G[(long)i * ld + j] * pre(i, j), EG);
  __syncthreads();
  e = kDigitNone;
  digit_gemm<true, true>(N, N, N, E1, ldd, 1, D, ld, 1, [e1](int) { return e1; }, [EG](int) { return EG; }, false, false,
                         [&e, G, ld](int i, int j, double v) {
                           G[(long)i * ld + j] = v;
                           e = max(e, digit_exp(v));
                         });
  const int ET = digit_cta_max(e, red);
  PQMC_FOR_2D(i, 0, N, j, 0, N) D[(long)i * ld + j] = digit_pack(G[(long)i * ld + j], ET);
  __syncthreads();
  digit_gemm<true, true>(N, N, N, D, ld, 1, E2, ldd, 1, [ET](int) { return ET; }, [e2](int) { return e2; }, false, false,
                         [G, ld](int i, int j, double v) { G[(long)i * ld + j] = v; });
  __syncthreads();
}

// e^{V} G_s e^{-V} (dir > 0) or e^{-V} G_s e^{V}, slice tau staged
template <typename T, bool RES>
__device__ __forceinline__ void scale_slice(Cta<T, RES>& x, int tau, int dir, int s) {
  const int N = x.c.N, ld = x.c.ld;
  T* G = x.G(s);
  if (dir > 0) {
    PQMC_FOR_2D(i, 0, N, j, 0, N) G[(long)i * ld + j] *= x.vexpT(tau, s, i) * x.vinvT(tau, s, j);
  } else {
    PQMC_FOR_2D(i, 0, N, j, 0, N) G[(long)i * ld + j] *= x.vexpT(tau, s, j) * x.vinvT(tau, s, i);
  }
}

template <bool kTc, bool RES>
__device__ __forceinline__ void wrap(Cta<double, RES>& x, int tau, int dir) {
  const ChainDesc& c = x.c;
  const bool gz = x.gutz(tau);
  x.stage(tau);
  for (int s = 0; s < x.nspec(); ++s) {
    if (!gz && dir > 0) {
      wrap_digits(x, s, c.dEm, c.eEm, c.dEp, c.eEp,
                  [&](int i, int j) { return x.vexpT(tau, s, i) * x.vinvT(tau, s, j); });
    } else {
      if (!gz) wrap_digits(x, s, c.dEp, c.eEp, c.dEm, c.eEm, [](int, int) { return 1.0; });
      scale_slice(x, tau, dir, s);
    }
  }
  __syncthreads();
}

template <bool kTc, bool RES>
__device__ __forceinline__ void wrap(Cta<float, RES>& x, int tau, int dir) {
  const ChainDesc& c = x.c;
  const int N = c.N, ld = c.ld;
  const bool gz = x.gutz(tau);
  float* Gt = x.Gt();
  const float* Em = x.Em();
  const float* Ep = x.Ep();
  if (!gz && RES && x.L.em) {
    // a chain resident in shared memory reads e^{-+dtau K} there: the two
    // tables are copied in from the L2-resident copy shared by all chains
    // (the wrap phase leaves room for them in the scratch)
    const int chunks = N * ld * (int)sizeof(float) / 16;
    int4* dm = reinterpret_cast<int4*>(x.scr + x.L.em);
    int4* dp = reinterpret_cast<int4*>(x.scr + x.L.ep);
    const int4* sm = reinterpret_cast<const int4*>(Em);
    const int4* sp = reinterpret_cast<const int4*>(Ep);
    for (int e = threadIdx.x; e < chunks; e += blockDim.x) {
      dm[e] = sm[e];
      dp[e] = sp[e];
    }
    Em = reinterpret_cast<const float*>(dm);
    Ep = reinterpret_cast<const float*>(dp);
    __syncthreads();
  }
  x.stage(tau);
  if (dir > 0) {
    for (int s = 0; s < x.nspec(); ++s) scale_slice(x, tau, +1, s);
    __syncthreads();
    if (gz) return;
    // Gt = e^{-dtau K} G, G = Gt e^{+dtau K}
    for (int s = 0; s < x.nspec(); ++s) {
      wrap_gemm<kTc, false>(x, N, Em, x.G(s), Gt, ld, EpiStore());
      __syncthreads();
      wrap_gemm<kTc, true>(x, N, Gt, Ep, x.G(s), ld, EpiStore());
      __syncthreads();
    }
  } else {
    if (!gz) {
      for (int s = 0; s < x.nspec(); ++s) {
        wrap_gemm<kTc, false>(x, N, Ep, x.G(s), Gt, ld, EpiStore());
        __syncthreads();
        wrap_gemm<kTc, true>(x, N, Gt, Em, x.G(s), ld, EpiStore());
        __syncthreads();
      }
    }
    for (int s = 0; s < x.nspec(); ++s) scale_slice(x, tau, -1, s);
    __syncthreads();
  }
}

// --------------------------------------------------------------------------
// FP64 stabilisation.

// log|prod_j d_j| and sign(prod_j d_j) of n values in shared memory, summed by
// warp 0 and broadcast through shared memory (collective).
template <typename T, bool RES>
__device__ __forceinline__ void log_det_of(Cta<T, RES>& x, const double* d, int n, int extra_sign_flips, double& logabs, double& sgn) {
  Smem<T>& sh = x.sh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (warp == 0) {
    double la = 0.0;
    int neg = 0;
    for (int j = lane; j < n; j += 32) {
      la += log(fabs(d[j]));
      neg += d[j] < 0 ? 1 : 0;
    }
    la = warp_sum(la);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) neg += __shfl_xor_sync(0xffffffffu, neg, o);
    if (lane == 0) {
      sh.red[0] = la;
      sh.red[1] = ((neg + extra_sign_flips) & 1) ? -1.0 : 1.0;
    }
  }
  __syncthreads();
  logabs = sh.red[0];
  sgn = sh.red[1];
  __syncthreads();
}

// Householder QR of the column-major N x n matrix M (ld ldm).  The explicit
// orthonormal factor goes to Q (column-major, ld N); log|det R| and sign(det R)
// are returned to every thread.  Each reflector is applied to all trailing
// columns in three CTA-wide phases (partial column dots over row chunks, one
// thread per column adds the chunks, a parallel rank-1 update), so no FP64
// work sits in warp-shuffle reductions.
template <typename T, bool RES>
__device__ __forceinline__ void householder_apply(Cta<T, RES>& x, int N, int lda, const double* v, double beta, double* A, int c0, int c1,
                                  int j) {
  double* part = x.qpart();
  double* w = x.qw();
  if (c1 <= c0) return;
  // thread (col, p): rows j + p, j + p + kQRParts, ...
  {
    const int p = threadIdx.x & (kQRParts - 1);
    for (int col = c0 + (int)(threadIdx.x / kQRParts); col < c1; col += (int)(blockDim.x / kQRParts)) {
      const double* a = A + (long)col * lda;
      double d0 = 0.0, d1 = 0.0;
      int i = j + p;
      for (; i + kQRParts < N; i += 2 * kQRParts) {
        d0 = fma(v[i], a[i], d0);
        d1 = fma(v[i + kQRParts], a[i + kQRParts], d1);
      }
      if (i < N) d0 = fma(v[i], a[i], d0);
      part[p * x.c.nmax + col] = d0 + d1;
    }
  }
  __syncthreads();
  for (int col = c0 + threadIdx.x; col < c1; col += blockDim.x) {
    const int nm = x.c.nmax;
    double q[kQRParts];
#pragma unroll
    for (int p = 0; p < kQRParts; ++p) q[p] = part[p * nm + col];
#pragma unroll
    for (int h = kQRParts / 2; h > 0; h >>= 1)
#pragma unroll
      for (int p = 0; p < h; ++p) q[p] += q[p + h];
    w[col] = q[0] * beta;
  }
  __syncthreads();
  {
    const int rows = N - j, total = rows * (c1 - c0);
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
      const int cl = e / rows, i = j + (e - cl * rows), col = c0 + cl;
      A[(long)col * lda + i] = fma(-v[i], w[col], A[(long)col * lda + i]);
    }
  }
  __syncthreads();
}

// reflector of column j (warp 0): v = x - alpha e_j stored over the column
template <typename T, bool RES>
__device__ __forceinline__ void householder_reflector(Cta<T, RES>& x, int N, int ldm, double* M, int j) {
  const int lane = threadIdx.x & 31;
  if ((threadIdx.x >> 5) == 0) {
    double* v = M + (long)j * ldm;
    double s = 0.0;
    for (int i = j + lane; i < N; i += 32) s = fma(v[i], v[i], s);
    s = warp_sum(s);
    if (lane == 0) {
      const double x0 = v[j];
      const double a = x0 > 0 ? -sqrt(s) : sqrt(s);
      const double v0 = x0 - a;
      const double vv = s - x0 * x0 + v0 * v0;
      v[j] = v0;
      x.qbeta()[j] = vv > 0 ? 2.0 / vv : 0.0;
      x.qalpha()[j] = a;
      if (a == 0.0) x.sh.err |= kErrStab;
    }
  }
  __syncthreads();
}

template <typename T, bool RES>
__device__ __forceinline__ void qr_householder(Cta<T, RES>& x, int N, int ldm, int n, double* M, double* Q, double& logabs, double& sgn) {
  for (int j = 0; j < n; ++j) {
    householder_reflector(x, N, ldm, M, j);
    householder_apply(x, N, ldm, M + (long)j * ldm, x.qbeta()[j], M, j + 1, n, j);
  }
  x.mark(kPhQR);
  PQMC_FOR_2D(col, 0, n, i, 0, N) Q[(long)col * N + i] = (i == col) ? 1.0 : 0.0;
  __syncthreads();
  for (int j = n - 1; j >= 0; --j) householder_apply(x, N, N, M + (long)j * ldm, x.qbeta()[j], Q, j, n, j);
  log_det_of(x, x.qalpha(), n, 0, logabs, sgn);
  x.mark(kPhQRForm);
}

// 1 / x by the geometric series: with y an approximation and e = 1 - x y,
// 1 / x = y / (1 - e) = y (1 + e + e^2 + ...); cut after e^2, which is Chebyshev's
// third-order iteration for the root of 1 / y - x (Householder, The Numerical
// Treatment of a Single Nonlinear Equation, 1970).  y is PTX's
// rcp.approx.ftz.f64, good to some 20 bits, so the terms left out are below 2^-60 and the result
// is within 0.5 + 2^-6 ulp.  Three dependent FMAs (65 cycles each) where the division takes
// 646 cycles on the pivots' serial chain; outside the approximation's range the division.
static __device__ __forceinline__ double recip64(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  if (e < 60 || e > 1980) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double r = fma(-x, y, 1.0);
  return fma(y, fma(r, r, r), y);
}

// f(k, i, load(k, i)) for k < n, i < N over the CTA, flat (no idle lanes in a
// row's tail), four loads in flight per thread
template <typename L, typename F>
__device__ __forceinline__ void for_flat4(int n, int N, L load, F f) {
  const int step = (int)blockDim.x, sq = step / N, sr = step - sq * N;
  int k = (int)threadIdx.x / N, i = (int)threadIdx.x - k * N;
  while (k < n) {
    int kk[4], ii[4];
    decltype(load(0, 0)) v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      kk[u] = k;
      ii[u] = i;
      if (k < n) v[u] = load(k, i);
      i += sr;
      k += sq;
      if (i >= N) { i -= N; ++k; }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (kk[u] < n) f(kk[u], ii[u], v[u]);
  }
}

// Cholesky QR of a stack block M (N x n) of the reduced-precision paths:
// C = M^T M = R^T R, Q = M R^{-1}
// (Stathopoulos & Wu, SIAM J. Sci. Comput. 23 (2002); the loss of
// orthogonality grows like eps cond(M)^2, Yamamoto et al., ETNA 44 (2015)).
// With two slices per stabilisation cond(M) stays near 1e2.  The two products,
// M^T M and M R^{-1}, run on the tensor cores from the digits of M
// (digit_gemm.cuh), or as FMA loops for few orbitals; the factor and its inverse
// come from one elimination of [C | I] on the FP64 pipe, both spins together, half
// of the CTA each.  Q goes column-major (ld N) to the stack block.  A block with a
// pivot below 1e-12 of its original diagonal entry (cond(M) above about 1e6)
// takes the Householder QR instead.  R has a positive diagonal, so only
// log|det R| = (1/2) sum_k log(pivot_k) is kept.
//
// The block's digits share one exponent, so the Gram matrix is off by about
// N 2^-58 of the largest element squared, and a column smaller by a factor r sees
// N r^2 2^-58 of its own diagonal.  That is below (r 2^-24)^2, what the FP32
// products leave of the large columns in the small one, for every N; a pivot
// that it spoils falls under the limit and takes the Householder QR.
//
// 72 sites, n = 36, one chain alone on its SM, both spins, per stabilisation: the
// Gram matrix, factor (two barriers, a division and a row scaling per column) and
// column-by-column Q on the FP64 pipe took 358 kcycles; this form takes 187,
// the overlap included.

// digits of a block into D (ld digit_ld(N)); the exponent comes back
template <typename T, bool RES, typename Elem>
__device__ __forceinline__ int pack_block(Cta<T, RES>& x, int N, int n, Elem M) {
  unsigned long long* D = reinterpret_cast<unsigned long long*>(x.scr + x.L.m64);
  const int ldd = digit_ld(N);
  int E = kDigitNone;
  for_flat4(N, n, M, [&](int, int, auto v) { E = max(E, digit_exp(v)); });
  E = digit_cta_max(E, reinterpret_cast<int*>(x.sh.red));
  for_flat4(N, n, M, [&](int i, int k, auto v) { D[(long)k * ldd + i] = digit_pack(v, E); });
  __syncthreads();
  return E;
}

// Elimination of [C | I] for both spins, the part of I that has filled in kept
// below the diagonal: step k takes row k, u_j = row_kj / p_k, from the rows below,
//     row_ij -= C_ki u_j   (C_ki = C_ik; column k, still zero: -C_ki / p_k).
// Row k then holds the Schur complements C_kj right of the diagonal and row
// k of L^{-1} (L unit lower, C = L diag(p) L^T) left of it.  One warp per spin
// runs ahead: it takes row k + 1 first, its pivot, reciprocal and u, while the
// others do the rest of step k: one barrier per column, the reciprocal's
// latency beside the other rows' FMAs (a flat index with constant row
// length: full FP64 warp instructions, no division).  The two warps that run
// ahead sit on different sub-partitions.
template <typename T, bool RES>
__device__ __forceinline__ void chol_eliminate(Cta<T, RES>& x) {
  Smem<T>& sh = x.sh;
  const int H = x.nspec() == 2 ? (int)blockDim.x >> 1 : (int)blockDim.x;
  const int s = (int)threadIdx.x / H, tid = (int)threadIdx.x - s * H, lane = threadIdx.x & 31;
  const int nw = H >> 5, w = tid >> 5, ahead = s < nw ? s : 0;
  const int n = x.nsig(s), ldc = digit_ld(x.nsig(s)), nmax = max(x.nsig(0), x.nsig(1));
  double* C = x.chol(s);
  double* u0 = C + (long)n * ldc;
  double* dlim = u0 + 2 * n;            // smallest pivot accepted
  double* pv = dlim + n;                // pivots
  if (tid == 0) sh.chol_bad[s] = 0;
  for (int k = tid; k < n; k += H) dlim[k] = 1e-12 * C[(long)k * ldc + k];
  __syncthreads();
  auto pivot_row = [&](int r) {
    double* un = u0 + (r & 1) * n;
    const double p = C[(long)r * ldc + r];
    // (positive doubles order like their bits)
    const long long pb = __double_as_longlong(p);
    const bool ok = pb > __double_as_longlong(dlim[r]) && pb < 0x7ff0000000000000ll;
    const double ip = ok ? recip64(p) : 0.0;
    if (lane == 0) {
      pv[r] = p;
      if (!ok) sh.chol_bad[s] = 1;
    }
    for (int j = lane; j < n; j += 32) un[j] = j == r ? ip : C[(long)r * ldc + j] * ip;
  };
  if (w == ahead && n > 0) pivot_row(0);
  __syncthreads();
  const bool bulk = nw == 1 || w != ahead;
  const int rest = nw == 1 ? H : H - 32, tr = nw == 1 ? tid : (w < ahead ? tid : tid - 32);
  const int sq = n > 0 ? rest / n : 0, sr = n > 0 ? rest - sq * n : 0;
  const int i0 = n > 0 && tr >= 0 ? tr / n : 0, j0 = tr - i0 * n;
  for (int k = 0; k + 1 < nmax; ++k) {
    if (k + 1 < n && !sh.chol_bad[s]) {
      const double* uk = u0 + (k & 1) * n;
      const double* Ck = C + (long)k * ldc;
      if (w == ahead) {
        const int r = k + 1;
        double* Cr = C + (long)r * ldc;
        const double m = Ck[r];
        for (int j = lane; j < n; j += 32) Cr[j] = fma(-m, uk[j], j == k ? 0.0 : Cr[j]);
        __syncwarp();
        pivot_row(r);
      }
      if (bulk) {
        int i = k + 2 + i0, j = j0;
        while (i < n) {
          // two elements in flight
          const int i1 = i, j1 = j;
          j += sr;
          i += sq;
          if (j >= n) { j -= n; ++i; }
          const bool two = i < n;
          const int i2 = two ? i : i1, j2 = two ? j : j1;
          double* p1 = C + i1 * ldc + j1;
          double* p2 = C + i2 * ldc + j2;
          const double f1 = Ck[i1], f2 = Ck[i2], u1 = uk[j1], u2 = uk[j2];
          const double a1 = j1 == k ? 0.0 : *p1, a2 = j2 == k ? 0.0 : *p2;
          const double v1 = fma(-f1, u1, a1), v2 = fma(-f2, u2, a2);
          *p1 = v1;
          if (two) {
            *p2 = v2;
            j += sr;
            i += sq;
            if (j >= n) { j -= n; ++i; }
          }
        }
      }
    }
    __syncthreads();
  }
  double* isq = pv + n;                 // 1 / sqrt(pivot)
  if (n > 0 && !sh.chol_bad[s])
    for (int k = tid; k < n; k += H) isq[k] = rsqrt(pv[k]);
  __syncthreads();
}

// Q = M R^{-1} of spin s to the stack block, from the block's digits (exponent
// E) and the elimination; log|det R| comes back.  The factor's digits take its
// place: column j of R^{-1} is row j of L^{-1} / sqrt(p_j), with 1 / sqrt(p_j)
// on the diagonal.
template <typename T, bool RES>
__device__ __forceinline__ double chol_form_q(Cta<T, RES>& x, int s, int E, double* Q) {
  Smem<T>& sh = x.sh;
  const int N = x.c.N, n = x.nsig(s), ldd = digit_ld(N), ldc = digit_ld(n);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  const unsigned long long* D = reinterpret_cast<const unsigned long long*>(x.scr + x.L.m64);
  double* C = x.chol(s);
  const double* pv = C + (long)n * ldc + 3 * n;
  const double* isq = pv + n;
  int* ex = reinterpret_cast<int*>(C + (long)n * ldc);       // (u's place)
  for (int j = warp; j < n; j += nw) {
    const double f = isq[j];
    double* row = C + (long)j * ldc;
    unsigned long long* X = reinterpret_cast<unsigned long long*>(row);
    int e = lane == 0 ? digit_exp(f) : kDigitNone;
    for (int c = lane; c < j; c += 32) e = max(e, digit_exp(row[c] * f));
    e = __reduce_max_sync(0xffffffffu, e);
    for (int c = lane; c < ldc; c += 32) X[c] = c < j ? digit_pack(row[c] * f, e) : c == j ? digit_pack(f, e) : kDigitZero;
    if (lane == 0) ex[j] = e;
  }
  if (warp == 0) {
    double la = 0.0;
    for (int k = lane; k < n; k += 32) la += log(pv[k]);
    la = warp_sum(la);
    if (lane == 0) sh.red[0] = 0.5 * la;
  }
  __syncthreads();
  const double logabs = sh.red[0];
  digit_gemm<false, true>(N, n, n, D, 1, ldd, reinterpret_cast<const unsigned long long*>(C), ldc, 1,
                          [E](int) { return E; }, [ex](int j) { return ex[j]; }, false, true,
                          [Q, N](int i, int j, double v) { Q[(long)j * N + i] = v; });
  __syncthreads();
  return logabs;
}

// Invert O_s (n_s x n_s, row-major) in place for both spins at once by
// Gauss-Jordan elimination with partial pivoting (Golub & Van Loan, section
// 3.2), one half of the CTA per spin.  Rows are not interchanged: step j
// takes the largest |A_ij| over the rows not used yet (row r_j), and at the end
// (O^{-1})_{j, r_c} = A_{r_j, c} (gj_rows; the caller reads the inverse through
// it).  A step is one barrier for the scaled pivot row and one for the
// elimination, one FP64 FMA per element over a flat index; meanwhile the
// half's first warp eliminates column j + 1 first and finds its pivot and
// reciprocal, so that their latency (shuffles, five dependent FP64 steps)
// passes beside the others' FMAs, which the FP64 pipe bounds: 2 n^2 / 32 warp
// instructions of 16 cycles (1300 cycles at n = 36; a step took 5.7 kcycles
// with the search, the interchange and a division between two barriers).
// Leaves log|det O_s| and sign(det O_s) in sh.gj_logabs, sh.gj_sign.
template <typename T, bool RES>
__device__ __forceinline__ void gj_invert2(Cta<T, RES>& x) {
  Smem<T>& sh = x.sh;
  const int half = x.nspec() == 2 ? (int)blockDim.x >> 1 : (int)blockDim.x;   // threads per species
  const int s = (int)threadIdx.x / half;
  const int tid = (int)threadIdx.x - s * half, lane = threadIdx.x & 31;
  const int nw = half >> 5, w = tid >> 5, ahead = s < nw ? s : 0;   // (on different sub-partitions)
  const bool first = w == ahead;
  const int n = x.nsig(s), nmax = max(x.nsig(0), x.nsig(1));
  double* A = x.Ob(s);
  double* f = x.gj_col(s);              // column j before step j, two steps in flight: f[(j & 1) n ..]
  double* R = x.gj_row(s);              // scaled pivot row of the step
  int* rows = x.gj_rows(s);
  unsigned used = 0;                    // bit b: row lane + 32 b has been a pivot row
  // column j at hand in f: pivot row and reciprocal (first warp of the half)
  auto pick = [&](int j) {
    const double* fj = f + (j & 1) * n;
    unsigned long long best = 0;
    int bi = -1;
    for (int i = lane, b = 0; i < n; i += 32, ++b) {
      // |x| is compared through the bit pattern with the sign cleared, which
      // orders non-negative doubles like their values
      const unsigned long long v = (unsigned long long)__double_as_longlong(fj[i]) & 0x7fffffffffffffffull;
      if (!((used >> b) & 1u) && (bi < 0 || v > best)) { best = v; bi = i; }
    }
    const unsigned hi = (unsigned)(best >> 32), top = __reduce_max_sync(0xffffffffu, bi < 0 ? 0u : hi);
    const unsigned lo = __reduce_max_sync(0xffffffffu, (bi >= 0 && hi == top) ? (unsigned)best : 0u);
    const bool mine = bi >= 0 && hi == top && (unsigned)best == lo;
    const int r = (int)__reduce_min_sync(0xffffffffu, mine ? (unsigned)bi : 0xffffffffu);   // ties to the lower row
    if ((r & 31) == lane) used |= 1u << (r >> 5);
    const double p = fj[r];
    if (lane == 0) {
      x.pval(s)[j] = p;
      rows[j] = r;
      sh.gj_ip[s] = p != 0.0 ? recip64(p) : 0.0;
      if (p == 0.0) atomicOr(&sh.err, kErrStab);
    }
  };
  if (first && n > 0) {
    for (int i = lane; i < n; i += 32) f[i] = A[(long)i * n];
    __syncwarp();
    pick(0);
  }
  const int rest = nw > 1 ? half - 32 : half, tr = nw == 1 || w < ahead ? tid : tid - 32;
  const int sq = n > 0 ? rest / n : 0, sr = n > 0 ? rest - sq * n : 0;
  const int i0 = n > 0 && tr >= 0 ? tr / n : 0, j0 = tr - i0 * n;
  __syncthreads();
  for (int j = 0; j < nmax; ++j) {
    const double* fj = f + (j & 1) * n;
    double* fn = f + ((j + 1) & 1) * n;
    const int r = j < n ? rows[j] : 0;
    if (j < n) {
      const double ip = sh.gj_ip[s];
      for (int c = tid; c < n; c += half) R[c] = c == j ? ip : A[(long)r * n + c] * ip;
    }
    __syncthreads();
    x.mark(kPhGJPivot);
    if (j < n) {
      if (first && j + 1 < n) {
        const double rn = R[j + 1];
        for (int i = lane; i < n; i += 32) {
          const double v = i == r ? rn : fma(-fj[i], rn, A[(long)i * n + j + 1]);
          A[(long)i * n + j + 1] = v;
          fn[i] = v;
        }
        __syncwarp();
        pick(j + 1);
      }
      if (!first || nw == 1) {
        int i = i0, c = j0;
        while (i < n) {
          // two elements in flight
          const int i1 = i, c1 = c;
          c += sr;
          i += sq;
          if (c >= n) { c -= n; ++i; }
          const bool two = i < n;
          const int i2 = two ? i : i1, c2 = two ? c : c1;
          double* p1 = A + i1 * n + c1;
          double* p2 = A + i2 * n + c2;
          const double f1 = fj[i1], f2 = fj[i2], r1 = R[c1], r2 = R[c2];
          const double a1 = c1 == j ? 0.0 : *p1, a2 = c2 == j ? 0.0 : *p2;
          const double v1 = i1 == r ? r1 : fma(-f1, r1, a1), v2 = i2 == r ? r2 : fma(-f2, r2, a2);
          if (c1 != j + 1) *p1 = v1;
          if (two && c2 != j + 1) *p2 = v2;
          if (two) {
            c += sr;
            i += sq;
            if (c >= n) { c -= n; ++i; }
          }
        }
      }
    }
    __syncthreads();
    x.mark(kPhGJElim);
  }
  // parity of the permutation j -> r_j: its inversions
  if (threadIdx.x < 2) sh.nswap[threadIdx.x] = 0;
  __syncthreads();
  {
    int inv = 0;
    for (int a = tid; a < n; a += half)
      for (int b = a + 1; b < n; ++b) inv += rows[a] > rows[b] ? 1 : 0;
    if (inv) atomicAdd(&sh.nswap[s], inv);
  }
  __syncthreads();
  for (int sp = 0; sp < 2; ++sp) {
    double la, sg;
    log_det_of(x, x.pval(sp), x.nsig(sp), sh.nswap[sp], la, sg);
    if (threadIdx.x == 0) {
      sh.gj_logabs[sp] = la;
      sh.gj_sign[sp] = sg;
    }
  }
  __syncthreads();
  x.mark(kPhGJTail);
}

// The inverse of spin s as a plain matrix, in place: row j from row r_j, then
// column r_c from column c, as interchanges by one warp (the FP64 path and the
// FP64 diagnostics; the reduced paths read through gj_rows instead).
template <typename T, bool RES>
__device__ __forceinline__ void gj_unpermute(Cta<T, RES>& x, int s) {
  const int n = x.nsig(s);
  double* A = x.Ob(s);
  const int* rows = x.gj_rows(s);
  int* at = x.gj_rows(s) + n;           // original row at each place
  int* swp = at + n;                    // place interchanged with j
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    for (int i = lane; i < n; i += 32) at[i] = i;
    __syncwarp();
    for (int j = 0; j < n; ++j) {
      // place j takes original row r_j: find where it is now (at or after j)
      unsigned p = 0xffffffffu;
      for (int i = j + lane; i < n; i += 32)
        if (at[i] == rows[j]) p = (unsigned)i;
      p = __reduce_min_sync(0xffffffffu, p);
      if ((int)p != j)
        for (int c = lane; c < n; c += 32) {
          const double t = A[(long)j * n + c];
          A[(long)j * n + c] = A[(long)p * n + c];
          A[(long)p * n + c] = t;
        }
      if (lane == 0) {
        at[p] = at[j];
        at[j] = rows[j];
        swp[j] = (int)p;
      }
      __syncwarp();
    }
    // columns: the same interchanges, last first (column r_c from column c)
    for (int j = n - 1; j >= 0; --j) {
      const int p = swp[j];
      if (p != j)
        for (int i = lane; i < n; i += 32) {
          const double t = A[(long)i * n + j];
          A[(long)i * n + j] = A[(long)i * n + p];
          A[(long)i * n + p] = t;
        }
      __syncwarp();
    }
  }
  __syncthreads();
}

static __device__ void copy_block(const double* src, double* dst, int n) {
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += blockDim.x) dst[e] = src[e];
  __syncthreads();
}

template <typename T, bool RES>
__device__ __forceinline__ double* stack_block(const Cta<T, RES>& x, double* base, int b, int s) {
  return base + ((long)b * 2 + s) * x.c.N * x.c.nmax;
}

// Calls f(element(i, k)) with the accessor of the block phase_stack left for
// spin s: a product in the path precision, or e^{V(s_tau0)} P in FP64 for the
// blocks at the ends of the projection.
template <typename T, bool RES, typename F>
__device__ __forceinline__ void with_block(Cta<T, RES>& x, int left, int s, F f) {
  const int ldn = x.ldn(s), N = x.c.N;
  if (x.sh.src == 2) {
    const double* P = x.c.P + (long)s * N * x.c.nmax;
    const int tau = left ? x.c.Ltau + 1 : 0;
    f([&x, P, tau, s, N](int i, int k) { return x.vexp(tau, s, i) * P[(long)k * N + i]; });
  } else {
    const T* Mt = x.sh.src ? x.Mt2() : x.Mt(s);
    f([Mt, ldn](int i, int k) { return Mt[(long)i * ldn + k]; });
  }
}
// M64 = that block, column-major
template <typename T, bool RES>
__device__ __forceinline__ void block_to_m64(Cta<T, RES>& x, int left, int s) {
  const int ldm = m64_ld(x.c.N);
  double* M = x.M64();
  with_block(x, left, s, [&](auto e) {
    PQMC_FOR_2D(k, 0, x.nsig(s), i, 0, x.c.N) M[(long)k * ldm + i] = (double)e(i, k);
  });
  __syncthreads();
}

// Right stack block b: QR of B_{b n} ... B_{(b-1)n+1} Q_R[b-1] (b >= 1) or of B_0 P (b = 0).
// Left stack block b holds (B_L(b n))^T = Q T^T: QR of
// B_{bn+1}^T ... B_{(b+1)n}^T Q_L[b+1] (b < nb) or of e^{V(s_{Ltau+1})} P (b = nb).
// phase_stack forms the block to factorise, of spin s (sh.src says where): the
// slice products run in the path precision on a row-major copy.
template <typename T, bool RES>
__device__ __noinline__ void phase_stack(int b, int left, int s) {
  auto x = this_cta<T, RES>();
  const ChainDesc& c = x.c;
  const int N = c.N, n_stab = c.n_stab;
  const int n = x.nsig(s), ldn = x.ldn(s);
  T* Mt = x.Mt(s);
  T* Mt2 = x.Mt2();
  constexpr bool f64 = std::is_same<T, double>::value;
  // Mt2 = e^{-dtau K} Mt: on the tensor cores in FP64 (digits of Mt in M64's
  // place).  The columns of a block grow apart by up to e^{6 dtau} per slice
  // and the product mixes rows only, so each column has its own exponent: a
  // shared one cost the small columns their digits (free fermions, 72 sites, 10
  // slices of dtau = 0.8: log det off by 2.7e-9, now by less than 1e-12).
  // It enters as a factor 2^e of the result: as a second exponent in the
  // digits' assembly it took 1.6% of a one-chain sweep of 18 sites.
  auto product = [&](const T* from, T* to) {
    if constexpr (f64) {
      const int ldd = digit_ld(N), ldk = N + (N & 1), e1 = c.eEm;
      unsigned long long* D = reinterpret_cast<unsigned long long*>(x.M64());
      double* sc = x.qbeta();                        // (the QR's vectors come later)
      for (int k = threadIdx.x >> 5; k < n; k += blockDim.x >> 5) {
        int e = kDigitNone;
        for (int i = threadIdx.x & 31; i < N; i += 32) e = max(e, digit_exp(from[(long)i * ldn + k]));
        e = __reduce_max_sync(0xffffffffu, e);
        for (int i = threadIdx.x & 31; i < N; i += 32) D[(long)k * ldk + i] = digit_pack(from[(long)i * ldn + k], e);
        // (2^{e - 1}: every exponent's is a normal number)
        if ((threadIdx.x & 31) == 0)
          sc[k] = __longlong_as_double(e == kDigitBad ? 0x7ff8000000000000ll : e == kDigitNone ? 0ll : (long long)(e + 1022) << 52);
      }
      __syncthreads();
      digit_gemm<true, true>(N, n, N, c.dEm, ldd, 1, D, ldk, 1, [e1](int) { return e1; }, [](int) { return 1; }, false,
                             false, [to, ldn, sc](int i, int j, double v) { to[(long)i * ldn + j] = v * sc[j]; });
    } else {
      cta_gemm_f32<false>(N, n, N, x.Em(), c.ld, from, ldn, to, ldn, EpiStore());
    }
  };
  int src = 0;
  if (left ? b == c.nb : b == 0) {
    const int tau = left ? c.Ltau + 1 : 0;
    x.stage(tau);
    src = 2;
  } else {
    const double* prev = left ? stack_block(x, c.Lst, b + 1, s) : stack_block(x, c.Rst, b - 1, s);
    PQMC_FOR_2D(k, 0, n, i, 0, N) Mt[(long)i * ldn + k] = (T)prev[(long)k * N + i];
    if (!left) {
      for (int tau = (b - 1) * n_stab + 1; tau <= b * n_stab; ++tau) {
        x.stage(tau);
        PQMC_FOR_2D(i, 0, N, k, 0, n) Mt[(long)i * ldn + k] *= x.vexpT(tau, s, i);
        __syncthreads();
        product(Mt, Mt2);
        __syncthreads();
        T* t = Mt; Mt = Mt2; Mt2 = t;
        src ^= 1;
      }
    } else {
      __syncthreads();
      for (int tau = (b + 1) * n_stab; tau > b * n_stab; --tau) {
        product(Mt, Mt2);
        x.stage(tau);
        PQMC_FOR_2D(i, 0, N, k, 0, n) Mt[(long)i * ldn + k] = x.vexpT(tau, s, i) * Mt2[(long)i * ldn + k];
        __syncthreads();
      }
    }
  }
  if (!f64 && src == 1) {
    // (an odd number of products upwards: Mt is the work buffer now)
    for (int e = threadIdx.x; e < N * ldn; e += blockDim.x) Mt2[e] = Mt[e];
    src = 0;
  }
  if (threadIdx.x == 0) x.sh.src = src;
  __syncthreads();
  if (f64) block_to_m64(x, left, s);
  x.mark(kPhStack);
}

// digits of the block of spin s and, with gram, its Gram matrix (upper triangle)
template <typename T, bool RES>
__device__ __noinline__ int phase_digits(int left, int s, bool gram) {
  auto x = this_cta<T, RES>();
  const int N = x.c.N, n = x.nsig(s), ldd = digit_ld(N), ldc = digit_ld(n);
  int E = 0;
  with_block(x, left, s, [&](auto e) { E = pack_block(x, N, n, e); });
  if (gram) {
    const unsigned long long* D = reinterpret_cast<const unsigned long long*>(x.scr + x.L.m64);
    double* C = x.chol(s);
    auto eM = [E](int) { return E; };
    digit_gemm<true, true>(n, n, N, D, ldd, 1, D, ldd, 1, eM, eM, true, false,
                           [C, ldc](int i, int j, double v) { C[(long)i * ldc + j] = v; });
    __syncthreads();
  }
  x.mark(kPhOverlap);
  return E;
}

// Up to 16 orbitals the reduced paths' three FP64 products of a stabilisation
// (Gram matrix, Q, overlap) are FMA loops, one element per thread: the fixed work
// of a digit tile (packing, fragments, assembly) is more than these few FMAs.
// ms per sweep by digits and by FMAs, 20 slices: 8 sites x 608 chains 1.65, 1.29; 18
// sites x 304 1.21, 1.01; 32 sites (n = 16) x 304 1.89, 1.66, packed densely (x 1216, 64
// threads) 13.5, 10.1; 72 sites with n = 19 4.67, 4.74; 50 sites (n = 25) x 608 6.41, 6.53; 64
// sites with n = 28 x 256 (120 slices) 21.5, 28.0.  One function for all of it and one
// for the product, loops rolled (unrolled and inlined: 11.5 for the dense case),
// because what they add to the code costs the larger chains 0.1 to 0.2% (inlined 0.2 to 0.6).
constexpr int kSmallOrbitals = 16;
template <typename T, bool RES>
__device__ __forceinline__ bool small_products(const Cta<T, RES>& x) {
  return x.c.nmax <= kSmallOrbitals;
}

// C(i, j) = sum_k A[i lda + k] B[j ldb + k] (with upper, only j >= i)
static __device__ __noinline__ void small_product(int M, int Nn, int K, const double* A, int lda, const double* B, int ldb,
                                                     bool upper, double* C, int ldc) {
#pragma unroll 1
  for (int e = threadIdx.x; e < M * Nn; e += blockDim.x) {
    const int i = e / Nn, j = e - i * Nn;
    if (upper && j < i) continue;
    const double* a = A + i * lda;
    const double* b = B + j * ldb;
    double v0 = 0.0, v1 = 0.0;
    int k = 0;
#pragma unroll 1
    for (; k + 1 < K; k += 2) {
      v0 = fma(a[k], b[k], v0);
      v1 = fma(a[k + 1], b[k + 1], v1);
    }
    if (k < K) v0 = fma(a[k], b[k], v0);
    C[i * ldc + j] = v0 + v1;
  }
}

// the block of spin s in M64 and, with gram, its Gram matrix
template <typename T, bool RES>
__device__ __forceinline__ void small_gram(Cta<T, RES>& x, int left, int s, bool gram) {
  const int N = x.c.N, n = x.nsig(s);
  block_to_m64(x, left, s);
  if (gram) {
    small_product(n, n, N, x.M64(), m64_ld(N), x.M64(), m64_ld(N), true, x.chol(s), digit_ld(n));
    __syncthreads();
  }
}
// Q = M R^{-1} from M64: q_ij = (m_ij + sum_{k < j} m_ik (L^{-1})_jk) / sqrt(p_j); log|det R| comes back
template <typename T, bool RES>
__device__ __forceinline__ double small_form_q(Cta<T, RES>& x, int s, double* Q) {
  const int N = x.c.N, n = x.nsig(s), ldc = digit_ld(n), ldm = m64_ld(N);
  const double* M = x.M64();
  const double* C = x.chol(s);
  const double* pv = C + (long)n * ldc + 3 * n;
  const double* isq = pv + n;
  if (threadIdx.x < 32) {
    const double la = warp_sum((int)threadIdx.x < n ? log(pv[threadIdx.x]) : 0.0);
    if (threadIdx.x == 0) x.sh.red[0] = 0.5 * la;
  }
#pragma unroll 1
  for (int e = threadIdx.x; e < N * n; e += blockDim.x) {
    const int j = e / N, i = e - j * N;
    double v = M[j * ldm + i];
#pragma unroll 1
    for (int k = 0; k < j; ++k) v = fma(M[k * ldm + i], C[j * ldc + k], v);
    Q[e] = v * isq[j];
  }
  __syncthreads();
  return x.sh.red[0];
}
template <typename T, bool RES>
__device__ __noinline__ void phase_factor() {
  auto x = this_cta<T, RES>();
  chol_eliminate(x);
  x.mark(kPhQR);
}
template <typename T, bool RES>
__device__ __noinline__ double phase_form_q(int b, int left, int s, int E) {
  auto x = this_cta<T, RES>();
  const double la = chol_form_q(x, s, E, stack_block(x, left ? x.c.Lst : x.c.Rst, b, s));
  x.mark(kPhQRForm);
  return la;
}
template <typename T, bool RES>
__device__ __noinline__ void phase_householder(int b, int left, int s, double* logabs, double* sgn) {
  auto x = this_cta<T, RES>();
  const int N = x.c.N, n = x.nsig(s);
  if (!std::is_same<T, double>::value) block_to_m64(x, left, s);
  qr_householder(x, N, m64_ld(N), n, x.M64(), x.Q64(), *logabs, *sgn);
  copy_block(x.Q64(), stack_block(x, left ? x.c.Lst : x.c.Rst, b, s), N * n);
  x.mark(kPhQR);
}

// the weight of stack block b of spin s, log|det R| and sign of R given
template <typename T, bool RES>
__device__ __forceinline__ void stack_weight(Cta<T, RES>& x, int b, int left, int s, double la, double sg) {
  const ChainDesc& c = x.c;
  if (threadIdx.x == 0) {
    double* lg = left ? c.Llog : c.Rlog;
    const bool first = left ? b == c.nb : b == 0;
    const int bp = left ? b + 1 : b - 1;
    lg[(b * 2 + s) * 2 + 0] = (first ? 0.0 : lg[(bp * 2 + s) * 2 + 0]) + la;
    lg[(b * 2 + s) * 2 + 1] = (first ? 1.0 : lg[(bp * 2 + s) * 2 + 1]) * sg;
  }
  __syncthreads();
}

// spins whose Cholesky factor broke down
template <typename T, bool RES>
__device__ __forceinline__ void householder_fallback(Cta<T, RES>& x, int b, int left, const bool bad[2]) {
  double la, sg;
  for (int s = 0; s < x.nspec(); ++s)
    if (bad[s]) {
      phase_householder<T, RES>(b, left, s, &la, &sg);
      stack_weight(x, b, left, s, la, sg);
    }
}

template <typename T, bool RES>
__device__ __forceinline__ void small_overlap(Cta<T, RES>& x, int b) {
  const int N = x.c.N;
  for (int s = 0; s < x.nspec(); ++s)
    small_product(x.nsig(s), x.nsig(s), N, stack_block(x, x.c.Lst, b, s), N, stack_block(x, x.c.Rst, b, s), N, false, x.Ob(s),
                  x.nsig(s));
  __syncthreads();
  x.mark(kPhOverlap);
}

// Cholesky QR of both species' blocks by the small products, or (left < 0) the overlap
template <typename T, bool RES>
__device__ __noinline__ void phase_small(int b, int left) {
  auto x = this_cta<T, RES>();
  if (left < 0) {
    small_overlap(x, b);
    return;
  }
  for (int s = 0; s < x.nspec(); ++s) small_gram(x, left, s, true);
  x.mark(kPhOverlap);
  phase_factor<T, RES>();
  const bool bad[2] = {x.sh.chol_bad[0] != 0, x.sh.chol_bad[1] != 0};
  for (int s = x.nspec() - 1; s >= 0; --s) {
    if (bad[s]) continue;
    if (s < x.nspec() - 1) small_gram(x, left, s, false);   // (M64 holds the last species' block)
    stack_weight(x, b, left, s, small_form_q(x, s, stack_block(x, left ? x.c.Lst : x.c.Rst, b, s)), 1.0);
  }
  x.mark(kPhQRForm);
  householder_fallback(x, b, left, bad);
}

// the new stack block b of both species
template <typename T, bool RES>
__device__ __forceinline__ void push_block(int b, int left) {
  auto x = this_cta<T, RES>();
  if constexpr (std::is_same<T, double>::value) {
    double la, sg;
    for (int s = 0; s < x.nspec(); ++s) {
      phase_stack<T, RES>(b, left, s);
      phase_householder<T, RES>(b, left, s, &la, &sg);
      stack_weight(x, b, left, s, la, sg);
    }
  } else {
    for (int s = 0; s < x.nspec(); ++s) phase_stack<T, RES>(b, left, s);
    if (small_products(x)) {
      phase_small<T, RES>(b, left);
      return;
    }
    int E = 0;
    for (int s = 0; s < x.nspec(); ++s) E = phase_digits<T, RES>(left, s, true);
    phase_factor<T, RES>();
    // the digits at hand are the last species'
    const bool bad[2] = {x.sh.chol_bad[0] != 0, x.sh.chol_bad[1] != 0};
    for (int s = x.nspec() - 1; s >= 0; --s) {
      if (bad[s]) continue;
      if (s < x.nspec() - 1) E = phase_digits<T, RES>(left, s, false);
      stack_weight(x, b, left, s, phase_form_q<T, RES>(b, left, s, E), 1.0);
    }
    householder_fallback(x, b, left, bad);
  }
}

// Fused epilogue of the G assembly: g = delta_ij - v, compare with the
// propagated G, overwrite it.
template <typename T>
struct EpiFresh {
  T* G;
  int ld;
  T* dmax;
  template <typename A, typename TC> __device__ void operator()(TC*, int, int, int i, int j, A v) const {
    const T g = (i == j ? T(1) : T(0)) - (T)v;
    T& ref = G[(long)i * ld + j];
    const T d = fabs(ref - g);
    *dmax = d > *dmax ? d : *dmax;
    ref = g;
  }
};

// Epilogue of the FP64 diagnostic assembly: g = delta_ij - v in FP64 against
// the propagated G (read only).
template <typename T>
struct EpiDiff64 {
  const T* G;
  int ld;
  double* dmax;
  double* gmax;      // largest |G_FP64| element
  template <typename A, typename TC> __device__ void operator()(TC*, int, int, int i, int j, A v) const {
    const double g = (i == j ? 1.0 : 0.0) - (double)v;
    const double d = fabs((double)G[(long)i * ld + j] - g);
    *dmax = d > *dmax ? d : *dmax;
    *gmax = fabs(g) > *gmax ? fabs(g) : *gmax;
  }
};

// G_fresh = 1 - Q_R X Q_L^T for spin s with X = (Q_L^T Q_R)^{-1} (FP64, n x n
// row-major at Xinv), in the path precision; the FP64 diagnostics of
// opts.dg_fp64 around it.
template <typename T, bool RES>
__device__ __forceinline__ void assemble_spin(Cta<T, RES>& x, int s, const double* QR, const double* QL, const double* Xinv, int ns,
                              bool record, T& dmax, double& dmax64) {
  const ChainDesc& c = x.c;
  Smem<T>& sh = x.sh;
  const int N = c.N, ld = c.ld;
  T* Y = x.Yb();
  const T* qr = reinterpret_cast<const T*>(QR);
  const T* ql = reinterpret_cast<const T*>(QL);
  if constexpr (!std::is_same<T, double>::value) {
    if ((c.dg64 == 1 || c.dg64 == 3) && record) {
      // Y64 = O^{-1} Q_L^T (n x N, FP64, in the space of the path-precision
      // copies of Q_R and Q_L, which are written after it), then
      // max |G - (1 - Q_R Y64)| over the propagated G (mode 3: divided by
      // max(1, max |G_FP64|), per spin)
      double* y64 = reinterpret_cast<double*>(x.QRt());
      cta_gemm<double>(ns, N, ns, Xinv, ns, 1, QL, N, 1, y64, N, 1, EpiStore());
      __syncthreads();
      double d_s = 0.0, g_s = 0.0;
      EpiDiff64<T> ed{x.G(s), ld, &d_s, &g_s};
      cta_gemm<double>(N, N, ns, QR, 1, N, y64, N, 1, (double*)nullptr, 0, 0, ed);
      if (c.dg64 == 3) {
        d_s = cta_max(d_s, sh.red);
        g_s = cta_max(g_s, sh.red);
        d_s /= fmax(1.0, g_s);
      }
      dmax64 = fmax(dmax64, d_s);
      __syncthreads();
    }
    T* qrt = x.QRt();
    T* qlt = x.QLt();
    for_flat4(ns, N, [QR, N](int k, int i) { return QR[(long)k * N + i]; },
              [qrt, ld](int k, int i, double v) { qrt[(long)k * ld + i] = (T)v; });
    for_flat4(ns, N, [QL, N](int k, int i) { return QL[(long)k * N + i]; },
              [qlt, ld](int k, int i, double v) { qlt[(long)k * ld + i] = (T)v; });
    qr = qrt;
    ql = qlt;
    __syncthreads();
  }
  if constexpr (std::is_same<T, double>::value) {
    cta_gemm<T>(ns, N, ns, Xinv, ns, 1, ql, N, 1, Y, ld, 1, EpiStore());
  } else {
    // O^{-1} to the path precision once (in the order of its rows and columns),
    // then a path-precision product
    T* ot = x.Ot();
    const int ldo = pad4(ns);
    if (c.dg64) {
      PQMC_FOR_2D(j, 0, ns, k, 0, ns) ot[(long)j * ldo + k] = (T)Xinv[(long)j * ns + k];
    } else {
      const int* rows = x.gj_rows(s);
      PQMC_FOR_2D(j, 0, ns, k, 0, ns) ot[(long)j * ldo + rows[k]] = (T)Xinv[(long)rows[j] * ns + k];
    }
    __syncthreads();
    cta_gemm_f32<true>(ns, N, ns, ot, ldo, ql, ld, Y, ld, EpiStore());
  }
  __syncthreads();
  EpiFresh<T> epi{x.G(s), ld, &dmax};
  if constexpr (std::is_same<T, double>::value) cta_gemm<T>(N, N, ns, qr, 1, N, Y, ld, 1, (T*)nullptr, 0, 0, epi);
  else cta_gemm_f32<false>(N, N, ns, qr, ld, Y, ld, nullptr, 0, epi);
  if constexpr (!std::is_same<T, double>::value) {
    if (c.dg64 == 2 && record) {
      // the refreshed G itself against G_FP64 (the path-precision copies of
      // Q_R and Q_L are no longer needed: Y64 takes their space)
      __syncthreads();
      double* y64 = reinterpret_cast<double*>(x.QRt());
      cta_gemm<double>(ns, N, ns, Xinv, ns, 1, QL, N, 1, y64, N, 1, EpiStore());
      __syncthreads();
      double g_s = 0.0;
      EpiDiff64<T> ed{x.G(s), ld, &dmax64, &g_s};
      cta_gemm<double>(N, N, ns, QR, 1, N, y64, N, 1, (double*)nullptr, 0, 0, ed);
    }
  }
  __syncthreads();
}

// O_s = Q_L^T Q_R of both spins, from the digits of the two blocks (columns of
// orthonormal matrices: exponent 1; should an element reach 2, the blocks are
// packed again against the largest).
template <typename T, bool RES>
__device__ __noinline__ void phase_overlap(int b) {
  auto x = this_cta<T, RES>();
  const ChainDesc& c = x.c;
  const int N = c.N, ldd = digit_ld(N);
  unsigned long long* DL = reinterpret_cast<unsigned long long*>(x.scr + x.L.dq);
  for (int s = 0; s < x.nspec(); ++s) {
    const int n = x.nsig(s);
    unsigned long long* DR = DL + (long)ldd * n;
    const double* QL = stack_block(x, c.Lst, b, s);
    const double* QR = stack_block(x, c.Rst, b, s);
    int E = 1;
    for (int pass = 0; pass < 2; ++pass) {
      int e = kDigitNone;
      auto pack = [&](const double* Q, unsigned long long* D) {
        for_flat4(n, N, [Q, N](int k, int i) { return Q[(long)k * N + i]; }, [&](int k, int i, double v) {
          e = max(e, digit_exp(v));
          D[(long)k * ldd + i] = digit_pack(v, E);
        });
      };
      pack(QL, DL);
      pack(QR, DR);
      const bool again = __syncthreads_or(e > E) != 0;
      if (!again) break;
      E = digit_cta_max(e, reinterpret_cast<int*>(x.sh.red));
      __syncthreads();
    }
    double* O = x.Ob(s);
    auto eQ = [E](int) { return E; };
    digit_gemm<true, true>(n, n, N, DL, ldd, 1, DR, ldd, 1, eQ, eQ, false, false,
                     [O, n](int i, int j, double v) { O[(long)i * n + j] = v; });
    __syncthreads();
  }
  x.mark(kPhOverlap);
}
template <typename T, bool RES>
__device__ __noinline__ void phase_inverse() {
  auto x = this_cta<T, RES>();
  gj_invert2(x);
  if (std::is_same<T, double>::value || x.c.dg64)
    for (int s = 0; s < x.nspec(); ++s) gj_unpermute(x, s);
  x.mark(kPhLU);
}
template <typename T, bool RES>
__device__ __noinline__ void phase_assemble(int b, bool record) {
  auto x = this_cta<T, RES>();
  const ChainDesc& c = x.c;
  Smem<T>& sh = x.sh;
  T dmax = T(0);
  double dmax64 = 0.0;
  double sign_total = 1.0;
  for (int s = 0; s < x.nspec(); ++s) {
    assemble_spin(x, s, stack_block(x, c.Rst, b, s), stack_block(x, c.Lst, b, s), x.Ob(s), x.nsig(s), record, dmax, dmax64);
    const double l_tot = c.Rlog[(b * 2 + s) * 2 + 0] + sh.gj_logabs[s] + c.Llog[(b * 2 + s) * 2 + 0];
    const double s_tot = c.Rlog[(b * 2 + s) * 2 + 1] * sh.gj_sign[s] * c.Llog[(b * 2 + s) * 2 + 1];
    if (threadIdx.x == 0) {
      sh.logw_spin[s] = l_tot;
      sh.sign_spin[s] = s_tot;
    }
    sign_total *= s_tot;
    __syncthreads();
  }
  x.mark(kPhAssemble);
  const double dm = cta_max((c.dg64 && record) ? dmax64 : (double)dmax, sh.red);
  if (threadIdx.x == 0) {
    for (int s = x.nspec(); s < 2; ++s) {
      sh.logw_spin[s] = 0.0;
      sh.sign_spin[s] = 1.0;
    }
    if (!isfinite(dm)) sh.err |= kErrNaN;
    if (record) {
      sh.dGmax = fmax(sh.dGmax, dm);
      c.dG[c.st->n_dG % kDGHistory] = dm;
      c.st->n_dG++;
    }
    c.st->sign_stack = sign_total;
  }
  __syncthreads();
}

// G <- 1 - Q_R (Q_L^T Q_R)^{-1} Q_L^T at stabilisation point b; records
// max |G - G_fresh| when record != 0, and the weight's log|det| and sign.
// With c.dg64 (reduced paths) the recorded error is max |G - G_FP64|, the
// propagated G against the same formula assembled in FP64 from the FP64
// factors; the G that replaces the propagated one is still the
// path-precision assembly, so the chain itself is unchanged.
template <typename T, bool RES>
__device__ __forceinline__ void refresh(int b, bool record) {
  bool small = false;
  if constexpr (!std::is_same<T, double>::value) {
    small = small_products(this_cta<T, RES>());
    if (small) phase_small<T, RES>(b, -1);
  }
  if (!small) phase_overlap<T, RES>(b);
  phase_inverse<T, RES>();
  phase_assemble<T, RES>(b, record);
}

// Two sums over i, j < N of the terms that term(i, j, a, b) adds (collective): one
// row at a time per warp, the rows' sums through the scratch (no phase's buffers
// are in use), so that the order of the additions, and with it the last bit
// of a record, does not depend on the number of threads, which the default takes
// from the batch.  Lanes of warp 0 leave with parts to add up over the warp, in a and b.
template <typename T, bool RES, typename F>
__device__ __forceinline__ void row_sums(Cta<T, RES>& x, F term, double& a, double& b) {
  const int N = x.c.N, lane = threadIdx.x & 31;
  double* rows = reinterpret_cast<double*>(x.scr);     // 2 N of them: less than any phase holds
  __syncthreads();
  for (int i = threadIdx.x >> 5; i < N; i += blockDim.x >> 5) {
    double p = 0.0, q = 0.0;
    for (int j = lane; j < N; j += 32) term(i, j, p, q);
    p = warp_sum(p);
    q = warp_sum(q);
    if (lane == 0) {
      rows[2 * i] = p;
      rows[2 * i + 1] = q;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32)
    for (int i = lane; i < N; i += 32) {
      a += rows[2 * i];
      b += rows[2 * i + 1];
    }
}

// Wick estimates of the spinless t-V model on the fresh G at the middle
// slice: E/site of Eq. (4), interaction energy/site
// V sum_<ij> [(n_i - 1/2)(n_j - 1/2) - G_ji G_ij] / N, kinetic/site, the weight
// sign, the running sign, and S_CDW = [(sum_i eps_i (n_i - 1/2))^2 +
// sum_ij eps_i eps_j (delta_ij - G_ji) G_ij] / N^2.
template <typename T, bool RES>
__device__ __forceinline__ void measure_tv(Cta<T, RES>& x) {
  const ChainDesc& c = x.c;
  Smem<T>& sh = x.sh;
  const int N = c.N, ld = c.ld;
  const T* G = x.G(0);
  double ek = 0.0, eb = 0.0, st = 0.0, ex = 0.0;
  row_sums(x, [&](int i, int j, double& k, double& e) {
    const double gji = (i == j ? 1.0 : 0.0) - (double)G[(long)j * ld + i];
    k += c.K64[(long)i * N + j] * gji;
    e += c.eps[i] * c.eps[j] * gji * (double)G[(long)i * ld + j];
  }, ek, ex);
  if (threadIdx.x < 32) {
    for (int i = threadIdx.x; i < N; i += 32) st += c.eps[i] * (0.5 - (double)G[(long)i * ld + i]);
    for (int b = threadIdx.x; b < c.nfld; b += 32) {
      const int i = c.bond_ends[2 * b], j = c.bond_ends[2 * b + 1];
      const double di = 0.5 - (double)G[(long)i * ld + i], dj = 0.5 - (double)G[(long)j * ld + j];
      eb += di * dj - (double)G[(long)j * ld + i] * (double)G[(long)i * ld + j];
    }
    ek = warp_sum(ek);
    eb = warp_sum(eb) * c.U;
    st = warp_sum(st);
    ex = warp_sum(ex);
  }
  if (threadIdx.x == 0) {
    const int m = c.st->n_meas;
    const double rec[kRecord] = {sh.sign_spin[0] * sh.sign_spin[1], (ek + eb) / N, eb / N, ek / N,
                                 sh.sign_running, (st * st + ex) / ((double)N * N)};
    for (int k = 0; k < kRecord; ++k) {
      if (m < c.max_meas) c.meas[(long)m * kRecord + k] = rec[k];
      c.last[k] = rec[k];
    }
    c.st->n_meas = m + 1;
  }
  __syncthreads();
}

// Wick estimates on the fresh G at the middle slice: E/site for Eq. (2),
// docc/site, kinetic/site, with the weight sign and the running sign, and the
// staggered S^z structure factor S = (1/N^2) sum_ij eps_i eps_j <S^z_i S^z_j>
// = [(sum_i eps_i m_i)^2 + sum_s sum_ij eps_i eps_j (delta_ij - G_s,ji) G_s,ij]
// / (4 N^2), m_i = n_i,up - n_i,dn (the spins are independent at fixed fields).
// grid_sums: the sums over i, j (ek, ex) formed elsewhere, n_sums pairs to add
// up (a chain swept by the whole GPU), or null.
template <typename T, bool RES>
__device__ __forceinline__ void measure(Cta<T, RES>& x, const double* grid_sums = nullptr, int n_sums = 0) {
  const ChainDesc& c = x.c;
  if (c.tv) {
    measure_tv(x);
    return;
  }
  Smem<T>& sh = x.sh;
  const int N = c.N, ld = c.ld;
  double ek = 0.0, dc = 0.0, st = 0.0, ex = 0.0;
  if (grid_sums) {
    for (int q = threadIdx.x < 32 ? (int)threadIdx.x : n_sums; q < n_sums; q += 32) {
      ek += grid_sums[2 * q];
      ex += grid_sums[2 * q + 1];
    }
  } else {
    row_sums(x, [&](int i, int j, double& kin, double& stag) {
      const double k = c.K64[(long)i * N + j];
      const double ee = c.eps[i] * c.eps[j];
      for (int s = 0; s < 2; ++s) {
        const double gji = (i == j ? 1.0 : 0.0) - (double)x.G(s)[(long)j * ld + i];
        kin += k * gji;
        stag += ee * gji * (double)x.G(s)[(long)i * ld + j];
      }
    }, ek, ex);
  }
  if (threadIdx.x < 32) {
    for (int i = threadIdx.x; i < N; i += 32) {
      const double g0 = (double)x.G(0)[(long)i * ld + i], g1 = (double)x.G(1)[(long)i * ld + i];
      dc += (1.0 - g0) * (1.0 - g1);
      st += c.eps[i] * (g1 - g0);
    }
    ek = warp_sum(ek);
    dc = warp_sum(dc);
    st = warp_sum(st);
    ex = warp_sum(ex);
  }
  if (threadIdx.x == 0) {
    const int m = c.st->n_meas;
    const double rec[kRecord] = {sh.sign_spin[0] * sh.sign_spin[1], (ek + c.U * dc) / N, dc / N, ek / N,
                                 sh.sign_running, (st * st + ex) / (4.0 * N * N)};
    for (int k = 0; k < kRecord; ++k) {
      if (m < c.max_meas) c.meas[(long)m * kRecord + k] = rec[k];
      c.last[k] = rec[k];
    }
    c.st->n_meas = m + 1;
  }
  __syncthreads();
}

// --------------------------------------------------------------------------
// sweeps

template <typename T, bool RES>
__device__ __noinline__ void phase_slice_tv(int tau, uint32_t sweep) {
  auto x = this_cta<T, RES>();
  update_slice_tv(x, tau, sweep);
}
template <typename T, bool RES, bool kTc>
__device__ __noinline__ void phase_wrap(int tau, int dir) {
  auto x = this_cta<T, RES>();
  wrap<kTc>(x, tau, dir);
  x.mark(kPhWrap);
}
template <typename T, bool RES>
__device__ __noinline__ void phase_measure() {
  auto x = this_cta<T, RES>();
  measure(x);
}

// The stabilisation at slice t (a multiple of n_stab): the new stack block,
// G from the stacks, the measurement at the middle slice.
template <typename T, bool RES>
__device__ __forceinline__ void stabilise(int t, int left, bool do_measure) {
  auto x = this_cta<T, RES>();
  const int b = t / x.c.n_stab;
  push_block<T, RES>(b, left);
  refresh<T, RES>(b, true);
  x.mark(kPhRefresh);
  if (do_measure && t == x.c.Ltau / 2) phase_measure<T, RES>();
  x.mark(kPhMeasure);
}

template <typename T, bool RES, bool kPair, bool kTc>
__device__ __forceinline__ void sweep_once(uint32_t sweep, bool do_measure) {
  auto x = this_cta<T, RES>();
  const int Lt = x.c.Ltau, n_stab = x.c.n_stab;
  const bool down = (sweep & 1u) != 0;
  for (int k = 0; k <= Lt + 1; ++k) {
    const int tau = down ? Lt + 1 - k : k;
    if (down) phase_wrap<T, RES, kTc>(tau, -1);
    if (x.c.tv) phase_slice_tv<T, RES>(tau, sweep);
    else update_slice<T, RES, kPair>(tau, sweep);
    if (!down) phase_wrap<T, RES, kTc>(tau, +1);
    const int t = down ? tau - 1 : tau;              // G is G(t) now
    if (t >= 0 && t <= Lt && t % n_stab == 0) stabilise<T, RES>(t, down ? 1 : 0, do_measure);
  }
}

// kTables: the slice exponentials too (the wrap and the stack products read them)
template <bool kTables = true, typename T, bool RES>
__device__ __forceinline__ void load_state(Cta<T, RES>& x) {
  if (threadIdx.x == 0) {
    const ChainState& st = *x.c.st;
    x.sh.sign_running = st.sign_running;
    x.sh.dGmax = st.max_dG;
    x.sh.n_prop = st.n_prop;
    x.sh.n_acc = st.n_acc;
    x.sh.acc_pos = st.acc_pos;
    x.sh.err = 0;
    x.sh.staged = -1;
    x.sh.sign_spin[0] = st.logw[0][1];
    x.sh.sign_spin[1] = st.logw[1][1];
    x.sh.logw_spin[0] = st.logw[0][0];
    x.sh.logw_spin[1] = st.logw[1][0];
  }
  if (kTables && threadIdx.x < 28) {
    const int k = threadIdx.x / 14, sp = (threadIdx.x / 7) % 2, m = threadIdx.x % 7 - 3;
    double v = 1.0;
    if (x.c.tv) {
      if (sp == 0) v = x.c.vtv[k][m + 3];
    } else if (m == 1 || m == -1) {
      v = x.c.vexp[k][sp][m > 0 ? 0 : 1];
    }
    x.sh.vtab[k][sp][m + 3] = v;
    x.sh.vt[k][sp][m + 3] = (T)v;
    x.sh.vti[k][sp][m + 3] = (T)(1.0 / v);
  }
  if (threadIdx.x < kPhases) x.sh.cyc[threadIdx.x] = 0;
  if (threadIdx.x == 0) x.sh.t_mark = clock64();
  __syncthreads();
}

template <typename T, bool RES>
__device__ __forceinline__ void store_state(Cta<T, RES>& x, int* err) {
  __syncthreads();
  if (threadIdx.x == 0) {
    ChainState& st = *x.c.st;
    st.sign_running = x.sh.sign_running;
    st.max_dG = x.sh.dGmax;
    st.n_prop = x.sh.n_prop;
    st.n_acc = x.sh.n_acc;
    st.acc_pos = x.sh.acc_pos;
    st.err |= x.sh.err;
    for (int s = 0; s < 2; ++s) {
      st.logw[s][0] = x.sh.logw_spin[s];
      st.logw[s][1] = x.sh.sign_spin[s];
    }
    for (int p = 0; p < kPhases; ++p) st.cycles[p] += x.sh.cyc[p];
    if (x.sh.err) atomicOr(err, x.sh.err);
  }
}

// Place G and the scratch: in shared memory after the fixed part when the
// chain's footprint fits in res_bytes (G is copied in), else in global memory.
// Every phase finds them again through this_cta.
template <typename T>
__device__ __forceinline__ Smem<T>& setup_cta(const ChainDesc& cg, size_t res_bytes, uint64_t seed) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<T>& sh = *reinterpret_cast<Smem<T>*>(smem_raw);
  // the descriptor is read all through the sweep: keep a shared-memory copy
  {
    const int words = (int)(sizeof(ChainDesc) / sizeof(int));
    const int* src = reinterpret_cast<const int*>(&cg);
    int* dst = reinterpret_cast<int*>(&sh.desc);
    for (int w = threadIdx.x; w < words; w += blockDim.x) dst[w] = src[w];
    __syncthreads();
  }
  const ChainDesc& c = sh.desc;
  const int ts = (int)sizeof(T);
  const bool res = resident_bytes(c.N, c.ld, c.nmax, ts, c.kb) <= res_bytes;
  if (threadIdx.x == 0) {
    sh.L = scratch_layout(c.N, c.ld, c.nmax, ts, c.kb);
    sh.res = res ? 1 : 0;
    sh.seed = seed;
    sh.scr_off = (uint32_t)(al16(sizeof(Smem<T>)) + al16(2 * (size_t)c.N * c.ld * ts));
    sh.tcs_off = 0;
    sh.tmem = 0;
  }
  if (res) {
    T* Gp = reinterpret_cast<T*>(smem_raw + al16(sizeof(Smem<T>)));
    const T* g = reinterpret_cast<const T*>(c.G);
    for (long e = threadIdx.x; e < 2L * c.N * c.ld; e += blockDim.x) Gp[e] = g[e];
  }
  __syncthreads();
  return sh;
}

template <typename T, bool RES>
__device__ __forceinline__ void write_back() {
  auto x = this_cta<T, RES>();
  __syncthreads();
  if (RES) {
    T* g = reinterpret_cast<T*>(x.c.G);
    for (long e = threadIdx.x; e < 2L * x.c.N * x.c.ld; e += blockDim.x) g[e] = x.Gp[e];
  }
  __syncthreads();
}

template <typename T, bool RES>
__device__ __forceinline__ void run_init(int* err, int b_at) {
  auto x = this_cta<T, RES>();
  Smem<T>& sh = x.sh;
  load_state(x);
  const int bt = b_at < 0 ? 0 : b_at;
  for (int b = x.c.nb; b >= bt; --b) push_block<T, RES>(b, 1);
  for (int b = 0; b <= bt; ++b) push_block<T, RES>(b, 0);
  refresh<T, RES>(bt, false);
  if (b_at < 0) {
    if (threadIdx.x == 0) sh.sign_running = sh.sign_spin[0] * sh.sign_spin[1];
    __syncthreads();
    phase_wrap<T, RES, false>(0, -1);
  }
  write_back<T, RES>();
  store_state(x, err);
}

// b_at < 0: initialisation from the chain's fields (left stack, right block
// 0, G at tau = -1 and the running sign). b_at >= 0: the left stack down to
// block b_at, the right stack up to it and G at the stabilisation point
// tau = b_at * n_stab, all from the fields (a recomputation the host wraps
// in a save and restore of the chain's state).
template <typename T, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB) init_kernel(const ChainDesc* chains, int chain0, uint64_t seed,
                                                          size_t res_bytes, int* err, int b_at) {
  Smem<T>& sh = setup_cta<T>(chains[chain0 + blockIdx.x], res_bytes, seed);
  if (sh.res) run_init<T, true>(err, b_at);
  else run_init<T, false>(err, b_at);
}

template <typename T, bool RES, bool kPair, bool kTc>
__device__ __forceinline__ void run_sweeps(uint32_t sweep0, int n_sweeps, int do_measure) {
  auto x = this_cta<T, RES>();
  Smem<T>& sh = x.sh;
  const long long t_start = clock64();
  for (int k = 0; k < n_sweeps; ++k) {
    sweep_once<T, RES, kPair, kTc>(sweep0 + (uint32_t)k, do_measure != 0);
    __syncthreads();
    if (sh.err) break;
  }
  if (threadIdx.x == 0) sh.cyc[kPhTotal] += clock64() - t_start;
}

template <typename T, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB) sweep_kernel(const ChainDesc* chains, uint64_t seed,
                                                       const uint32_t* sweep_ctr, int n_sweeps, int do_measure,
                                                       size_t res_bytes, int* err, int tc_on) {
  if (chains[blockIdx.x].st->err) return;
  constexpr bool kPair = TPB * MINB <= 512;   // 128 registers per thread: room for the one-warp decisions
  const uint32_t sweep0 = *sweep_ctr;
  Smem<T>& sh = setup_cta<T>(chains[blockIdx.x], res_bytes, seed);
  if (sh.res) {
    auto x = this_cta<T, true>();
    load_state(x);
    run_sweeps<T, true, kPair, (TPB == 512)>(sweep0, n_sweeps, do_measure);
    write_back<T, true>();
    store_state(x, err);
  } else {
    auto x = this_cta<T, false>();
    load_state(x);
    if constexpr (std::is_same<T, float>::value && TPB == 512) {
      // BF16X3 chains kept in global memory run their products on the tensor
      // cores: a staging area after the dynamic shared memory the launch
      // reserves for it, and TMEM columns held until the CTA ends
      if (tc_on && x.c.tc) {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        const size_t fbb = flipbuf_bytes((int)sizeof(T));
        const uint32_t base = smem_addr(smem_raw);
        const uint32_t at = base + (uint32_t)(al16(sizeof(Smem<T>)) + (res_bytes > fbb ? res_bytes : fbb));
        const uint32_t off = ((at + 127) & ~127u) - base;
        const uint32_t tmem = tc_alloc(smem_raw + off);
        if (threadIdx.x == 0) {
          sh.tcs_off = off;
          sh.tmem = tmem;
        }
        __syncthreads();
      }
    }
    run_sweeps<T, false, kPair, (TPB == 512)>(sweep0, n_sweeps, do_measure);
    if constexpr (std::is_same<T, float>::value && TPB == 512) {
      if (sh.tcs_off) tc_free(sh.tmem);
    }
    write_back<T, false>();
    store_state(x, err);
  }
}

// --------------------------------------------------------------------------
// launch templates, instantiated by the per-path translation units

template <typename T>
static size_t dyn_smem(size_t res) {
  const size_t fbb = flipbuf_bytes((int)sizeof(T));
  return al16(sizeof(Smem<T>)) + (res > fbb ? res : fbb);
}

template <typename T, int TPB, int MINB>
static cudaError_t launch_init_t(const ChainDesc* d_chains, int chain0, int n, uint64_t seed, size_t res, int* d_err,
                                 cudaStream_t stream, int b_at) {
  const size_t sm = dyn_smem<T>(res);
  cudaError_t e = cudaFuncSetAttribute(init_kernel<T, TPB, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  init_kernel<T, TPB, MINB><<<n, TPB, sm, stream>>>(d_chains, chain0, seed, res, d_err, b_at);
  return cudaGetLastError();
}

// Advances the device-side sweep index after a sweep launch (sweep.cu).
cudaError_t launch_advance(uint32_t* sweep_ctr, int n, cudaStream_t stream);

// tc_on: the launch reserves the tensor-core staging area (BF16X3 on
// 512-thread CTAs)
template <typename T, int TPB, int MINB>
static size_t sweep_smem(size_t res, int tc_on) {
  return dyn_smem<T>(res) + ((std::is_same<T, float>::value && TPB == 512 && tc_on) ? kTcBytes + 128 : 0);
}

template <typename T, int TPB, int MINB>
static cudaError_t prepare_sweep_t(size_t res, int tc_on) {
  return cudaFuncSetAttribute(sweep_kernel<T, TPB, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sweep_smem<T, TPB, MINB>(res, tc_on));
}

template <typename T, int TPB, int MINB>
static cudaError_t launch_sweep_t(const ChainDesc* d_chains, int n, uint64_t seed, uint32_t* sweep_ctr, int n_sweeps,
                                  int measure, size_t res, int* d_err, cudaStream_t stream, int tc_on) {
  sweep_kernel<T, TPB, MINB><<<n, TPB, sweep_smem<T, TPB, MINB>(res, tc_on), stream>>>(
      d_chains, seed, sweep_ctr, n_sweeps, measure, res, d_err, tc_on);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_advance(sweep_ctr, n_sweeps, stream);
}

// Defines launch_init_<P>, prepare_sweep_<P> and launch_sweep_<P> over the
// CTA shapes that PQMC_TPB_DISPATCH (defined by the including unit) selects.
#define PQMC_DEFINE_LAUNCHERS(P)                                                                                  \
  cudaError_t launch_init_##P(int tpb, const ChainDesc* d_chains, int chain0, int n, uint64_t seed, size_t res,    \
                              int* d_err, cudaStream_t stream, int b_at) {                                         \
    PQMC_TPB_DISPATCH(launch_init_t, d_chains, chain0, n, seed, res, d_err, stream, b_at);                          \
  }                                                                                                                \
  cudaError_t prepare_sweep_##P(int tpb, size_t res, int tc_on) { PQMC_TPB_DISPATCH(prepare_sweep_t, res, tc_on); } \
  cudaError_t launch_sweep_##P(int tpb, const ChainDesc* d_chains, int n, uint64_t seed, uint32_t* sweep_ctr,      \
                               int n_sweeps, int measure, size_t res, int* d_err, cudaStream_t stream, int tc_on) { \
    PQMC_TPB_DISPATCH(launch_sweep_t, d_chains, n, seed, sweep_ctr, n_sweeps, measure, res, d_err, stream, tc_on);  \
  }

// Per-path launchers (one translation unit each).
#define PQMC_DECLARE_LAUNCHERS(P)                                                                                 \
  cudaError_t launch_init_##P(int tpb, const ChainDesc* d_chains, int chain0, int n, uint64_t seed, size_t res,    \
                              int* d_err, cudaStream_t stream, int b_at);                                          \
  cudaError_t prepare_sweep_##P(int tpb, size_t res, int tc_on);                                                  \
  cudaError_t launch_sweep_##P(int tpb, const ChainDesc* d_chains, int n, uint64_t seed, uint32_t* sweep_ctr,      \
                               int n_sweeps, int measure, size_t res, int* d_err, cudaStream_t stream, int tc_on);
PQMC_DECLARE_LAUNCHERS(f64)
PQMC_DECLARE_LAUNCHERS(f32)
PQMC_DECLARE_LAUNCHERS(f32_256)
PQMC_DECLARE_LAUNCHERS(f32_512)
PQMC_DECLARE_LAUNCHERS(f32_dense)

}  // namespace pqmc
