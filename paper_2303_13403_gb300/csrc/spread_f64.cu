// Spread sweep (spread.cuh): the FP64 path's kernel sequence and the FP64
// stabilisation steps that both paths call.
#include "spread.cuh"

#include <cooperative_groups.h>

namespace pqmc {

namespace {

__device__ __forceinline__ SpBuf<double> fp64_bufs(const ChainDesc& c, int tsize) {
  return SpBuf<double>(c.spread, c.N, c.ld, c.nmax, tsize);
}
__device__ __forceinline__ int nsig_of(const ChainDesc& c, int s) { return s == 0 ? c.nup : c.ndn; }

// Digits of M64 (b < 0, q = 0) or of stack blocks b, Q_L (q = 0) and Q_R (q = 1),
// one column per CTA with the column's own exponent (grid: column of q = 0, then
// of q = 1; spin; chain): the columns of M64 grow apart by up to e^{6 dtau} per
// slice, and the Gram matrix has to keep the small ones' diagonal (against the
// block's largest element a pivot of free fermions, 72 sites, 10 slices of
// dtau = 0.8, failed).  A thread holds its rows in registers between the search
// and the packing.
__global__ void __launch_bounds__(256) sp_digits_kernel(const ChainDesc* chains, int b, int tsize) {
  __shared__ int red[8];
  constexpr int kRows = kMaxN / 256;
  static_assert(kMaxN % 256 == 0, "rows per thread");
  const ChainDesc& c = chains[blockIdx.z];
  if (c.st->err) return;
  const int s = blockIdx.y, n = nsig_of(c, s), N = c.N;
  const int q = blockIdx.x >= c.nmax ? 1 : 0, k = blockIdx.x - q * c.nmax;
  if (k >= n) return;
  SpBuf<double> sp = fp64_bufs(c, tsize);
  const double* col = (b < 0 ? sp.m64(s) : (q == 0 ? c.Lst : c.Rst) + ((long)b * 2 + s) * N * c.nmax) + (long)k * N;
  double v[kRows];
  int e = kDigitNone;
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int i = threadIdx.x + 256 * r;
    v[r] = i < N ? col[i] : 0.0;
    e = max(e, digit_exp(v[r]));
  }
  e = digit_cta_max(e, red);
  unsigned long long* D = sp.dq(s, q) + (long)k * digit_ld(N);
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int i = threadIdx.x + 256 * r;
    if (i < N) D[i] = digit_pack(v[r], e);
  }
  if (threadIdx.x == 0) sp.dexp(s, q)[k] = e;
}

// One 32 x 32 block of the Gram matrix (b < 0, upper triangle) or of O per CTA
// (digit_gemm.cuh; 648 x 324: 36 MMAs per 16-deep step on 8 warps, against the FP64
// pipe's 74% in a tiled FMA product).
__global__ void __launch_bounds__(256) sp_digit_gemm_kernel(const ChainDesc* chains, int b, int tsize) {
  const ChainDesc& c = chains[blockIdx.z];
  if (c.st->err) return;
  const int s = blockIdx.y, n = nsig_of(c, s), N = c.N, ldd = digit_ld(N), ldn = c.nmax;
  const int tn = (c.nmax + 31) >> 5;
  const int i0 = 32 * (int)(blockIdx.x / tn), j0 = 32 * (int)(blockIdx.x % tn);
  if (i0 >= n || j0 >= n || (b < 0 && i0 > j0)) return;
  SpBuf<double> sp = fp64_bufs(c, tsize);
  const int qb = b < 0 ? 0 : 1;
  const unsigned long long* A = sp.dq(s, 0) + (long)i0 * ldd;
  const unsigned long long* B = sp.dq(s, qb) + (long)j0 * ldd;
  const int* ea = sp.dexp(s, 0) + i0;
  const int* eb = sp.dexp(s, qb) + j0;
  double* C = (b < 0 ? sp.c64(s) : sp.o64(s)) + (long)i0 * ldn + j0;
  digit_gemm<true, true>(min(32, n - i0), min(32, n - j0), N, A, ldd, 1, B, ldd, 1, [ea](int i) { return ea[i]; },
                         [eb](int j) { return eb[j]; }, false, false,
                         [C, ldn](int i, int j, double v) { C[(long)i * ldn + j] = v; });
}

// Cholesky factor, diagonal block of panel p (one CTA per spin, chain), and its
// inverse, by the elimination of [C | I] in shared memory (chol_eliminate):
// step k takes row k, u_j = row_kj / p_k, from the rows below; right of the
// diagonal stay the Schur complements (R_kj = C_kj / sqrt(p_k)), left of it the
// rows of L^{-1} (R_PP^{-1} = L^{-T} diag(p)^{-1/2}).  Warp 0 runs one step ahead (row
// k + 1, its pivot and reciprocal), so a column costs one barrier and the
// reciprocal's latency passes beside the other rows' FMAs; factor and
// back substitution as two chains of 32 steps took 42.6 us, this form 17.0.  Panel 0 first
// records the Gram diagonal and clears the chain's breakdown flag and log det R.
__global__ void __launch_bounds__(256) chol_panel_kernel(const ChainDesc* chains, int p, int tsize) {
  __shared__ double A[kSpPanel][kSpPanel + 1];
  __shared__ double u[2][kSpPanel];
  __shared__ double pv[kSpPanel], isq[kSpPanel], dlim[kSpPanel];
  __shared__ int bad;
  const ChainDesc& c = chains[blockIdx.y];
  if (c.st->err) return;
  const int s = blockIdx.x, n = nsig_of(c, s), ldn = c.nmax;
  const int p0 = p * kSpPanel;
  if (p0 >= n) return;
  const int p1 = min(p0 + kSpPanel, n), bw = p1 - p0;
  SpBuf<double> sp = fp64_bufs(c, tsize);
  double* C = sp.c64(s);
  double* d0 = sp.d0(s);
  if (p == 0) {
    for (int k = threadIdx.x; k < n; k += blockDim.x) d0[k] = C[(long)k * ldn + k];
    if (threadIdx.x == 0) {
      sp.bad()[s] = 0;
      sp.lchol()[s] = 0.0;
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < kSpPanel * kSpPanel; e += blockDim.x) {
    const int i = e / kSpPanel, j = e % kSpPanel;
    A[i][j] = (i < bw && j < bw && j >= i) ? C[(long)(p0 + i) * ldn + p0 + j] : 0.0;
  }
  if ((int)threadIdx.x < bw) dlim[threadIdx.x] = 1e-12 * d0[p0 + threadIdx.x];
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  auto pivot_row = [&](int r) {
    const double piv = A[r][r];
    // (positive doubles order like their bits)
    const long long pb = __double_as_longlong(piv);
    const bool ok = pb > __double_as_longlong(dlim[r]) && pb < 0x7ff0000000000000ll;
    const double ip = ok ? recip64(piv) : 0.0;
    if (lane == 0) {
      pv[r] = piv;
      if (!ok) bad = 1;
    }
    u[r & 1][lane] = lane == r ? ip : A[r][lane] * ip;
  };
  if (warp == 0) pivot_row(0);
  __syncthreads();
  // (every step runs to its barrier whatever the pivots are: warp 0 sets bad
  // one step ahead, so it is read only after the last barrier; past a bad
  // pivot the rows take u = 0)
  for (int k = 0; k + 1 < bw; ++k) {
    const double uk = u[k & 1][lane];
    if (warp == 0) {
      const int r = k + 1;
      A[r][lane] = fma(-A[k][r], uk, lane == k ? 0.0 : A[r][lane]);
      __syncwarp();
      pivot_row(r);
    } else {
      for (int i = k + 1 + warp; i < bw; i += 7) A[i][lane] = fma(-A[k][i], uk, lane == k ? 0.0 : A[i][lane]);
    }
    __syncthreads();
  }
  if (bad) {
    if (threadIdx.x == 0) sp.bad()[s] = 1;
    return;
  }
  if ((int)threadIdx.x < bw) isq[threadIdx.x] = rsqrt(pv[threadIdx.x]);
  if (threadIdx.x < 32) {
    // log det R_PP: one logarithm per lane, summed over the warp
    double la = (int)threadIdx.x < bw ? log(pv[threadIdx.x]) : 0.0;
    la = warp_sum(la);
    if (threadIdx.x == 0) sp.lchol()[s] += 0.5 * la;
  }
  __syncthreads();
  double* Ri = sp.rinv(s) + (long)p * kSpPanel * kSpPanel;
  for (int e = threadIdx.x; e < kSpPanel * kSpPanel; e += blockDim.x) {
    const int i = e / kSpPanel, j = e % kSpPanel;
    const bool in = i < bw && j < bw;
    if (in && i <= j) C[(long)(p0 + i) * ldn + p0 + j] = i == j ? pv[i] * isq[i] : A[i][j] * isq[i];
    Ri[e] = !in || i > j ? 0.0 : i == j ? isq[i] : A[j][i] * isq[j];
  }
}

// Q = M R^{-1}, one warp per row i of M: panel by panel, t = m_P - q_{<P} R_{<P,P}
// (lane j: column p0 + j), then q_P = t R_PP^{-1}; the eight rows of a CTA
// are written to the column-major stack block together
__global__ void __launch_bounds__(256) qform_kernel(const ChainDesc* chains, int left, int b, int tsize) {
  __shared__ double q[8][kMaxSigma];
  const ChainDesc& c = chains[blockIdx.z];
  if (c.st->err) return;
  const int s = blockIdx.y, n = nsig_of(c, s), ldn = c.nmax, N = c.N;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i0 = blockIdx.x * 8, i = i0 + w;
  SpBuf<double> sp = fp64_bufs(c, tsize);
  const double* M = sp.m64(s);
  const double* C = sp.c64(s);
  const double* Ri = sp.rinv(s);
  if (i < N) {
    for (int p0 = 0; p0 < n; p0 += kSpPanel) {
      const int bw = min(kSpPanel, n - p0), j = lane;
      double t = 0.0;
      if (j < bw) {
        double a0 = M[(long)(p0 + j) * N + i], a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int l = 0;
        for (; l + 4 <= p0; l += 4) {
          a0 = fma(-q[w][l], C[(long)l * ldn + p0 + j], a0);
          a1 = fma(-q[w][l + 1], C[(long)(l + 1) * ldn + p0 + j], a1);
          a2 = fma(-q[w][l + 2], C[(long)(l + 2) * ldn + p0 + j], a2);
          a3 = fma(-q[w][l + 3], C[(long)(l + 3) * ldn + p0 + j], a3);
        }
        for (; l < p0; ++l) a0 = fma(-q[w][l], C[(long)l * ldn + p0 + j], a0);
        t = (a0 + a1) + (a2 + a3);
      }
      const double* Rp = Ri + (long)(p0 / kSpPanel) * kSpPanel * kSpPanel;
      double acc = 0.0;
      for (int l = 0; l < bw; ++l) {
        const double tl = __shfl_sync(0xffffffffu, t, l);
        if (l <= j && j < bw) acc = fma(tl, Rp[l * kSpPanel + j], acc);
      }
      if (j < bw) q[w][p0 + j] = acc;
      __syncwarp();
    }
  }
  __syncthreads();
  double* Q = (left ? c.Lst : c.Rst) + ((long)b * 2 + s) * N * c.nmax;
  const int rows = min(8, N - i0);
  for (int e = threadIdx.x; e < n * 8; e += blockDim.x) {
    const int k = e >> 3, r = e & 7;
    if (r < rows) Q[(long)k * N + i0 + r] = q[r][k];
  }
}

// Gauss-Jordan panel p (columns P = [p0, p1)) of O, one cluster of kGJRanks CTAs
// per spin and chain: for each column j of P the largest |O_ij| over the rows
// not used yet (ties to the lower row), then the elimination of column j
// restricted to the panel's columns (the rest of the row operations is the
// block update that follows, from the block row saved at the end).  The rows
// are dealt out to the cluster's CTAs and stay in their shared memory; a step
// costs one cluster barrier: every CTA hands its best candidate, the whole
// panel row, to all eight (distributed shared memory), and each takes the
// best of the eight and eliminates its own rows.  (One CTA per spin had n x 16
// FP64 FMAs per column on one SM and two barriers with a division between
// them: 71.7 us per panel at n = 324, this form 27.9.)  Rows are interchanged once, at the end: the
// panel's interchanges composed into one permutation of at most 2 bw rows
// (place rows[e] takes row src[e]), applied to the panel as it is written back
// and to the other columns, which the CTAs share.
constexpr int kGJRanks = 8;
constexpr int kGJRows = kMaxSigma / kGJRanks;     // rows per CTA
static_assert(kMaxSigma % kGJRanks == 0 && kGJRows == 4 * 16 && kSpGJ == 16, "four rows per thread and column");
// a CTA's candidate: the scaled pivot row it would give (16), the pivot, its
// absolute value's bits and its row
constexpr int kGJWords = kSpGJ + 3;

__global__ void __cluster_dims__(kGJRanks, 1, 1) __launch_bounds__(256)
    gj_panel_kernel(const ChainDesc* chains, int p, int tsize) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ double Ap[kGJRows][kSpGJ + 1];
  __shared__ unsigned long long cand[2][kGJRanks][kGJWords];   // two steps in flight
  __shared__ int used[kGJRows], place[kGJRows], pivrow[kSpGJ];
  __shared__ int rows[2 * kSpGJ], src[2 * kSpGJ], nrows;
  const ChainDesc& c = chains[blockIdx.y];
  if (c.st->err) return;                            // (the whole cluster)
  const int s = blockIdx.x / kGJRanks, rank = blockIdx.x % kGJRanks, n = nsig_of(c, s), ldn = c.nmax;
  const int p0 = p * kSpGJ;
  if (p0 >= n) return;
  const int p1 = min(p0 + kSpGJ, n), bw = p1 - p0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = threadIdx.x % kSpGJ, r0 = threadIdx.x / kSpGJ;
  const int nl = rank < n ? (n - rank + kGJRanks - 1) / kGJRanks : 0;   // local row l: rank + 8 l
  SpBuf<double> sp = fp64_bufs(c, tsize);
  double* A = sp.o64(s);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int l = r0 + 16 * q;
    if (l < nl) Ap[l][col] = col < bw ? A[(long)(rank + kGJRanks * l) * ldn + p0 + col] : 0.0;
  }
  for (int l = threadIdx.x; l < kGJRows; l += blockDim.x) {
    used[l] = rank + kGJRanks * l < p0 ? 1 : 0;     // rows before the panel are pivot rows already
    place[l] = rank + kGJRanks * l;
  }
  cl.sync();                                        // every CTA of the cluster runs before its memory is written
  for (int jj = 0; jj < bw; ++jj) {
    const int j = p0 + jj;
    auto cd = cand[jj & 1];
    if (warp == 0) {
      // this CTA's candidate, handed to every CTA; its owner takes the
      // reciprocal and scales the row, so that the choice below is integer work
      unsigned long long best = 0;
      int bl = -1;
      for (int l = lane; l < nl; l += 32) {
        const unsigned long long v = (unsigned long long)__double_as_longlong(Ap[l][jj]) & 0x7fffffffffffffffull;
        if (!used[l] && (bl < 0 || v > best)) { best = v; bl = l; }
      }
      const unsigned hi = __reduce_max_sync(0xffffffffu, bl < 0 ? 0u : (unsigned)(best >> 32));
      const unsigned lo = __reduce_max_sync(0xffffffffu, bl >= 0 && (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
      const bool mine = bl >= 0 && (unsigned)(best >> 32) == hi && (unsigned)best == lo;
      const unsigned l = __reduce_min_sync(0xffffffffu, mine ? (unsigned)bl : 0xffffffffu);   // ties to the lower row
      const bool any = l != 0xffffffffu;
      const double pvt = any ? Ap[l][jj] : 0.0;
      const double ip = pvt != 0.0 ? recip64(pvt) : 0.0;
      const double x = lane == jj ? ip : any && lane < kSpGJ ? Ap[l][lane] * ip : 0.0;
      unsigned long long w = (unsigned long long)__double_as_longlong(lane == kSpGJ ? pvt : x);
      if (lane == kSpGJ + 1) w = ((unsigned long long)hi << 32) | lo;
      if (lane == kSpGJ + 2) w = any ? (unsigned long long)(rank + kGJRanks * (int)l) : 0x7fffffffull;
      if (lane < kGJWords) {
#pragma unroll
        for (int t = 0; t < kGJRanks; ++t) *cl.map_shared_rank(&cd[rank][lane], t) = w;
      }
    }
    cl.sync();
    // the best of the eight, ties to the lower row
    int b;
    {
      const int row = lane < kGJRanks ? (int)cd[lane][kSpGJ + 2] : 0x7fffffff;
      const unsigned long long best = lane < kGJRanks && row != 0x7fffffff ? cd[lane][kSpGJ + 1] : 0ull;
      const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
      const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
      const bool top = (unsigned)(best >> 32) == hi && (unsigned)best == lo;
      const unsigned low = __reduce_min_sync(0xffffffffu, top ? (unsigned)row : 0xffffffffu);
      b = __ffs((int)__ballot_sync(0xffffffffu, top && (unsigned)row == low)) - 1;
    }
    const int r = (int)cd[b][kSpGJ + 2];
    const double pvt = __longlong_as_double((long long)cd[b][kSpGJ]);
    const double x = __longlong_as_double((long long)cd[b][col]);
    // eliminate column j: v = add - f_i x, one FP64 instruction per element
    double f[4], v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int l = r0 + 16 * q;
      if (l < nl) {
        f[q] = Ap[l][jj];
        v[q] = col == jj ? 0.0 : Ap[l][col];
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int l = r0 + 16 * q;
      if (l < nl) Ap[l][col] = rank + kGJRanks * l == r ? x : fma(-f[q], x, v[q]);
    }
    if (threadIdx.x == 0) {
      pivrow[jj] = r;
      if (r % kGJRanks == rank) used[r / kGJRanks] = 1;
      if (rank == 0) {
        sp.pval(s)[j] = pvt;
        if (pvt == 0.0) sp.bad()[s] = 1;
      }
    }
    __syncthreads();
  }
  // the interchanges: entry e (lane e) is place rows[e] and the row it takes
  if (warp == 0) {
    int pl = lane < bw ? p0 + lane : -1, id = pl, m = bw;
    for (int jj = 0; jj < bw; ++jj) {
      const int r = pivrow[jj];
      const unsigned at = __ballot_sync(0xffffffffu, lane < m && id == r);
      const int other = __shfl_sync(0xffffffffu, id, jj);          // the row now at place p0 + jj
      int e = __ffs((int)at) - 1;
      if (at == 0) {                                               // row r is still at place r
        e = m++;
        if (lane == e) { pl = r; id = r; }
      }
      const int pr = __shfl_sync(0xffffffffu, pl, e);
      if (e != jj) {
        if (lane == e) id = other;
        if (lane == jj) id = r;
      }
      if (rank == 0 && lane == 0) sp.perm(s)[p0 + jj] = pr;
    }
    if (lane < m) {
      rows[lane] = pl;
      src[lane] = id;
      if (id % kGJRanks == rank) place[id / kGJRanks] = pl;
    }
    if (lane == 0) nrows = m;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int l = r0 + 16 * q;
    if (l < nl && col < bw) A[(long)place[l] * ldn + p0 + col] = Ap[l][col];
  }
  // the other columns, and the block row of the update (rows[e] = p0 + e for e < bw)
  const int m = nrows;
  double* Tb = sp.tgj(s);
  static_assert(kMaxSigma <= 64 * kGJRanks, "one column per 64 threads and rank");
  const int cc = rank * 64 + (int)(threadIdx.x & 63), eg = (int)(threadIdx.x >> 6) * 8;   // eight entries per thread
  const bool mover = cc < n && (cc < p0 || cc >= p1);
  double mv[8];
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (mover && eg + e < m) mv[e] = A[(long)src[eg + e] * ldn + cc];
  __syncthreads();                                  // a column's rows are all read before one is written
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (mover && eg + e < m) {
      A[(long)rows[eg + e] * ldn + cc] = mv[e];
      if (eg + e < bw) Tb[(long)(eg + e) * ldn + cc] = mv[e];
    }
}

// row i: the interchanges of the elimination applied to the columns, last first
__global__ void __launch_bounds__(128) gj_unswap_kernel(const ChainDesc* chains, int tsize) {
  const ChainDesc& c = chains[blockIdx.z];
  if (c.st->err) return;
  const int s = blockIdx.y, n = nsig_of(c, s), ldn = c.nmax;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  SpBuf<double> sp = fp64_bufs(c, tsize);
  double* A = sp.o64(s) + (long)i * ldn;
  const int* perm = sp.perm(s);
  for (int j = n - 1; j >= 0; --j) {
    const int q = perm[j];
    if (q != j) {
      const double t = A[j];
      A[j] = A[q];
      A[q] = t;
    }
  }
}

}  // namespace

cudaError_t sp_dgemm(SpGemm& g, int mode, int max_m, int max_n, cudaStream_t st) {
  return sp_gemm_t<double>(g, mode, max_m, max_n, st);
}

cudaError_t sp_digit_products(const ChainDesc* d, int nc, int N, int nmax, int b, int tsize, cudaStream_t st) {
  const int t = (nmax + 31) / 32;
  (void)N;
  sp_digits_kernel<<<dim3((b < 0 ? 1 : 2) * nmax, 2, nc), 256, 0, st>>>(d, b, tsize);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  sp_digit_gemm_kernel<<<dim3(t * t, 2, nc), 256, 0, st>>>(d, b, tsize);
  return cudaGetLastError();
}

cudaError_t sp_chol_panel(const ChainDesc* d, int nc, int nmax, int p, int tsize, cudaStream_t st) {
  (void)nmax;
  chol_panel_kernel<<<dim3(2, nc), 256, 0, st>>>(d, p, tsize);
  return cudaGetLastError();
}

cudaError_t sp_qform(const ChainDesc* d, int nc, int N, int nmax, int left, int b, int tsize, cudaStream_t st) {
  (void)nmax;
  qform_kernel<<<dim3((N + 7) / 8, 2, nc), 256, 0, st>>>(d, left, b, tsize);
  return cudaGetLastError();
}

cudaError_t sp_gj_panel(const ChainDesc* d, int nc, int nmax, int p, int tsize, cudaStream_t st) {
  (void)nmax;
  gj_panel_kernel<<<dim3(2 * kGJRanks, nc), 256, 0, st>>>(d, p, tsize);
  return cudaGetLastError();
}

cudaError_t sp_gj_unswap(const ChainDesc* d, int nc, int nmax, int tsize, cudaStream_t st) {
  gj_unswap_kernel<<<dim3((nmax + 127) / 128, 2, nc), 128, 0, st>>>(d, tsize);
  return cudaGetLastError();
}

cudaError_t spread_sweep_f64(const SpreadPlan& p, int mode, int measure, cudaStream_t st) {
  return spread_sweep_t<double>(p, mode, measure, st);
}

}  // namespace pqmc
