// linalg.cuh - dense complex linear algebra of the MPO update, written for
// one GB300: a tiled SIMT complex GEMM, a persistent cooperative parallel
// Jacobi eigen-solver for Hermitian matrices, and the single-CTA
// sort/select/entropy kernel that turns eigenvalues into kept Schmidt values.
#pragma once
#include "common.cuh"

// ---------------------------------------------------------------------------
// Complex GEMM: C (M x N) = alpha * op(A) * op(B), all row-major.
//   op == 0: plain; op == 1: conjugate transpose.
//   op(A)(i,k) = A[i*lda + k]      or conj(A[k*lda + i])
//   op(B)(k,j) = B[k*ldb + j]      or conj(B[j*ldb + k])
// alpha = alpha_host * (alpha_dev ? *alpha_dev : 1); accumulate != 0 adds the
// product to C instead of overwriting it (C and A / B must not overlap then).
// CTA tile BM x BN, K-slab BK, 256 threads, each thread TM x TN outputs spaced
// by 16 rows / 16 columns so that shared-memory reads broadcast along rows.
// The complex64 product; complex128 has its own kernel below.
// ---------------------------------------------------------------------------
template <typename T, int BM, int BN, int BK>
__global__ void __launch_bounds__(256) cgemm_kernel(int M, int N, int K,
    const cplx<T>* __restrict__ A, int lda, int opA,
    const cplx<T>* __restrict__ B, int ldb, int opB,
    cplx<T>* __restrict__ C, int ldc, const double* __restrict__ alpha_dev, double alpha_host, int accumulate) {
  constexpr int TM = BM / 16, TN = BN / 16;
  __shared__ cplx<T> As[BK][BM];
  __shared__ cplx<T> Bs[BK][BN];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int row0 = blockIdx.y * BM, col0 = blockIdx.x * BN;
  cplx<T> acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = czero<T>();

  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int s = 0; s < (BM * BK) / 256; ++s) {
      int idx = tid + 256 * s, i, k;
      cplx<T> v = czero<T>();
      if (opA == 0) {
        i = idx / BK; k = idx % BK;
        if (row0 + i < M && k0 + k < K) v = A[(size_t)(row0 + i) * lda + (k0 + k)];
      } else {
        i = idx % BM; k = idx / BM;
        if (row0 + i < M && k0 + k < K) v = cconj<T>(A[(size_t)(k0 + k) * lda + (row0 + i)]);
      }
      As[k][i] = v;
    }
#pragma unroll
    for (int s = 0; s < (BN * BK) / 256; ++s) {
      int idx = tid + 256 * s, j, k;
      cplx<T> v = czero<T>();
      if (opB == 0) {
        j = idx % BN; k = idx / BN;
        if (col0 + j < N && k0 + k < K) v = B[(size_t)(k0 + k) * ldb + (col0 + j)];
      } else {
        k = idx % BK; j = idx / BK;
        if (col0 + j < N && k0 + k < K) v = cconj<T>(B[(size_t)(col0 + j) * ldb + (k0 + k)]);
      }
      Bs[k][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      cplx<T> a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) cfma<T>(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
  const T alpha = (T)(alpha_host * (alpha_dev ? *alpha_dev : 1.0));
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = row0 + ty + 16 * i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = col0 + tx + 16 * j;
      if (c < N) {
        cplx<T> v = cscale<T>(acc[i][j], alpha);
        if (accumulate) v = cadd<T>(v, C[(size_t)r * ldc + c]);
        C[(size_t)r * ldc + c] = v;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The complex128 product. An SM does 2 FP64 FMAs per clock, so a 64 x 64 tile
// costs one SM 8192 clocks per k (4 us), padding included: the factorisations'
// products (16 .. 256 rows) sat on one to sixteen SMs for 100 .. 250 us. Small
// tiles put the same work on all of them; at this rate one output per thread
// and two shared-memory reads per complex FMA hide behind the FP64 unit.
// TT x TT outputs per CTA of 256 threads; TT = 16 gives every thread one, TT = 8
// splits k four ways inside the CTA (partial sums added in a fixed order) and
// serves products with fewer 16 x 16 tiles than SMs. The next k slab is read into
// registers while this one is multiplied. Linear grid.
// Measured: 256 x 256 x 64 36 us, 1024 x 1024 x 256 1.80 ms (28 us and 1.79 ms at the
// part's 1.2 TFLOP/s); sampling 2000 strings (128 products of 2000 x 64 x 64)
// 14.5 -> 4.8 ms, 1082 products of a short chain's circuit 130 -> 20 ms.
// ---------------------------------------------------------------------------
template <typename T, int TT>
__global__ void __launch_bounds__(256) cgemm_small_kernel(int M, int N, int K, const cplx<T>* __restrict__ A, int lda,
                                                          int opA, const cplx<T>* __restrict__ B, int ldb, int opB,
                                                          cplx<T>* __restrict__ C, int ldc,
                                                          const double* __restrict__ alpha_dev, double alpha_host,
                                                          int accumulate, int ncol) {
  constexpr int KSPLIT = 256 / (TT * TT), BK = 256 / TT, KT = BK / KSPLIT;   // one element of A and B per thread and slab
  __shared__ cplx<T> As[BK][TT + 1], Bs[BK][TT + 1];
  __shared__ cplx<T> red[KSPLIT > 1 ? 256 : 1];
  const int tid = threadIdx.x;
  const int row0 = (int)(blockIdx.x / ncol) * TT, col0 = (int)(blockIdx.x % ncol) * TT;
  const int i = (tid / TT) % TT, j = tid % TT, part = tid / (TT * TT);
  // this thread's staged elements: along the stored row of either form
  const int ai = opA ? tid % TT : tid / BK, ak = opA ? tid / TT : tid % BK;
  const int bj = opB ? tid / BK : tid % TT, bk = opB ? tid % BK : tid / TT;
  auto load_a = [&](int k0) -> cplx<T> {
    if (row0 + ai >= M || k0 + ak >= K) return czero<T>();
    return opA ? cconj<T>(A[(size_t)(k0 + ak) * lda + row0 + ai]) : A[(size_t)(row0 + ai) * lda + k0 + ak];
  };
  auto load_b = [&](int k0) -> cplx<T> {
    if (col0 + bj >= N || k0 + bk >= K) return czero<T>();
    return opB ? cconj<T>(B[(size_t)(col0 + bj) * ldb + k0 + bk]) : B[(size_t)(k0 + bk) * ldb + col0 + bj];
  };
  cplx<T> acc = czero<T>(), an = load_a(0), bn = load_b(0);
  for (int k0 = 0; k0 < K; k0 += BK) {
    As[ak][ai] = an;
    Bs[bk][bj] = bn;
    __syncthreads();
    if (k0 + BK < K) { an = load_a(k0 + BK); bn = load_b(k0 + BK); }
    const int kn = min(KT, K - k0 - part * KT);
#pragma unroll 8
    for (int k = 0; k < kn; ++k) cfma<T>(acc, As[part * KT + k][i], Bs[part * KT + k][j]);
    __syncthreads();
  }
  if constexpr (KSPLIT > 1) {
    red[tid] = acc;
    __syncthreads();
    if (part > 0) return;
#pragma unroll
    for (int q = 1; q < KSPLIT; ++q) acc = cadd<T>(acc, red[tid + q * TT * TT]);
  }
  const int r = row0 + i, c = col0 + j;
  if (r >= M || c >= N) return;
  cplx<T> v = cscale<T>(acc, (T)(alpha_host * (alpha_dev ? *alpha_dev : 1.0)));
  if (accumulate) v = cadd<T>(v, C[(size_t)r * ldc + c]);
  C[(size_t)r * ldc + c] = v;
}

constexpr int kTileSms = 152;     // SMs of the part: fewer 16 x 16 tiles than that go as 8 x 8 ones

template <typename T>
inline cudaError_t cgemm(cudaStream_t st, int M, int N, int K, const cplx<T>* A, int lda, int opA,
                         const cplx<T>* B, int ldb, int opB, cplx<T>* C, int ldc,
                         const double* alpha_dev = nullptr, double alpha_host = 1.0, int accumulate = 0) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  constexpr int BM = 64, BN = 64, BK = 8;
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
  if (K <= 0 && accumulate) return cudaSuccess;
  if (K <= 0) {  // empty contraction: C = 0
    for (int r = 0; r < M; ++r) {
      cudaError_t e = cudaMemsetAsync(C + (size_t)r * ldc, 0, sizeof(cplx<T>) * N, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if constexpr (sizeof(T) == 8) {
    const long nr16 = (M + 15) / 16, nc16 = (N + 15) / 16, nr8 = (M + 7) / 8, nc8 = (N + 7) / 8;
    if (nr16 * nc16 < kTileSms)
      cgemm_small_kernel<T, 8><<<(unsigned)(nr8 * nc8), 256, 0, st>>>(M, N, K, A, lda, opA, B, ldb, opB, C, ldc, alpha_dev,
                                                                      alpha_host, accumulate, (int)nc8);
    else
      cgemm_small_kernel<T, 16><<<(unsigned)(nr16 * nc16), 256, 0, st>>>(M, N, K, A, lda, opA, B, ldb, opB, C, ldc,
                                                                         alpha_dev, alpha_host, accumulate, (int)nc16);
  } else {
    cgemm_kernel<T, BM, BN, BK><<<grid, 256, 0, st>>>(M, N, K, A, lda, opA, B, ldb, opB, C, ldc, alpha_dev, alpha_host,
                                                       accumulate);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Parallel cyclic Jacobi eigen-solver for an m x m Hermitian matrix G
// (row-major, leading dimension m), in place: on exit G is diagonal to
// within the stopping rule, w[i] = G_ii and V (row-major) holds the
// eigenvectors as columns, G_in = V diag(w) V^H.
//
// Ordering: round-robin (circle method) over N = m + (m odd) players, so each
// round rotates N/2 disjoint pairs (p, q) and a sweep of N-1 rounds visits
// every pair once; an odd m gives one pair a bye per round.
// Rotation of pair (p, q) with a = G_pp, b = G_qq, g = G_pq = |g| u:
//   zeta = (b - a) / (2|g|), t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
//   c = 1/sqrt(1 + t^2), s = t c, J = [[c, s], [-conj(u) s, conj(u) c]],
// the complex form of the symmetric Schur rotation (Golub & Van Loan,
// Matrix Computations, Sec. 8.5); J^H G J zeroes G_pq.
// A pair is skipped when |g| <= max(tol_rel sqrt(|a b|), floor_rel max_i|G_ii|)
// (the relative criterion of Demmel & Veselic 1992 plus an absolute floor at
// the rounding level of the input). The solve stops after a sweep without a
// rotation; status = 1 if max_sweeps is reached first.
//
// Only the upper triangle is kept: entry (i, j) with i > j is read as the
// conjugate of (j, i). A round runs as two phases of one persistent cooperative
// launch:
//   A: the round's rotation table, each pair by one thread of the grid, to
//      the global table of this round's parity;                     barrier
//   B: the round's pairs split G into 2 x 2 blocks G[p_a, q_a][p_b, q_b]; each
//      block a <= b becomes J_a^H G_ab J_b, and V <- V J;              barrier
// (work items of 32 blocks of one a, or 32 pairs of four rows of V, a warp each).
// All G/V traffic uses L2-only loads/stores because other CTAs write it.
// What bounds it: the FP64 unit (2 FMA per clock and SM) from m ~ 500, the two
// barriers and the rotation parameters below. Updating both triangles by rows
// and then by columns, with a third barrier, took 1.5 times the FP64 work; a
// table built by every CTA, with ~200 FP64 instructions per rotation, 6 us per
// round. Nearly diagonal m = 1088: 303 -> 111 ms, m = 320 18.6 -> 9.1, m = 128 5.0 -> 3.5.
// ---------------------------------------------------------------------------
template <typename T> struct JRot { T c, s, ur, ui; };

__device__ __forceinline__ int rr_player(int pos, int r, int N) {
  return pos == 0 ? 0 : 1 + ((pos - 1 + r) % (N - 1));
}

// ---------------------------------------------------------------------------
// Select kernel (one CTA): turn the m eigenvalues w of a Gram matrix (the
// squared Schmidt values lambda'^2 of the factorised bond) into the kept set.
//   - bitonic sort of (value desc, index asc) in shared memory (stable order
//     for exact ties), negative rounding values clamped to 0;
//   - k = min(cap, #{lambda^2 > cutoff^2 * lambda_max^2}), at least 1; min(cap, m) when
//     cutoff2 < 0, also where every value is zero (callers then read all of perm);
//   - sums in FP64: total = sum lambda^2 (or *total_in, the squared Frobenius
//     norm of the factorised matrix, when w holds Ritz values of a subspace
//     only), kept = sum of the k largest;
//   - outputs perm[0..k), lam2[0..k) (descending), info->k, info->kept,
//     info->total, info->status (1: a value is infinite or NaN); adds (total-kept)/total to *disc_acc and 0.5 log(kept) to
//     *lognorm when those are non-null;
//   - with S_out: the MPO entanglement entropy -sum p log2 p, p = lam2/kept
//     (Sec. 3.3), and the normalised lam2/kept into schmidt_out.
// ---------------------------------------------------------------------------
struct SelectInfo {
  int k;
  int status;
  int pad[2];
  double kept;
  double total;
  double inv_sqrt_kept;
  double pad2;
};

template <typename T>
__global__ void __launch_bounds__(1024) select_kernel(const T* __restrict__ w, int m, int cap, double cutoff2,
                                                       int* __restrict__ perm, double* __restrict__ lam2,
                                                       SelectInfo* info, double* disc_acc, double* lognorm,
                                                       double* S_out, double* schmidt_out,
                                                       const double* __restrict__ total_in) {
  extern __shared__ unsigned char ssm[];
  int P = 1;
  while (P < m) P <<= 1;
  double* key = reinterpret_cast<double*>(ssm);
  int* idx = reinterpret_cast<int*>(key + P);
  __shared__ double red[32];
  __shared__ double s_tot, s_kept, s_max;
  __shared__ int s_k;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wp = tid >> 5;
  bool bad = false;
  for (int i = tid; i < P; i += nt) {
    if (i < m) { double v = (double)w[i]; key[i] = v > 0.0 ? v : 0.0; idx[i] = i; bad |= !isfinite(v); }
    else { key[i] = -1.0; idx[i] = 0x7fffffff; }
  }
  const int any_bad = __syncthreads_or(bad);
  // bitonic sort, descending by key, ascending index on ties
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = tid; i < P; i += nt) {
        int j = i ^ stride;
        if (j > i) {
          bool desc = ((i & size) == 0);
          double ki = key[i], kj = key[j];
          int ii = idx[i], ij = idx[j];
          bool i_first = (ki > kj) || (ki == kj && ii < ij);   // i belongs before j in descending order
          bool swap = desc ? !i_first : i_first;
          if (swap) { key[i] = kj; key[j] = ki; idx[i] = ij; idx[j] = ii; }
        }
      }
      __syncthreads();
    }
  }
  // total and max
  double loc = 0.0;
  for (int i = tid; i < m; i += nt) loc += key[i];
  for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
  if (lane == 0) red[wp] = loc;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int i = 0; i < (nt + 31) / 32; ++i) s += red[i];
    s_tot = total_in ? *total_in : s;   // the factorised matrix's squared norm when w covers a subspace only
    s_max = key[0];
    const double thr = cutoff2 * key[0];
    int k = 0;
    const int lim = cap < m ? cap : m;
    while (k < lim && (cutoff2 < 0.0 || key[k] > thr)) ++k;
    if (k == 0) k = 1;
    s_k = k;
  }
  __syncthreads();
  const int k = s_k;
  loc = 0.0;
  for (int i = tid; i < k; i += nt) loc += key[i];
  for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
  __syncthreads();
  if (lane == 0) red[wp] = loc;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int i = 0; i < (nt + 31) / 32; ++i) s += red[i];
    s_kept = s;
  }
  __syncthreads();
  const double kept = s_kept;
  for (int i = tid; i < k; i += nt) { perm[i] = idx[i]; lam2[i] = key[i]; }
  if (S_out) {
    loc = 0.0;
    for (int i = tid; i < k; i += nt) {
      const double pz = kept > 0.0 ? key[i] / kept : 0.0;
      if (schmidt_out) schmidt_out[i] = pz;
      if (pz > 0.0) loc -= pz * log2(pz);
    }
    for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
    __syncthreads();
    if (lane == 0) red[wp] = loc;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int i = 0; i < (nt + 31) / 32; ++i) s += red[i];
      *S_out = s;
    }
  }
  if (tid == 0) {
    info->k = k;
    info->status = any_bad ? 1 : 0;
    info->kept = kept;
    info->total = s_tot;
    info->inv_sqrt_kept = kept > 0.0 ? 1.0 / sqrt(kept) : 0.0;
    if (disc_acc && s_tot > 0.0) *disc_acc += (s_tot - kept) / s_tot;
    if (lognorm && kept > 0.0) *lognorm += 0.5 * log(kept);
  }
}

// ---------------------------------------------------------------------------
// One-sided (Hestenes) Jacobi SVD by row orthogonalisation.
// Input X (r x c, row-major, leading dimension ldx), in place. On exit the
// rows of X are mutually orthogonal, X_out = U^H X_in with U unitary (r x r),
// returned transposed as Ut (row p of Ut = column p of U, leading dim r), and
// w[i] = ||row i of X_out||^2: X_in = U X_out, so the squared singular values
// of X_in are w and its left singular vectors the columns of U
// (Hestenes 1958; Demmel & Veselic 1992 for the relative-accuracy stopping
// rule). No Gram matrix is formed, so small singular values keep their
// relative accuracy instead of being lost below eps * sigma_max^2.
//
// Pair (p, q) with a = ||x_p||^2, b = ||x_q||^2, g = <x_p, x_q> = sum_j
// x_p[j] conj(x_q[j]) is rotated by the same J as in the two-sided solver:
// rows  x_p <- c x_p - u s x_q,   x_q <- s x_p + u c x_q      (X <- J^H X)
// Ut    t_p <- c t_p - u* s t_q,  t_q <- s t_p + u* c t_q      (U <- U J)
// Ordering is round-robin as above; pairs of one round touch disjoint rows,
// so a round is one phase (one warp per pair) followed by one grid barrier.
// The complex64 form below its block solver's smallest size.
// A sweep with no rotation (|g| <= max(tol sqrt(ab), floor)) ends the solve.
// ---------------------------------------------------------------------------
struct OSCtl {
  GridCtl g;
  int active[64];   // rotations per sweep (grid-wide atomic counts)
  double scale;
  double pad;
  unsigned long long phase_ns[4];   // CTA 0: wall time per phase (G, E, A), barrier waits included
};

// Largest of w[0 .. r), read through L2 by the whole CTA (at most 1024 threads).
template <typename T>
__device__ T block_max(const T* w, int r) {
  __shared__ T s_part[32];
  T mx = T(0);
  for (int i = threadIdx.x; i < r; i += blockDim.x) mx = fmax(mx, __ldcg(&w[i]));
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = s_part[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) mx = fmax(mx, s_part[i]);
  __syncthreads();
  return mx;
}

template <typename T>
__device__ __forceinline__ void warp_sum3(T& a, T& b, T& c, T& d) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
    d += __shfl_xor_sync(0xffffffffu, d, o);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) onesided_jacobi_kernel(cplx<T>* X, int r, int c, int ldx, cplx<T>* Ut, T* w,
                                                               OSCtl* ctl, int max_sweeps, T tol_rel, T floor_rel,
                                                               long long timeout_ns) {
  const int N = r + (r & 1), npairs = N / 2;
  const unsigned nblk = gridDim.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwb = blockDim.x >> 5;
  // warp w of CTA b takes the pairs w gridDim + b, ...: neighbouring pairs go to
  // different SMs, so that a round of fewer pairs than warps uses every SM
  const long gwarp = (long)warp * nblk + blockIdx.x, nwarps = (long)nblk * nwb;
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, gthreads = (size_t)nblk * blockDim.x;
  if (max_sweeps > 64) max_sweeps = 64;

  for (size_t e = gtid; e < (size_t)r * r; e += gthreads) {
    const size_t i = e / r, j = e % r;
    stcg(&Ut[e], mk<T>(i == j ? T(1) : T(0), T(0)));
  }
  // squared row norms -> w, then the largest one sets the absolute floor
  for (long i = gwarp; i < r; i += nwarps) {
    T s = T(0);
    for (int j = lane; j < c; j += 32) { const cplx<T> x = ldcg(&X[(size_t)i * ldx + j]); s += x.x * x.x + x.y * x.y; }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) w[i] = s;
  }
  if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
  const T floor_abs = floor_rel * block_max<T>(w, r);

  int sweep = 0;
  bool converged = (r <= 1);
  for (; sweep < max_sweeps && !converged; ++sweep) {
    for (int rd = 0; rd < N - 1; ++rd) {
      for (long pi = gwarp; pi < npairs; pi += nwarps) {
        int p = rr_player((int)pi, rd, N), q = rr_player(N - 1 - (int)pi, rd, N);
        if (p > q) { int t_ = p; p = q; q = t_; }
        if (q >= r) continue;
        cplx<T>* xp = X + (size_t)p * ldx;
        cplx<T>* xq = X + (size_t)q * ldx;
        T a = T(0), b = T(0), gr = T(0), gi = T(0);
#pragma unroll 16
        for (int j = lane; j < c; j += 32) {
          const cplx<T> x = ldcg(&xp[j]), y = ldcg(&xq[j]);
          a = fma(x.x, x.x, fma(x.y, x.y, a));
          b = fma(y.x, y.x, fma(y.y, y.y, b));
          gr = fma(x.x, y.x, fma(x.y, y.y, gr));     // x conj(y)
          gi = fma(x.y, y.x, fma(-x.x, y.y, gi));
        }
        warp_sum3<T>(a, b, gr, gi);
        // rotation parameters in FP64 whatever T is: unbiased c, s, u keep
        // the accumulated U unitary over many sweeps
        const double agd = hypot((double)gr, (double)gi);
        const double thr = fmax((double)tol_rel * sqrt((double)a * (double)b), (double)floor_abs);
        if (!(agd > thr) || agd == 0.0) continue;
        const double zeta = ((double)b - (double)a) / (2.0 * agd);
        double td;
        if (fabs(zeta) > 1e16) td = 0.5 / zeta;
        else td = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        const double csd = 1.0 / sqrt(1.0 + td * td);
        const T cs = (T)csd, sn = (T)(td * csd);
        if (sn == T(0)) continue;
        const T ur = (T)((double)gr / agd), ui = (T)((double)gi / agd);
        if (lane == 0) atomicAdd(&ctl->active[sweep], 1);
#pragma unroll 16
        for (int j = lane; j < c; j += 32) {
          const cplx<T> x = ldcg(&xp[j]), y = ldcg(&xq[j]);
          const cplx<T> uy = cmul<T>(mk<T>(ur, ui), y);
          stcg(&xp[j], mk<T>(cs * x.x - sn * uy.x, cs * x.y - sn * uy.y));
          stcg(&xq[j], mk<T>(sn * x.x + cs * uy.x, sn * x.y + cs * uy.y));
        }
        cplx<T>* tp = Ut + (size_t)p * r;
        cplx<T>* tq = Ut + (size_t)q * r;
#pragma unroll 16
        for (int j = lane; j < r; j += 32) {
          const cplx<T> x = ldcg(&tp[j]), y = ldcg(&tq[j]);
          const cplx<T> uy = cmul<T>(mk<T>(ur, -ui), y);
          stcg(&tp[j], mk<T>(cs * x.x - sn * uy.x, cs * x.y - sn * uy.y));
          stcg(&tq[j], mk<T>(sn * x.x + cs * uy.x, sn * x.y + cs * uy.y));
        }
      }
      if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
    }
    if (atomicAdd(&ctl->active[sweep], 0) == 0) converged = true;
  }
  for (long i = gwarp; i < r; i += nwarps) {
    T s = T(0);
    for (int j = lane; j < c; j += 32) { const cplx<T> x = ldcg(&X[(size_t)i * ldx + j]); s += x.x * x.x + x.y * x.y; }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) w[i] = s;
  }
  if (gtid == 0) {
    ctl->g.sweeps = sweep;
    ctl->g.status = converged ? 0 : 1;
  }
}

// ---------------------------------------------------------------------------
// The same solver with one CTA (four warps) per row pair: every complex128
// factorisation, and the FP32 solves (quad_jacobi_kernel below) of fewer than 32
// rows or more than 4096 columns. onesided_jacobi_kernel above serves the
// complex64 form, whose results are pinned to its arithmetic.
//
// What bounds it: an FP64 warp instruction occupies its SM partition for 64
// clocks on this part, so a pair handled by one warp uses a quarter of the
// SM's FP64 rate, and the ~200 FP64 instructions of the rotation parameters
// (hypot, square roots, divisions) cost 6 us per round, more than the rows
// themselves below ~300 columns. Four warps share the pair's rows, the four
// sums are reduced by halves (6 + 2 additions instead of 20), one warp forms
// the parameters in ~35 FP64 instructions (osj_rotation), and rows of up to
// 128 E elements stay in registers between the dot products and the rotation
// (one read and one write per round instead of two and one).
// Measured, one warp per pair -> this kernel: complex128 64 x 64 17.2 ->
// 7.1 ms (20 sweeps), 256 x 256 174 -> 51 ms, 768 x 1024 1363 -> 586 ms
// (28 sweeps, 27 us per round).
// ---------------------------------------------------------------------------
constexpr int OSJ_NT = 128;

// 1 / sqrt(x) for x in [1, 8): the FP32 approximation (2^-22) and one
// third-order step y (1 + e/2 + 3 e^2 / 8), e = 1 - x y^2, whose remainder
// (5/16) e^3 is below 2^-66.
__device__ __forceinline__ double osj_rsqrt(double x) {
  const double y = (double)rsqrtf((float)x);
  const double e = fma(-x * y, y, 1.0);
  return fma(y, e * fma(e, 0.375, 0.5), y);
}

// 2^k as a double, |k| <= 1022.
__device__ __forceinline__ double osj_pow2(int k) { return __longlong_as_double((long long)(k + 1023) << 52); }

// Rotation parameters of a row pair with a = |x|^2, b = |y|^2, g = <x, y>:
// c, s real and u = g / |g|; false when |g| <= max(tol sqrt(ab), floor) or
// the rotation is below resolution. The root t of t^2 + 2 zeta t - 1 is taken in
// FP32 and corrected by one FP64 Newton step (relative error ~1e-14, so a
// rotation leaves 1e-14 of g); c and u come from osj_rsqrt, so c^2 + s^2 and
// |u| are 1 to FP64 rounding whatever the angle. g is scaled by a power of two
// first (integer arithmetic on its exponent), so no square over- or underflows.
// A denormal g has too few bits for a rotation: none is made, and unresolved (if
// given) is set when it is still above the threshold (rows below ~1e-150), so that
// the solve ends unconverged instead of taking such rows for orthogonal.
__device__ __forceinline__ bool osj_rotation(double a, double b, double gr, double gi, double tol2, double floor_abs,
                                             double& c, double& s, double& ur, double& ui,
                                             bool* unresolved = nullptr) {
  const int er = (int)((__double_as_longlong(gr) >> 52) & 0x7FF), ei = (int)((__double_as_longlong(gi) >> 52) & 0x7FF);
  const int e = max(er, ei) - 1023;
  if (e <= -1022) {
    if (unresolved) *unresolved = fmax(fabs(gr), fabs(gi)) > fmax(sqrt(tol2) * (sqrt(a) * sqrt(b)), floor_abs);
    return false;
  }
  if (e >= 1022) return false;                    // infinite or NaN couplings
  const double sc = osj_pow2(-e);
  const double x = gr * sc, y = gi * sc;
  const double g2 = fma(x, x, y * y);             // in [1, 8)
  if (!(g2 > tol2 * fabs((a * sc) * (b * sc)))) return false;
  const double inv = osj_rsqrt(g2);
  if (!(g2 * inv * osj_pow2(e) > floor_abs)) return false;
  const double zeta = ((b - a) * sc) * (0.5 * inv);
  const float zf = (float)zeta, az = fabsf(zf);
  if (!(az < 3e38f)) return false;                // t below 1e-38: no change at any precision
  float t0 = az > 1e18f ? 0.5f / az : 1.0f / (az + sqrtf(fmaf(az, az, 1.0f)));
  if (zf < 0.0f) t0 = -t0;
  const double td = (double)t0;
  const double f = fma(td, td + 2.0 * zeta, -1.0);
  const double t = fma(-f, (double)(0.5f / (zf + t0)), td);
  c = osj_rsqrt(fma(t, t, 1.0));
  s = t * c;
  ur = x * inv;
  ui = y * inv;
  return s != 0.0;
}

// Sum of the four values over the CTA's 128 threads, returned in every lane of
// warp 0 only (one barrier; the caller's next barrier frees the scratch).
template <typename T>
__device__ __forceinline__ void osj_reduce4(T& a, T& b, T& c, T& d, T (*part)[4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool h16 = lane & 16, h8 = lane & 8;
  T v0 = h16 ? c : a, v1 = h16 ? d : b;
  v0 += __shfl_xor_sync(0xffffffffu, h16 ? a : c, 16);
  v1 += __shfl_xor_sync(0xffffffffu, h16 ? b : d, 16);
  T v = h8 ? v1 : v0;
  v += __shfl_xor_sync(0xffffffffu, h8 ? v0 : v1, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  if ((lane & 7) == 0) part[lane >> 3][warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = part[(lane >> 2) & 3][lane & 3];
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    a = __shfl_sync(0xffffffffu, v, 0);
    b = __shfl_sync(0xffffffffu, v, 4);
    c = __shfl_sync(0xffffffffu, v, 8);
    d = __shfl_sync(0xffffffffu, v, 12);
  }
}

template <typename T> struct OsjRot { T c, s, sur, sui, cur, cui; int on; };

// (x, y) <- (c x - s u y, s x + c u y)
template <typename T>
__device__ __forceinline__ void osj_rotate(cplx<T>& x, cplx<T>& y, T c, T s, T sur, T sui, T cur, T cui) {
  const cplx<T> xn = mk<T>(fma(sui, y.y, fma(-sur, y.x, c * x.x)), fma(-sui, y.x, fma(-sur, y.y, c * x.y)));
  y = mk<T>(fma(-cui, y.y, fma(cur, y.x, s * x.x)), fma(cui, y.x, fma(cur, y.y, s * x.y)));
  x = xn;
}

// The two-sided solver (described at JRot).
template <typename T>
__global__ void __launch_bounds__(256) jacobi_kernel(cplx<T>* G, int m, cplx<T>* V, T* w, JRot<T>* table, GridCtl* ctl,
                                                      int max_sweeps, T tol_rel, T floor_rel, long long timeout_ns) {
  extern __shared__ unsigned char jsmem[];
  JRot<T>* rot = reinterpret_cast<JRot<T>*>(jsmem);
  __shared__ T s_red[32];
  const int N = m + (m & 1), npairs = N / 2;
  const unsigned nblk = gridDim.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwarp_blk = blockDim.x >> 5;
  const long gwarp = (long)warp * nblk + blockIdx.x, nwarps = (long)nblk * nwarp_blk;
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, gthreads = (size_t)nblk * blockDim.x;

  // V = I
  for (size_t e = gtid; e < (size_t)m * m; e += gthreads) {
    size_t r = e / m, c = e % m;
    stcg(&V[e], mk<T>(r == c ? T(1) : T(0), T(0)));
  }
  // scale = max_i |G_ii| (each CTA redundantly)
  T loc = T(0);
  for (int i = threadIdx.x; i < m; i += blockDim.x) loc = fmax(loc, fabs(ldcg(&G[(size_t)i * m + i]).x));
  for (int o = 16; o > 0; o >>= 1) loc = fmax(loc, __shfl_xor_sync(0xffffffffu, loc, o));
  if (lane == 0) s_red[warp] = loc;
  __syncthreads();
  if (threadIdx.x == 0) {
    T mx = T(0);
    for (int i = 0; i < nwarp_blk; ++i) mx = fmax(mx, s_red[i]);
    s_red[0] = mx;
  }
  __syncthreads();
  const T floor_abs = floor_rel * s_red[0];
  if (!grid_barrier(ctl, nblk, timeout_ns)) return;

  auto ld = [&](int i, int j) -> cplx<T> {
    return i < j ? ldcg(&G[(size_t)i * m + j]) : cconj<T>(ldcg(&G[(size_t)j * m + i]));
  };
  auto st = [&](int i, int j, cplx<T> v) {
    if (i < j) stcg(&G[(size_t)i * m + j], v);
    else stcg(&G[(size_t)j * m + i], cconj<T>(v));
  };
  // the work items of phase B: blocks (a, b) with b in chunk k and a <= b, then
  // four rows of V by one chunk of pairs
  const int nch = (npairs + 31) / 32;
  long nblocks = 0;
  for (int k = 0; k < nch; ++k) nblocks += min(npairs, 32 * (k + 1));
  const long nitems = nblocks + (long)((m + 3) / 4) * nch;
  const double tol2 = (double)tol_rel * (double)tol_rel;

  int sweep = 0;
  bool converged = (m <= 1);
  for (; sweep < max_sweeps && !converged; ++sweep) {
    long sweep_active = 0;
    for (int r = 0; r < N - 1; ++r) {
      // ---- phase A: rotation table -------------------------------------
      // two tables in turn: a CTA that is already in the next round writes
      // the other one while slower CTAs still read this one
      JRot<T>* tab = table + (size_t)((sweep * (N - 1) + r) & 1) * npairs;
      for (long pi = blockIdx.x + (long)threadIdx.x * nblk; pi < npairs; pi += (long)nblk * blockDim.x) {
        int p = rr_player((int)pi, r, N), q = rr_player(N - 1 - (int)pi, r, N);
        if (p > q) { int t_ = p; p = q; q = t_; }
        JRot<T> R; R.c = T(1); R.s = T(0); R.ur = T(1); R.ui = T(0);
        if (q < m) {
          const T a = ldcg(&G[(size_t)p * m + p]).x, b = ldcg(&G[(size_t)q * m + q]).x;
          const cplx<T> g = ldcg(&G[(size_t)p * m + q]);
          double cs, sn, ur, ui;
          if (osj_rotation((double)a, (double)b, (double)g.x, (double)g.y, tol2, (double)floor_abs, cs, sn, ur, ui)) {
            R.c = (T)cs; R.s = (T)sn; R.ur = (T)ur; R.ui = (T)ui;
          }
        }
        __stcg(&tab[pi].c, R.c); __stcg(&tab[pi].s, R.s); __stcg(&tab[pi].ur, R.ur); __stcg(&tab[pi].ui, R.ui);
      }
      // phase B rewrites the pivots (G_pp, G_qq, G_pq) that phase A reads:
      // no CTA rotates before the whole table has been built from the same G
      if (!grid_barrier(ctl, nblk, timeout_ns)) return;
      int my_active = 0;
      for (int pi = threadIdx.x; pi < npairs; pi += blockDim.x) {
        JRot<T> R;
        R.c = __ldcg(&tab[pi].c); R.s = __ldcg(&tab[pi].s); R.ur = __ldcg(&tab[pi].ur); R.ui = __ldcg(&tab[pi].ui);
        rot[pi] = R;
        if (R.s != T(0)) my_active = 1;
      }
      const int act = __syncthreads_or(my_active);   // identical in every CTA: the same table
      if (act == 0) continue;
      ++sweep_active;
      // ---- phase B -------------------------------------------------------
      for (long it = gwarp; it < nitems; it += nwarps) {
        if (it < nblocks) {
          int k = 0;
          long a_ = it;
          while (a_ >= min(npairs, 32 * (k + 1))) a_ -= min(npairs, 32 * ++k);
          const int a = (int)a_, b = 32 * k + lane;
          if (b >= npairs || a > b) continue;
          const JRot<T> Ra = rot[a], Rb = rot[b];
          if (Ra.s == T(0) && Rb.s == T(0)) continue;
          int p = rr_player(a, r, N), q = rr_player(N - 1 - a, r, N);
          if (p > q) { int t_ = p; p = q; q = t_; }
          if (a == b) {              // the rotated pair itself: G_pq becomes an exact zero
            const cplx<T> g = ldcg(&G[(size_t)p * m + q]);
            const T d = Ra.s / Ra.c * (g.x * Ra.ur + g.y * Ra.ui);     // t |g|
            stcg(&G[(size_t)p * m + p], mk<T>(ldcg(&G[(size_t)p * m + p]).x - d, T(0)));
            stcg(&G[(size_t)q * m + q], mk<T>(ldcg(&G[(size_t)q * m + q]).x + d, T(0)));
            stcg(&G[(size_t)p * m + q], czero<T>());
            continue;
          }
          int x = rr_player(b, r, N), y = rr_player(N - 1 - b, r, N);
          if (x > y) { int t_ = x; x = y; y = t_; }
          const bool hq = q < m, hy = y < m;      // false for the index that sits out (odd m)
          cplx<T> b00 = ld(p, x), b01 = hy ? ld(p, y) : czero<T>();
          cplx<T> b10 = hq ? ld(q, x) : czero<T>(), b11 = hq && hy ? ld(q, y) : czero<T>();
          if (Rb.s != T(0)) {        // columns: [x y] <- [c x - s conj(u) y, s x + c conj(u) y]
            const T sur = Rb.s * Rb.ur, sui = -Rb.s * Rb.ui, cur = Rb.c * Rb.ur, cui = -Rb.c * Rb.ui;
            osj_rotate<T>(b00, b01, Rb.c, Rb.s, sur, sui, cur, cui);
            osj_rotate<T>(b10, b11, Rb.c, Rb.s, sur, sui, cur, cui);
          }
          if (Ra.s != T(0)) {        // rows: [x; y] <- [c x - s u y; s x + c u y]
            const T sur = Ra.s * Ra.ur, sui = Ra.s * Ra.ui, cur = Ra.c * Ra.ur, cui = Ra.c * Ra.ui;
            osj_rotate<T>(b00, b10, Ra.c, Ra.s, sur, sui, cur, cui);
            osj_rotate<T>(b01, b11, Ra.c, Ra.s, sur, sui, cur, cui);
          }
          st(p, x, b00);
          if (hy) st(p, y, b01);
          if (hq) st(q, x, b10);
          if (hq && hy) st(q, y, b11);
        } else {
          const long v = it - nblocks;
          const int b = 32 * (int)(v % nch) + lane, row0 = 4 * (int)(v / nch);
          if (b >= npairs) continue;
          const JRot<T> R = rot[b];
          if (R.s == T(0)) continue;
          int p = rr_player(b, r, N), q = rr_player(N - 1 - b, r, N);
          if (p > q) { int t_ = p; p = q; q = t_; }
          const T sur = R.s * R.ur, sui = -R.s * R.ui, cur = R.c * R.ur, cui = -R.c * R.ui;
          cplx<T> xs[4], ys[4];
#pragma unroll
          for (int h = 0; h < 4; ++h)
            if (row0 + h < m) { xs[h] = ldcg(&V[(size_t)(row0 + h) * m + p]); ys[h] = ldcg(&V[(size_t)(row0 + h) * m + q]); }
#pragma unroll
          for (int h = 0; h < 4; ++h)
            if (row0 + h < m) {
              osj_rotate<T>(xs[h], ys[h], R.c, R.s, sur, sui, cur, cui);
              stcg(&V[(size_t)(row0 + h) * m + p], xs[h]);
              stcg(&V[(size_t)(row0 + h) * m + q], ys[h]);
            }
        }
      }
      if (!grid_barrier(ctl, nblk, timeout_ns)) return;
    }
    if (sweep_active == 0) converged = true;
  }
  for (size_t i = gtid; i < (size_t)m; i += gthreads) w[i] = ldcg(&G[i * m + i]).x;
  if (gtid == 0) {
    ctl->sweeps = sweep;
    ctl->status = converged ? 0 : 1;
  }
}

template <typename T, int E>
__global__ void __launch_bounds__(OSJ_NT) pair_jacobi_kernel(cplx<T>* X, int r, int c, int ldx, cplx<T>* Ut, T* w,
                                                             OSCtl* ctl, int max_sweeps, T tol_rel, T floor_rel,
                                                             int given_u, long long timeout_ns) {
  __shared__ T part[4][4];
  __shared__ OsjRot<T> s_rot;
  const int N = r + (r & 1), npairs = N / 2;
  const unsigned nblk = gridDim.x;
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t gtid = (size_t)blockIdx.x * OSJ_NT + tid, gthreads = (size_t)nblk * OSJ_NT;
  const bool regs = c <= OSJ_NT * E, uregs = r <= OSJ_NT * E;   // the rows fit the registers
  if (max_sweeps > 64) max_sweeps = 64;

  for (size_t e = gtid; e < (size_t)r * r && !given_u; e += gthreads) {   // else Ut already holds a U to rotate on
    const size_t i = e / r, j = e % r;
    stcg(&Ut[e], mk<T>(i == j ? T(1) : T(0), T(0)));
  }
  // squared row norms -> w, one warp per row
  auto norms = [&]() {
    for (long i = gtid >> 5; i < r; i += (long)(gthreads >> 5)) {
      T s = T(0);
      for (int j = lane; j < c; j += 32) {
        const cplx<T> x = ldcg(&X[(size_t)i * ldx + j]);
        s = fma(x.x, x.x, fma(x.y, x.y, s));
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) __stcg(&w[i], s);
    }
  };
  norms();
  if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
  const double floor_abs = (double)(floor_rel * block_max<T>(w, r));
  const double tol2 = (double)tol_rel * (double)tol_rel;

  int sweep = 0;
  bool converged = (r <= 1);
  for (; sweep < max_sweeps && !converged; ++sweep) {
    for (int rd = 0; rd < N - 1; ++rd) {
      for (int pi = blockIdx.x; pi < npairs; pi += nblk) {
        int p = rr_player(pi, rd, N), q = rr_player(N - 1 - pi, rd, N);
        if (p > q) { int t_ = p; p = q; q = t_; }
        if (q >= r) continue;
        cplx<T>* xp = X + (size_t)p * ldx;
        cplx<T>* xq = X + (size_t)q * ldx;
        T a = T(0), b = T(0), gr = T(0), gi = T(0);
        auto dots = [&](cplx<T> x, cplx<T> y) {
          a = fma(x.x, x.x, fma(x.y, x.y, a));
          b = fma(y.x, y.x, fma(y.y, y.y, b));
          gr = fma(x.x, y.x, fma(x.y, y.y, gr));     // x conj(y)
          gi = fma(x.y, y.x, fma(-x.x, y.y, gi));
        };
        cplx<T>* tp = Ut + (size_t)p * r;
        cplx<T>* tq = Ut + (size_t)q * r;
        cplx<T> rx[E], ry[E];
        // short rows: U's two rows are fetched together with X's, so that their
        // L2 round trip runs under the reduction and the rotation parameters
        constexpr int EU = E <= 2 ? E : 1;
        cplx<T> ux[EU], uy[EU];
        if (E <= 2 && uregs) {
#pragma unroll
          for (int e = 0; e < EU; ++e) {
            const int j = tid + OSJ_NT * e;
            ux[e] = j < r ? ldcg(&tp[j]) : czero<T>();
            uy[e] = j < r ? ldcg(&tq[j]) : czero<T>();
          }
        }
        if (regs) {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int j = tid + OSJ_NT * e;
            rx[e] = j < c ? ldcg(&xp[j]) : czero<T>();
            ry[e] = j < c ? ldcg(&xq[j]) : czero<T>();
          }
#pragma unroll
          for (int e = 0; e < E; ++e)
            if (OSJ_NT * e < c) dots(rx[e], ry[e]);
        } else {
#pragma unroll 4
          for (int j = tid; j < c; j += OSJ_NT) dots(ldcg(&xp[j]), ldcg(&xq[j]));
        }
        osj_reduce4<T>(a, b, gr, gi, part);
        if (tid < 32) {
          double cs, sn, ur, ui;
          bool unresolved = false;
          const bool on = osj_rotation((double)a, (double)b, (double)gr, (double)gi, tol2, floor_abs, cs, sn, ur, ui,
                                       &unresolved) && (T)sn != T(0);
          if (tid == 0) {
            s_rot.on = on;
            if (unresolved) atomicAdd(&ctl->active[sweep], 1);
            if (on) {
              s_rot.c = (T)cs; s_rot.s = (T)sn;
              s_rot.sur = (T)(sn * ur); s_rot.sui = (T)(sn * ui);
              s_rot.cur = (T)(cs * ur); s_rot.cui = (T)(cs * ui);
              atomicAdd(&ctl->active[sweep], 1);
            }
          }
        }
        __syncthreads();
        if (!s_rot.on) continue;
        const T cs = s_rot.c, sn = s_rot.s, sur = s_rot.sur, sui = s_rot.sui, cur = s_rot.cur, cui = s_rot.cui;
        if (regs) {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int j = tid + OSJ_NT * e;
            if (j < c) {
              osj_rotate<T>(rx[e], ry[e], cs, sn, sur, sui, cur, cui);
              stcg(&xp[j], rx[e]);
              stcg(&xq[j], ry[e]);
            }
          }
        } else {
#pragma unroll 4
          for (int j = tid; j < c; j += OSJ_NT) {
            cplx<T> x = ldcg(&xp[j]), y = ldcg(&xq[j]);
            osj_rotate<T>(x, y, cs, sn, sur, sui, cur, cui);
            stcg(&xp[j], x);
            stcg(&xq[j], y);
          }
        }
        // U <- U J: the conjugate phase
        if (E <= 2 && uregs) {
#pragma unroll
          for (int e = 0; e < EU; ++e) {
            const int j = tid + OSJ_NT * e;
            if (j < r) {
              osj_rotate<T>(ux[e], uy[e], cs, sn, sur, -sui, cur, -cui);
              stcg(&tp[j], ux[e]);
              stcg(&tq[j], uy[e]);
            }
          }
        } else if (uregs) {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int j = tid + OSJ_NT * e;
            rx[e] = j < r ? ldcg(&tp[j]) : czero<T>();
            ry[e] = j < r ? ldcg(&tq[j]) : czero<T>();
          }
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int j = tid + OSJ_NT * e;
            if (j < r) {
              osj_rotate<T>(rx[e], ry[e], cs, sn, sur, -sui, cur, -cui);
              stcg(&tp[j], rx[e]);
              stcg(&tq[j], ry[e]);
            }
          }
        } else {
#pragma unroll 4
          for (int j = tid; j < r; j += OSJ_NT) {
            cplx<T> x = ldcg(&tp[j]), y = ldcg(&tq[j]);
            osj_rotate<T>(x, y, cs, sn, sur, -sui, cur, -cui);
            stcg(&tp[j], x);
            stcg(&tq[j], y);
          }
        }
      }
      if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
    }
    if (atomicAdd(&ctl->active[sweep], 0) == 0) converged = true;
  }
  norms();
  if (gtid == 0) {
    ctl->g.sweeps = sweep;
    ctl->g.status = converged ? 0 : 1;
  }
}

// ---------------------------------------------------------------------------
// Row Jacobi in FP32 on blocks of RB rows, the precision form's Rayleigh-Ritz
// solve: the same rotations as above, row pair by row pair (no Gram of the block,
// so the relative accuracy of the row method stays), but a CTA holds two blocks
// in registers and rotates all RB^2 pairs between them (at the first round of a
// sweep the pairs inside each block too) before it writes them back.
// Why: at 2048 rows the pair form reads and writes X and U once per round,
// 128 MB at 13 TB/s of L2, and passes a grid barrier for each; blocks of four
// divide both by four. RB pairs are rotated at a time: their 4 RB sums are
// reduced together and one lane each forms the rotations, in FP32 (c and 1 / |g|
// by one Newton step, so c^2 + s^2 and |u| are 1 to FP32 rounding; the solve's
// vectors are orthonormalised in FP64 afterwards). U takes the recorded
// rotations in one pass. Rows of up to 256 E columns.
// Measured in the precision form, pair kernel -> this one: 2048 rows 166 -> 82 ms,
// 512 rows 18.5 -> 5.3 ms.
// ---------------------------------------------------------------------------
constexpr int QJ_NT = 256;

__device__ __forceinline__ float qj_rsqrt(float x) {
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.0f), y);
}

// osj_rotation in FP32.
__device__ __forceinline__ bool qj_rotation(float a, float b, float gr, float gi, float tol2, float floor_abs, float& c,
                                            float& s, float& ur, float& ui) {
  const int er = (__float_as_int(gr) >> 23) & 0xFF, ei = (__float_as_int(gi) >> 23) & 0xFF;
  const int e = max(er, ei) - 127;
  if (e <= -126 || e >= 126) return false;
  const float sc = __int_as_float((127 - e) << 23);
  const float x = gr * sc, y = gi * sc;
  const float g2 = fmaf(x, x, y * y);
  if (!(g2 > tol2 * ((a * sc) * (b * sc)))) return false;
  const float inv = qj_rsqrt(g2);
  if (!(g2 * inv * __int_as_float((127 + e) << 23) > floor_abs)) return false;
  const float z = ((b - a) * sc) * (0.5f * inv), az = fabsf(z);
  if (!(az < 3e38f)) return false;
  float t = az > 1e18f ? 0.5f / az : 1.0f / (az + sqrtf(fmaf(az, az, 1.0f)));
  if (z < 0.0f) t = -t;
  c = qj_rsqrt(fmaf(t, t, 1.0f));
  s = t * c;
  ur = x * inv;
  ui = y * inv;
  return s != 0.0f;
}

template <int RB, int E>
__global__ void __launch_bounds__(QJ_NT) quad_jacobi_kernel(float2* X, int r, int c, int ldx, float2* Ut, float* w, OSCtl* ctl,
                                                            int max_sweeps, float tol_rel, float floor_rel,
                                                            long long timeout_ns) {
  constexpr int NV = 4 * RB;                       // sums of one step
  constexpr int NSTEP = 2 * RB - 1;                // steps of a round: RB - 1 inside the blocks, RB across
  __shared__ float part[QJ_NT / 32][NV];
  __shared__ float4 s_rot[NSTEP][RB];              // c, s, u; s = 0: no rotation
  __shared__ int s_any;
  const int nb = (r + RB - 1) / RB, N = nb + (nb & 1), npairs = N / 2;
  const unsigned nblk = gridDim.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t gtid = (size_t)blockIdx.x * QJ_NT + tid, gthreads = (size_t)nblk * QJ_NT;
  if (max_sweeps > 64) max_sweeps = 64;

  for (size_t e = gtid; e < (size_t)r * r; e += gthreads) {
    const size_t i = e / r, j = e % r;
    stcg(&Ut[e], make_float2(i == j ? 1.0f : 0.0f, 0.0f));
  }
  auto norms = [&]() {
    for (long i = gtid >> 5; i < r; i += (long)(gthreads >> 5)) {
      float s = 0.0f;
      for (int j = lane; j < c; j += 32) {
        const float2 x = ldcg(&X[(size_t)i * ldx + j]);
        s = fmaf(x.x, x.x, fmaf(x.y, x.y, s));
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) __stcg(&w[i], s);
    }
  };
  norms();
  if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
  const float floor_abs = floor_rel * block_max<float>(w, r);
  const float tol2 = tol_rel * tol_rel;

  int sweep = 0;
  bool converged = (r <= 1);
  for (; sweep < max_sweeps && !converged; ++sweep) {
    const int nround = N > 1 ? N - 1 : 1;
    for (int rd = 0; rd < nround; ++rd) {
      for (int pi = blockIdx.x; pi < npairs; pi += nblk) {
        const int P = rr_player(pi, rd, N), Q = rr_player(N - 1 - pi, rd, N);
        if ((P >= nb || Q >= nb) && rd > 0) continue;      // sits out (its own rows are rotated at the first round)
        auto row_of = [&](int i) -> int {                  // block row i of the CTA; r if there is none
          const int g = i < RB ? P * RB + i : Q * RB + (i - RB);
          return g < r ? g : r;
        };
        float2 x[2 * RB][E];
        auto load = [&](const float2* M, int ld, int n) {
#pragma unroll
          for (int i = 0; i < 2 * RB; ++i) {
            const int g = row_of(i);
#pragma unroll
            for (int e = 0; e < E; ++e) {
              const int j = tid + QJ_NT * e;
              x[i][e] = g < r && j < n ? ldcg(&M[(size_t)g * ld + j]) : make_float2(0.f, 0.f);
            }
          }
        };
        auto store = [&](float2* M, int ld, int n) {
#pragma unroll
          for (int i = 0; i < 2 * RB; ++i) {
            const int g = row_of(i);
#pragma unroll
            for (int e = 0; e < E; ++e) {
              const int j = tid + QJ_NT * e;
              if (g < r && j < n) stcg(&M[(size_t)g * ld + j], x[i][e]);
            }
          }
        };
        load(X, ldx, c);
        if (tid == 0) s_any = 0;
        // step k < RB - 1: pairs (i, i ^ (k + 1)) inside both blocks; then
        // (i, RB + (i ^ (k - RB + 1))) across. Pair q's rows: first, second
#pragma unroll
        for (int k = 0; k < NSTEP; ++k) {
          constexpr int H = RB / 2;
          if (k < RB - 1 && rd > 0) continue;
          auto first = [&](int q) -> int {
            if (k >= RB - 1) return q;
            const int blk = q / H, n = q % H, m = k + 1;   // the n-th i with i < i ^ m
            int cnt = 0, f = 0;
#pragma unroll
            for (int i = 0; i < RB; ++i)
              if (i < (i ^ m)) { if (cnt == n) f = i; ++cnt; }
            return blk * RB + f;
          };
          auto second = [&](int q) -> int { return k >= RB - 1 ? RB + (q ^ (k - RB + 1)) : first(q) ^ (k + 1); };
          float v[NV];
#pragma unroll
          for (int q = 0; q < RB; ++q) {
            float a = 0.f, b = 0.f, gr = 0.f, gi = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) {
              const float2 p0 = x[first(q)][e], p1 = x[second(q)][e];
              a = fmaf(p0.x, p0.x, fmaf(p0.y, p0.y, a));
              b = fmaf(p1.x, p1.x, fmaf(p1.y, p1.y, b));
              gr = fmaf(p0.x, p1.x, fmaf(p0.y, p1.y, gr));
              gi = fmaf(p0.y, p1.x, fmaf(-p0.x, p1.y, gi));
            }
            v[4 * q] = a; v[4 * q + 1] = b; v[4 * q + 2] = gr; v[4 * q + 3] = gi;
          }
          // halves: after the step of width h a lane keeps the values whose bit agrees with its own
          int o = 16;
#pragma unroll
          for (int h = NV / 2; h >= 1; h >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < h; ++i) {
              const float keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
              v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          constexpr int LPV = 32 / NV;      // lanes that share a value now
#pragma unroll
          for (int h = LPV / 2; h >= 1; h >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], h);
          if ((lane % LPV) == 0) part[warp][lane / LPV] = v[0];
          __syncthreads();
          if (warp == 0) {
            float t = 0.f;
#pragma unroll
            for (int u = 0; u < QJ_NT / 32; ++u) t += part[u][lane % NV];
            const int q = lane % RB;
            const float a = __shfl_sync(0xffffffffu, t, 4 * q), b = __shfl_sync(0xffffffffu, t, 4 * q + 1);
            const float gr = __shfl_sync(0xffffffffu, t, 4 * q + 2), gi = __shfl_sync(0xffffffffu, t, 4 * q + 3);
            float cs = 1.f, sn = 0.f, ur = 1.f, ui = 0.f;
            const bool on = qj_rotation(a, b, gr, gi, tol2, floor_abs, cs, sn, ur, ui);
            if (lane < RB) s_rot[k][q] = on ? make_float4(cs, sn, ur, ui) : make_float4(1.f, 0.f, 1.f, 0.f);
            const unsigned any = __ballot_sync(0xffffffffu, on && lane < RB);
            if (lane == 0 && any) {
              s_any = 1;
              atomicAdd(&ctl->active[sweep], __popc(any));
            }
          }
          __syncthreads();
#pragma unroll
          for (int q = 0; q < RB; ++q) {
            const float4 R = s_rot[k][q];
            if (R.y == 0.f) continue;
            const float sur = R.y * R.z, sui = R.y * R.w, cur = R.x * R.z, cui = R.x * R.w;
#pragma unroll
            for (int e = 0; e < E; ++e) osj_rotate<float>(x[first(q)][e], x[second(q)][e], R.x, R.y, sur, sui, cur, cui);
          }
        }
        if (s_any) {
          store(X, ldx, c);
          load(Ut, r, r);
#pragma unroll
          for (int k = 0; k < NSTEP; ++k) {
            constexpr int H = RB / 2;
            if (k < RB - 1 && rd > 0) continue;
            auto first = [&](int q) -> int {
              if (k >= RB - 1) return q;
              const int blk = q / H, n = q % H, m = k + 1;
              int cnt = 0, f = 0;
#pragma unroll
              for (int i = 0; i < RB; ++i)
                if (i < (i ^ m)) { if (cnt == n) f = i; ++cnt; }
              return blk * RB + f;
            };
            auto second = [&](int q) -> int { return k >= RB - 1 ? RB + (q ^ (k - RB + 1)) : first(q) ^ (k + 1); };
#pragma unroll
            for (int q = 0; q < RB; ++q) {
              const float4 R = s_rot[k][q];
              if (R.y == 0.f) continue;
              const float sur = R.y * R.z, sui = -R.y * R.w, cur = R.x * R.z, cui = -R.x * R.w;   // U <- U J: the conjugate phase
#pragma unroll
              for (int e = 0; e < E; ++e) osj_rotate<float>(x[first(q)][e], x[second(q)][e], R.x, R.y, sur, sui, cur, cui);
            }
          }
          store(Ut, r, r);
        }
        __syncthreads();            // s_any and s_rot are free for the next pair
      }
      if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
    }
    if (atomicAdd(&ctl->active[sweep], 0) == 0) converged = true;
  }
  norms();
  if (gtid == 0) {
    ctl->g.sweeps = sweep;
    ctl->g.status = converged ? 0 : 1;
  }
}

// ---------------------------------------------------------------------------
// LQ preconditioning of the complex128 SVD (Drmac & Veselic, SIAM J. Matrix
// Anal. Appl. 29 (2008), without pivoting): with A = L Q (L r x r lower
// triangular, Q with orthonormal rows) the row Jacobi runs on R = L^H instead
// of A. R = W (Sigma U^H) gives A = U Sigma (W^H Q): U from the normalised rows
// of the result, the rows Sigma W^H Q from the accumulated W and the
// reflectors of Q, both orthonormal to FP64 rounding.
// Why: the rows of L^H are graded and nearly orthogonal, so the solve needs
// about half the sweeps (23 -> 11 on a 256 x 256 block of decaying spectrum),
// and each of them rotates rows of r instead of c elements.
// lq_kernel: one cooperative launch, one barrier per Householder step; every
// CTA forms the step's norm itself while it takes its first row's dot product
// (one reduction for both), so nothing waits for a broadcast.
// Truncated SVD, row Jacobi on A -> with the LQ step: 128 x 128 13.7 -> 8.5 ms,
// 256 x 256 52 -> 21 ms, 577 x 600 260 -> 119 ms, 1024 x 1024 1244 -> 539 ms.
//
// FP32 start. From kPreMinRows rows on, the FP32 solver first runs on fl32(R)
// (scaled to a largest entry near 1), and the FP64 solve starts from W^H R and W,
// W the FP32 left factor made orthonormal to FP64 rounding: with E = (I - W^H W)
// / 2, W (I + E + 3/2 E^2 + 5/2 E^3) is off by 35/8 E^4. E is the drift of the FP32
// rotations and grows with the rows: 2-norm 1.1e-4 at 1024, 4.3e-4 at 4096, where
// 35/8 E^4 left rows of X off by 2.8e-13. The host therefore reads its largest row
// sum (a bound of the 2-norm, 2.5 to 3.5 times as large here) while the products
// above run, and above kStartOnce takes one Newton-Schulz step more, above
// kStartMax no start at all. The FP64 unit runs at 1/64 of the FP32 rate, so its sweeps are what the solve costs, and
// five (the last of them quiet) remain of eleven; it stops by the same test as
// without the start. Truncated SVD, LQ only -> with the start: 64 x 64 4.1 -> 2.8 ms,
// 256 x 256 21.5 -> 17.5 ms, 577 x 600 116 -> 88 ms, 1024 x 1024 542 -> 350 ms;
// 768 x 1024 with a spectrum over three decades 253 -> 115 ms (FP64 solve 57, FP32
// 21, products 16, LQ step and rows 21).
// ---------------------------------------------------------------------------
// *out = the largest biased exponent among the real and imaginary parts of a
// matrix of n entries (zeroed before the launch).
__global__ void __launch_bounds__(256) max_exp_kernel(const double2* __restrict__ R, size_t n, int* __restrict__ out) {
  int v = 0;
  for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (size_t)gridDim.x * 256) {
    const double2 x = R[e];
    v = max(v, max((int)((__double_as_longlong(x.x) >> 52) & 0x7FF), (int)((__double_as_longlong(x.y) >> 52) & 0x7FF)));
  }
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0 && v > 0) atomicMax(out, v);
}

// out = fl32(R 2^-e), e the exponent found above (an all-zero R stays zero).
__global__ void __launch_bounds__(256) scale_fp32_kernel(const double2* __restrict__ R, size_t n, const int* __restrict__ ex,
                                                         float2* __restrict__ out) {
  const int be = *ex;
  const double sc = be > 0 && be < 2046 ? __longlong_as_double((long long)(2046 - be) << 52) : 1.0;   // 2^(1023 - be)
  for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (size_t)gridDim.x * 256) {
    const double2 x = R[e];
    out[e] = make_float2((float)(x.x * sc), (float)(x.y * sc));
  }
}

// G (m x m, a Gram matrix) <- E = (I - G) / 2, one CTA per row; *out = the largest
// row sum of |E_ij| (FP32 bits, zeroed before the launch; a NaN stays one).
__global__ void __launch_bounds__(256) half_defect_kernel(double2* __restrict__ G, int m, unsigned int* __restrict__ out) {
  __shared__ float part[8];
  const int i = blockIdx.x;
  float sum = 0.0f;
  for (int j = threadIdx.x; j < m; j += 256) {
    double2 g = G[(size_t)i * m + j];
    g.x = 0.5 * ((i == j ? 1.0 : 0.0) - g.x);
    g.y = -0.5 * g.y;
    G[(size_t)i * m + j] = g;
    const float x = (float)g.x, y = (float)g.y;
    sum += sqrtf(fmaf(x, x, y * y));
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) sum += part[q];
    atomicMax(out, __float_as_uint(fabsf(sum)));
  }
}

// out (c x r) = in (r x c)^T in FP64, 32 x 32 tiles through shared memory.
template <typename S>
__global__ void transpose_kernel(const S* __restrict__ in, int r, int c, double2* __restrict__ out) {
  __shared__ double2 tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int i = by + yy, j = bx + threadIdx.x;
    if (i < r && j < c) { const S v = in[(size_t)i * c + j]; tile[yy][threadIdx.x] = make_double2((double)v.x, (double)v.y); }
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int j = bx + yy, i = by + threadIdx.x;
    if (j < c && i < r) out[(size_t)j * r + i] = tile[threadIdx.x][yy];
  }
}

// 1 / sqrt(x) for a normal positive x.
__device__ __forceinline__ double lq_rsqrt(double x) {
  const int e = ((int)(__double_as_longlong(x) >> 52) - 1023) & ~1;
  return osj_rsqrt(x * osj_pow2(-e)) * osj_pow2(-(e >> 1));
}

// Z (r x c) <- X with row j's reflector z_j left in columns j .. c - 1 (its
// first entry in zd[j]), H_j = I - f_j z_j^H z_j; Y (r x r) <- L^H. r <= c.
// A row whose squared norm is not above 1e-300 (less than that, denormal squares
// cost it its accuracy) counts as zero; ctl->g.sweeps receives the largest biased exponent
// of such a squared norm plus 1, 0 if there was none but exact zeros, and the caller refuses
// the factorisation when that is not negligible beside the whole (rows below ~1e-150).
template <int E>
__global__ void __launch_bounds__(OSJ_NT) lq_kernel(const double2* __restrict__ X, int ldx, int r, int c, double2* Z,
                                                    double2* Y, double* f, double2* zd, OSCtl* ctl,
                                                    long long timeout_ns) {
  __shared__ double part[4][4];
  __shared__ double2 s_coef, s_z0;
  __shared__ double s_f;
  const unsigned nblk = gridDim.x;
  const int tid = threadIdx.x;
  const bool regs = c <= OSJ_NT * E;
  int dropped = 0;
  for (int i = blockIdx.x; i < r; i += nblk) {
    for (int k = tid; k < c; k += OSJ_NT) stcg(&Z[(size_t)i * c + k], X[(size_t)i * ldx + k]);
    for (int k = tid; k < r; k += OSJ_NT) stcg(&Y[(size_t)i * r + k], czero<double>());
  }
  if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
  for (int j = 0; j < r; ++j) {
    const double2* zj = Z + (size_t)j * c;
    int i = blockIdx.x;                       // this CTA's first row below the pivot
    if (i <= j) i += ((j - i) / (int)nblk + 1) * (int)nblk;
    if (i < r || blockIdx.x == 0) {
      const int e0 = j / OSJ_NT;              // columns below j are final
      double2 z[E], a[E];
      double n2 = 0.0, dr = 0.0, di = 0.0, none = 0.0;
      double2* row = Z + (size_t)(i < r ? i : j) * c;
      auto dot = [&](double2 av, double2 zv) {     // sum a conj(z)
        dr = fma(av.x, zv.x, fma(av.y, zv.y, dr));
        di = fma(av.y, zv.x, fma(-av.x, zv.y, di));
      };
      if (regs) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int k = tid + OSJ_NT * e;
          const bool in = k >= j && k < c;
          z[e] = in ? ldcg(&zj[k]) : czero<double>();
          a[e] = in && i < r ? ldcg(&row[k]) : czero<double>();
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (e >= e0 && OSJ_NT * e < c) {
            n2 = fma(z[e].x, z[e].x, fma(z[e].y, z[e].y, n2));
            dot(a[e], z[e]);
          }
      } else {
        for (int k = tid + OSJ_NT * e0; k < c; k += OSJ_NT) {
          if (k < j) continue;
          const double2 zv = ldcg(&zj[k]);
          n2 = fma(zv.x, zv.x, fma(zv.y, zv.y, n2));
          if (i < r) dot(ldcg(&row[k]), zv);
        }
      }
      osj_reduce4<double>(n2, dr, di, none, part);
      if (tid < 32) {
        // z = x + phase(x_0) |x| e_0, f = 1 / (|x| (|x| + |x_0|)), L_jj = -phase |x|
        const double2 x0 = ldcg(&zj[j]);
        double2 ph = make_double2(1.0, 0.0);
        double nrm = 0.0, fj = 0.0;
        if (n2 > 1e-300) {
          const double inv = lq_rsqrt(n2);
          nrm = n2 * inv;
          const double ux = x0.x * inv, uy = x0.y * inv;      // x_0 / |x|
          const double u2 = fma(ux, ux, uy * uy);
          double au = 0.0;
          if (u2 > 1e-300) {
            const double iu = lq_rsqrt(u2);
            au = u2 * iu;
            ph = make_double2(ux * iu, uy * iu);
          }
          fj = inv * lq_rsqrt(1.0 + au);                       // f = (fj)^2
          fj = fj * fj;
        } else if (n2 > 0.0) {
          dropped = max(dropped, (int)(__double_as_longlong(n2) >> 52) + 1);
        }
        const double2 ps = make_double2(ph.x * nrm, ph.y * nrm);
        const double2 z0 = cadd<double>(x0, ps);
        const double2 aij = i < r ? ldcg(&row[j]) : czero<double>();
        double2 d = cadd<double>(make_double2(dr, di), cmul<double>(aij, cconj<double>(ps)));
        if (tid == 0) {
          s_coef = cscale<double>(d, fj);
          s_z0 = z0;
          s_f = fj;
          if (blockIdx.x == 0) {
            f[j] = fj;
            stcg(&zd[j], z0);
            stcg(&Y[(size_t)j * r + j], make_double2(-ps.x, ps.y));   // conj(L_jj)
          }
        }
      }
      __syncthreads();
      const double2 z0 = s_z0;
      const double fj = s_f;
      for (;;) {
        if (i >= r) break;
        const double2 co = s_coef;
        auto update = [&](double2 av, double2 zv, int k) {
          const double2 v = make_double2(fma(co.y, zv.y, fma(-co.x, zv.x, av.x)), fma(-co.y, zv.x, fma(-co.x, zv.y, av.y)));
          if (k == j) stcg(&Y[(size_t)j * r + i], cconj<double>(v));
          else stcg(&row[k], v);
        };
        if (regs) {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int k = tid + OSJ_NT * e;
            if (k >= j && k < c) update(a[e], k == j ? z0 : z[e], k);
          }
        } else {
          for (int k = tid + OSJ_NT * e0; k < c; k += OSJ_NT)
            if (k >= j) update(ldcg(&row[k]), k == j ? z0 : ldcg(&zj[k]), k);
        }
        i += nblk;
        if (i >= r) break;
        row = Z + (size_t)i * c;
        dr = di = 0.0;
        if (regs) {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const int k = tid + OSJ_NT * e;
            a[e] = k >= j && k < c ? ldcg(&row[k]) : czero<double>();
          }
#pragma unroll
          for (int e = 0; e < E; ++e)
            if (e >= e0 && OSJ_NT * e < c) dot(a[e], tid + OSJ_NT * e == j ? z0 : z[e]);
        } else {
          for (int k = tid + OSJ_NT * e0; k < c; k += OSJ_NT)
            if (k >= j) dot(ldcg(&row[k]), k == j ? z0 : ldcg(&zj[k]));
        }
        double n_ = 0.0, m_ = 0.0;
        osj_reduce4<double>(dr, di, n_, m_, part);
        if (tid == 0) s_coef = make_double2(fj * dr, fj * di);
        __syncthreads();
      }
    }
    if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
  }
  if (blockIdx.x == 0 && tid == 0) ctl->g.sweeps = dropped;
}

// Row j of the factorisation from the Jacobi result (Y rows Sigma U^H, Wt row j
// = column j of W, w = sigma^2): X row j = sigma_j w_j^H Q = sigma_j [w_j^H 0]
// H_{r-1} .. H_0, and Uc row j = conj(column j of U) (may be Y). One CTA per row; the row
// stays in registers while the reflectors stream past (each is read ahead
// while the previous one's dot product is reduced).
template <int E>
__global__ void __launch_bounds__(OSJ_NT) lq_apply_kernel(const double2* __restrict__ Z, int r, int c,
                                                          const double* __restrict__ f, const double2* __restrict__ zd,
                                                          const double2* __restrict__ Wt, const double2* Y, double2* Uc,
                                                          const double* __restrict__ w, double2* __restrict__ X, int ldx) {
  __shared__ double part[2][2][4];
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool regs = c <= OSJ_NT * E;
  double2* xr = X + (size_t)j * ldx;
  // sum of (re, im) over the CTA in every thread: one barrier, scratch in turn
  auto reduce2 = [&](double re, double im, int buf) -> double2 {
    const bool hi = lane & 16;
    double v = hi ? im : re;
    v += __shfl_xor_sync(0xffffffffu, hi ? re : im, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 15) == 0) part[buf][lane >> 4][warp] = v;
    __syncthreads();
    v = part[buf][(lane >> 2) & 1][lane & 3];
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    return make_double2(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 4));
  };
  const double sig = sqrt(w[j]);
  if (regs) {
    double2 y[E], z[E], zn[E];
    auto load = [&](int k, double2* dst) {
      const double2* zk = Z + (size_t)k * c;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int l = tid + OSJ_NT * e;
        dst[e] = l > k && l < c ? zk[l] : (l == k ? zd[k] : czero<double>());
      }
    };
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int l = tid + OSJ_NT * e;
      y[e] = l < r ? cconj<double>(Wt[(size_t)j * r + l]) : czero<double>();
    }
    load(r - 1, zn);
    for (int k = r - 1; k >= 0; --k) {
      const double fk = f[k];
#pragma unroll
      for (int e = 0; e < E; ++e) z[e] = zn[e];
      if (k > 0) load(k - 1, zn);
      const int e0 = k / OSJ_NT;
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (e >= e0 && OSJ_NT * e < c) {
          re = fma(y[e].x, z[e].x, fma(y[e].y, z[e].y, re));
          im = fma(y[e].y, z[e].x, fma(-y[e].x, z[e].y, im));
        }
      const double2 d = reduce2(re, im, k & 1);
      const double cr = fk * d.x, ci = fk * d.y;
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (e >= e0 && OSJ_NT * e < c) {
          y[e].x = fma(ci, z[e].y, fma(-cr, z[e].x, y[e].x));
          y[e].y = fma(-ci, z[e].x, fma(-cr, z[e].y, y[e].y));
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int l = tid + OSJ_NT * e;
      if (l < c) xr[l] = cscale<double>(y[e], sig);
    }
  } else {
    for (int l = tid; l < c; l += OSJ_NT) xr[l] = l < r ? cconj<double>(Wt[(size_t)j * r + l]) : czero<double>();
    for (int k = r - 1; k >= 0; --k) {
      const double2* zk = Z + (size_t)k * c;
      const double2 z0 = zd[k];
      const double fk = f[k];
      double re = 0.0, im = 0.0;
      const int l0 = tid + OSJ_NT * (k / OSJ_NT);
      for (int l = l0; l < c; l += OSJ_NT) {
        if (l < k) continue;
        const double2 zv = l == k ? z0 : zk[l], yv = xr[l];
        re = fma(yv.x, zv.x, fma(yv.y, zv.y, re));
        im = fma(yv.y, zv.x, fma(-yv.x, zv.y, im));
      }
      const double2 d = reduce2(re, im, k & 1);
      const double cr = fk * d.x, ci = fk * d.y;
      for (int l = l0; l < c; l += OSJ_NT) {
        if (l < k) continue;
        const double2 zv = l == k ? z0 : zk[l], yv = xr[l];
        xr[l] = make_double2(fma(ci, zv.y, fma(-cr, zv.x, yv.x)), fma(-ci, zv.x, fma(-cr, zv.y, yv.y)));
      }
    }
    for (int l = tid; l < c; l += OSJ_NT) xr[l] = cscale<double>(xr[l], sig);
  }
  const double inv = sig > 0.0 ? 1.0 / sig : 0.0;
  for (int l = tid; l < r; l += OSJ_NT) {
    double2 v = cscale<double>(Y[(size_t)j * r + l], inv);
    if (!(sig > 0.0)) v = make_double2(l == j ? 1.0 : 0.0, 0.0);
    Uc[(size_t)j * r + l] = v;
  }
}

// ---------------------------------------------------------------------------
// Gather of selected rows: element (j, i) = f_j * op(src[perm[j] * lds + i]),
// i < len, j < k (k = min(info->k, k_cap)), op = conj if conj_ else identity;
// written to out[j * ldo + i] (transpose == 0) or out[i * ldo + j] (== 1).
// f_j by mode: 0 -> 1; 1 -> 1/sqrt(lam2_j); 2 -> sqrt(lam2_j / kept);
//              3 -> 1/sqrt(kept).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void gather_rows_kernel(const cplx<T>* __restrict__ src, int lds, int len, const int* __restrict__ perm,
                                  const double* __restrict__ lam2, const SelectInfo* __restrict__ info, int k_cap,
                                  int transpose, int conj_, int mode, cplx<T>* __restrict__ out, int ldo) {
  const int k = info->k < k_cap ? info->k : k_cap;
  const size_t total = (size_t)len * k;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    int i, j;
    if (transpose) { i = (int)(e / k); j = (int)(e % k); }
    else { j = (int)(e / len); i = (int)(e % len); }
    double f = 1.0;
    if (mode == 1) f = lam2[j] > 0.0 ? 1.0 / sqrt(lam2[j]) : 0.0;
    else if (mode == 2) f = info->kept > 0.0 ? sqrt(lam2[j] / info->kept) : 0.0;
    else if (mode == 3) f = info->inv_sqrt_kept;
    cplx<T> v = src[(size_t)perm[j] * lds + i];
    if (conj_) v = cconj<T>(v);
    v = cscale<T>(v, (T)f);
    if (transpose) out[(size_t)i * ldo + j] = v;
    else out[(size_t)j * ldo + i] = v;
  }
}

// out (c x r) = in (r x c)^H, 32 x 32 tiles through shared memory.
template <typename T>
__global__ void conj_transpose_kernel(const cplx<T>* __restrict__ in, int r, int c, int ldi, cplx<T>* __restrict__ out, int ldo) {
  __shared__ cplx<T> tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int i = by + yy, j = bx + threadIdx.x;
    if (i < r && j < c) tile[yy][threadIdx.x] = in[(size_t)i * ldi + j];
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int j = bx + yy, i = by + threadIdx.x;
    if (j < c && i < r) out[(size_t)j * ldo + i] = cconj<T>(tile[threadIdx.x][yy]);
  }
}


// Shared-memory address of a generic pointer (for cp.async).
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---------------------------------------------------------------------------
// Block one-sided Jacobi SVD (row blocks of JB rows; a pair holds 2 JB rows).
// Same contract as onesided_jacobi_kernel: X (r x c) <- U^H X with rows
// mutually orthogonal, Ut = U^T, w = squared row norms.
//
// Rows are grouped in nb = ceil(r / JB) blocks, paired round-robin (bye for
// odd nb). For the pair (P, Q) of a round:
//   G = X_PQ X_PQ^H (2JB x 2JB), diagonalised as G = J diag J^H by an in-CTA
//   cyclic Jacobi, then X_PQ <- J^H X_PQ and Ut_PQ <- J^T Ut_PQ;
// this orthogonalises all 2JB rows of the pair at once (block Jacobi; the
// rotations are applied as small dense products, so each round streams X once
// instead of once per row pair). A pair is left alone when every cross entry
// satisfies |G_ij| <= max(tol sqrt(G_ii G_jj), floor * max_k G_kk).
// One round = three phases of a persistent cooperative launch:
//   G: Gram partials over column chunks (pair x chunk work items)   barrier
//   E: per pair, sum partials, skip test, inner Jacobi -> J         barrier
//   A: per pair x chunk, apply J to X and to Ut                     barrier
// ---------------------------------------------------------------------------
constexpr int JB = 16;           // rows per block
constexpr int JP = 2 * JB;       // rows per pair
constexpr int JCW = 512;         // columns per Gram / apply work item

// Integer state of the block Jacobi for r rows: the per-pair rotate flags of
// a round, then for each block the round stamp of its last rotation, then
// for each block a flag "own rows not known orthogonal", then for each block
// pair (P, Q) the stamp of the round that last found it orthogonal (N x N,
// N = the padded block count).
__host__ __device__ constexpr size_t bj_state_ints(int r) {
  return (size_t)(((r + JB - 1) / JB + (((r + JB - 1) / JB) & 1)) / 2) +
         2 * (size_t)((r + JB - 1) / JB + (((r + JB - 1) / JB) & 1)) +
         (size_t)((r + JB - 1) / JB + (((r + JB - 1) / JB) & 1)) * (size_t)((r + JB - 1) / JB + (((r + JB - 1) / JB) & 1));
}


// In-CTA cyclic Jacobi of the pair's 2JB x 2JB Gram in the working precision
// TI (FP64 arithmetic runs at 1/64 of the FP32 rate on this part, so nothing
// here is promoted). The tolerance is set at the rounding level of TI and the
// sweep count is capped, because J is re-derived in every outer round and an
// inexact inner solve only costs outer sweeps. The rounding drift of the
// accumulated rotations is removed afterwards by bj_polish_unitary.
template <typename TI> __device__ __forceinline__ TI rsqrt_fast(TI x);
template <> __device__ __forceinline__ float rsqrt_fast<float>(float x) { return rsqrtf(x); }
template <> __device__ __forceinline__ double rsqrt_fast<double>(double x) { return rsqrt(x); }

// Rotation parameters of the 2 x 2 Hermitian block [[a, g], [conj g, b]]
// (rows p, q of G): c, s real and u = g / |g|, chosen so that the rotation
// R = [[c, s], [-s conj(u), c conj(u)]] zeroes the off-diagonal entry of
// R^H G R; s = 0 when |g|^2 <= max(tol^2 |a b|, floor^2) (square-root free
// skip test).
template <typename TI>
__device__ __forceinline__ void bj_rot_params(const cplx<TI>* G, int p, int q, TI tol2, TI flo2, TI& c_, TI& s_,
                                              TI& ur, TI& ui) {
  constexpr int LD = JP + 1;
  const TI a_ = G[p * LD + p].x, b_ = G[q * LD + q].x;
  const TI gx = G[p * LD + q].x, gy = G[p * LD + q].y;
  const TI g2 = gx * gx + gy * gy;
  c_ = TI(1); s_ = TI(0); ur = TI(1); ui = TI(0);
  if (g2 > fmax(tol2 * fabs(a_ * b_), flo2) && g2 > TI(0)) {
    const TI inv = rsqrt_fast<TI>(g2);                              // 1 / |g|
    const TI zeta = (b_ - a_) * TI(0.5) * inv;
    TI t;
    if constexpr (sizeof(TI) == 4) {
      // FP32: approximate divide and square root (a few ulp); any t gives
      // an exactly normalised (c, s) up to rsqrt rounding, and an inexact
      // angle only leaves a slightly larger off-diagonal for later rounds
      const float az = fabsf(zeta);
      if (az > 1.0f / eps_of<float>::value) t = __fdividef(0.5f, zeta);
      else {
        const float q = fmaf(zeta, zeta, 1.0f);
        t = __fdividef(1.0f, az + q * rsqrtf(q));
        if (!(zeta >= 0.0f)) t = -t;
      }
    } else {
      if (fabs(zeta) > TI(1) / eps_of<TI>::value) t = TI(0.5) / zeta;
      else t = (zeta >= TI(0) ? TI(1) : TI(-1)) / (fabs(zeta) + sqrt(TI(1) + zeta * zeta));
    }
    c_ = rsqrt_fast<TI>(TI(1) + t * t);
    s_ = t * c_;
    ur = gx * inv; ui = gy * inv;
  }
}

// Pair solve: one round of the cyclic parallel Jacobi as 2 x 2 block updates: the round's
// JP/2 disjoint rotations partition the indices into pairs, so the JP x JP
// matrix splits into (JP/2)^2 blocks B_ab = G[{p_a, q_a}][{p_b, q_b}], each
// updated on its own as B_ab <- R_a^H B_ab R_b. Thread (a, b) derives both
// rotations from the old matrix and writes the new block into the other
// buffer, so a round needs one barrier instead of three (parameters, column
// pass, row pass). Requires blockDim.x == (JP/2)^2.
//
// In-CTA cyclic Jacobi of the pair's 2JB x 2JB Gram in the working precision
// TI (FP64 arithmetic runs at 1/64 of the FP32 rate on this part, so nothing
// here is promoted). The tolerance is set at the rounding level of TI and the
// sweep count is capped, because J is re-derived in every outer round and an
// inexact inner solve only costs outer sweeps. The rounding drift of the
// accumulated rotations is removed afterwards by bj_polish_unitary. G0 holds
// the input; G1 is scratch of the same shape; both are overwritten. Returns
// 1 when a sweep found nothing left to rotate (the result is diagonal to the
// tolerance), 0 when max_sweeps ran out first. order[rd * NR + a] holds pair a of
// round rd (bj_fill_order): six player indices modulo JP - 1 were a third of a
// round's instructions.
__device__ __forceinline__ void bj_fill_order(uchar2* order) {
  for (int e = threadIdx.x; e < (JP - 1) * (JP / 2); e += blockDim.x) {
    const int rd = e / (JP / 2), a = e % (JP / 2);
    const int p = rr_player(a, rd, JP), q = rr_player(JP - 1 - a, rd, JP);
    order[e] = make_uchar2((unsigned char)min(p, q), (unsigned char)max(p, q));
  }
}

template <typename TI>
__device__ int bj_inner_eig(cplx<TI>* G0, cplx<TI>* G1, cplx<TI>* Vs /*JP x JP, ld JP+1*/, double tol,
                             double floor_abs, int max_sweeps, const uchar2* order) {
  constexpr int LD = JP + 1, NR = JP / 2;
  static_assert(NR * NR == 256, "one thread per 2 x 2 block");
  const int tid = threadIdx.x, ia = tid / NR, ib = tid % NR;
  for (int e = tid; e < JP * JP; e += blockDim.x) {
    const int i = e / JP, j = e % JP;
    Vs[i * LD + j] = mk<TI>(i == j ? TI(1) : TI(0), TI(0));
  }
  __syncthreads();
  const TI tol2 = (TI)(tol * tol), flo2 = (TI)(floor_abs * floor_abs);
  cplx<TI>* Gc = G0;
  cplx<TI>* Gn = G1;
  for (int sw = 0; sw < max_sweeps; ++sw) {
    int any = 0;
    for (int rd = 0; rd < JP - 1; ++rd) {
      const uchar2 oa = order[rd * NR + ia], ob = order[rd * NR + ib];
      const int pa = oa.x, qa = oa.y, pb = ob.x, qb = ob.y;
      // lane l of every warp derives rotation l % NR; threads fetch the two
      // they need by shuffle (no block barrier for a shared table)
      TI cl, sl, url, uil;
      {
        const int lr = (tid & 31) % NR;
        const uchar2 ol = order[rd * NR + lr];
        bj_rot_params<TI>(Gc, ol.x, ol.y, tol2, flo2, cl, sl, url, uil);
      }
      // every warp derives the same table from the same matrix, so a round
      // with nothing to rotate is skipped by all threads alike (no writes,
      // no barrier); the function therefore ends with a barrier, so that no
      // thread reuses G0 / G1 (the caller's polish scratch) while another is
      // still reading the last skipped rounds' table
      if (!__any_sync(0xffffffffu, sl != TI(0))) continue;
      const TI ca = __shfl_sync(0xffffffffu, cl, ia), sa = __shfl_sync(0xffffffffu, sl, ia);
      const TI ura = __shfl_sync(0xffffffffu, url, ia), uia = __shfl_sync(0xffffffffu, uil, ia);
      const TI cb = __shfl_sync(0xffffffffu, cl, ib), sb = __shfl_sync(0xffffffffu, sl, ib);
      const TI urb = __shfl_sync(0xffffffffu, url, ib), uib = __shfl_sync(0xffffffffu, uil, ib);
      cplx<TI> b00 = Gc[pa * LD + pb], b01 = Gc[pa * LD + qb], b10 = Gc[qa * LD + pb], b11 = Gc[qa * LD + qb];
      if (sb != TI(0)) {        // columns: [x y] <- [c x - s conj(u) y, s x + c conj(u) y]
        const cplx<TI> ub = mk<TI>(urb, -uib);
        const cplx<TI> y0 = cmul<TI>(ub, b01), y1 = cmul<TI>(ub, b11);
        b01 = mk<TI>(sb * b00.x + cb * y0.x, sb * b00.y + cb * y0.y);
        b00 = mk<TI>(cb * b00.x - sb * y0.x, cb * b00.y - sb * y0.y);
        b11 = mk<TI>(sb * b10.x + cb * y1.x, sb * b10.y + cb * y1.y);
        b10 = mk<TI>(cb * b10.x - sb * y1.x, cb * b10.y - sb * y1.y);
      }
      if (sa != TI(0)) {        // rows: [x; y] <- [c x - s u y; s x + c u y]
        const cplx<TI> ua = mk<TI>(ura, uia);
        const cplx<TI> y0 = cmul<TI>(ua, b10), y1 = cmul<TI>(ua, b11);
        b10 = mk<TI>(sa * b00.x + ca * y0.x, sa * b00.y + ca * y0.y);
        b00 = mk<TI>(ca * b00.x - sa * y0.x, ca * b00.y - sa * y0.y);
        b11 = mk<TI>(sa * b01.x + ca * y1.x, sa * b01.y + ca * y1.y);
        b01 = mk<TI>(ca * b01.x - sa * y1.x, ca * b01.y - sa * y1.y);
        if (ia == ib) {         // the rotated diagonal block: exact zeros, real diagonal
          b01 = czero<TI>(); b10 = czero<TI>(); b00.y = TI(0); b11.y = TI(0);
        }
      }
      Gn[pa * LD + pb] = b00; Gn[pa * LD + qb] = b01; Gn[qa * LD + pb] = b10; Gn[qa * LD + qb] = b11;
      if (sb != TI(0)) {        // V <- V R_b on rows ia and ia + NR
        const cplx<TI> ub = mk<TI>(urb, -uib);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          cplx<TI>* R = Vs + (ia + h * NR) * LD;
          const cplx<TI> x = R[pb], uy = cmul<TI>(ub, R[qb]);
          R[pb] = mk<TI>(cb * x.x - sb * uy.x, cb * x.y - sb * uy.y);
          R[qb] = mk<TI>(sb * x.x + cb * uy.x, sb * x.y + cb * uy.y);
        }
      }
      any |= __syncthreads_or(sb != TI(0));
      cplx<TI>* t_ = Gc; Gc = Gn; Gn = t_;
    }
    if (!any) {
      __syncthreads();   // rounds skipped without a barrier: no thread may leave while others still read Gc
      return 1;
    }
  }
  __syncthreads();
  return 0;
}

// One Newton-Schulz step V <- V (3 I - V^H V) / 2 (Higham, Functions of
// Matrices, Sec. 8.3): for V = Q (I + E) with small Hermitian E the result is
// unitary to O(|E|^2) + rounding, so the per-pair rotation J carries no
// accumulated drift into the U of the SVD. S and W are JP x JP scratch
// (leading dimension JP+1) in shared memory.
template <typename TI>
__device__ void bj_polish_unitary(cplx<TI>* Vs, cplx<TI>* S, cplx<TI>* W) {
  constexpr int LD = JP + 1;
  const int tid = threadIdx.x;
  for (int e = tid; e < JP * JP; e += blockDim.x) {      // S = V^H V
    const int i = e / JP, j = e % JP;
    cplx<TI> acc = czero<TI>();
#pragma unroll 8
    for (int k = 0; k < JP; ++k) cfma<TI>(acc, cconj<TI>(Vs[k * LD + i]), Vs[k * LD + j]);
    S[i * LD + j] = acc;
  }
  __syncthreads();
  for (int e = tid; e < JP * JP; e += blockDim.x) {      // W = V (3 I - S) / 2
    const int i = e / JP, j = e % JP;
    cplx<TI> acc = czero<TI>();
#pragma unroll 8
    for (int k = 0; k < JP; ++k) {
      cplx<TI> m = cscale<TI>(S[k * LD + j], TI(-0.5));
      if (k == j) m.x += TI(1.5);
      cfma<TI>(acc, Vs[i * LD + k], m);
    }
    W[i * LD + j] = acc;
  }
  __syncthreads();
  for (int e = tid; e < JP * JP; e += blockDim.x) Vs[(e / JP) * LD + (e % JP)] = W[(e / JP) * LD + (e % JP)];
  __syncthreads();
}

// Newton-Schulz steps until V is unitary to rounding: each step first forms
// S = V^H V and tests max |S - I| <= tol, then applies the step; the loop
// ends after the first step taken from a state that passed the test (leaving
// a defect of about tol^2 plus rounding) or after max_steps steps. The
// iteration converges for |S - I| < 1 (Higham, Functions of Matrices, 8.3).
template <typename TI>
__device__ void bj_polish_unitary_to(cplx<TI>* Vs, cplx<TI>* S, cplx<TI>* W, TI tol, int max_steps) {
  constexpr int LD = JP + 1;
  const int tid = threadIdx.x;
  for (int it = 0; it < max_steps; ++it) {
    int bad = 0;
    for (int e = tid; e < JP * JP; e += blockDim.x) {
      const int i = e / JP, j = e % JP;
      cplx<TI> acc = czero<TI>();
#pragma unroll 8
      for (int k = 0; k < JP; ++k) cfma<TI>(acc, cconj<TI>(Vs[k * LD + i]), Vs[k * LD + j]);
      S[i * LD + j] = acc;
      if (!(fabs(acc.x - (i == j ? TI(1) : TI(0))) <= tol && fabs(acc.y) <= tol)) bad = 1;
    }
    const int any_bad = __syncthreads_or(bad);
    for (int e = tid; e < JP * JP; e += blockDim.x) {
      const int i = e / JP, j = e % JP;
      cplx<TI> acc = czero<TI>();
#pragma unroll 8
      for (int k = 0; k < JP; ++k) {
        cplx<TI> m = cscale<TI>(S[k * LD + j], TI(-0.5));
        if (k == j) m.x += TI(1.5);
        cfma<TI>(acc, Vs[i * LD + k], m);
      }
      W[i * LD + j] = acc;
    }
    __syncthreads();
    for (int e = tid; e < JP * JP; e += blockDim.x) Vs[(e / JP) * LD + (e % JP)] = W[(e / JP) * LD + (e % JP)];
    __syncthreads();
    if (!any_bad) break;
  }
}

// Asynchronous global -> shared copies (cp.async): BYTES per copy, the tail
// beyond src_bytes zero-filled, so rows past the matrix read as zeros.
template <int BYTES>
__device__ __forceinline__ void cp_async_zfill(void* dst, const void* src, int src_bytes) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" :: "r"(smem_addr(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" :: "r"(smem_addr(dst)), "l"(src), "n"(BYTES),
                 "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" :: "n"(N) : "memory"); }

template <typename T> struct BJ_GW { static constexpr int value = sizeof(T) == 4 ? 128 : 64; };
constexpr int BJ_NB = 4;   // phase-G staging ring: sub-chunks in flight per CTA
__device__ __forceinline__ bool tid_is_zero() { return threadIdx.x == 0; }

// Dynamic shared memory of block_jacobi_kernel<T>: the larger of the phase-G
// staging ring and the phase E/A matrices, then the cross-block reduction
// buffer.
template <typename T>
constexpr int block_jacobi_smem_bytes() {
  constexpr int GW = BJ_GW<T>::value;
  constexpr int TS = GW + 1;
  constexpr int RING = BJ_NB * JP * TS * (int)sizeof(cplx<T>);
  constexpr int GV = 3 * JP * (JP + 1) * (int)sizeof(cplx<T>);
  constexpr int RED = 8 * 16 * 40 * (int)sizeof(T);
  return (RING > GV ? RING : GV) + RED;
}

template <typename T>
__global__ void __launch_bounds__(256) block_jacobi_kernel(cplx<T>* X, int r, int c, int ldx, cplx<T>* Ut, T* w,
                                                            cplx<T>* Gpart, cplx<T>* Jbuf, int* act_flag, OSCtl* ctl,
                                                            int max_sweeps, T tol_rel, T floor_rel, long long timeout_ns) {
  constexpr int LD = JP + 1;
  // Dynamic shared memory (block_jacobi_smem_bytes<T>()): a ring of BJ_NB
  // phase-G tiles of JP rows x TS columns; phases E and A reuse the same
  // bytes for the pair Gram Gs, the rotation Vs and the polish scratch; the
  // cross-block reduction buffer follows.
  constexpr int GW = BJ_GW<T>::value;                    // staged columns in phase G
  // padded row stride: GW + 1 puts the rows that one warp reads at the same
  // column in distinct banks (8-byte rows at 2 x 129 words, 16-byte at 4 x 65)
  constexpr int TS = GW + 1;
  constexpr int RING = BJ_NB * JP * TS * (int)sizeof(cplx<T>), GV = 3 * JP * (JP + 1) * (int)sizeof(cplx<T>);
  extern __shared__ __align__(128) unsigned char smraw[];
  cplx<T>* ring = reinterpret_cast<cplx<T>*>(smraw);
  T* red = reinterpret_cast<T*>(smraw + (RING > GV ? RING : GV));   // [8][16][40]
  cplx<T>* Gs = reinterpret_cast<cplx<T>*>(smraw);     // phase E: the pair Gram; phase A: J^H or J^T
  cplx<T>* Vs = Gs + JP * LD;

  cplx<T>* Js = reinterpret_cast<cplx<T>*>(red);        // phase A: J^H or J^T (ld JP+1)
  __shared__ uchar2 s_order[(JP - 1) * (JP / 2)];
  bj_fill_order(s_order);                               // read after the first grid barrier
  const int nb = (r + JB - 1) / JB, N = nb + (nb & 1), npairs = N / 2;
  const int nch = (c + JCW - 1) / JCW, nchu = (r + JCW - 1) / JCW;
  const unsigned nblk = gridDim.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwb = blockDim.x >> 5;
  const long gwarp = (long)blockIdx.x * nwb + warp, nwarps = (long)nblk * nwb;
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + tid, gthreads = (size_t)nblk * blockDim.x;
  if (max_sweeps > 64) max_sweeps = 64;

  for (size_t e = gtid; e < (size_t)r * r; e += gthreads) {
    const size_t i = e / r, j = e % r;
    stcg(&Ut[e], mk<T>(i == j ? T(1) : T(0), T(0)));
  }
  // round stamps (round g = sweep (N - 1) + rd + 1): a pair whose blocks are
  // both unchanged since the round that found it orthogonal stays orthogonal,
  // so cross-only sweeps skip its Gram and its test
  int* last_mod = act_flag + npairs;
  int* wdirty = last_mod + N;   // 1: the block's own rows were left by an inexact pair solve
  int* last_clean = wdirty + N;
  // every block starts unverified: its first pair forms the full Gram
  for (size_t e = gtid; e < 2 * (size_t)N + (size_t)N * N; e += gthreads) last_mod[e] = (e >= (size_t)N && e < 2 * (size_t)N) ? 1 : 0;
  for (long i = gwarp; i < r; i += nwarps) {
    T s = T(0);
    for (int j = lane; j < c; j += 32) { const cplx<T> x = ldcg(&X[(size_t)i * ldx + j]); s += x.x * x.x + x.y * x.y; }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) w[i] = s;
  }
  if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
  const T floor_abs = floor_rel * block_max<T>(w, r);

  int sweep = 0;
  bool converged = (r <= 1);
  bool verify = false;   // this sweep forms full Grams to confirm convergence
  for (; sweep < max_sweeps && !converged; ++sweep) {
    // a verification pass is one round of full Grams (two when a block sits
    // out round 0): every round pairs each block once, so it re-checks the
    // rows inside every block; the cross blocks were just found orthogonal
    const int nrounds = verify ? ((nb & 1) ? 2 : 1) : N - 1;
    for (int rd = 0; rd < nrounds; ++rd) {
      unsigned long long tph = (blockIdx.x == 0 && tid == 0) ? global_timer_ns() : 0ull;
      // ---- phase G: partial Grams of each pair over column chunks ---------
      // A pair with an unverified block (every block until its first pair
      // solve, and after an inexact one) and every pair of a verification
      // pass form the full 2JB x 2JB Gram. Otherwise each block's own rows
      // are mutually orthogonal (a pair solve orthogonalises all its rows,
      // and a block's rows change only when it is paired), so only the
      // JB x JB cross block X_P X_Q^H and the row norms are formed; the
      // diagonal blocks are taken as diagonal.
      const bool full_gram = verify;
      const long nitems = (long)npairs * nch;
      // The CTA's work is the sequence of (item, sub-chunk) stages of its
      // items; a ring of BJ_NB tiles keeps BJ_NB stages in flight (cp.async,
      // no register staging), refilling each tile as soon as its stage has
      // been consumed, across item boundaries.
      const int gstamp = sweep * (N - 1) + rd + 1;
      auto pair_dirty = [&](int P_, int Q_) -> bool {
        return __ldcg(&last_clean[(size_t)P_ * N + Q_]) <= max(__ldcg(&last_mod[P_]), __ldcg(&last_mod[Q_]));
      };
      // a pair forms its full Gram in full sweeps, and whenever one of its
      // blocks was left by a pair solve that ran out of inner sweeps (its own
      // rows are then not known to be orthogonal, which cross-only Grams
      // assume)
      auto pair_full = [&](int P_, int Q_) -> bool {
        return full_gram || __ldcg(&wdirty[P_]) != 0 || __ldcg(&wdirty[Q_]) != 0;
      };
      auto item_valid = [&](long it) -> bool {
        const int pi_ = (int)(it / nch);
        int P_ = rr_player(pi_, rd, N), Q_ = rr_player(N - 1 - pi_, rd, N);
        if (P_ > Q_) { const int t_ = P_; P_ = Q_; Q_ = t_; }
        return Q_ < nb && (pair_full(P_, Q_) || pair_dirty(P_, Q_));
      };
      long p_item = blockIdx.x;   // producer cursor
      int p_sub = 0;
      while (p_item < nitems && !item_valid(p_item)) p_item += nblk;
      auto issue = [&](int buf) {
        if (p_item >= nitems) return;
        const int pi_ = (int)(p_item / nch), ch_ = (int)(p_item % nch);
        int P_ = rr_player(pi_, rd, N), Q_ = rr_player(N - 1 - pi_, rd, N);
        if (P_ > Q_) { const int t_ = P_; P_ = Q_; Q_ = t_; }
        const int c0_ = ch_ * JCW, c1_ = min(c, c0_ + JCW), k0 = c0_ + p_sub * GW;
        cplx<T>* tile = ring + buf * JP * TS;
        constexpr int PER = JP * GW / 256;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const int e_ = tid + 256 * u, i = e_ / GW, k = e_ % GW;
          const int row = (i < JB ? P_ * JB + i : Q_ * JB + (i - JB));
          const bool in = row < r && k0 + k < c1_;
          cp_async_zfill<(int)sizeof(cplx<T>)>(&tile[i * TS + k], in ? (const void*)&X[(size_t)row * ldx + k0 + k]
                                                                     : (const void*)X,
                                               in ? (int)sizeof(cplx<T>) : 0);
        }
        if (++p_sub == (c1_ - c0_ + GW - 1) / GW) {
          p_sub = 0;
          do { p_item += nblk; } while (p_item < nitems && !item_valid(p_item));
        }
      };
#pragma unroll
      for (int q = 0; q < BJ_NB; ++q) { issue(q); cp_async_commit(); }
      int jseq = 0;               // consumer position in the stage sequence
      for (long item = blockIdx.x; item < nitems; item += nblk) {
        if (!item_valid(item)) continue;
        const int pi = (int)(item / nch), ch = (int)(item % nch);
        int P = rr_player(pi, rd, N), Q = rr_player(N - 1 - pi, rd, N);
        if (P > Q) { int t_ = P; P = Q; Q = t_; }
        const bool fullp = pair_full(P, Q);
        // full: thread (ti, tj) owns G[ti + 16a][tj + 16b];
        // cross: k-slice g = tid / 16 (k = g, g + 16, ...), member m = tid % 16
        // owns C[4 mi + i][4 mj + j], mi = m / 4, mj = m % 4, and the norms of
        // rows 4 mi + mj and JB + 4 mj + mi (each row's norm on one member)
        const int ti = tid >> 4, tj = tid & 15;
        const int mi = (tid & 15) >> 2, mj = tid & 3;
        cplx<T> acc[4][4];
        T nrmP = T(0), nrmQ = T(0);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = czero<T>();
        const int c0 = ch * JCW, c1 = min(c, c0 + JCW);
        const int nsub = (c1 - c0 + GW - 1) / GW;
        for (int s = 0; s < nsub; ++s, ++jseq) {
          cp_async_wait<BJ_NB - 1>();
          __syncthreads();
          const cplx<T>* tile = ring + (jseq % BJ_NB) * JP * TS;
          const int kn = min(GW, c1 - (c0 + s * GW));
          if (fullp) {
#pragma unroll 4
            for (int k = 0; k < kn; ++k) {
              const cplx<T> a0 = tile[ti * TS + k], a1 = tile[(ti + 16) * TS + k];
              const cplx<T> b0 = cconj<T>(tile[tj * TS + k]), b1 = cconj<T>(tile[(tj + 16) * TS + k]);
              cfma<T>(acc[0][0], a0, b0); cfma<T>(acc[0][1], a0, b1);
              cfma<T>(acc[1][0], a1, b0); cfma<T>(acc[1][1], a1, b1);
            }
          } else {
            for (int k = (tid >> 4); k < kn; k += 16) {
              cplx<T> av[4], bv[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                av[i] = tile[(4 * mi + i) * TS + k];
                bv[i] = tile[(JB + 4 * mj + i) * TS + k];
              }
              const cplx<T> np_ = tile[(4 * mi + mj) * TS + k], nq_ = tile[(JB + 4 * mj + mi) * TS + k];
              nrmP += np_.x * np_.x + np_.y * np_.y;
              nrmQ += nq_.x * nq_.x + nq_.y * nq_.y;
#pragma unroll
              for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) cfma<T>(acc[i][j], av[i], cconj<T>(bv[j]));
            }
          }
          __syncthreads();                      // the tile is free: refill it
          issue(jseq % BJ_NB);
          cp_async_commit();
        }
        cplx<T>* Gp = Gpart + ((size_t)pi * nch + ch) * JP * JP;
        if (fullp) {
#pragma unroll
          for (int a_ = 0; a_ < 2; ++a_)
#pragma unroll
            for (int b_ = 0; b_ < 2; ++b_) stcg(&Gp[(ti + 16 * a_) * JP + tj + 16 * b_], acc[a_][b_]);
        } else {
          // reduce the 16 k-slices in a fixed order (deterministic, so the
          // same input always gives the same factorisation): half-warp pairs
          // by shuffle, then the 8 warps through shared memory
          constexpr int NV = 34;                                 // 16 complex + 2 norms
          T vals[NV];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) { vals[2 * (4 * i + j)] = acc[i][j].x; vals[2 * (4 * i + j) + 1] = acc[i][j].y; }
          vals[32] = nrmP;
          vals[33] = nrmQ;
#pragma unroll
          for (int v = 0; v < NV; ++v) vals[v] += __shfl_xor_sync(0xffffffffu, vals[v], 16);
          if ((tid & 31) < 16) {
#pragma unroll
            for (int v = 0; v < NV; ++v) red[((tid >> 5) * 16 + (tid & 15)) * NV + v] = vals[v];
          }
          __syncthreads();
          for (int e = tid; e < JP * JP; e += blockDim.x) {
            const int i = e / JP, j = e % JP;
            cplx<T> v = czero<T>();
            if ((i < JB) != (j < JB)) {
              const bool upper = i < JB;
              const int pi_ = upper ? i : j, qj = upper ? j - JB : i - JB;
              const int m = (pi_ >> 2) * 4 + (qj >> 2), o = 2 * (4 * (pi_ & 3) + (qj & 3));
              T sr = T(0), si = T(0);
              for (int w = 0; w < 8; ++w) { sr += red[(w * 16 + m) * NV + o]; si += red[(w * 16 + m) * NV + o + 1]; }
              v = mk<T>(sr, upper ? si : -si);
            } else if (i == j) {
              T s = T(0);
              if (i < JB) { for (int w = 0; w < 8; ++w) s += red[(w * 16 + i) * NV + 32]; }        // member i
              else {
                const int q = i - JB, m = 4 * (q & 3) + (q >> 2);                                   // 4 mi + mj, mj = q / 4, mi = q % 4
                for (int w = 0; w < 8; ++w) s += red[(w * 16 + m) * NV + 33];
              }
              v = mk<T>(s, T(0));
            }
            stcg(&Gp[e], v);
          }
          __syncthreads();
        }
      }
      cp_async_wait<0>();
      __syncthreads();
      if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
      if (blockIdx.x == 0 && tid == 0) { unsigned long long t2 = global_timer_ns(); ctl->phase_ns[0] += t2 - tph; tph = t2; }
      // ---- phase E: per pair, reduce, test, inner eigen-solve ---------------
      for (long pi = blockIdx.x; pi < npairs; pi += nblk) {
        int P = rr_player((int)pi, rd, N), Q = rr_player(N - 1 - (int)pi, rd, N);
        if (P > Q) { int t_ = P; P = Q; Q = t_; }
        const bool full_e = Q < nb && pair_full(P, Q);
        if (Q >= nb || (!full_e && !pair_dirty(P, Q))) { if (tid == 0) act_flag[pi] = 0; continue; }
        // FP64 only where its rounding matters (an FP64 warp instruction holds
        // its SM partition for 64 clocks): sums of zero-padded loads and maxima
        // taken in FP64 cost 18 of the 56 us of a pair solve
        for (int e = tid; e < JP * JP; e += blockDim.x) {
          const cplx<T>* src = Gpart + (size_t)pi * nch * JP * JP + e;
          if (nch == 1) {
            const cplx<T> v = ldcg(src);
            Gs[(e / JP) * LD + (e % JP)] = mk<T>(v.x + T(0), v.y + T(0));
            continue;
          }
          double sr = 0.0, si = 0.0;
          for (int ch0 = 0; ch0 < nch; ch0 += 8) {   // up to eight loads in flight
            cplx<T> v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = ch0 + u < nch ? ldcg(src + (size_t)(ch0 + u) * JP * JP) : czero<T>();
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (ch0 + u < nch) { sr += (double)v[u].x; si += (double)v[u].y; }
          }
          Gs[(e / JP) * LD + (e % JP)] = mk<T>((T)sr, (T)si);
        }
        __shared__ int s_need;
        if (tid == 0) s_need = 0;
        __syncthreads();
        // the test: |G_ij| > max(tol sqrt(G_ii G_jj), floor); the floor is
        // the larger of the global one (initial largest row) and floor_rel
        // times the pair's largest row norm, the level to which a rotation
        // derived from this pair's Gram resolves its entries (rows gain norm
        // as the sweeps concentrate it, so the initial scale alone can sit
        // below what the pair solve can reach and the sweeps never end)
        static_assert(JP == 32, "one diagonal entry per lane");
        const T dl = Gs[lane * LD + lane].x;
        T gpm = fmax(T(0), dl);
        for (int o = 16; o > 0; o >>= 1) gpm = fmax(gpm, __shfl_xor_sync(0xffffffffu, gpm, o));
        const double pfloor = fmax((double)floor_abs, (double)floor_rel * (double)gpm);
        for (int e = tid; e < (full_e ? JP * JP : JB * JB); e += blockDim.x) {
          const int i = full_e ? e / JP : e / JB, j = full_e ? e % JP : JB + e % JB;
          if (i >= j) continue;
          const double aij = hypot(Gs[i * LD + j].x, Gs[i * LD + j].y);
          const double thr = fmax((double)tol_rel * sqrt(fabs(Gs[i * LD + i].x * Gs[j * LD + j].x)), pfloor);
          if (aij > thr) s_need = 1;
        }
        __syncthreads();
        const int need = s_need;
        if (need) {
          // Near convergence the pair Gram is diag + a small cross block: one
          // first-order step J = I + E, E_ij = G_ij / (G_jj - G_ii) on the
          // cross entries (E skew-Hermitian), made unitary to rounding by
          // Newton-Schulz steps (J^H J = I - E^2 to start), leaves O(|E|^2)
          // off-diagonals -- quadratic like the Jacobi endgame but with O(1)
          // sequential steps. Those O(|E|^2) residues also land inside the
          // blocks, which cross-only sweeps assume orthogonal, so the step is
          // taken only where they stay below the convergence test: every
          // cross |E_ij| < 0.01 (so |J^H J - I| <= 512 * 1e-4 and the polish
          // converges in a few steps) and JB max|E|^2 max_k G_kk <=
          // max(tol min_k G_kk, floor); outside full-Gram sweeps; else the
          // inner solve.
          int first_order = 0, exact = 1;
          if (!full_e) {
            T gmn = dl;
            for (int o = 16; o > 0; o >>= 1) gmn = fmin(gmn, __shfl_xor_sync(0xffffffffu, gmn, o));
            const double gmin = (double)gmn, gmax = (double)gpm;
            const double e2lim = gmax > 0.0 ? fmax((double)tol_rel * gmin, pfloor) / (JB * gmax) : 0.0;
            int ok = 1;
            for (int e = tid; e < JB * JB; e += blockDim.x) {
              const int i = e / JB, j = JB + e % JB;
              const double gap = fabs((double)Gs[j * LD + j].x - (double)Gs[i * LD + i].x);
              const double gx = (double)Gs[i * LD + j].x, gy = (double)Gs[i * LD + j].y;
              const double g2 = gx * gx + gy * gy;
              if (!(g2 < 1e-4 * gap * gap && g2 <= e2lim * gap * gap)) ok = 0;
            }
            first_order = __syncthreads_and(ok);
          }
          if (first_order) {
            for (int e = tid; e < JP * JP; e += blockDim.x) {
              const int i = e / JP, j = e % JP;
              cplx<T> v = mk<T>(i == j ? T(1) : T(0), T(0));
              if (i < JB && j >= JB) {                 // E_ij = G_ij / (G_jj - G_ii)
                const T den = Gs[j * LD + j].x - Gs[i * LD + i].x;
                v = cscale<T>(Gs[i * LD + j], T(1) / den);
              } else if (i >= JB && j < JB) {          // E_ij = -conj(E_ji)
                const T den = Gs[i * LD + i].x - Gs[j * LD + j].x;
                v = cscale<T>(cconj<T>(Gs[j * LD + i]), T(-1) / den);
              }
              Vs[i * LD + j] = v;
            }
            __syncthreads();
            bj_polish_unitary_to<T>(Vs, Gs, Vs + JP * LD, T(8.0 * eps_of<T>::value * 5.66), 6);
          } else {
            exact = bj_inner_eig<T>(Gs, Vs + JP * LD, Vs, 4.0 * (double)eps_of<T>::value * sqrt((double)JP),
                                    32.0 * (double)eps_of<T>::value * (double)gpm, 3, s_order);
            // FP32: remove the rounding drift of J (FP64 rotations keep it at 1e-16)
            if constexpr (sizeof(T) == 4) bj_polish_unitary<T>(Vs, Gs, Vs + JP * LD);
          }
          for (int e = tid; e < JP * JP; e += blockDim.x) stcg(&Jbuf[(size_t)pi * JP * JP + e], Vs[(e / JP) * LD + (e % JP)]);
          if (tid == 0) {
            act_flag[pi] = 1;
            last_mod[P] = gstamp;
            last_mod[Q] = gstamp;
            wdirty[P] = wdirty[Q] = exact ? 0 : 1;
            atomicAdd(&ctl->active[sweep], 1);
          }
        } else if (tid == 0) {
          act_flag[pi] = 0;
          last_clean[(size_t)P * N + Q] = gstamp;
          if (full_e) wdirty[P] = wdirty[Q] = 0;   // verified by the full Gram
        }
        __syncthreads();
      }
      if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
      if (blockIdx.x == 0 && tid == 0) { unsigned long long t2 = global_timer_ns(); ctl->phase_ns[1] += t2 - tph; tph = t2; }
      // ---- phase A: X_PQ <- J^H X_PQ, Ut_PQ <- J^T Ut_PQ -----------------
      // Work items are (active pair, 512-column chunk of X or of Ut), staged
      // GW columns at a time through the same cp.async ring as phase G. Each
      // thread forms a 4 x (GW/32) complex micro-tile of the product: rows
      // 4 ty .. 4 ty + 3 (J from shared memory, a broadcast within the warp)
      // by columns tx + 32 b (consecutive across the warp), eight shared
      // loads per 16 (FP32) complex multiply-adds.
      {
        constexpr int NBC = GW / 32;                         // columns per thread
        const long aitems = (long)npairs * (nch + nchu);
        auto a_valid = [&](long it) -> bool { return __ldcg(&act_flag[(int)(it / (nch + nchu))]) != 0; };
        long p_item = blockIdx.x;
        int p_sub = 0;
        while (p_item < aitems && !a_valid(p_item)) p_item += nblk;
        auto issue = [&](int buf) {
          if (p_item >= aitems) return;
          const int pi_ = (int)(p_item / (nch + nchu)), ch_ = (int)(p_item % (nch + nchu));
          int P_ = rr_player(pi_, rd, N), Q_ = rr_player(N - 1 - pi_, rd, N);
          if (P_ > Q_) { const int t_ = P_; P_ = Q_; Q_ = t_; }
          const bool onU_ = ch_ >= nch;
          const cplx<T>* M_ = onU_ ? Ut : X;
          const int ld_ = onU_ ? r : ldx, ncol_ = onU_ ? r : c;
          const int c0_ = (onU_ ? ch_ - nch : ch_) * JCW, c1_ = min(ncol_, c0_ + JCW), k0 = c0_ + p_sub * GW;
          cplx<T>* tile = ring + buf * JP * TS;
          constexpr int PER = JP * GW / 256;
#pragma unroll
          for (int u = 0; u < PER; ++u) {
            const int e_ = tid + 256 * u, i = e_ / GW, k = e_ % GW;
            const int row = (i < JB ? P_ * JB + i : Q_ * JB + (i - JB));
            const bool in = row < r && k0 + k < c1_;
            cp_async_zfill<(int)sizeof(cplx<T>)>(&tile[i * TS + k],
                                                 in ? (const void*)&M_[(size_t)row * ld_ + k0 + k] : (const void*)M_,
                                                 in ? (int)sizeof(cplx<T>) : 0);
          }
          if (++p_sub == (c1_ - c0_ + GW - 1) / GW) {
            p_sub = 0;
            do { p_item += nblk; } while (p_item < aitems && !a_valid(p_item));
          }
        };
#pragma unroll
        for (int q = 0; q < BJ_NB; ++q) { issue(q); cp_async_commit(); }
        const int ty = tid >> 5, tx = tid & 31;
        int jseq = 0;
        // J of the CTA's next item is loaded into registers while the current
        // item computes, so its L2 round trip is off the critical path
        constexpr int JPER = JP * JP / 256;
        cplx<T> jpre[JPER];
        auto load_j = [&](long it) {
          const int pi_ = (int)(it / (nch + nchu));
#pragma unroll
          for (int u = 0; u < JPER; ++u) {
            const int e = tid + 256 * u, i = e / JP, k = e % JP;
            jpre[u] = ldcg(&Jbuf[(size_t)pi_ * JP * JP + k * JP + i]);
          }
        };
        long item = blockIdx.x;
        while (item < aitems && !a_valid(item)) item += nblk;
        if (item < aitems) load_j(item);
        for (; item < aitems;) {
          const int pi = (int)(item / (nch + nchu)), ch = (int)(item % (nch + nchu));
          int P = rr_player(pi, rd, N), Q = rr_player(N - 1 - pi, rd, N);
          if (P > Q) { int t_ = P; P = Q; Q = t_; }
          const bool onU = ch >= nch;
          cplx<T>* M = onU ? Ut : X;
          const int ld = onU ? r : ldx, ncol = onU ? r : c;
          const int c0 = (onU ? ch - nch : ch) * JCW, c1 = min(ncol, c0 + JCW);
#pragma unroll
          for (int u = 0; u < JPER; ++u) {
            // Js[i][k] = (J^H)[i][k] = conj(J[k][i])  or  (J^T)[i][k] = J[k][i]
            const int e = tid + 256 * u, i = e / JP, k = e % JP;
            Js[i * LD + k] = onU ? jpre[u] : cconj<T>(jpre[u]);
          }
          long next = item + nblk;
          while (next < aitems && !a_valid(next)) next += nblk;
          if (next < aitems) load_j(next);
          int orow[4];
#pragma unroll
          for (int a_ = 0; a_ < 4; ++a_) {
            const int i = 4 * ty + a_;
            orow[a_] = i < JB ? P * JB + i : Q * JB + (i - JB);
          }
          const int nsub = (c1 - c0 + GW - 1) / GW;
          for (int s = 0; s < nsub; ++s, ++jseq) {
            cp_async_wait<BJ_NB - 1>();
            __syncthreads();                    // the stage (and, first time, Js) is visible
            const cplx<T>* tile = ring + (jseq % BJ_NB) * JP * TS;
            cplx<T> acc[4][NBC];
#pragma unroll
            for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
              for (int b_ = 0; b_ < NBC; ++b_) acc[a_][b_] = czero<T>();
#pragma unroll 4
            for (int k = 0; k < JP; ++k) {
              cplx<T> jv[4], xv[NBC];
#pragma unroll
              for (int a_ = 0; a_ < 4; ++a_) jv[a_] = Js[(4 * ty + a_) * LD + k];
#pragma unroll
              for (int b_ = 0; b_ < NBC; ++b_) xv[b_] = tile[k * TS + tx + 32 * b_];
#pragma unroll
              for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
                for (int b_ = 0; b_ < NBC; ++b_) cfma<T>(acc[a_][b_], jv[a_], xv[b_]);
            }
            const int k0 = c0 + s * GW;
#pragma unroll
            for (int a_ = 0; a_ < 4; ++a_) {
              if (orow[a_] >= r) continue;
#pragma unroll
              for (int b_ = 0; b_ < NBC; ++b_) {
                const int col = k0 + tx + 32 * b_;
                if (col < c1) stcg(&M[(size_t)orow[a_] * ld + col], acc[a_][b_]);
              }
            }
            __syncthreads();                    // stage consumed: refill it
            issue(jseq % BJ_NB);
            cp_async_commit();
          }
          item = next;
        }
        cp_async_wait<0>();
        __syncthreads();
      }
      if (!grid_barrier(&ctl->g, nblk, timeout_ns)) return;
      if (blockIdx.x == 0 && tid == 0) ctl->phase_ns[2] += global_timer_ns() - tph;
    }
    // a quiet sweep ends the solve only if it checked every block's own rows:
    // sweep 0 (each block's first pair forms its full Gram) or a verification
    // pass; a quiet cross-only sweep triggers a verification pass
    const bool quiet = atomicAdd(&ctl->active[sweep], 0) == 0;
    const bool was_full = (sweep == 0) || verify;
    if (quiet && was_full) converged = true;
    verify = quiet && !was_full;
  }
  for (long i = gwarp; i < r; i += nwarps) {
    T s = T(0);
    for (int j = lane; j < c; j += 32) { const cplx<T> x = ldcg(&X[(size_t)i * ldx + j]); s += x.x * x.x + x.y * x.y; }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) w[i] = s;
  }
  if (gtid == 0) {
    ctl->g.sweeps = sweep;
    ctl->g.status = converged ? 0 : 1;
  }
}
