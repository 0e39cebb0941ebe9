// mixed.cuh - kernels of the precision form ("mixed"): the truncated SVD of
// a complex128 matrix A (App. A) with FP64-class products on the tensor cores
// and FP32 solves, refined to FP64 accuracy:
//
//   subspace iteration from a seeded Gaussian start, Q <- orth(A orth(A^H Q)),
//        orth = mixed-precision Cholesky QR (FP64-class Gram, FP32 Cholesky of
//        the diagonally scaled Gram, FP64-class product), Newton-Schulz steps
//        Q <- Q (3 I - Q^H Q) / 2 for the final orthonormality;
//   FP32 Rayleigh-Ritz (one-sided Jacobi) on the iterated subspace, and a
//        first-order correction of its leading directions for the coupling
//        the FP32 solve leaves to the rest of the subspace;
//   FP64 Rayleigh-Ritz on those directions: B = Q'^H A, H = B B^H and the FP64
//        Hermitian Jacobi eigen-solve H = V Lambda^2 V^H; left factor Q' V,
//        rows V^H B.
//
// The products are the engine's complex GEMM; these kernels convert, gather,
// draw the start basis, form the Newton-Schulz multiplier and the Cholesky QR
// factors, reduce norms and defects, make a Gram matrix Hermitian and form
// the first-order correction.
#pragma once
#include "common.cuh"

// out (r x c, FP32, ld c) = fl32(in (r x c, FP64, ld ldi)).
__global__ void to_fp32_kernel(const double2* __restrict__ in, int r, int c, int ldi, float2* __restrict__ out) {
  const size_t total = (size_t)r * c;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t i = e / c, j = e % c;
    const double2 v = in[i * ldi + j];
    out[e] = make_float2((float)v.x, (float)v.y);
  }
}

// Q (r x m, FP64, row-major) column j = column perm[j] of U, where the FP32
// one-sided Jacobi returns Ut = U^T (row p of Ut = column p of U, ld r).
__global__ void promote_columns_kernel(const float2* __restrict__ Ut, int r, const int* __restrict__ perm, int m,
                                       double2* __restrict__ Q) {
  const size_t total = (size_t)r * m;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / m), j = (int)(e % m);
    const float2 v = Ut[(size_t)perm[j] * r + i];
    Q[e] = make_double2((double)v.x, (double)v.y);
  }
}

// G (m x m) <- (I - G) / 2 in place: the Newton-Schulz correction
// (Higham, Functions of Matrices, Sec. 8.3).
__global__ void ns_multiplier_kernel(double2* __restrict__ G, int m) {
  const size_t total = (size_t)m * m;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / m), j = (int)(e % m);
    double2 g = G[e];
    g.x = 0.5 * ((i == j ? 1.0 : 0.0) - g.x);
    g.y = -0.5 * g.y;
    G[e] = g;
  }
}

// ---------------------------------------------------------------------------
// Mixed-precision Cholesky QR, the small factor: from the Gram G = Y^H Y (m x m,
// complex128) to W = D L^{-H} (complex128, upper triangular), with
// D = diag(G)^{-1/2} (0 for a zero column) and A = fl32(D G D) + shift I =
// L L^H factored in FP32 (Golub & Van Loan, Matrix Computations, Sec. 4.2).
// Y W then has Gram L^{-1} (D G D) L^{-H}, close to the identity.
//
// One cooperative launch, right-looking over 64 x 64 tiles on [A | I], which
// turns into [L^H | L^{-1}]: step j multiplies the tiles below A_jj by L_jj^{-H}
// and row j of the right half by L_jj^{-1} (barrier), then subtracts rank 64
// from everything below; CTA 0 meanwhile updates A_{j+1,j+1} first and factors
// it, so the serial 64 x 64 factorisation runs under the tile products
// (barrier). The factorisation holds its tile and the tile of L^{-1} in
// registers (4 x 4 of each per thread) and passes one barrier per column.
// What bounds it: FP32 FMAs for m >= 1024 (m^3 / 3 tile flops), else the chain
// of 2 m / 64 barriers and tile latencies. A pass at m = 2048 took 8.4 ms as 156
// launches (recursive halving, a 64 x 64 base case of 130 us), 2.4 ms now; at
// m = 512 1.5 -> 0.44 ms.
// A non-positive pivot sets status[0] to 1 (the factorisation goes on with a tiny
// one, so that no NaN is produced), a barrier that timed out to 2. status[1]
// receives max |L^{-1}_ij|^2 (FP32 bits), the caller's measure of how far Y was
// from orthogonal columns: 1 when they already were.
// ---------------------------------------------------------------------------
constexpr int CH = 64;                 // tile
constexpr int CHP = CH + 2;            // padded row of a staged tile (16-byte rows)
constexpr int CHOL_SMEM = 2 * CH * CHP * (int)sizeof(float2);

// Stage the CH x CH tile at (r0, c0) of M (ld m, zero outside m x m) as
// dst[k][i]: trans != 0 puts the tile's columns along k (dst[k][i] = M[r0 + i][c0 + k]),
// 0 its rows (dst[k][i] = M[r0 + k][c0 + i]).
__device__ __forceinline__ void chol_stage(float2* dst, const float2* M, int m, int r0, int c0, int trans) {
#pragma unroll 4
  for (int e = threadIdx.x; e < CH * CH; e += 256) {
    const int r = e >> 6, c = e & 63;
    const float2 v = r0 + r < m && c0 + c < m ? ldcg(&M[(size_t)(r0 + r) * m + c0 + c]) : make_float2(0.f, 0.f);
    if (trans) dst[c * CHP + r] = v;
    else dst[r * CHP + c] = v;
  }
}

// acc[a][b] = sum_k As[k][4 ty + a] op(Bs[k][4 tx + b]), op = conjugate if conjb.
__device__ __forceinline__ void chol_tile(float2 (&acc)[4][4], const float2* As, const float2* Bs, bool conjb) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  const float sg = conjb ? -1.0f : 1.0f;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);
#pragma unroll 8
  for (int k = 0; k < CH; ++k) {
    float2 av[4], bv[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 x = *reinterpret_cast<const float4*>(&As[k * CHP + 4 * ty + 2 * h]);
      const float4 y = *reinterpret_cast<const float4*>(&Bs[k * CHP + 4 * tx + 2 * h]);
      av[2 * h] = make_float2(x.x, x.y); av[2 * h + 1] = make_float2(x.z, x.w);
      bv[2 * h] = make_float2(y.x, sg * y.y); bv[2 * h + 1] = make_float2(y.z, sg * y.w);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) cfma<float>(acc[a][b], av[a], bv[b]);
  }
}

// Factor the Hermitian tile a (this thread's 4 x 4 part; rows and columns from
// m on read as identity) and leave the lower triangular L^{-1} in r.
__device__ __forceinline__ void chol_factor(float2 (&a)[4][4], float2 (&r)[4][4], float2* buf, float* diag, int* status) {
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) r[i][k] = make_float2(ty == tx && i == k ? 1.f : 0.f, 0.f);
  for (int jb = 0; jb < CH / 4; ++jb) {
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int j = 4 * jb + jj;
      float2* col = buf + (j & 1) * 2 * CH;    // column j of A, row j of the right half; two buffers in turn
      float2* row = col + CH;
      if (tx == jb) {
#pragma unroll
        for (int i = 0; i < 4; ++i) col[4 * ty + i] = a[i][jj];
      }
      if (ty == jb) {
#pragma unroll
        for (int k = 0; k < 4; ++k) row[4 * tx + k] = r[jj][k];
      }
      __syncthreads();
      float d = col[j].x;
      if (!(d > 0.f)) {
        if (tid == 0) atomicMax(status, 1);
        d = 1e-30f;
      }
      if (tid == 0) diag[j] = d;
      const float inv = 1.0f / d;
      float2 f[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 c = col[4 * ty + i];
        f[i] = 4 * ty + i > j ? make_float2(c.x * inv, c.y * inv) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 c = col[4 * tx + k], w = row[4 * tx + k];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // a_ik -= f_i conj(a_kj), r_ik -= f_i r_jk
          a[i][k].x = fmaf(-f[i].x, c.x, fmaf(-f[i].y, c.y, a[i][k].x));
          a[i][k].y = fmaf(-f[i].y, c.x, fmaf(f[i].x, c.y, a[i][k].y));
          r[i][k].x = fmaf(-f[i].x, w.x, fmaf(f[i].y, w.y, r[i][k].x));
          r[i][k].y = fmaf(-f[i].x, w.y, fmaf(-f[i].y, w.x, r[i][k].y));
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float s = rsqrtf(diag[4 * ty + i]);
#pragma unroll
    for (int k = 0; k < 4; ++k) r[i][k] = 4 * tx + k <= 4 * ty + i ? make_float2(s * r[i][k].x, s * r[i][k].y) : make_float2(0.f, 0.f);
  }
}

__global__ void __launch_bounds__(256) cholqr_factor_kernel(const double2* __restrict__ G, int m, float shift, float2* A,
                                                            float2* Li, double2* __restrict__ W, int* status, GridCtl* ctl,
                                                            long long timeout_ns) {
  extern __shared__ __align__(16) unsigned char csm[];
  float2* As = reinterpret_cast<float2*>(csm);
  float2* Bs = As + CH * CHP;
  __shared__ double s_d[2 * CH];
  __shared__ float s_diag[CH];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, nb = (m + CH - 1) / CH;
  const int nblk = (int)gridDim.x, bid = (int)blockIdx.x;
  auto barrier = [&]() -> bool {
    if (grid_barrier(ctl, gridDim.x, timeout_ns)) return true;
    if (tid == 0) atomicMax(status, 2);
    return false;
  };
  // column scales of tiles ti and tk -> s_d
  auto scales = [&](int ti, int tk) {
    __syncthreads();
    if (tid < 2 * CH) {
      const int i = (tid < CH ? ti : tk) * CH + (tid & (CH - 1));
      const double g = i < m ? G[(size_t)i * m + i].x : 0.0;
      s_d[tid] = g > 1e-300 ? rsqrt(g) : 0.0;
    }
    __syncthreads();
  };
  // this thread's part of a finished tile of L^{-1}: to Li and, conjugate
  // transposed and scaled, to W; the tile of W across the diagonal is zero
  auto finish = [&](int j, int k, const float2 (&r)[4][4]) {
    scales(k, k);
    float mx = 0.0f;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int gi = j * CH + 4 * ty + a, gk = k * CH + 4 * tx + b;
        if (gi >= m || gk >= m) continue;
        stcg(&Li[(size_t)gi * m + gk], r[a][b]);
        mx = fmaxf(mx, r[a][b].x * r[a][b].x + r[a][b].y * r[a][b].y);
        if (gk <= gi) {
          const double d = s_d[4 * tx + b];
          W[(size_t)gk * m + gi] = make_double2(d * (double)r[a][b].x, -d * (double)r[a][b].y);
        }
        if (gk < gi) W[(size_t)gi * m + gk] = make_double2(0.0, 0.0);
      }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) atomicMax(&status[1], __float_as_int(mx));
  };

  // after a barrier of an earlier launch that timed out the word holds a partial
  // count, and barriers would end before all have arrived
  if (*(volatile int*)&ctl->err) {
    if (tid == 0) atomicMax(status, 2);
    return;
  }
  if (bid == 0 && tid == 0) status[1] = 0;   // before the first barrier; written after it
  // A = fl32(D G D) + shift I, lower tiles
  for (int q = bid; q < nb * (nb + 1) / 2; q += nblk) {
    int i = 0, k = q;
    while (k > i) k -= ++i;
    scales(i, k);
    for (int e = tid; e < CH * CH; e += 256) {
      const int r = e >> 6, c = e & 63, gr = i * CH + r, gc = k * CH + c;
      if (gr >= m || gc >= m) continue;
      const double2 g = G[(size_t)gr * m + gc];
      const double dd = s_d[r] * s_d[CH + c];
      stcg(&A[(size_t)gr * m + gc], make_float2((float)(dd * g.x) + (gr == gc ? shift : 0.0f), (float)(dd * g.y)));
    }
  }
  if (!barrier()) return;

  float2 acc[4][4];
  // diagonal tile j, less the product in acc, factored by this CTA
  auto diagonal = [&](int j) {
    float2 a[4][4], r[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int gi = j * CH + 4 * ty + x, gk = j * CH + 4 * tx + y;
        // the upper triangle is not used (column j of the tile is read below the pivot)
        float2 v = gi < m && gk < m ? ldcg(&A[(size_t)gi * m + gk]) : make_float2(gi == gk ? 1.f : 0.f, 0.f);
        a[x][y] = csub<float>(v, acc[x][y]);
      }
    __syncthreads();
    chol_factor(a, r, As, s_diag, status);
    finish(j, j, r);
  };
  if (bid == 0) {
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[x][y] = make_float2(0.f, 0.f);
    diagonal(0);
  }
  if (!barrier()) return;
  for (int j = 0; j < nb; ++j) {
    // panel: L_ij = A_ij L_jj^{-H} (i > j), (L^{-1})_jk = L_jj^{-1} R_jk (k < j)
    for (int q = bid; q < nb; q += nblk) {
      if (q == j) continue;
      __syncthreads();
      if (q > j) {
        chol_stage(As, A, m, q * CH, j * CH, 1);
        chol_stage(Bs, Li, m, j * CH, j * CH, 1);
      } else {
        chol_stage(As, Li, m, j * CH, j * CH, 1);
        chol_stage(Bs, Li, m, j * CH, q * CH, 0);
      }
      __syncthreads();
      chol_tile(acc, As, Bs, q > j);
      if (q > j) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const int gi = q * CH + 4 * ty + x, gk = j * CH + 4 * tx + y;
            if (gi < m && gk < m) stcg(&A[(size_t)gi * m + gk], acc[x][y]);
          }
      } else {
        finish(j, q, acc);
      }
    }
    if (j + 1 == nb) break;
    if (!barrier()) return;
    // rank-64 update of the rows below: A_ik -= L_ij L_kj^H (j < k <= i) and
    // R_ik -= L_ij (L^{-1})_jk (k <= j; R_ij starts here); CTA 0 takes the next
    // diagonal tile, the others the rest
    const int lanes = nblk > 1 ? nblk - 1 : 1, me = nblk > 1 ? bid - 1 : 0;
    if (bid == 0) {
      __syncthreads();
      chol_stage(As, A, m, (j + 1) * CH, j * CH, 1);
      __syncthreads();
      chol_tile(acc, As, As, true);
      diagonal(j + 1);
    }
    if (me >= 0) {
      int total = 0;
      for (int i = j + 1; i < nb; ++i) total += i + 1;
      for (int q = me; q < total; q += lanes) {
        int i = j + 1, k = q;
        while (k > i) k -= ++i;
        if (i == j + 1 && k == i) continue;
        const bool right = k <= j;
        __syncthreads();
        chol_stage(As, A, m, i * CH, j * CH, 1);
        if (right) chol_stage(Bs, Li, m, j * CH, k * CH, 0);
        else chol_stage(Bs, A, m, k * CH, j * CH, 1);
        __syncthreads();
        chol_tile(acc, As, Bs, !right);
        float2* C = right ? Li : A;
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const int gi = i * CH + 4 * ty + x, gk = k * CH + 4 * tx + y;
            if (gi >= m || gk >= m) continue;
            const float2 c0 = k == j ? make_float2(0.f, 0.f) : ldcg(&C[(size_t)gi * m + gk]);
            stcg(&C[(size_t)gi * m + gk], csub<float>(c0, acc[x][y]));
          }
      }
    }
    if (!barrier()) return;
  }
}

// Seeded complex Gaussian start basis for the subspace iteration: entry e
// draws two uniforms from the SplitMix64 sequence (Steele, Lea & Flood 2014)
// at counter 2e, 2e+1 of the given seed and turns them into a standard
// complex normal by the Box-Muller transform.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void gauss_start_kernel(double2* __restrict__ out, size_t n, unsigned long long seed) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const unsigned long long a = splitmix64(seed + 2 * e), b = splitmix64(seed + 2 * e + 1);
    const double u1 = ((double)(a >> 11) + 1.0) * (1.0 / 9007199254740993.0);   // (0, 1]
    const double u2 = (double)(b >> 11) * (1.0 / 9007199254740992.0);           // [0, 1)
    const double rad = sqrt(-log(u1));
    double sn, cs;
    sincospi(2.0 * u2, &sn, &cs);
    out[e] = make_double2(rad * cs, rad * sn);
  }
}

// *out += sum |A_ij|^2 over an r x c complex128 matrix (leading dimension
// lda), accumulated in FP64: grid-stride partial sums, one atomicAdd per CTA
// (*out zeroed beforehand).
__global__ void __launch_bounds__(256) frob2_kernel(const double2* __restrict__ A, int r, int c, int lda,
                                                    double* __restrict__ out) {
  __shared__ double red[8];
  double s = 0.0;
  const size_t total = (size_t)r * c;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const double2 v = A[(e / c) * lda + e % c];
    s += v.x * v.x + v.y * v.y;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < 8; ++i) v += red[i];
    atomicAdd(out, v);
  }
}

// H (m x m) <- (H + H^H) / 2 in place: the Gram matrix of the Rayleigh-Ritz
// step made exactly Hermitian (its two triangles come from separately rounded
// products) before the Hermitian eigen-solver, which reads one triangle.
__global__ void hermitise_kernel(double2* __restrict__ H, int m) {
  const size_t total = (size_t)m * m;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / m), j = (int)(e % m);
    if (j < i) continue;
    if (j == i) { H[e].y = 0.0; continue; }
    const double2 a = H[e], b = H[(size_t)j * m + i];
    const double2 v = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
    H[e] = v;
    H[(size_t)j * m + i] = make_double2(v.x, -v.y);
  }
}

// First-order correction of the leading approximate eigenvectors (one
// refinement step of Ogita & Aishima, Japan J. Indust. Appl. Math. 35 (2018)):
// with the approximate eigenvector matrix V (m x m), S = V^H H V and G = V^H V
// (both FP64-accurate), R = I - G and lambda_i = S_ii / (1 - R_ii), the leading
// columns i < mp gain
//   E_ji = (S_ji + lambda_i R_ji) / (lambda_i - lambda_j)
// of column j, which removes their error along it to first order. Towards the
// remaining columns (j >= mp) that is what keeps the FP32 solve's couplings out
// of the kept subspace; pairs with a relative gap below 1e-2 (inside a cluster
// at the edge, only in the margin beyond the kept directions) get the
// orthogonality term R_ji / 2 alone, and so do pairs with |E_ji| > 1e-2: couplings of
// 3e-5 give at most 3e-3 there, so both values are rounding of zeros (a rank
// below mp), and E_ji their ratio, of any size. Among the leading columns it saves the FP64
// eigen-solve that follows a sweep; there a pair is taken where |E_ji| <= 1e-3, so
// that V_P (I + E_PP) stays within reach of the Newton-Schulz steps, else R_ji / 2.
// A pair without a gap is never taken: exactly equal values with no coupling
// (zero rows, equal rows, a multiple of the identity) have 0 / 0 there, and any
// basis of their span is one of eigenvectors.
// Output (m x mp): rows j < mp are I + E_PP, the others E_RP.
__global__ void partition_correction_kernel(const double2* __restrict__ S, const double2* __restrict__ G, int m, int mp,
                                            double2* __restrict__ E) {
  const size_t total = (size_t)m * mp;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(e / mp), i = (int)(e % mp);
    if (i == j) { E[e] = make_double2(1.0, 0.0); continue; }
    const double li = S[(size_t)i * m + i].x / G[(size_t)i * m + i].x;
    const double lj = S[(size_t)j * m + j].x / G[(size_t)j * m + j].x;
    const double2 s = S[(size_t)j * m + i];
    const double2 g = G[(size_t)j * m + i];
    const double2 rji = make_double2(-g.x, -g.y);      // (I - G)_ji, j != i
    const double gap = li - lj;
    const double2 num = make_double2(s.x + li * rji.x, s.y + li * rji.y);
    const double an = fmax(fabs(num.x), fabs(num.y)), ag = fabs(gap);
    const bool far = j < mp ? ag > 0.0 && an <= 1e-3 * ag : ag > 1e-2 * fmax(fabs(li), fabs(lj)) && an <= 1e-2 * ag;
    E[e] = far ? make_double2(num.x / gap, num.y / gap) : make_double2(0.5 * rji.x, 0.5 * rji.y);
  }
}

// *out = max_ij |G_ij - delta_ij| over an m x m complex128 matrix: the
// orthonormality defect of a basis whose Gram matrix is G. Grid-stride
// maxima, one atomicMax per CTA on the bit pattern (order-preserving for
// non-negative doubles); *out zeroed beforehand.
__global__ void __launch_bounds__(256) defect_kernel(const double2* __restrict__ G, int m, double* __restrict__ out) {
  __shared__ double red[8];
  double s = 0.0;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)m * m; e += (size_t)gridDim.x * blockDim.x) {
    const size_t i = e / m, j = e % m;
    const double2 g = G[e];
    s = fmax(s, hypot(g.x - (i == j ? 1.0 : 0.0), g.y));
  }
  for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < 8; ++i) v = fmax(v, red[i]);
    atomicMax((unsigned long long*)out, (unsigned long long)__double_as_longlong(v));
  }
}
