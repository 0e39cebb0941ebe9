// ozgemm.cuh - FP64-accurate complex GEMM on the tcgen05 tensor cores from
// BF16 split products with FP32 accumulation (the error-free splitting
// scheme of Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012):
//
//   C (M x N, complex128) = alpha op(A) op(B) (+ C),  op = plain or ^H.
//
// Splitting. Every row i of op(A) (every column j of op(B)) gets a power of
// two 2^e_i bounding its entries; each real entry x = v / 2^e_i in (-1, 1)
// is written as sum_{t=1..S} a_t 2^{-7t} with integers |a_1| <= 128,
// |a_t| <= 64 for t >= 2 (the balanced base-128 digits of round(x 2^{7S})),
// so every slice value a_t 2^{-7t} is exact in BF16 and every product
// a_t b_u 2^{-7(t+u)} is exact in FP32. Keeping the products with
// t + u <= S + 1 leaves a relative error of about 2^{-7S} of |row| |column|.
//
// Complex as real: op(A)' = [Re | Im] (M x 2K), and the rows of op(B)'^T
// interleave the output's real and imaginary parts: row 2j = [Re b_j | -Im
// b_j], row 2j+1 = [Im b_j | Re b_j], so a real output column pair
// (2j, 2j+1) is the complex column j.
//
// Accumulation. The products of one level L = t + u are summed in their own
// TMEM accumulator: within a level every product is an integer multiple of
// 2^{-7L}, and over a K chunk of KC real terms those integer sums are at most
// 2^24, so each chunk's sum is exact whatever the alignment and
// rounding inside the tensor core's FP32 accumulation (levels of different
// units must not share an accumulator: their small terms would fall below
// the accumulator's resolution, an error growing with K). After each chunk
// every level is drained to double-float (hi, lo) FP32 registers; the tile's
// value (hi + lo) 2^{e_i + f_j} is formed in FP64 once at the end.
//
// Operand layout. The split kernels write the slices in the order in which the
// MMA kernel reads them: one stage is 16 complex k, its real parts, then (the
// next stage) its imaginary parts, 16 real K each, in the K-major no-swizzle
// core-matrix layout (8 rows x 16 bytes per core matrix, SBO = 128 B between
// 8-row groups, LBO between the two K groups of 8):
//   A: [row block of 128][stage][slice][K group][128 rows][8]   24 KB per stage
//   B: [column block of 64][stage][K group][slice][64 rows][8]  12 KB per stage
// so a stage is three bulk copies, and the slices of B follow one another as
// rows: one MMA multiplies an A slice by two neighbouring B slices (N = 128).
//
// Accumulators. Level t + u of a slice pair has 64 TMEM columns; pairs of
// levels (2p, 2p + 1) are the fixed 128-column accumulators, so every MMA on an
// accumulator has the same shape and they execute in issue order. A slice of
// odd index meets the pair that starts one level lower with a zero slice
// ahead of B's first one in shared memory: 12 MMAs (24 slice products, 3 of
// them zero) per 16 real K. With N = 64, one product each, the A operand is
// read from shared memory 21 times instead of 12, more than its bandwidth.
//
// A persistent CTA (grid <= SMs) walks over 128 x 64 real tiles (128 rows x 32
// complex columns): one warp issues the bulk copies (five stages ahead), one
// thread the MMAs, eight warps drain the accumulators and write C, so the
// copies of the next tile run under the epilogue of this one. Every wait is
// bounded.
// What bounds it: most likely L2, whose reads run at 7.9 TB/s. A stage of 16 real K
// takes 768 clocks of the tensor pipe and 1056 of shared memory (the MMAs read
// 96 KB, the copies write 36 KB, at 128 B per clock) but 1343 in all, and a CTA pair
// with 23 % less shared-memory traffic was no faster (6.8 ms per call instead of
// 6.0). 4096 x 2048 x 4096: 13.75 ms with cp.async loads one stage ahead and N = 64
// MMAs, 4.92 ms now (tensor pipe 54 % active, 55.9 TFLOP/s of FP64-accurate work).
#pragma once
#include <cuda_bf16.h>
#include "common.cuh"
#include "tcgemm.cuh"

namespace oz {
constexpr int S = 6;                         // slices per operand (about 43 bits)
constexpr int BM = 128, BN = 64;             // real tile: 128 rows x 64 real (32 complex) columns
constexpr int KS = 16;                       // real K per stage: one MMA deep
// real K per exact chunk: a level's products sum to at most 2^15 units per K
// (|a_1| <= 128, |a_t| <= 64: 2 * 2^13 + 4 * 2^12 at level 7), 2^24 per chunk
constexpr int KC = 512;
static_assert((long long)KC * (2 * 128 * 64 + (S - 2) * 64 * 64) <= 1ll << 24, "a chunk's sums must be exact in FP32");
constexpr int SPC = KC / KS;                 // stages per chunk
constexpr int A_STAGE = S * 2 * BM * 16;     // 24 KB in global and shared memory
constexpr int B_STAGE = 2 * S * BN * 16;     // 12 KB in global memory
constexpr int B_KG = (S + 1) * BN * 16;      // one K group of B in shared memory, zero slice first
constexpr int STAGE_BYTES = A_STAGE + 2 * B_KG;
constexpr int NSTAGE = 5;
constexpr int SMEM_BYTES = NSTAGE * STAGE_BYTES + 1024;
constexpr int A_LBO = BM * 16;               // byte step between the K groups of 8
constexpr int NDRAIN = 8;                    // drain warps: 4 TMEM lane groups x 2 column halves
constexpr int NT = 32 * (NDRAIN + 2);
constexpr int TCOLS = 512;                   // TMEM allocation (power of two >= S * BN)
static_assert(S * BN <= TCOLS, "accumulators exceed the TMEM allocation");
constexpr int MAXSPLIT = 8;                  // parts of a tile's K range
constexpr int MAXITEMS = 256;                // (tile, part) items of a split product, at most the SMs
constexpr size_t PART_BYTES = (size_t)BM * BN * sizeof(double);   // a part's sums

// Shared-memory matrix descriptor, K-major, no swizzle: start address, LBO
// (byte step between the core matrices of consecutive K groups), SBO = 128 B
// (step between 8-row groups), descriptor version 1.
__device__ __forceinline__ uint64_t desc(uint32_t addr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((128 >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
}  // namespace oz

// Scaling exponents. raw[i] = the largest biased FP64 exponent field among
// the real and imaginary parts of row i of op(A) (or column j of op(B)),
// gathered with integer atomicMax (raw zeroed beforehand); the scaling
// exponent is then oz_ex(raw) = raw - 1022 (the frexp exponent of the row's
// largest entry, so every |x| < 2^oz_ex), or 0 for a zero row.
__device__ __forceinline__ int oz_ex(int raw) { return raw > 0 ? raw - 1022 : 0; }
__device__ __forceinline__ int oz_bexp(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF); }

// One operand of a product: the stored matrix, its form and its slices.
struct OzOp {
  const double2* X;
  int ld, op;        // op 0: as stored, 1: conjugate transpose
  int n;             // rows of op(A) / columns of op(B)
  int* raw;          // exponents
  __nv_bfloat16* sl;
};

// The stored matrices (R rows x C columns) are scanned in 32-column x 256-row
// tiles, block (32, 8); by_row = 1 reduces along each stored row (raw indexed by
// stored row), 0 along each stored column. One atomic per warp-row or per
// tile column. Blocks below na scan A, the rest B.
__global__ void oz_exp_kernel(OzOp a, OzOp b, int K, int na) {
  __shared__ int red[8][33];
  const bool isB = (int)blockIdx.x >= na;
  const OzOp o = isB ? b : a;
  const int by_row = isB ? o.op : 1 - o.op;              // the K index runs along the stored row
  const int R = by_row ? o.n : K, C = by_row ? K : o.n;
  const int id = isB ? blockIdx.x - na : blockIdx.x, nx = (C + 31) / 32;
  const int c = (id % nx) * 32 + threadIdx.x, r0 = (id / nx) * 256, ty = threadIdx.y;
  int mcol = 0;
  for (int r = r0 + ty; r < min(R, r0 + 256); r += 8) {
    int v = 0;
    if (c < C) {
      const double2 x = o.X[(size_t)r * o.ld + c];
      v = max(oz_bexp(x.x), oz_bexp(x.y));
    }
    if (by_row) {
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, s));
      if (threadIdx.x == 0 && v > 0) atomicMax(&o.raw[r], v);
    } else {
      mcol = max(mcol, v);
    }
  }
  if (!by_row) {
    red[ty][threadIdx.x] = mcol;
    __syncthreads();
    if (ty == 0) {
      int v = red[0][threadIdx.x];
#pragma unroll
      for (int i = 1; i < 8; ++i) v = max(v, red[i][threadIdx.x]);
      if (c < C && v > 0) atomicMax(&o.raw[c], v);
    }
  }
}

// The S slices of x / 2^ex (|x| < 2^ex) by integer arithmetic on the FP64
// bits: N = round(x 2^(7S - ex)), |N| <= 2^(7S), written in balanced base-128
// digits N = sum_t a_t 2^(7(S - t)) (a_t in [-64, 63] for t >= 2 and
// |a_1| <= 128); out[t] = a_{t+1} 2^{-7(t+1)}, exact in BF16. The error
// |x / 2^ex - sum| <= 2^(-7S - 1). No FP64 arithmetic (that unit runs at
// 1/64 of the FP32 rate on this part).
__device__ __forceinline__ void oz_slices(double v, int ex, float* out) {
  const long long bits = __double_as_longlong(v);
  const int be = (int)((bits >> 52) & 0x7FF);
  long long n = 0;
  if (be > 0) {
    const long long mant = (bits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
    const int sh = 1075 - 7 * oz::S + ex - be;     // right shift taking mant 2^(be-1075) to units of 2^(ex - 7S)
    if (sh < 63) {
      const long long mag = sh > 0 ? (mant + (1ll << (sh - 1))) >> sh : mant << (-sh);
      n = bits < 0 ? -mag : mag;
    }
  }
#pragma unroll
  for (int t = oz::S - 1; t >= 1; --t) {
    const long long d = ((n + 64) & 127) - 64;
    out[t] = __int2float_rn((int)d) * __int_as_float((127 - 7 * (t + 1)) << 23);
    n = (n - d) >> 7;
  }
  out[0] = __int2float_rn((int)n) * __int_as_float((127 - 7) << 23);
}

// Slices of both operands in the stage layout above, zero outside the matrix.
// One block of 128 threads takes 16 complex k (both stages) of 32 rows of
// op(A), or of 16 columns of op(B): the 32 interleaved rows 2j = [Re b_j |
// -Im b_j], 2j + 1 = [Im b_j | Re b_j]. Through shared memory, so that either
// form is read coalesced; a thread then forms 8 K values of one row and stage
// and writes 16 bytes per slice, 512 consecutive bytes per warp. Blocks below
// na take A (nka = stages / 2 blocks per 32 rows), the rest B.
__global__ void __launch_bounds__(128) oz_split_kernel(OzOp a, OzOp b, int K, int nkb, int na) {
  __shared__ double2 tile[32][17];
  const bool isB = (int)blockIdx.x >= na;
  const OzOp o = isB ? b : a;
  const int id = isB ? blockIdx.x - na : blockIdx.x, kb = id % nkb, rb = id / nkb;
  const int tid = threadIdx.x, k0 = kb * 16, i0 = rb * (isB ? 16 : 32), ni = isB ? 16 : 32;
  const bool along = isB ? o.op == 1 : o.op == 0;   // k runs along the stored row
  for (int e = tid; e < ni * 16; e += 128) {
    const int i = along ? e >> 4 : e % ni, k = along ? e & 15 : e / ni;
    double2 v = make_double2(0.0, 0.0);
    if (i0 + i < o.n && k0 + k < K) {
      v = along ? o.X[(size_t)(i0 + i) * o.ld + k0 + k] : o.X[(size_t)(k0 + k) * o.ld + i0 + i];
      if (o.op) v.y = -v.y;
    }
    tile[i][k] = v;
  }
  __syncthreads();
  const int q = tid & 31, cg = (tid >> 5) & 1, im = tid >> 6;   // row, K group of 8, stage
  const int i = isB ? q >> 1 : q;
  const int ex = i0 + i < o.n ? oz_ex(o.raw[i0 + i]) : 0;
  const bool take_im = isB ? ((q & 1) != im) : im != 0;         // B: even rows [Re, -Im], odd rows [Im, Re]
  const float sign = isB && im && !(q & 1) ? -1.0f : 1.0f;
  uint32_t pk[oz::S][4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float s0[oz::S], s1[oz::S];
    const double2 v0 = tile[i][8 * cg + 2 * h], v1 = tile[i][8 * cg + 2 * h + 1];
    oz_slices(take_im ? v0.y : v0.x, ex, s0);
    oz_slices(take_im ? v1.y : v1.x, ex, s1);
#pragma unroll
    for (int t = 0; t < oz::S; ++t) {
      const __nv_bfloat162 p2 = __floats2bfloat162_rn(sign * s0[t], sign * s1[t]);
      pk[t][h] = *reinterpret_cast<const uint32_t*>(&p2);
    }
  }
  unsigned char* base = reinterpret_cast<unsigned char*>(o.sl);
  const int stage = 2 * kb + im;
  if (!isB) {
    base += ((size_t)(rb >> 2) * (2 * nkb) + stage) * oz::A_STAGE + cg * oz::A_LBO + ((rb & 3) * 32 + q) * 16;
#pragma unroll
    for (int t = 0; t < oz::S; ++t)
      *reinterpret_cast<uint4*>(base + t * 2 * oz::A_LBO) = make_uint4(pk[t][0], pk[t][1], pk[t][2], pk[t][3]);
  } else {
    base += ((size_t)(rb >> 1) * (2 * nkb) + stage) * oz::B_STAGE + cg * (oz::B_STAGE / 2) + ((rb & 1) * 32 + q) * 16;
#pragma unroll
    for (int t = 0; t < oz::S; ++t)
      *reinterpret_cast<uint4*>(base + t * oz::BN * 16) = make_uint4(pk[t][0], pk[t][1], pk[t][2], pk[t][3]);
  }
}

// (hi, lo) += x for exact x (Knuth's two-sum; the rounding error of hi + x
// goes to lo).
__device__ __forceinline__ void df_add(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bb = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  hi = s;
  lo = __fadd_rn(lo, err);
}

// The tile list of a product. General: row blocks in groups of 16 and the
// column blocks of a group in turn, so the tiles in flight at one time share
// their operands in L2.
// kHerm (op(A) op(B) Hermitian, e.g. a Gram): only the tiles that reach the
// diagonal or lie above it; the epilogue writes the mirror image too.
// kUpper (op(B) upper triangular, zero below the diagonal): a tile's K loop ends
// with its last column; column blocks from the longest down.
// Both halve the work of a Cholesky QR pass (Y^H Y and Y W).
struct OzTiles {
  enum { kGeneral = 0, kHerm = 1, kUpper = 2 };
  int nrb, ncb, nkb;      // row blocks, column blocks, blocks of 16 complex k
  int mode;
  // K parts per tile. A product with fewer tiles than SMs splits K between CTAs,
  // one item each: the parts' sums go to global memory and the CTA that finishes a
  // tile last adds them in order of k, so the result does not depend on the timing.
  int splits;
  __host__ __device__ __forceinline__ int count() const {
    if (mode != kHerm) return nrb * ncb;
    int n = 0;
    for (int rb = 0; rb < nrb && 4 * rb < ncb; ++rb) n += ncb - 4 * rb;
    return n;
  }
  __device__ __forceinline__ void tile(int id, int& rb, int& cb) const {
    if (mode == kHerm) {            // row 128 rb <= column 32 cb + 31
      rb = 0;
      while (id >= ncb - 4 * rb) id -= ncb - 4 * rb++;
      cb = 4 * rb + id;
      return;
    }
    if (mode == kUpper) {
      cb = ncb - 1 - id / nrb;
      rb = id % nrb;
      return;
    }
    const int per = 16 * ncb, g = id / per, h = min(16, nrb - 16 * g), w = id - g * per;
    rb = 16 * g + w % h;
    cb = w / h;
  }
  __device__ __forceinline__ int stages(int cb) const { return 2 * (mode == kUpper ? min(nkb, 2 * cb + 2) : nkb); }
  // the item's tile, its part and its range of stages
  __device__ __forceinline__ void item(int id, int& rb, int& cb, int& s0, int& s1) const {
    tile(id / splits, rb, cb);
    const int n = stages(cb), q = id % splits;
    s0 = n * q / splits;
    s1 = n * (q + 1) / splits;
  }
};

#define OZ_LD32(v, taddr)                                                                                      \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15," \
               "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"                      \
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),           \
                 "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),       \
                 "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]),    \
                 "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),    \
                 "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])                                            \
               : "r"(taddr))

// grid <= SMs, oz::NT threads, dynamic smem oz::SMEM_BYTES. status: set to 1 if
// an mbarrier wait ran past timeout_ns (the CTA's remaining tiles are then left
// unwritten).
__global__ void __launch_bounds__(oz::NT, 1) oz_mma_kernel(OzTiles tl, OzOp a, OzOp b, double2* __restrict__ C, int ldc,
                                                           double alpha, int accumulate, double2* part, int* counters,
                                                           int* status, long long timeout_ns) {
  using namespace oz;
  extern __shared__ __align__(1024) unsigned char oz_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[NSTAGE], empty[NSTAGE], acc_full, acc_empty, part_done, last_known;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail, s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(tcg::saddr(&tmem_base)), "n"(TCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < NSTAGE; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(tcg::saddr(&full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(tcg::saddr(&empty[i])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(tcg::saddr(&acc_full)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(tcg::saddr(&acc_empty)), "n"(NDRAIN));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(tcg::saddr(&part_done)), "n"(NDRAIN));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(tcg::saddr(&last_known)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  // the zero slice ahead of B's first one, in both K groups of every stage
  for (int e = tid; e < NSTAGE * 2 * BN; e += NT) {
    unsigned char* z = sm + (e / (2 * BN)) * STAGE_BYTES + A_STAGE + ((e / BN) & 1) * B_KG + (e % BN) * 16;
    *reinterpret_cast<uint4*>(z) = make_uint4(0, 0, 0, 0);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = tmem_base;
  const int ntiles = tl.count() * tl.splits;
  volatile int* fail = &s_fail;
  // limit of the waits for this CTA's own copies and MMAs at the end: microseconds,
  // which a caller's shorter limit must not cut
  const long long drain_ns = max(timeout_ns, 1000000000ll);

  if (warp == NDRAIN) {
    // ---- producer: three bulk copies per stage --------------------------
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int id = blockIdx.x; id < ntiles && ok; id += gridDim.x) {
        int rb, cb, s0, s1;
        tl.item(id, rb, cb, s0, s1);
        const unsigned char* pa = reinterpret_cast<const unsigned char*>(a.sl) + (size_t)rb * 2 * tl.nkb * A_STAGE;
        const unsigned char* pb = reinterpret_cast<const unsigned char*>(b.sl) + (size_t)cb * 2 * tl.nkb * B_STAGE;
        for (int s = s0; s < s1; ++s, ++it) {
          const int slot = it % NSTAGE;
          if (it >= NSTAGE && !tcg::wait_parity(tcg::saddr(&empty[slot]), (uint32_t)(it / NSTAGE - 1) & 1u, timeout_ns)) ok = false;
          if (!ok || *fail) { ok = false; break; }
          const uint32_t st = tcg::saddr(sm + slot * STAGE_BYTES), bar = tcg::saddr(&full[slot]);
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "n"(A_STAGE + B_STAGE) : "memory");
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                       :: "r"(st), "l"(pa + (size_t)s * A_STAGE), "n"(A_STAGE), "r"(bar) : "memory");
#pragma unroll
          for (int g = 0; g < 2; ++g)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         :: "r"(st + A_STAGE + g * B_KG + BN * 16), "l"(pb + (size_t)s * B_STAGE + g * (B_STAGE / 2)),
                            "n"(B_STAGE / 2), "r"(bar) : "memory");
        }
      }
      if (!ok) s_fail = 1;
      // copies still in flight land before the CTA may end
      for (int j = max(0, it - NSTAGE); j < it; ++j)
        (void)tcg::wait_parity(tcg::saddr(&full[j % NSTAGE]), (uint32_t)(j / NSTAGE) & 1u, drain_ns);
    }
  } else if (warp == NDRAIN + 1) {
    // ---- MMA issue --------------------------------------------------------
    if (lane == 0) {
      // kind::f16 instruction descriptor: D FP32 (bit 4), A and B BF16 (bits 7, 10), K-major, N >> 3, M >> 4
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * BN) >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      int it = 0, chunk = 0;
      bool ok = true;
      for (int id = blockIdx.x; id < ntiles && ok; id += gridDim.x) {
        int rb, cb, s0, s1;
        tl.item(id, rb, cb, s0, s1);
        const int nst = s1 - s0;
        for (int s = 0; s < nst; ++s, ++it) {
          const int slot = it % NSTAGE;
          const bool first = s % SPC == 0;
          if (first && chunk > 0) {     // the drain warps have read the previous chunk
            if (!tcg::wait_parity(tcg::saddr(&acc_empty), (uint32_t)(chunk - 1) & 1u, timeout_ns)) ok = false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          if (!ok || *fail || !tcg::wait_parity(tcg::saddr(&full[slot]), (uint32_t)(it / NSTAGE) & 1u, timeout_ns)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = tcg::saddr(sm + slot * STAGE_BYTES);
#pragma unroll
          for (int p = 0; p < S / 2; ++p) {
#pragma unroll
            for (int t = 0; t < 2 * p + 2; ++t) {
              // levels 2p, 2p + 1 from slice t of A and slices 2p - t, 2p - t + 1 of B (row 64 (u + 1); u = -1: zeros)
              const uint64_t da = oz::desc(st + t * 2 * A_LBO, A_LBO);
              const uint64_t db = oz::desc(st + A_STAGE + (2 * p - t + 1) * BN * 16, B_KG);
              const uint32_t en = (first && t == 0) ? 0u : 1u;
              asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                           :: "r"(tbase + 2 * BN * p), "l"(da), "l"(db), "r"(idesc), "r"(en));
            }
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(tcg::saddr(&empty[slot])) : "memory");
          if ((s + 1) % SPC == 0 || s + 1 == nst) {
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(tcg::saddr(&acc_full)) : "memory");
            ++chunk;
          }
        }
      }
      if (!ok) s_fail = 1;
      // MMAs still in flight finish before TMEM is released
      for (int j = max(0, it - NSTAGE); j < it; ++j)
        (void)tcg::wait_parity(tcg::saddr(&empty[j % NSTAGE]), (uint32_t)(j / NSTAGE) & 1u, drain_ns);
    }
  } else {
    // ---- drain and epilogue ------------------------------------------------
    const int lg = warp & 3, half = warp >> 2;      // rows 32 lg .., real columns 32 half .. of each level
    const uint32_t tl0 = tbase + ((uint32_t)(32 * lg) << 16) + 32 * half;
    uint32_t pphase = 0;
    int chunk = 0;
    bool ok = true;
    for (int id = blockIdx.x; id < ntiles && ok; id += gridDim.x) {
      int rb, cb, s0, s1;
      tl.item(id, rb, cb, s0, s1);
      const int nch = (s1 - s0 + SPC - 1) / SPC;
      float hi[32], lo[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) { hi[j] = 0.f; lo[j] = 0.f; }
      for (int q = 0; q < nch; ++q, ++chunk) {
        ok = tcg::wait_parity(tcg::saddr(&acc_full), (uint32_t)chunk & 1u, timeout_ns) && !*fail;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t v[2][32];
        OZ_LD32(v[0], tl0);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int l = 0; l < S; ++l) {
          if (l + 1 < S) OZ_LD32(v[(l + 1) & 1], tl0 + BN * (l + 1));
#pragma unroll
          for (int j = 0; j < 32; ++j) df_add(hi[j], lo[j], __uint_as_float(v[l & 1][j]));
          if (l + 1 < S) asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (l + 2 == S) {            // the last level is in registers: the accumulators are free
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tcg::saddr(&acc_empty)) : "memory");
          }
        }
      }
      if (!ok) break;
      double2 sum[16];
#pragma unroll
      for (int q = 0; q < 16; ++q)
        sum[q] = make_double2((double)hi[2 * q] + (double)lo[2 * q], (double)hi[2 * q + 1] + (double)lo[2 * q + 1]);
      if (tl.splits > 1) {
        // item's block of part: [complex column][128 rows], so a warp writes 512
        // consecutive bytes; the drain warps meet on mbarriers (bounded waits)
        double2* mine = part + (size_t)id * (BM * BN / 2) + (size_t)(16 * half) * BM + 32 * lg + lane;
#pragma unroll
        for (int q = 0; q < 16; ++q) stcg(&mine[(size_t)q * BM], sum[q]);
        __threadfence();
        const int tile = id / tl.splits;
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tcg::saddr(&part_done)) : "memory");
        ok = __all_sync(0xffffffffu, tcg::wait_parity(tcg::saddr(&part_done), pphase, timeout_ns));
        if (!ok) break;
        if (tid == 0) {
          __threadfence();      // the other warps' stores, known here through the mbarrier, before the count
          s_last = atomicAdd(&counters[tile], 1) == tl.splits - 1;
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tcg::saddr(&last_known)) : "memory");
        }
        ok = __all_sync(0xffffffffu, tcg::wait_parity(tcg::saddr(&last_known), pphase, timeout_ns));
        if (!ok) break;
        pphase ^= 1u;
        if (!s_last) continue;
        __threadfence();
        if (tid == 0) counters[tile] = 0;            // for the next launch
        const double2* all = part + (size_t)tile * tl.splits * (BM * BN / 2) + (size_t)(16 * half) * BM + 32 * lg + lane;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          double2 v = ldcg(&all[(size_t)q * BM]);
          for (int p = 1; p < tl.splits; ++p) v = cadd<double>(v, ldcg(&all[(size_t)p * (BM * BN / 2) + (size_t)q * BM]));
          sum[q] = v;
        }
      }
      const int row = rb * BM + 32 * lg + lane;
      const int er = row < a.n ? oz_ex(a.raw[row]) : 0;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int j = cb * (BN / 2) + 16 * half + q;   // complex column: real part 2q, imaginary 2q + 1
        if (row >= a.n || j >= b.n) continue;
        const int sc = er + oz_ex(b.raw[j]);
        double re = ldexp(sum[q].x, sc) * alpha;
        double im = ldexp(sum[q].y, sc) * alpha;
        if (tl.mode == OzTiles::kHerm) {
          if (row > j) continue;
          if (row < j) C[(size_t)j * ldc + row] = make_double2(re, -im);
        }
        double2* dst = &C[(size_t)row * ldc + j];
        if (accumulate) { const double2 cv = *dst; re += cv.x; im += cv.y; }
        *dst = make_double2(re, im);
      }
    }
    if (!ok) s_fail = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && s_fail) atomicExch(status, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tbase), "n"(TCOLS));
}
