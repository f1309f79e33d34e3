// FP64 Toeplitz products of whole time lines (64 .. 1024 steps): the FP64
// smoother's half-sweep (Sec. 3 Eq. red-black, Sec. 6 Eq. red-black_2d) and
// one-point solve, u_p = k * b_p with b_p = f_p + h^-2 sum of neighbour lines, and
// the time term T_M u_p of the FP64 defect.
//
// GB300 issues two FP64 operations per clock and SM, so the FFT form of the
// product (about 78 FP64 instructions per value at M = 1024) keeps that pipe
// busy and cannot run faster.  Here both factors are cut into eight slices of
// eight bits and multiplied as integers on tcgen05.mma (kind::f16), the
// error-free splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59,
// 2012) on fp16 tensor cores as in Mukunoki, Ozaki, Ogita and Imamura (ISC 2020):
//   b = 2^(E-6) sum_j B_j 2^(-8j),  k = 2^(F-6) sum_i K_i 2^(-8i),  i, j = 0..7,
// with balanced digits of at most 128 (64 for the leading one), exact in fp16,
// E and F the exponents of the largest |b| of the line and |k| of the column.
// s_p, the sum of the products with i + j = p for p = 0..7, is an FP32
// accumulator of integers; a segment of the sum is as long as keeps it within
// 2^24 for any b (bounded at set-up with the column's own digits), so every s_p is
// exact.  Segments are added in two 64-bit integers per
// value and the total is rounded to FP64 once.  What is dropped, the products
// with i + j > 7, is about 2^-59 (largest |k|) (largest |b|); the half-sweep's
// error against 64-bit sums is that of the final rounding (about 1e-16 of the
// line's scale; the FFT form's is 2e-16 to 4e-16).
//
// Two kernels per half-sweep:
//  k_toep_gather  forms b (FP64), the line's exponent and the eight digits,
//                 written as fp16 in the layout the MMA reads (16 bytes a value);
//  k_toep_mma     one CTA per SM.  An item is NL lines x 128 output steps: the
//                 MMA's 128 rows are output steps, its columns the lines, once
//                 per order p = i + j.  The orders 0 .. 3 and 4 .. 7 are an
//                 accumulator each: one instruction multiplies slice i of the
//                 column with the slices j = p - i of the lines for the four
//                 orders of an accumulator (N = 4 NL; slices j < 0 are a pad of
//                 zeros before the lines' slices).
// The PTX ISA orders two tcgen05.mma only where both have the same accumulator and
// the same shape (and come from one thread); others may overlap and lose a sum.  So
// every MMA of an accumulator has one shape and one issuing thread.  The zeros cost
// 48 blocks of four orders where the triangle i + j <= 7 has 36.
// Because the time index of a chunk of 32 steps is stored reversed, element
// (row, kk) of the Toeplitz operand depends on row + kk only, so its 8 x 8 core
// matrices depend on one index and all blocks of all lags are windows into one
// array of M/8 + 15 cores per slice (leading and stride byte offsets both 128
// bytes): the whole operand (143 KB at M = 1024) stays in shared memory.
// Far from the diagonal k is small and its leading digits vanish; the first
// slice that is not zero from a lag on is recorded per 64 lags at set-up, and
// the slices before it are neither loaded nor multiplied (on a fine level about
// half the products remain).
// Lines are processed in slabs, which bounds the digits' memory.
//
// Warp roles in k_toep_mma: warps 0-15 fold and store (tcgen05.ld), warp 16 loads
// chunks of digits by bulk copies into a ring, warps 17 and 18 issue the MMAs; the
// accumulator is double-buffered (2 x 8 NL columns).  Every wait is bounded.
//
// Measured (2-D, finest half-sweep, alpha = 0.5; 255 x 255, M = 1024): FFT form
// 4.8 ms; k_toep_gather 0.27 ms (0.22 ms of it FP64 sums at the pipe's rate) and
// k_toep_mma 0.74 ms, bound by its MMAs (tensor pipe 69 % of the active clocks, each
// reading as many clocks of shared memory as it multiplies) and by folding (seven
// conversions a value and segment at a quarter of the rate, tcgen05.ld latency).  With
// MMAs of eight widths, which nothing keeps in order, it took 0.58 ms (63 %).  The ring's
// depth does not bound it: 2, 3, 4 and 8 stages 284, 270, 270 and 271 us for gather and
// products of 127 x 127 x 1024, 391, 378, 378, 381 us of 255 x 255 x 512.
//
// Where there are too few lines to fill the chip the product is a sum of FP64
// products (k_toep_direct): one launch, 4.5 us for one line of 512 steps (FFT form
// 26 us, the tensor-core pair 21 us).
#include <cuda_fp16.h>

#include <climits>

#include "mgwr_common.cuh"
#include "mgwr_tma.cuh"

namespace mgwr {

namespace {

constexpr int kSlices = 8;
constexpr int kTile = 128;     // output steps of an item: the MMA's M
constexpr int kChunk = 32;     // time steps per shared-memory chunk (two K = 16 steps)
constexpr int kMaxStages = 8;  // chunks in flight, as many as shared memory holds
constexpr int kFoldThreads = 512;
constexpr int kLoader = 512, kIssuer = 544;  // first threads of warps 16 and 17
constexpr int kOrders = 4;                    // orders of an accumulator
constexpr int kIssuers = kSlices / kOrders;   // one warp per accumulator
constexpr int kThreads = kIssuer + 32 * kIssuers;

__host__ __device__ constexpr int cores(int M) { return (M < kTile ? kTile : M) / 8 + 15; }
__host__ __device__ constexpr size_t slice_bytes(int M) { return (size_t)cores(M) * 128; }
// band blob: the slices, then BandHead
__host__ __device__ constexpr size_t blob_bytes(int M) { return kSlices * slice_bytes(M) + 32; }

struct BandHead {
  unsigned long long first;
  int F;
  short shift;   // low bits dropped when the two sums are joined: |y| < 2^(62 + shift) units
  short chunks;  // chunks from the diagonal down that have a nonzero slice
  unsigned starts;  // bit c: a segment starts with chunk c
  unsigned pad;
};

__device__ __forceinline__ const BandHead* band_head(const unsigned char* blob, int M) {
  return reinterpret_cast<const BandHead*>(blob + kSlices * slice_bytes(M));
}

// Chunk c of tile tau holds the 32 steps from s0 = 128 tau + 96 - 32 c (M >= 128;
// M - 32 - 32 c below): c counts from the diagonal down.
__device__ __forceinline__ int tile_chunks(int M, int tau) {
  return M < kTile ? M / kChunk : 4 * tau + 4;
}
__host__ __device__ __forceinline__ int chunk_lag0(int M, int c) {  // t0 - s0
  return kChunk * c - (M < kTile ? M - kChunk : kTile - kChunk);
}
// smallest lag that chunks 2 x and 2 x + 1 multiply
__device__ __forceinline__ int pair_lag(int M, int x) {
  const int lag = chunk_lag0(M, 2 * x) - (kChunk - 1);
  return lag > 0 ? lag : 0;
}
// first core of chunk c's window
__device__ __forceinline__ int chunk_core(int M, int c) { return (chunk_lag0(M, c) + 96) / 8; }
// first nonzero slice of chunk c
__device__ __forceinline__ int first_slice(unsigned long long first, int c) {
  return (int)(first >> (4 * (c >> 1))) & 15;
}
// the chunk after the segment that starts with chunk c
__device__ __forceinline__ int segment_end(unsigned starts, int c, int nc) {
  const unsigned later = c + 1 < 32 ? starts >> (c + 1) : 0u;
  const int end = later != 0 ? c + __ffs((int)later) : nc;
  return end < nc ? end : nc;
}

// exponent field of |x| (1 for zero and subnormals, 2047 for inf and NaN)
__device__ __forceinline__ int exp_field(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7FF;
  return e > 0 ? e : 1;
}

// The digits of x against the largest exponent field ef of its line: the
// integer q = x 2^(62 - (ef - 1022)), |q| < 2^62 (bits below it rounded), plus 128
// in every byte: byte j (from the low end) minus 128 is digit 7 - j.
__device__ __forceinline__ unsigned long long biased_digits(double x, int ef) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e0 = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if (e0 > 0) m |= 1ull << 52;
  int r = ef - (e0 > 0 ? e0 : 1);  // right shift of m 2^9
  r = r > 63 ? 63 : r;
  const unsigned long long q = ((m << 9) + ((1ull << r) >> 1)) >> r;
  const unsigned long long s = (b >> 63) ? 0ull - q : q;
  return s + 0x8080808080808080ull;
}

// Two values' digits of one byte position as fp16 pairs (x low, y high).
__device__ __forceinline__ unsigned digit_pair(unsigned x, unsigned y, unsigned sel) {
  const unsigned t = (__byte_perm(x, y, sel) & 0x00FF00FFu) | 0x64006400u;  // 1024 + byte
  const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&t), __float2half2_rn(1152.f));
  return *reinterpret_cast<const unsigned*>(&v);
}

// ---- set-up ---------------------------------------------------------------------

// The band of one column (blockIdx.x): core g holds k[8g - 127 + r + c] at row
// r, column c, per slice; the first nonzero slice by lag; the exponent F.
__global__ void __launch_bounds__(256)
    k_toep_band(const double* __restrict__ cols, unsigned char* __restrict__ blob, int M) {
  __shared__ short dig[kSlices][1024];
  __shared__ int s_ef, s_last[kSlices];
  __shared__ double s_sum[8];
  // per chunk: most that one step's digits add to |s_7| and, less, to |s_2|
  __shared__ int s_prefix[1025], s_scan[8], s_all[32], s_top[32];
  const double* k = cols + (size_t)blockIdx.x * M;
  unsigned char* out = blob + (size_t)blockIdx.x * blob_bytes(M);
  if (threadIdx.x == 0) s_ef = 1;
  if (threadIdx.x < kSlices) s_last[threadIdx.x] = -1;
  __syncthreads();
  int ef = 1;
  for (int m = threadIdx.x; m < M; m += 256) ef = max(ef, exp_field(k[m]));
  atomicMax(&s_ef, ef);
  __syncthreads();
  ef = s_ef;
  double sum = 0.0;
  for (int m = threadIdx.x; m < M; m += 256) {
    const unsigned long long q = biased_digits(k[m], ef);
    sum += fabs(k[m]);
#pragma unroll
    for (int i = 0; i < kSlices; ++i) {
      const int v = (int)((q >> (8 * (7 - i))) & 0xFF) - 128;
      dig[i][m] = (short)v;
      if (v != 0) atomicMax(&s_last[i], m);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  for (int x = threadIdx.x; x < kSlices * cores(M) * 64; x += 256) {
    const int i = x / (cores(M) * 64), rest = x - i * cores(M) * 64;
    const int g = rest >> 6, r = (rest >> 3) & 7, c = rest & 7;
    const int lag = 8 * g - 127 + r + c;
    const int v = lag >= 0 && lag < M ? dig[i][lag] : 0;
    *reinterpret_cast<__half*>(out + i * slice_bytes(M) + g * 128 + r * 16 + c * 2) =
        __int2half_rn(v);
  }
  // A chunk adds to |s_7| at most sum_{i < 7} 128 W_i + 64 W_7 (the leading digit of b
  // is at most 64) and to |s_2| at most 128 (W_0 + W_1) + 64 W_2, W_i the largest sum
  // of the 32 consecutive |K_i| that a row of its window multiplies.
  const int chunks = M / kChunk;
  if (threadIdx.x < 32) s_all[threadIdx.x] = s_top[threadIdx.x] = 0;
  for (int i = 0; i < kSlices; ++i) {
    __syncthreads();
    int own[4], acc = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int m = 4 * threadIdx.x + q;
      acc += m < M ? abs((int)dig[i][m]) : 0;
      own[q] = acc;
    }
    int incl = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if ((threadIdx.x & 31) >= o) incl += up;
    }
    if ((threadIdx.x & 31) == 31) s_scan[threadIdx.x >> 5] = incl;
    __syncthreads();
    int before = incl - acc;
    for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += s_scan[w];
    if (threadIdx.x == 0) s_prefix[0] = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * threadIdx.x + q < M) s_prefix[4 * threadIdx.x + q + 1] = before + own[q];
    __syncthreads();
    // eight threads per chunk; row r multiplies lags chunk_lag0 - 31 + r .. chunk_lag0 + r
    const int c = threadIdx.x >> 3;
    int most = 0;
    if (c < chunks)
      for (int r = threadIdx.x & 7; r < kTile; r += 8) {
        const int hi = min(M, max(0, chunk_lag0(M, c) + r + 1));
        const int lo = min(M, max(0, chunk_lag0(M, c) + r + 1 - kChunk));
        most = max(most, s_prefix[hi] - s_prefix[lo]);
      }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    if (c < chunks && (threadIdx.x & 7) == 0) {
      s_all[c] += most * (i == kSlices - 1 ? 64 : 128);
      if (i < 3) s_top[c] += most * (i == 2 ? 64 : 128);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long first = 0;
    const int pairs = M < kTile ? 1 : M / kChunk / 2;
    for (int x = 0; x < pairs; ++x) {
      int i = 0;
      while (i < kSlices && s_last[i] < pair_lag(M, x)) ++i;
      if (pair_lag(M, x) == 0) i = 0;  // the diagonal always runs (a zero column gives zeros)
      first |= (unsigned long long)i << (4 * x);
    }
    // |y| <= |k|_1 2^E = 2^(E + F) 2^g, in units of 2^(E + F - 68): 2^(68 + g)
    double total = 0.0;
    for (int w = 0; w < 8; ++w) total += s_sum[w];
    const int g = exp_field(total) - ef + 2;
    BandHead* h = reinterpret_cast<BandHead*>(out + kSlices * slice_bytes(M));
    h->first = first;
    h->F = ef - 1022;
    h->shift = (short)(6 + (g < 1 ? 1 : g > 20 ? 20 : g));
    int live = 0;
    while (live < pairs && first_slice(first, 2 * live) < kSlices) ++live;
    h->chunks = (short)(2 * live);
    // segments: within 2^24 for every order, and 256 |s_2| + |s_3| within 2^31
    unsigned starts = 1;
    int all = 0, top = 0;
    for (int c = 0; c < chunks; ++c) {
      if (c > 0 && (all + s_all[c] > (1 << 24) || top + s_top[c] > 8000000)) {
        starts |= 1u << c;
        all = top = 0;
      }
      all += s_all[c];
      top += s_top[c];
    }
    h->starts = starts;
    h->pad = 0;
  }
}

// ---- gather ---------------------------------------------------------------------

struct Geometry {
  int d, n, M, par, npts;  // npts: lines of the colour (par < 0: of the grid) per instance
  int per_inst;            // groups of NL lines per instance
  int group0, groups;      // the slab: groups group0 .. group0 + groups - 1 of all instances
  size_t fstride;          // values of one instance's field
  size_t bstride;          // bytes from one instance's band to the next
  bool zero_u;             // u is zero: no neighbour sums
};

// the k-th line of a launch
__device__ __forceinline__ int launch_point(const Geometry& G, int k, int& i, int& j) {
  if (G.par >= 0) return colour_point(k, G.d, G.n, G.par, i, j);
  return k;  // every point; its place in the grid is not needed
}

// b of steps m .. m + W - 1 of point p (line start `base`, neighbours by flag).
template <int W>
__device__ __forceinline__ void gather_steps(const double* __restrict__ f,
                                             const double* __restrict__ u, size_t at, size_t M,
                                             size_t nM, bool w, bool e, bool s, bool t,
                                             double hinv2, double (&b)[W]) {
  double a[W];
#pragma unroll
  for (int q = 0; q < W; q += 2) {
    const double2 x =
        w ? __ldg(reinterpret_cast<const double2*>(u + at - M + q)) : make_double2(0.0, 0.0);
    a[q] = x.x;
    a[q + 1] = x.y;
  }
  auto add = [&](const double* src) {
#pragma unroll
    for (int q = 0; q < W; q += 2) {
      const double2 x = __ldg(reinterpret_cast<const double2*>(src + q));
      a[q] += x.x;
      a[q + 1] += x.y;
    }
  };
  if (e) add(u + at + M);
  if (s) add(u + at - nM);
  if (t) add(u + at + nM);
#pragma unroll
  for (int q = 0; q < W; q += 2) {
    const double2 x = __ldg(reinterpret_cast<const double2*>(f + at + q));
    b[q] = fma(hinv2, a[q], x.x);
    b[q + 1] = fma(hinv2, a[q + 1], x.y);
  }
}

// One block per LPB lines: thread t holds line t % LPB, the octet t / LPB of its
// steps.  LPB = 4 or 8 writes whole 32-byte sectors; small grids take fewer lines
// per block, so that the FP64 sums of a line (four operations a value, two a clock
// and SM: what bounds this kernel) spread over the SMs.
// PLAIN: b is the line of f itself (the defect's time term of a field).
template <int NL, int LPB, bool PLAIN>
__global__ void __launch_bounds__(512, 3)
    k_toep_gather(const double* __restrict__ f, const double* __restrict__ u,
                  const unsigned char* __restrict__ band, unsigned char* __restrict__ dig,
                  int* __restrict__ lexp, Geometry G, double hinv2) {
  __shared__ int red[16][LPB];
  const int T = blockDim.x;
  const int g = blockIdx.x / (NL / LPB);
  const int inst = (G.group0 + g) / G.per_inst;
  const int x = threadIdx.x % LPB;
  const int line = (blockIdx.x - g * (NL / LPB)) * LPB + x;  // of the group
  const int k = (G.group0 + g - inst * G.per_inst) * NL + line;
  const int M = G.M;
  double b[8];
  int ef = 1;
  if (k < G.npts) {
    int i = 0, j = 0;
    const int p = launch_point(G, k, i, j);
    const size_t base = inst * G.fstride + (size_t)p * M;
    const bool sums = !PLAIN && !G.zero_u;
    gather_steps<8>(f, u, base + 8 * (threadIdx.x / LPB), M, (size_t)G.n * M, sums && i > 0,
                    sums && i < G.n - 1, sums && G.d == 2 && j > 0,
                    sums && G.d == 2 && j < G.n - 1, hinv2, b);
#pragma unroll
    for (int q = 0; q < 8; ++q) ef = max(ef, exp_field(b[q]));
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) b[q] = 0.0;
  }
  // the line's largest exponent: lanes of equal line, then the block's warps
#pragma unroll
  for (int o = LPB; o < 32; o <<= 1) ef = max(ef, __shfl_xor_sync(0xffffffffu, ef, o));
  if ((threadIdx.x & 31) < LPB) red[threadIdx.x >> 5][x] = ef;
  __syncthreads();
  for (int w = 0; w < (T >> 5); ++w) ef = max(ef, red[w][x]);
  if (threadIdx.x < LPB) {
    const BandHead* h = band_head(band + inst * G.bstride, M);
    // exponent of one unit of the joined sums (INT_MIN: infinities or NaN in the line)
    lexp[g * NL + line] = ef == 2047 ? INT_MIN : ef - 1022 + h->F - 68 + h->shift;
  }
  unsigned lo[8], hi[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const unsigned long long z = biased_digits(b[q], ef);
    lo[q] = (unsigned)z;
    hi[q] = (unsigned)(z >> 32);
  }
  // chunk oct / 4; steps reversed within it: core 3 - oct % 4, column 7 - q
  const int oct = threadIdx.x / LPB;
  unsigned char* out = dig + ((size_t)g * (M / kChunk) + (oct >> 2)) * kSlices * NL * 64 +
                       (line >> 3) * 512 + (3 - (oct & 3)) * 128 + (line & 7) * 16;
#pragma unroll
  for (int j = 0; j < kSlices; ++j) {
    const unsigned sel =
        (j & 3) == 0 ? 0x0703u : (j & 3) == 1 ? 0x0602u : (j & 3) == 2 ? 0x0501u : 0x0400u;
    unsigned v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)  // columns 2c and 2c + 1
      v[c] = j < 4 ? digit_pair(hi[7 - 2 * c], hi[6 - 2 * c], sel)
                   : digit_pair(lo[7 - 2 * c], lo[6 - 2 * c], sel);
    *reinterpret_cast<uint4*>(out + j * NL * 64) = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

// Few lines: the product as FP64 sums.  A block holds OB output steps of one
// line from its end and OB from its start (so all blocks sum the same number of
// terms); a warp's lanes are the steps (and 32 / OB phases of the sum), its eight
// warps share the sum, and b up to the last step is in shared memory.  FP64 issue
// bounds it (two operations a clock and SM).  With the lanes of a step reducing by
// shuffles, and one tile a block, the reductions took as much of the pipe as the
// products: 16 lines of 512 steps 13.6 us, now 7.7 us; 25 lines 16.6, now 11.6 us.
template <int OB>
__global__ void __launch_bounds__(256)
    k_toep_direct(const double* __restrict__ f, double* __restrict__ u, double* __restrict__ delta,
                  const double* __restrict__ cols, size_t cstride, Geometry G, double hinv2) {
  constexpr int kTerms = 256 / OB;  // terms of the sums that the block takes at a time
  __shared__ double sb[1024], sk[1024], part[512];
  const int M = G.M;
  const int inst = blockIdx.x / G.npts;
  const int k = blockIdx.x - inst * G.npts;
  int i = 0, j = 0;
  const int p = colour_point(k, G.d, G.n, G.par, i, j);
  const size_t base = inst * G.fstride + (size_t)p * M;
  const int first[2] = {M - OB - (int)blockIdx.y * OB, (int)blockIdx.y * OB};
  cols += inst * cstride;
  for (int m = 2 * threadIdx.x; m < first[0] + OB; m += 512) {
    double b[2];
    gather_steps<2>(f, u, base + m, M, (size_t)G.n * M, i > 0 && !G.zero_u,
                    i < G.n - 1 && !G.zero_u, G.d == 2 && j > 0 && !G.zero_u,
                    G.d == 2 && j < G.n - 1 && !G.zero_u, hinv2, b);
    sb[m] = b[0];
    sb[m + 1] = b[1];
    const double2 c = __ldg(reinterpret_cast<const double2*>(cols + m));
    sk[m] = c.x;
    sk[m + 1] = c.y;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int t0 = first[h], t = t0 + threadIdx.x % OB;
    double a[2] = {0.0, 0.0};
    int s = threadIdx.x / OB;
#pragma unroll 2
    for (; s + kTerms < t0; s += 2 * kTerms) {
      a[0] = fma(sk[t - s], sb[s], a[0]);
      a[1] = fma(sk[t - s - kTerms], sb[s + kTerms], a[1]);
    }
    for (; s < t0 + OB; s += kTerms)
      if (s < t) a[0] = fma(sk[t - s], sb[s], a[0]);
    part[256 * h + threadIdx.x] = a[0] + a[1];
  }
  __syncthreads();
  if (threadIdx.x >= 64) return;
  const int lane = threadIdx.x & 31, h = threadIdx.x >> 5;
  const int t = (h == 0 ? first[0] : first[1]) + lane % OB;
  double y[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) y[w] = part[256 * h + 32 * w + lane];
#pragma unroll
  for (int x = 4; x > 0; x >>= 1)
#pragma unroll
    for (int w = 0; w < x; ++w) y[w] += y[w + x];
#pragma unroll
  for (int o = OB; o < 32; o <<= 1) y[0] += __shfl_xor_sync(0xffffffffu, y[0], o);
  y[0] = fma(sk[0], sb[t], y[0]);  // the largest product last
  if (lane < OB) {
    if (delta != nullptr) delta[base + t] = y[0] - u[base + t];
    u[base + t] = y[0];
  }
}

// ---- products ---------------------------------------------------------------------

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes; `lead`
// bytes to the next core along K, `stride` bytes to the next eight rows.
__device__ __forceinline__ uint64_t operand(unsigned addr, unsigned lead, unsigned stride) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)(lead >> 4) << 16 |
         (uint64_t)(stride >> 4) << 32 | (uint64_t)1 << 46;
}

// FP32 accumulator, fp16 A and B, both K-major, 128 rows, `n` columns.
__device__ __forceinline__ constexpr uint32_t mma_shape(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(unsigned tmem, uint64_t da, uint64_t db, uint32_t shape,
                                        unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(da), "l"(db), "r"(shape), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_load4(unsigned addr, unsigned (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr));
}

__device__ __forceinline__ void tmem_clear4(unsigned addr) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%1,%1,%1};" ::"r"(addr), "r"(0)
               : "memory");
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// A wait of the whole warp, its outcome uniform across the lanes.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, unsigned parity) {
  return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity) ? 1 : 0) != 0;
}

// The value of lane 0, uniform across the warp (the MMA's operands then live in
// uniform registers).
__device__ __forceinline__ unsigned uniform(unsigned x) { return __shfl_sync(0xffffffffu, x, 0); }

// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile(
      "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(p));
  return p != 0;
}

// hi 2^32 + 256 lo, less its last `shift` bits (|result| < 2^62), times 2^e, rounded
// once to FP64 (half away from zero) with integer operations only.
__device__ __forceinline__ double join(long long hi, long long lo, int shift, int e) {
  const long long v =
      (hi << (32 - shift)) + (shift > 8 ? ((lo >> (shift - 9)) + 1) >> 1 : lo << (8 - shift));
  if (e <= -1000 || e >= 900) {
    // INT_MIN: an infinity or NaN in the line, whose finite values have no digits left
    return e == INT_MIN ? __longlong_as_double(0x7FF8000000000000ll) : scalbn((double)v, e);
  }
  if (v == 0) return 0.0;
  const unsigned long long sign = (unsigned long long)v & 0x8000000000000000ull;
  const unsigned long long mag = (unsigned long long)(v < 0 ? -v : v);
  const int z = __clzll((long long)mag);
  const unsigned long long m = mag << z;  // leading bit at 63
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1);  // 53 bits, carrying into 2^53
  return __longlong_as_double(
      (long long)(sign | (((unsigned long long)(e + 63 - z + 1022) << 52) + r)));
}

// Work order of a CTA.  Many groups: a contiguous run of them, every tile of
// each (the band is reloaded only where the instance changes).  Few: items
// dealt one by one, the longest tiles first.
struct Items {
  int groups, tiles, dealt;
  __device__ __forceinline__ bool get(int it, int& g, int& tau) const {
    if (dealt) {
      const int x = blockIdx.x + it * gridDim.x;
      if (x >= groups * tiles) return false;
      const int q = x / groups;
      tau = tiles - 1 - q;
      g = x - q * groups;
      return true;
    }
    const int a = (int)((long long)groups * blockIdx.x / gridDim.x);
    const int b = (int)((long long)groups * (blockIdx.x + 1) / gridDim.x);
    g = a + it / tiles;
    tau = tiles - 1 - it % tiles;
    return g < b;
  }
};

// Zeros before a chunk's digits in shared memory: the slices j = p - i of an
// accumulator's orders run from -(kOrders - 1) (order 0 of slice kOrders - 1, order
// kOrders of slice 2 kOrders - 1) to kSlices - 1.
static_assert(kSlices == 2 * kOrders, "slices reach from -(kOrders - 1) to kSlices - 1");
__host__ __device__ constexpr int pad_bytes(int NL) { return (kOrders - 1) * NL * kChunk * 2; }

template <int NL>
__global__ void __launch_bounds__(kThreads, 1)
    k_toep_mma(double* __restrict__ u, double* __restrict__ delta,
               const unsigned char* __restrict__ band, const unsigned char* __restrict__ dig,
               const int* __restrict__ lexp, Geometry G, Items items, int stages,
               unsigned* __restrict__ gave_up) {
  constexpr int kCols = kSlices * NL;               // columns of the accumulators of a segment
  constexpr unsigned kTmem = 2 * kCols;             // 512 or 256
  constexpr int kStage = kCols * kChunk * 2;        // bytes of a chunk's digits
  constexpr int kPad = pad_bytes(NL);               // zeros before them: slices -3 .. -1
  constexpr int kSlot = kPad + kStage;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // band: full / empty; chunk ring: full / empty; accumulators: full / empty
  __shared__ __align__(8) uint64_t bars[2 + 2 * kMaxStages + 4];
  uint64_t* const band_full = bars;
  uint64_t* const band_empty = bars + 1;
  uint64_t* const full = bars + 2;
  uint64_t* const empty = full + kMaxStages;
  uint64_t* const acc_full = empty + kMaxStages;
  uint64_t* const acc_empty = acc_full + 2;
  __shared__ unsigned tmem_slot;
  const int M = G.M;
  unsigned char* const sBand = smem_raw;
  unsigned char* const sRing = smem_raw + kSlices * slice_bytes(M);

  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == kLoader) {
    mbar_init(band_full, 1);
    mbar_init(band_empty, kIssuers);
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kIssuers);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], kIssuers);
      mbar_init(&acc_empty[a], kFoldThreads / 32);
    }
    mbar_fence_init();
  }
  if (warp == kIssuer / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = tmem_slot;
  if (warp < kFoldThreads / 32) {
    const unsigned at = tmem + ((unsigned)(32 * (warp & 3)) << 16);
    for (int c = (warp >> 2) * 4; c < 2 * kCols; c += 16) tmem_clear4(at + (unsigned)c);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    tc_fence_before();
    for (int x = threadIdx.x; x < stages * (kPad / 16); x += kFoldThreads) {
      const int slot = x / (kPad / 16);
      *reinterpret_cast<uint4*>(sRing + slot * kSlot + (x - slot * (kPad / 16)) * 16) =
          make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
  }
  __syncthreads();
  tc_fence_after();
  bool ok = true;
  int g = 0, tau = 0;

  if (warp == kLoader / 32) {
    if (threadIdx.x == kLoader) {
      int cur = -1, bands = 0, chunks = 0, slot = 0, round = 0;
      for (int it = 0; ok && items.get(it, g, tau); ++it) {
        const int inst = (G.group0 + g) / G.per_inst;
        const unsigned char* blob = band + inst * G.bstride;
        if (inst != cur) {
          if (bands > 0) ok = mbar_wait_bounded(band_empty, (unsigned)((bands - 1) & 1));
          if (!ok) break;
          mbar_arrive_expect_tx(band_full, (unsigned)(kSlices * slice_bytes(M)));
          bulk_copy_g2s(sBand, blob, (unsigned)(kSlices * slice_bytes(M)), band_full);
          ++bands;
          cur = inst;
        }
        const unsigned long long first = band_head(blob, M)->first;
        const int tc = tile_chunks(M, tau);
        const int nc = min(tc, (int)band_head(blob, M)->chunks);
        // digits of the tile's last chunk (c = 0), then backwards in time
        const unsigned char* src = dig + ((size_t)g * (M / kChunk) + tc - 1) * kStage;
        for (int c = 0; c < nc; ++c, src -= kStage) {
          const int i0 = first_slice(first, c);
          if (round > 0) ok = mbar_wait_bounded(&empty[slot], (unsigned)((round - 1) & 1));
          if (!ok) break;
          const unsigned bytes = (unsigned)((kSlices - i0) * NL * kChunk * 2);
          mbar_arrive_expect_tx(&full[slot], bytes);
          bulk_copy_g2s(sRing + slot * kSlot + kPad, src, bytes, &full[slot]);
          ++chunks;
          if (++slot == stages) slot = 0, ++round;
        }
      }
      if (!ok) {
        // copies in flight land before the CTA can end
        if (bands > 0) (void)mbar_wait_bounded(band_full, (unsigned)((bands - 1) & 1));
        for (int x = chunks > stages ? chunks - stages : 0; x < chunks; ++x)
          (void)mbar_wait_bounded(&full[x % stages], (unsigned)((x / stages) & 1));
      }
    }
    __syncwarp();
  } else if (warp >= kIssuer / 32) {
    // Each issuer takes one accumulator, both K steps of every chunk (the order of an
    // accumulator's MMAs is its thread's; waits and bookkeeping of one warp for both
    // would leave the tensor cores idle).  Accumulators start at zero (cleared by the
    // warps that read them).  A whole warp walks the items (uniform control flow), one
    // lane issues.
    const bool lead = elect_one();
    const int half = warp - kIssuer / 32;
    const unsigned tmem_u = uniform(tmem);
    int cur = -1, bands = 0, seg = 0, slot = 0, round = 0, last = -1, last_round = 0;
    const unsigned sb = (unsigned)slice_bytes(M) >> 4;
    const uint64_t opA = operand(0, 128, 128) + (smem_u32(sBand) >> 4);
    // slice `kOrders half` of the first slot: the window of slice i = 0
    const uint64_t opB = operand(0, 128, 512) +
                         ((smem_u32(sRing) + (unsigned)(kPad + half * kOrders * NL * kChunk * 2)) >> 4);
    constexpr uint32_t kShape = mma_shape(kOrders * NL);
    constexpr unsigned kWindow = NL * kChunk * 2 / 16;  // one slice on, in 16-byte units
    for (int it = 0; ok && items.get(it, g, tau); ++it) {
      const int inst = (G.group0 + g) / G.per_inst;
      if (inst != cur) {
        if (cur >= 0 && lead) mma_commit(band_empty);  // when all products with the old band are done
        ok = warp_wait(band_full, (unsigned)(bands & 1));
        if (!ok) break;
        ++bands;
        cur = inst;
      }
      const BandHead* head = band_head(band + inst * G.bstride, M);
      const unsigned long long f64 = head->first;
      const unsigned long long first =
          (unsigned long long)uniform((unsigned)(f64 >> 32)) << 32 | uniform((unsigned)f64);
      const int nc = min(tile_chunks(M, tau), (int)uniform((unsigned)head->chunks));
      const unsigned starts = uniform(head->starts);
      for (int c = 0; ok && c < nc; ++seg) {
        const int end = segment_end(starts, c, nc);
        const int a = seg & 1;
        const unsigned dst = tmem_u + (unsigned)(a * kCols + half * kOrders * NL);
        if (seg >= 2) ok = warp_wait(&acc_empty[a], (unsigned)((seg / 2 - 1) & 1));
        for (; ok && c < end; ++c) {
          ok = warp_wait(&full[slot], (unsigned)(round & 1));
          if (!ok) break;
          tc_fence_after();
          if (lead) {
            const int i0 = first_slice(first, c);
            const uint64_t da = opA + (unsigned)chunk_core(M, c) * 8;
            const uint64_t db = opB + (unsigned)slot * (kSlot / 16);
#pragma unroll
            for (int k = 0; k < kChunk / 16; ++k)  // 16 steps: two cores of either operand
#pragma unroll
              for (int i = 0; i < kSlices; ++i)
                if (i >= i0 && i < kOrders * (half + 1))
                  mma_f16(dst, da + (uint64_t)(i * sb + k * 16), db - (uint64_t)(i * kWindow) + k * 16,
                          kShape, 1u);
            mma_commit(&empty[slot]);
            if (c + 1 == end) mma_commit(&acc_full[a]);
          }
          __syncwarp();
          last = slot;
          last_round = round;
          if (++slot == stages) slot = 0, ++round;
        }
      }
    }
    // after a failure, what was issued finishes before the accumulators are released
    if (!ok && last >= 0) (void)mbar_wait_bounded(&empty[last], (unsigned)(last_round & 1));
  } else {
    // warp w: steps 32 (w % 4) .. +31 of the tile, lines of quarter w / 4
    constexpr int kMine = NL / 4;
    const int lane = threadIdx.x & 31;
    const int mine = (warp >> 2) * kMine;
    const unsigned lane_row = (unsigned)(32 * (warp & 3)) << 16;
    int seg = 0;
    for (int it = 0; ok && items.get(it, g, tau); ++it) {
      const int inst = (G.group0 + g) / G.per_inst;
      const BandHead* head = band_head(band + inst * G.bstride, M);
      const unsigned long long first = head->first;
      const int shift = head->shift;
      const unsigned starts = head->starts;
      const int nc = min(tile_chunks(M, tau), (int)head->chunks);
      // lane x holds the point and exponent of line x of this quarter
      const int k = (G.group0 + g - inst * G.per_inst) * NL + mine + (lane & (kMine - 1));
      int p = -1, e = 0;
      if (k < G.npts) {
        int i = 0, j = 0;
        p = launch_point(G, k, i, j);
        e = lexp[g * NL + mine + (lane & (kMine - 1))];
      }
      long long hi[kMine], lo[kMine];
#pragma unroll
      for (int x = 0; x < kMine; ++x) hi[x] = lo[x] = 0;
      for (int c = 0; c < nc;) {
        const int i0 = first_slice(first, c);
        const int a = seg & 1;
        ok = warp_wait(&acc_full[a], (unsigned)((seg / 2) & 1));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int x0 = 0; x0 < kMine; x0 += 4) {
          unsigned v[kSlices][4];
#pragma unroll
          for (int p = 0; p < kSlices; ++p) {
            if (p >= i0) {
              tmem_load4(tmem + lane_row + (unsigned)(a * kCols + p * NL + mine + x0), v[p]);
            } else {
#pragma unroll
              for (int x = 0; x < 4; ++x) v[p][x] = 0u;
            }
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int p = 0; p < kSlices; ++p)
            if (p >= i0) tmem_clear4(tmem + lane_row + (unsigned)(a * kCols + p * NL + mine + x0));
          // s_0 .. s_3 into hi (|256 s_0 + s_1|, |256 s_2 + s_3| < 2^31), the rest into lo
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            auto s = [&](int p) { return __float2int_rn(__uint_as_float(v[p][x])); };
            long long& h = hi[x0 + x];
            long long& l = lo[x0 + x];
            if (i0 < 4) {
              h = mad_wide(s(0) * 256 + s(1), 65536, h);
              h = mad_wide(s(2) * 256 + s(3), 1, h);
            }
            // s_6 + s_7 / 256 to the nearest integer: 2^-61 of (largest |k|) (largest |b|)
            const int s67 = __float2int_rn(
                fmaf(__uint_as_float(v[7][x]), 0.00390625f, __uint_as_float(v[6][x])));
            l = mad_wide(s(4), 65536, l);
            l = mad_wide(s(5), 256, l);
            l = mad_wide(s67, 1, l);
          }
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[a]);
        ++seg;
        c = segment_end(starts, c, nc);
      }
      if (!ok) break;
      const int t = kTile * tau + 32 * (warp & 3) + lane;
#pragma unroll
      for (int x = 0; x < kMine; ++x) {
        const int px = __shfl_sync(0xffffffffu, p, x);
        const int ex = __shfl_sync(0xffffffffu, e, x);
        if (px < 0 || t >= M) continue;
        const double y = join(hi[x], lo[x], shift, ex);
        const size_t at = inst * G.fstride + (size_t)px * M + t;
        if (delta != nullptr) delta[at] = y - u[at];
        u[at] = y;
      }
    }
  }
  if (!ok) atomicOr(gave_up, kGaveUpToep);
  tc_fence_before();
  __syncthreads();
  if (warp == kIssuer / 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem)
                 : "memory");
}

// Bytes of a slab's digits.  Both kernels are bound by arithmetic, so writing the digits
// to HBM and reading them back costs nothing, while every slab leaves SMs idle at the
// end of two launches: 255 x 255 x 1024 solves with slabs of 32, 64, 128, 256 and 600 MB
// (the last: one slab) took 101, 87, 82.3, 79.2 and 78.8 ms (products at 0.58 of the 0.74
// ms a half-sweep they take now).
constexpr size_t kSlabBytes = size_t(256) << 20;
constexpr size_t kLineValue = 2 * kSlices;  // bytes of digits per value

// Lines per group: 32, or 16 while that leaves SMs without an item.
int lines_per_group(int M, int npts, int batch) {
  const long long items = (long long)((npts + 31) / 32) * batch * ((M + kTile - 1) / kTile);
  return items >= sm_count() ? 32 : 16;
}

// Lines of a slab: a colour of every instance (a defect, on all points, takes two
// slabs), at most kSlabBytes of digits.
size_t slab_lines(int M, int d, int n, int batch) {
  const size_t pts = (size_t)(d == 1 ? n : n * n);
  const size_t lines = ((pts + 1) / 2 + 31) / 32 * 32 * batch;
  const size_t most = kSlabBytes / ((size_t)M * kLineValue);
  return lines < most ? lines : most;
}

// Groups per slab of equal slabs.
int slab_groups(const Geometry& G, int batch, int NL, int groups) {
  const int most = (int)(slab_lines(G.M, G.d, G.n, batch) / NL);
  const int slabs = (groups + most - 1) / most;
  return (groups + slabs - 1) / slabs;
}

template <int NL, bool PLAIN>
cudaError_t gather_launch(const double* f, const double* u, const unsigned char* band,
                          unsigned char* dig, int* lexp, const Geometry& G, double hinv2,
                          cudaStream_t s) {
  const int M = G.M;
#define MGWR_GATHER(LPB)                                                                  \
  k_toep_gather<NL, LPB, PLAIN><<<(unsigned)(G.groups * (NL / LPB)), LPB * M / 8, 0, s>>>( \
      f, u, band, dig, lexp, G, hinv2)
  if (M >= 256 && G.groups * (NL / 4) < 2 * sm_count()) {
    MGWR_GATHER(1);
  } else if (M == 128 && G.groups * (NL / 8) < 2 * sm_count()) {
    MGWR_GATHER(2);
  } else if (M >= 512 || (M == 64 && G.groups * (NL / 8) < 2 * sm_count())) {
    MGWR_GATHER(4);
  } else {
    MGWR_GATHER(8);
  }
#undef MGWR_GATHER
  return counted(cudaGetLastError());
}

template <int NL>
cudaError_t slab_launch(const double* f, double* u, double* delta, const unsigned char* band,
                        unsigned char* scratch, const Geometry& G, double hinv2, unsigned* gave_up,
                        cudaStream_t s) {
  const int M = G.M;
  unsigned char* dig = scratch;
  int* lexp = reinterpret_cast<int*>(scratch + (size_t)G.groups * NL * M * kLineValue);
  cudaError_t e = G.par >= 0 ? gather_launch<NL, false>(f, u, band, dig, lexp, G, hinv2, s)
                             : gather_launch<NL, true>(f, u, band, dig, lexp, G, hinv2, s);
  if (e != cudaSuccess) return e;
  Items items;
  items.groups = G.groups;
  items.tiles = (M + kTile - 1) / kTile;
  items.dealt = G.groups < 4 * sm_count();
  const long long count = items.dealt ? (long long)G.groups * items.tiles : G.groups;
  const unsigned grid = (unsigned)(count < sm_count() ? count : sm_count());
  constexpr size_t kSlot = (size_t)pad_bytes(NL) + (size_t)kSlices * NL * kChunk * 2;
  const size_t band_bytes = kSlices * slice_bytes(M);
  int stages = (int)((226 * 1024 - band_bytes) / kSlot);
  if (stages > kMaxStages) stages = kMaxStages;
  // at least half the SM's shared memory and one byte: one CTA per SM, whose
  // accumulators take its tensor memory (NL = 32)
  size_t smem = band_bytes + stages * kSlot;
  if (smem < 116 * 1024) smem = 116 * 1024;
  e = prepare_smem(k_toep_mma<NL>, smem);
  if (e != cudaSuccess) return e;
  k_toep_mma<NL><<<grid, kThreads, smem, s>>>(u, delta, band, dig, lexp, G, items, stages,
                                             gave_up);
  return counted(cudaGetLastError());
}

// Few lines: the FP64 sums (about 4 us + 2 us a million multiply-adds) instead of
// the tensor-core pair (14.0, 15.5, 17.3, 21.5 and 29.5 us at M = 64 .. 1024 for any
// grid up to one item per SM, and a second launch).  Measured, sums against pair
// without that launch: M = 64, 1023 lines (2.1 M) 11.8 / 14.0 us; M = 128, 255 lines
// (2.1 M) 11.5 / 15.5; M = 256, 127 lines (4.2 M) 16.4 / 17.3; M = 512, 31 lines
// (4.1 M) 13.2 / 21.4, 64 lines (8.4 M) 22.7 / 21.7; M = 1024, 15 lines (7.9 M) 22.1 /
// 30.2, 32 lines 40 / 30.2.
bool few_lines(long long lines, int M) {
  return lines * M * M / 2 <= (1ll << 21) + (1ll << 13) * M;
}

// Groups of lines of a launch over all instances (an instance's last group is padded).
long long line_groups(int npts, int batch, int M) {
  const int NL = lines_per_group(M, npts, batch);
  return (long long)((npts + NL - 1) / NL) * batch;
}

// Batches of few lines an instance and 512 or 1024 steps: the pair's groups are mostly
// padding (every instance has a column of its own), the transform takes one block per
// 1024 / M line pairs.  Measured, us, pair / transform: M = 1024, one line each of 64,
// 512, 4096 instances 99 / 48, 559 / 167, 4460 / 1078; three lines 94 / 49, 536 / 296,
// 4271 / 2224; five of 512 552 / 470; seven of 512 and 4096 535 / 586, 4276 / 4456;
// M = 512, one to three lines of 64, 512, 4096 46 / 28, 195 / 160, 1325 / 1049; seven
// of 512 195 / 280; M = 256 and below the pair throughout (one line of 512 84 / 131).
bool transform_pays(int npts, int batch, int M) {
  if (M < 512) return false;
  const long long pairs = (npts + 1) / 2, per_block = 1024 / M;
  const long long blocks = (pairs + per_block - 1) / per_block * batch;
  // hundredths of us
  const long long pair = 2000 + line_groups(npts, batch, M) * (M == 1024 ? 104 : 32);
  const long long least = M == 1024 ? 4800 : 2700;
  const long long transform = (M == 1024 ? 2000 : 1200) + 28 * blocks;
  return pair > (transform > least ? transform : least);
}

// Steps per tile of the FP64 sums: the one whose rounds of blocks (one per SM) take
// least, a block costing its tile's sums and about five steps' worth for the rest
// (M = 512, tiles of 8, 16, 32: 4 lines 4.7, 5.6, 7.6 us; 8 lines 6.3, 5.7, 7.6;
// 16 lines 10.3, 8.4, 7.7; 25 lines 14.1, 11.6, 12.6).
int direct_tile(long long lines, int M) {
  int best = 0;
  long long least = 0;
  for (int tile = 8; tile <= 32; tile *= 2) {
    const long long rounds = (lines * (M / (2 * tile)) + sm_count() - 1) / sm_count();
    const long long cost = rounds * (tile + 5);
    if (best == 0 || cost < least) {
      best = tile;
      least = cost;
    }
  }
  return best;
}

// Every line of a launch, in slabs of groups.
cudaError_t product(const double* f, double* u, double* delta, const unsigned char* band,
                    unsigned char* scratch, Geometry G, int batch, double hinv2, unsigned* gave_up,
                    cudaStream_t s) {
  const int NL = lines_per_group(G.M, G.npts, batch);
  G.per_inst = (G.npts + NL - 1) / NL;
  const int total = G.per_inst * batch;
  const int step = slab_groups(G, batch, NL, total);
  for (int g0 = 0; g0 < total; g0 += step) {
    G.group0 = g0;
    G.groups = total - g0 < step ? total - g0 : step;
    const cudaError_t e =
        NL == 32 ? slab_launch<32>(f, u, delta, band, scratch, G, hinv2, gave_up, s)
                 : slab_launch<16>(f, u, delta, band, scratch, G, hinv2, gave_up, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// r = f - r - h^-2 sum (u_p - u_q), r holding T_M u; every difference formed before the
// sum.  A group of threads per line, 16-byte accesses.  Nine FP64 operations a value
// bound it (66.6 million values: 1.0 ms of the pipe).
__global__ void __launch_bounds__(256)
    k_defect_finish(const double* __restrict__ u, const double* __restrict__ f,
                    double* __restrict__ r, int d, int n, int M, int log_tpl, int npts,
                    double hinv2, unsigned long long* __restrict__ norm_bits, size_t fstride) {
  __shared__ double red[8];
  const int tpl = 1 << log_tpl;
  const int p = blockIdx.x * (256 >> log_tpl) + (threadIdx.x >> log_tpl);
  u += blockIdx.y * fstride;
  f += blockIdx.y * fstride;
  r += blockIdx.y * fstride;
  double amax = 0.0;
  if (p < npts) {
    const int i = d == 1 ? p : p % n, j = d == 1 ? 0 : p / n;
    const bool w = i > 0, e = i < n - 1, s = d == 2 && j > 0, t = d == 2 && j < n - 1;
    const size_t nM = (size_t)n * M;
    auto ld = [](const double* q) { return *reinterpret_cast<const double2*>(q); };
    for (int m = 2 * (threadIdx.x & (tpl - 1)); m < M; m += 2 * tpl) {
      const size_t at = (size_t)p * M + m;
      const double2 c = ld(u + at), fv = ld(f + at), y = ld(r + at);
      const double2 z = make_double2(0.0, 0.0);
      const double2 qw = w ? ld(u + at - M) : z, qe = e ? ld(u + at + M) : z;
      double2 sum = make_double2((c.x - qw.x) + (c.x - qe.x), (c.y - qw.y) + (c.y - qe.y));
      if (d == 2) {
        const double2 qs = s ? ld(u + at - nM) : z, qt = t ? ld(u + at + nM) : z;
        sum.x += (c.x - qs.x) + (c.x - qt.x);
        sum.y += (c.y - qs.y) + (c.y - qt.y);
      }
      const double2 out = make_double2((fv.x - y.x) - hinv2 * sum.x, (fv.y - y.y) - hinv2 * sum.y);
      *reinterpret_cast<double2*>(r + at) = out;
      amax = absmax_nan(fabs(out.x), absmax_nan(fabs(out.y), amax));
    }
  }
  if (norm_bits == nullptr) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = absmax_nan(__shfl_xor_sync(0xffffffffu, amax, o), amax);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int x = 1; x < 8; ++x) amax = absmax_nan(red[x], amax);
    atomic_max_nonneg(norm_bits + blockIdx.y, amax);
  }
}

}  // namespace

size_t toep_band_bytes(int M) { return blob_bytes(M); }

cudaError_t launch_toep_band(const double* cols, unsigned char* blob, int M, size_t lines,
                             cudaStream_t s) {
  k_toep_band<<<(unsigned)lines, 256, 0, s>>>(cols, blob, M);
  return counted(cudaGetLastError());
}

size_t toep_slab_bytes(int M) {
  return kSlabBytes / ((size_t)M * kLineValue) * ((size_t)M * kLineValue + sizeof(int));
}

size_t toep_scratch_bytes(const LevelShape& ls) {
  return slab_lines(ls.M, ls.d, ls.n, ls.batch) * ((size_t)ls.M * kLineValue + sizeof(int));
}

cudaError_t launch_sweep_toep(const double* f, double* u, double* delta, const double* cols,
                              size_t cstride, const unsigned char* band, size_t bstride,
                              unsigned char* scratch, const LevelShape& ls, int par, double hinv2,
                              unsigned* gave_up, cudaStream_t s, bool zero_u) {
  if (!toep_length(ls.M)) return cudaErrorInvalidValue;
  const int npts = colour_count(ls.d, ls.n, par);
  if (npts == 0 || ls.batch == 0) return cudaSuccess;
  Geometry G;
  G.d = ls.d;
  G.n = ls.n;
  G.M = ls.M;
  G.par = par;
  G.npts = npts;
  G.fstride = ls.field_stride();
  G.bstride = bstride;
  G.zero_u = zero_u;
  const long long lines = (long long)npts * ls.batch;
  if (toep_form(ls, par) == kToepSums) {
    G.per_inst = G.group0 = G.groups = 0;
#define MGWR_DIRECT(OB)                                                                     \
  k_toep_direct<OB><<<dim3((unsigned)lines, ls.M / (2 * OB)), 256, 0, s>>>(f, u, delta, cols, \
                                                                           cstride, G, hinv2)
    // by one instance's lines, so that a batch sums as one instance does
    const int tile = direct_tile(npts, ls.M);
    if (tile == 8)
      MGWR_DIRECT(8);
    else if (tile == 16)
      MGWR_DIRECT(16);
    else
      MGWR_DIRECT(32);
#undef MGWR_DIRECT
    return counted(cudaGetLastError());
  }
  return product(f, u, delta, band, scratch, G, ls.batch, hinv2, gave_up, s);
}

ToepForm toep_form(const LevelShape& ls, int par) {
  const int npts = colour_count(ls.d, ls.n, par);
  if (few_lines((long long)npts * ls.batch, ls.M)) return kToepSums;
  return transform_pays(npts, ls.batch, ls.M) ? kToepTransform : kToepProduct;
}

// Few lines keep the transform's defect (one launch).
bool toep_defect(const LevelShape& ls) {
  const int npts = ls.d == 1 ? ls.n : ls.n * ls.n;
  return toep_length(ls.M) && (long long)npts * ls.batch * ls.M * ls.M / 2 > (1ll << 22) &&
         !transform_pays(npts, ls.batch, ls.M);
}

cudaError_t launch_defect_toep(const double* u, const double* f, double* r,
                               const unsigned char* band, unsigned char* scratch,
                               const LevelShape& ls, double hinv2, unsigned long long* norm_bits,
                               unsigned* gave_up, cudaStream_t s) {
  if (!toep_length(ls.M)) return cudaErrorInvalidValue;
  if (ls.batch == 0) return cudaSuccess;
  Geometry G;
  G.d = ls.d;
  G.n = ls.n;
  G.M = ls.M;
  G.par = -1;
  G.npts = ls.d == 1 ? ls.n : ls.n * ls.n;
  G.fstride = ls.field_stride();
  G.bstride = blob_bytes(ls.M);
  G.zero_u = false;
  const cudaError_t e = product(u, r, nullptr, band, scratch, G, ls.batch, 0.0, gave_up, s);
  if (e != cudaSuccess) return e;
  const int per = ls.M / 2, tpl = per < 64 ? per : 64;
  const unsigned blocks = (unsigned)((G.npts + 256 / tpl - 1) / (256 / tpl));
  k_defect_finish<<<dim3(blocks, (unsigned)ls.batch), 256, 0, s>>>(
      u, f, r, ls.d, ls.n, ls.M, ilog2(tpl), G.npts, hinv2, norm_bits, G.fstride);
  return counted(cudaGetLastError());
}

}  // namespace mgwr
