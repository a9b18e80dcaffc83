// fp64_digits.cu -- the grouped FP64 triple product on the 16-bit tensor cores
// by exact digit arithmetic.
//
// GB300's FP64 units (DFMA and DMMA alike) issue 2 FMAs per clock and SM, its
// mma.sync f16 path 1024 (measured: 1.06 TFLOP/s against 600 TFLOP/s), so an
// FP64 product is cheaper as a sum of exact 16-bit products.  The scheme is
// the error-free splitting of Ozaki, Ogita, Oishi and Rump (Numerical
// Algorithms 59, 2012) with one power-of-two scale per operand row:
//     x = 2^(E-63) v,  v a 64-bit integer = sum_{i<7} d_i 2^(56-8i) + (< 2^8),
// the d_i balanced base-256 digits in [-128, 127], exact in f16.  Products of
// digits are at most 2^14; a sum over K = 32 of the pairs of equal weight
// s = i + j (at most 7 of them) stays below 2^22, so it is an exact integer in
// an FP32 accumulator that starts at 1.5 * 2^23, read off its mantissa without
// a conversion.  The pairs with s <= 7 are kept (34 of them).
// The eight integers of an output are put together in a 64-bit integer.
//
// Digits hold an entry to 2^-56 of its row's largest, an FMA chain to 2^-53 of
// itself: norms come out as exact as the chain's, but an output that hangs on
// small entries alone (a weakly weighted state behind a diagonal operator) would
// not.  So every piece of a tile carries a certificate: for each output a lower
// bound S of sum |alpha||L||X||R| and an upper bound E of what the digits left
// out, both kept with the sums.  Where E exceeds the rounding errors that an FMA
// chain may make in the same products, sum (K + L) 2^-53 S (K and L the lengths
// of the two contractions), the piece is given to the FMA kernel, which runs
// behind this one (k_tasks_fp64_failed).  S comes from one more digit pair: the
// leading digits' magnitudes less a half.  E is, in units of 2^-56 of the
// scales of A's and B's rows and X's block,
//     sum_k |b_k| (sum_l |x_kl| + 0.033 L + rounding of T's sums)    A's last digit, dropped pairs
//   + sum_k |t_k| + max |t| (0.05 K + 0.6)                           B's last digit, T's last bits, dropped pairs
// with |a|, |b|, |x| < 1 after scaling (magnitudes of rows of X are summed where
// they are cut).  On dense operators S (K + L) 8 is 5 to 50 times E; with
// states weighted over three decades 1 of 400 pieces fails (24 orbitals, D = 512
// in 9 sectors), where blocks have few states one of ten (the same, all sectors).
// Magnitudes that the fixed-point form cannot hold (infinities, NaN, vector
// entries of 2^330 and more or blocks below 2^-700, operators of 2^50 and more,
// rows or products far below the rest) are failures like any other.
//
// One CTA owns one output tile of one block and walks the block's products in
// a fixed order, as the DFMA classes do.  With A the operand of the tile's
// "a" side (op(R) and its columns, or op(L) and its rows; chosen per tile), X
// oriented to match and B the other operand, a product is
//     GEMM1  T[a][k] = sum_l A[a][l] X[k][l]     (64-bit integers per row a)
//     GEMM2  Y[a][b] += alpha sum_k T[a][k] B[b][k]
// Each warp owns 16 rows a.  GEMM1's accumulators are fragments whose layout
// is that of GEMM2's A operand, so T is normalised per row, cut into digits
// again and used from registers.
//
// The digits are cut beforehand (images, below), so the kernel is for lists that
// are kept; lists that run once or have no room for images, lists whose first
// product fails in more than a fifth of its work, and the adjoint, whose operands
// change between calls, stay with the FMA kernel.  The kernel is bound by the
// integer work around the MMAs (joining the weight sums, cutting T) and by the 8
// to 12 warps that registers and shared memory leave an SM to hide its latencies.
// One H_eff*psi, DFMA tile classes -> here (time, useful rate; in brackets
// without certificates):
//   24 orbitals, D = 512, all sectors (blocks <= 26):  36.5 -> 19.3 ms, 0.89 TFLOP/s [15.9]
//   24 orbitals, D = 512, 9 sectors (blocks <= 68):     153 -> 52 ms, 2.2 TFLOP/s    [47]
//   13 orbitals, D = 260, 3 sectors (blocks <= 99):    3.03 -> 0.83 ms, 2.6 TFLOP/s  [0.78]
// (cuBLAS DGEMM: 1.10 TFLOP/s).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "cuda_backend.h"

namespace tns {
namespace {

constexpr int DG_N = 7;                        // digits of an operand
constexpr int DG_S = 8;                        // weights s = i + j kept: 0 .. 7
constexpr unsigned DG_MAGIC = 0x4B400000u;     // bits of 1.5 * 2^23
constexpr float DG_LIMIT = 0.96f * 8.f;        // 2^-53 in units of 2^-56, less the roundings of the certificate itself
constexpr int DG_EMIN = 322;                   // smallest scale of a vector block (2^-700)
constexpr int DG_DEPTH = 60;                   // rows' scales are at most this far below 1 (operators) or their block's (vectors)
constexpr int DG_EMAX = (1023 + 330) << 20;    // high word from which on a vector entry leaves the fixed-point form
constexpr int DG_OPMAX = (1023 + 50) << 20;    // the same for an operator entry (ranges of the certificate)

__device__ __forceinline__ uint32_t sm_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void mma_acc(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the first product of an accumulator: starts at the integer base
__device__ __forceinline__ void mma_first(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  const float c = __uint_as_float(DG_MAGIC);
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c));
}

// digit p (0 = most significant) of two biased 64-bit integers as f16x2
template <int P>
__device__ __forceinline__ uint32_t digit2(uint32_t h0, uint32_t l0, uint32_t h1, uint32_t l1) {
  constexpr uint32_t sel = P % 4 == 0 ? 0x7733 : P % 4 == 1 ? 0x6622 : P % 4 == 2 ? 0x5511 : 0x4400;
  const uint32_t u = (__byte_perm(P < 4 ? h0 : l0, P < 4 ? h1 : l1, sel) & 0x00ff00ffu) | 0x64006400u;  // 1024 + byte
  const uint32_t off = 0x64806480u;                                                                    // 1152
  const __half2 d = __hsub2(*(const __half2*)&u, *(const __half2*)&off);
  return *(const uint32_t*)&d;
}

// the weight sums of one output as an integer, sum_s i_s 2^(43 - 8 s) to the
// nearest, below 2^62.1
__device__ __forceinline__ long long dg_join(float f0, float f1, float f2, float f3, float f4, float f5, float f6,
                                             float f7) {
  constexpr unsigned c = DG_MAGIC * 257u;
  auto two = [](float hi, float lo, unsigned off) {
    return (int)((unsigned)__float_as_int(hi) * 256u + (unsigned)__float_as_int(lo) - off);
  };
  const int P = two(f0, f1, c), Q = two(f2, f3, c), R = two(f4, f5, c), U = two(f6, f7, c - (1u << 12));
  const int V = R + (U >> 16);
  const unsigned long long hi = (unsigned long long)((unsigned)P * 8u + (unsigned)(Q >> 13)) << 32 | ((unsigned)Q << 19);
  const unsigned long long lo = (unsigned long long)(unsigned)(V >> 29) << 32 | ((unsigned)V << 3 | ((unsigned)U >> 13 & 7u));
  return (long long)(hi + lo);
}

// v 2^(e - 1085) as the nearest double: the leading one goes to bit 62, so that
// rounding may carry into bit 63 and from there into the exponent
__device__ __forceinline__ double dg_double(long long v, int e) {
  const long long sg = v >> 63;
  const unsigned long long m = (unsigned long long)((v ^ sg) - sg);
  uint32_t h = (uint32_t)(m >> 32), l = (uint32_t)m;
  const bool low = h == 0;
  h = low ? l : h;
  l = low ? 0u : l;
  const int z = __clz((int)h);
  const uint32_t hs = __funnelshift_lc(l, h, z), ls = l << (z & 31);
  const uint32_t half = __funnelshift_r(ls, hs, 1);  // sums have few bits more than a double: ties are common, and go to even
  const unsigned long long r = ((unsigned long long)(hs >> 1) << 32 | half) + (0x1ffu + (half >> 10 & 1u));
  const uint32_t rh = (uint32_t)(r >> 32), rl = (uint32_t)r;
  uint32_t dh = ((uint32_t)sg & 0x80000000u) | ((uint32_t)((e - z - (low ? 32 : 0)) << 20) + (rh >> 10));
  uint32_t dl = __funnelshift_r(rl, rh, 10);
  if (h == 0) dh = dl = 0u;
  return __hiloint2double((int)dh, (int)dl);
}

// ---------------------------------------------------------------------------
// Every distinct operand of the list has an image: its digits, cut once, in
// units of 8 rows x 8 columns x 7 planes of f16 core matrices (896 bytes; row
// groups outermost, columns padded to 16), after the scales of its rows.  The
// vectors are cut once per call, each block in the orientation its products
// read, into 8 digits (all 64 bits of v; the pair (0, 7) joins the others).
// The scales of X cannot go to the columns of B, which are cut before X is
// known, so T is brought to a common scale over k as it is normalised: a shift
// per element by the distance of its row of X from the block's largest.
// ---------------------------------------------------------------------------
constexpr int IM_UNIT = DG_N * 128;  // bytes of one 8 x 8 unit of an operator
constexpr int IM_NX = 8;             // digits of the vector and of T
constexpr int IM_XUNIT = IM_NX * 128;
constexpr int IM_SLOW = 0x7fffffff;  // scale of a block that the fixed-point form cannot hold
constexpr int IM_ZERO = 0;           // scale of a block of zeros

__host__ __device__ inline int im_oct(int cols) { return (cols + 15) / 16 * 2; }
__host__ __device__ inline int im_head(int rows) { return ((rows + 7) / 8 * 8 * 4 + 127) / 128 * 128; }
__host__ __device__ inline long long im_bytes(int rows, int cols) {
  return im_head(rows) + (long long)((rows + 7) / 8) * im_oct(cols) * IM_UNIT;
}

// an image of a vector block has the sums of its rows' magnitudes (floats, in
// units of the rows' scales) between the scales and the digits
__host__ __device__ inline int im_xhead(int rows) { return 2 * im_head(rows); }

struct DgRec {  // a product in the orientation of its tile
  uint32_t a, b, x;  // images of A (rows a) and B (rows b) in the operator arena, of X in the vector arena; 128-byte units
  int xb;            // scale index of X
  double alpha;
  int K, L, f, pad;  // f: 1 A is the identity, 2 B is, 4 an operator does not fit the fixed-point form
};
struct DgImage {  // an operand to cut: op(M) is rows x cols, element (r, c) = src[r * sr + c * sc]
  const double* src;
  int rows, cols, sr, sc;
  uint32_t off;
  int slow;
};
struct DgXBlock {  // a block of the vector, in one orientation
  long long src;
  int rows, cols, sr, sc;
  uint32_t off;
  int pad;
};

// one row's 8 columns as digits: E the row's scale
template <int N>
__device__ __forceinline__ void im_cut(const double (&x)[8], int E, unsigned char* at) {
  uint32_t hi[8], lo[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const uint32_t h = (uint32_t)__double2hiint(x[e]), l = (uint32_t)__double2loint(x[e]);
    const int sh = max(0, min(E - (int)((h & 0x7fffffffu) >> 20), 63));
    const unsigned long long v = (((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 | l) << 10) >> sh;
    const uint32_t sg = (uint32_t)((int)h >> 31);
    const unsigned long long b =
        ((unsigned long long)((uint32_t)(v >> 32) ^ sg) << 32 | ((uint32_t)v ^ sg)) + 0x8080808080808080ull;
    hi[e] = (uint32_t)(b >> 32);
    lo[e] = (uint32_t)b;
  }
#define IM_PUT(P)                                                                                                  \
  *(uint4*)(at + (P) * 128) = make_uint4(digit2<P>(hi[0], lo[0], hi[1], lo[1]), digit2<P>(hi[2], lo[2], hi[3], lo[3]), \
                                         digit2<P>(hi[4], lo[4], hi[5], lo[5]), digit2<P>(hi[6], lo[6], hi[7], lo[7]))
  IM_PUT(0);
  IM_PUT(1);
  IM_PUT(2);
  IM_PUT(3);
  IM_PUT(4);
  IM_PUT(5);
  IM_PUT(6);
  if (N > 7) IM_PUT(7);
#undef IM_PUT
}

__device__ __forceinline__ int im_scale(int mx, int least) { return max((mx + 0x2100) >> 20, least); }
// the scale of a row of zeros where the largest is top: 2^(it - top), as the bits of a float, is 0
__device__ __forceinline__ int im_none(int top) { return top - 127; }
__device__ __forceinline__ float im_pow2(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }  // -127 <= e <= 127
constexpr int IM_ONE = 1022;  // the scale of magnitudes below 1

// high word of a magnitude, at least 1 where the value is not zero
__device__ __forceinline__ int im_high(double x) {
  return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0 ? 1 : 0);
}

// the image of a matrix by a CTA of 4 warps, a warp per group of 8 rows: the
// rows' scales (and sums, for a vector block), then their digits; returns the
// largest high word seen
template <int N>
__device__ __forceinline__ int im_rows(const double* __restrict__ src, int rows, int cols, int sr, int sc, int groups,
                                       int top_scale, int least, unsigned char* img) {
  const int oc = im_oct(cols), lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r7 = lane & 7, q = lane >> 3;
  int* scale = (int*)img;
  unsigned char* units = img + (N == IM_NX ? im_xhead(8 * groups) : im_head(8 * groups));
  int top = 0;
  for (int rg = warp; rg < groups; rg += 4) {
    const int row = 8 * rg + r7;
    int mx = 0;
    if (row < rows)
      for (int c = q; c < cols; c += 4)
        mx = max(mx, im_high(__ldg(src + (long long)row * sr + (long long)c * sc)));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    top = max(top, mx);
    const int E = im_scale(mx, least);
    if (q == 0) scale[row] = mx ? E : im_none(top_scale);
    float sum = 0.f;
    for (int o = q; o < oc; o += 4) {
      double x[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        x[e] = (row < rows && 8 * o + e < cols) ? __ldg(src + (long long)row * sr + (long long)(8 * o + e) * sc) : 0.0;
      im_cut<N>(x, E, units + ((long long)rg * oc + o) * (N * 128) + r7 * 16);
      if (N == IM_NX)
#pragma unroll
        for (int e = 0; e < 8; ++e) {  // 1.m 2^(exponent - E), rounded up
          const int h = im_high(x[e]);
          if (h) sum += __uint_as_float((uint32_t)max((h >> 20) - E + 126, 1) << 23 | (uint32_t)(h & 0xfffff) << 3 | 7u);
        }
    }
    if (N == IM_NX) {
      sum += __shfl_xor_sync(0xffffffffu, sum, 8);
      sum += __shfl_xor_sync(0xffffffffu, sum, 16);
      if (q == 0) ((float*)(img + im_head(8 * groups)))[row] = sum;
    }
  }
  return top;
}

__global__ void __launch_bounds__(128) k_dg_ops(DgImage* __restrict__ jobs, unsigned char* arena) {
  DgImage& J = jobs[blockIdx.x];
  if (im_rows<DG_N>(J.src, J.rows, J.cols, J.sr, J.sc, (J.rows + 7) / 8, IM_ONE, IM_ONE - DG_DEPTH,
                    arena + (long long)J.off * 128) >= DG_OPMAX)
    J.slow = 1;
}

// vector images: one CTA per block, orientation and vector.  The first one
// clears the counts of pieces without a certificate, whose kernels come later.
__global__ void __launch_bounds__(128) k_dg_x(const DgXBlock* __restrict__ blocks, int nblk, const double* xv,
                                              long long xs, unsigned char* arena, long long xbytes, int* scales,
                                              int* failed) {
  const DgXBlock B = blocks[blockIdx.x];
  const double* X = xv + (long long)blockIdx.y * xs + B.src;
  unsigned char* img = arena + (long long)blockIdx.y * xbytes + (long long)B.off * 128;
  const int n = B.rows * B.cols;
  __shared__ int red[4];
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kDgClasses) failed[threadIdx.x] = 0;
  int mx = 0;
  for (int e = threadIdx.x; e < n; e += 128) mx = max(mx, im_high(X[e]));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = max(max(red[0], red[1]), max(red[2], red[3]));
  const int ex = im_scale(mx, DG_EMIN);
  if (threadIdx.x == 0) scales[(long long)blockIdx.y * nblk + blockIdx.x] = mx == 0 ? IM_ZERO : mx >= DG_EMAX ? IM_SLOW : ex;
  // GEMM1 takes X in pairs of row groups
  im_rows<IM_NX>(X, B.rows, B.cols, B.sr, B.sc, (B.rows + 15) / 16 * 2, ex, max(ex - DG_DEPTH, DG_EMIN), img);
}

// ---- planning on the device: distinct operands by a hash table of (address,
// stored transposed), image offsets by atomic addition (their order does not
// matter), then one record per product ---------------------------------------
struct DgPlanState {
  unsigned long long units;  // 128-byte units of the operator arena used so far
  unsigned long long xunits;
  int njobs, nx, fail, pad;
};

// the first half of MurmurHash3's 64-bit finaliser (Appleby, public domain)
__device__ __forceinline__ unsigned im_hash(unsigned long long k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  return (unsigned)k;
}

__device__ __forceinline__ unsigned long long im_key(const Task& t, int side) {
  return (unsigned long long)(uintptr_t)(side ? t.R : t.L) | ((t.flags & (side ? TF_RT : TF_LT)) ? 1ull : 0ull);
}

constexpr int IM_PROBES = 64;

__global__ void k_dg_find(const Task* __restrict__ tasks, const Group* __restrict__ groups,
                          const unsigned char* __restrict__ aside, unsigned long long* keys, int* slot_job,
                          unsigned mask, DgImage* jobs, int max_jobs, int* xtab, unsigned long long xtab_n, DgXBlock* xblocks,
                          int max_x, DgPlanState* st) {
  const Group G = groups[blockIdx.x];
  const int bl = aside[blockIdx.x];
  for (int ti = G.t0 + threadIdx.x; ti < G.t1; ti += blockDim.x) {
    const Task t = tasks[ti];
    if ((t.flags & (TF_XV | TF_XT | TF_XI)) != TF_XV || 2ull * (size_t)t.X >= xtab_n) {  // not a product on the vector
      st->fail = 1;
      continue;
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (t.flags & (side ? TF_RI : TF_LI)) continue;
      const unsigned long long key = im_key(t, side);
      unsigned h = im_hash(key) & mask;
      int p = 0;
      for (; p < IM_PROBES; ++p, h = (h + 1) & mask) {
        unsigned long long old = keys[h];
        if (old == key) break;
        if (old != 0) continue;
        old = atomicCAS(&keys[h], 0ull, key);
        if (old == key) break;
        if (old != 0) continue;
        const int j = atomicAdd(&st->njobs, 1);
        if (j >= max_jobs) {
          st->fail = 1;
          break;
        }
        DgImage J;
        J.src = side ? t.R : t.L;
        J.rows = side ? t.r : t.q;
        J.cols = side ? t.n : t.m;
        const bool tr = (t.flags & (side ? TF_RT : TF_LT)) != 0;
        J.sr = tr ? 1 : J.cols;
        J.sc = tr ? J.rows : 1;
        J.off = (uint32_t)atomicAdd(&st->units, (unsigned long long)(im_bytes(J.rows, J.cols) / 128));
        J.slow = 0;
        jobs[j] = J;
        slot_job[h] = j;
        break;
      }
      if (p == IM_PROBES) st->fail = 1;
    }
    // the vector block in the orientation (k, l) of this tile; a block that
    // stands in A's place is needed the other way round
    const int o = ((t.flags & (bl ? TF_LI : TF_RI)) && !(t.flags & (bl ? TF_RI : TF_LI))) ? 1 - bl : bl;
    int* slot = xtab + 2 * (long long)(size_t)t.X + o;
    if (*slot == 0 && atomicCAS(slot, 0, -1) == 0) {
      const int j = atomicAdd(&st->nx, 1);
      if (j >= max_x) {
        st->fail = 1;
        continue;
      }
      DgXBlock B;
      B.src = (long long)(size_t)t.X;
      B.rows = o ? t.n : t.m;
      B.cols = o ? t.m : t.n;
      B.sr = o ? 1 : t.n;
      B.sc = o ? t.n : 1;
      B.off = (uint32_t)atomicAdd(&st->xunits, (unsigned long long)((im_xhead((B.rows + 15) / 16 * 16) + (B.rows + 15) / 16 * 2 * im_oct(B.cols) * IM_XUNIT) / 128));
      B.pad = 0;
      xblocks[j] = B;
      *slot = j + 1;
    }
  }
}

__global__ void k_dg_records(const Task* __restrict__ tasks, const Group* __restrict__ groups,
                             const unsigned char* __restrict__ aside, const unsigned long long* __restrict__ keys,
                             const int* __restrict__ slot_job, unsigned mask, const DgImage* __restrict__ jobs,
                             const int* __restrict__ xtab, const DgXBlock* __restrict__ xblocks, DgRec* recs,
                             DgPlanState* st) {
  const Group G = groups[blockIdx.x];
  const int bl = aside[blockIdx.x];
  for (int ti = G.t0 + threadIdx.x; ti < G.t1; ti += blockDim.x) {
    const Task t = tasks[ti];
    DgRec r;
    r.a = r.b = 0;
    r.f = 0;
    r.pad = 0;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const bool is_a = (side == 0) == (bl != 0);
      if (t.flags & (side ? TF_RI : TF_LI)) {
        r.f |= is_a ? 1 : 2;
        continue;
      }
      const unsigned long long key = im_key(t, side);
      unsigned h = im_hash(key) & mask;
      int p = 0;
      while (p < IM_PROBES && keys[h] != key) {
        h = (h + 1) & mask;
        ++p;
      }
      if (p == IM_PROBES) {
        st->fail = 1;
        continue;
      }
      const DgImage J = jobs[slot_job[h]];
      if (J.rows != (side ? t.r : t.q) || J.cols != (side ? t.n : t.m)) st->fail = 1;
      if (J.slow) r.f |= 4;
      (is_a ? r.a : r.b) = J.off;
    }
    const int o = (r.f & 3) == 1 ? 1 - bl : bl;
    r.xb = xtab[2 * (long long)(size_t)t.X + o] - 1;
    const DgXBlock B = xblocks[r.xb];
    if (B.rows != (o ? t.n : t.m) || B.cols != (o ? t.m : t.n)) st->fail = 1;
    r.x = B.off;
    r.alpha = t.alpha;
    r.K = bl ? t.n : t.m;
    r.L = bl ? t.m : t.n;
    recs[ti] = r;
  }
}

// lower bounds of the magnitudes of two entries from their leading digits: the
// digits below it make up less than half of one
__device__ __forceinline__ uint32_t dg_low(uint32_t d) {
  const __half2 v = __hmax2(__hsub2(__habs2(*(const __half2*)&d), __floats2half2_rn(0.5f, 0.5f)), __floats2half2_rn(0.f, 0.f));
  return *(const uint32_t*)&v;
}
// their magnitudes, and upper bounds of them
__device__ __forceinline__ uint32_t dg_abs(uint32_t d) { return d & 0x7fff7fffu; }
__device__ __forceinline__ uint32_t dg_high(uint32_t d) {
  const __half2 v = __hadd2(__habs2(*(const __half2*)&d), __floats2half2_rn(0.51f, 0.51f));
  return *(const uint32_t*)&v;
}
__device__ __forceinline__ uint32_t dg_pack(float x, float y) {
  const __half2 v = __floats2half2_rn(x, y);
  return *(const uint32_t*)&v;
}
__device__ __forceinline__ uint32_t dg_mul(uint32_t x, uint32_t y) {
  const __half2 v = __hmul2(*(const __half2*)&x, *(const __half2*)&y);
  return *(const uint32_t*)&v;
}
// s plus two floats, at most 2^15
__device__ __forceinline__ uint32_t dg_more(uint32_t s, float x, float y) {
  const __half2 m = __floats2half2_rn(32768.f, 32768.f);
  const __half2 v = __hmin2(__hadd2(*(const __half2*)&s, __floats2half2_rn(fminf(x, 32768.f), fminf(y, 32768.f))), m);
  return *(const uint32_t*)&v;
}

template <int W_, int NBT_, int DBT_, int LK_, int KM_, int CTAS_>
struct ImCfg {
  static constexpr int W = W_, NBT = NBT_, DBT = DBT_, LK = LK_, KM = KM_, CTAS = CTAS_;
  static constexpr int NT = 32 * W, AR = 16 * W, BR = 8 * NBT;
  static constexpr int GU = W == 4 ? KM / 8 : 1;  // bodies of GEMM1, eight rows of X each
  static constexpr int LO = LK / 8, KO = KM / 8;              // octets staged
  static constexpr int off_x = (AR / 8) * LO * IM_UNIT;       // X after A in the first slot; a vector in A's place takes both
  static constexpr int off_b = off_x + (KM / 8) * LO * IM_XUNIT;
  static constexpr int off_y = off_b + NBT * KO * IM_UNIT;    // the tile's sums
  static constexpr int off_d = off_y + AR * BR * 8;           // their certificates; beyond DBT tiles one per two columns
  static constexpr int off_e = off_d + AR * (8 * DBT * 4 + 8 * (NBT - DBT) * 2);           // row scales of A, B and X, row sums of X
  static constexpr int total = off_e + 4 * (AR + BR + 2 * KM);
  static_assert(CTAS * (total + 1024) <= 228 * 1024, "resident CTAs");
  static_assert(KM == LK && off_b >= (AR / 8) * LO * IM_XUNIT, "chunks; the first slot holds the vector in A's place");
};

__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// `rows` runs of n 16-byte pieces, a warp per run.  Out of line: inlined, the
// kernel's copies are a third of the code that its warps fetch again for every
// product.
template <int W>
__device__ __noinline__ void im_copy(uint32_t dst, const unsigned char* src, int n, int rows, int sstride, int dstride) {
  const int warp = W == 1 ? 0 : threadIdx.x >> 5, lane = threadIdx.x & 31;
  src += (long long)warp * sstride + lane * 16;
  dst += (uint32_t)(warp * dstride + lane * 16);
#pragma unroll 1
  for (int r = warp; r < rows; r += W) {
#pragma unroll 1
    for (int i = lane; i < n; i += 32) cp16(dst + (uint32_t)(i - lane) * 16, src + (i - lane) * 16);
    src += (long long)W * sstride;
    dst += W * dstride;
  }
}

// The kernel's size counts: its warps run through all of it for every product,
// and with every loop over a tile unrolled it was 80 KB of code, a quarter of
// the time fetches of it (24 orbitals, D = 512, all sectors 27.2 ms, 9 sectors
// 53.4).  Loops that are not held in registers stay rolled (22.7 and 50.9 ms),
// the two places that copy the next operands are one, and the two smaller
// classes run GEMM1 in one body over X's rows (20.8 ms; the 64-class is slower
// with it, 51.8).
template <class C>
__global__ void __launch_bounds__(C::NT, C::CTAS)
    k_tasks_im(const DgRec* __restrict__ recs, const Task* __restrict__ tasks, const Group* __restrict__ groups,
               const Tile* __restrict__ tiles, int tile0, const unsigned char* __restrict__ ops,
               const unsigned char* __restrict__ xin, long long xbytes, const int* __restrict__ xscale, int nxb,
               const double* xv, double* yv, long long xs, long long ys, double* part, long long psize, int nv,
               int* nfailed, int* failed) {
  constexpr int W = C::W, NBT = C::NBT, LK = C::LK, KM = C::KM, NT = C::NT, LO = C::LO, KO = C::KO;
  constexpr int KT = KM / 8;
  extern __shared__ __align__(128) unsigned char sm[];
  const uint32_t sA = sm_u32(sm), sX = sm_u32(sm + C::off_x), sB = sm_u32(sm + C::off_b);
  const int* const eA = (const int*)(sm + C::off_e);
  const int* const eB = eA + C::AR;
  const int* const eX = eB + C::BR;
  const float* const xsum = (const float*)(eX + KM);
  const uint32_t sEA = sm_u32(eA), sEB = sm_u32(eB), sEX = sm_u32(eX), sXS = sm_u32(xsum);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int mj = lane >> 3, mr16 = (lane & 7) * 16;
  const Tile TL = tiles[tile0 + blockIdx.x / nv];
  const Group G = groups[TL.g];
  const int vec = blockIdx.x % nv;
  const unsigned char* xi = xin + (long long)vec * xbytes;
  const int* xsc = xscale + (long long)vec * nxb;
  const bool bl = TL.aside != 0;
  const int na = bl ? TL.nrows : TL.ncols, nb = bl ? TL.ncols : TL.nrows;
  const int a0 = bl ? TL.row0 : TL.col0, b0 = bl ? TL.col0 : TL.row0;
  const int arows = bl ? G.q : G.r, brows = bl ? G.r : G.q;  // rows of the A and B operands
  const int nbt = (nb + 7) >> 3, arg = (na + 7) >> 3;
  const bool mine = 16 * warp < na;
  // Y sits in shared memory, two 16-byte pairs a lane and 8-column tile: four
  // accesses to some 200 other instructions, which leaves the loop over the
  // tiles rolled (unrolled over registers its code missed the instruction
  // cache) and 8 NBT registers free
  double2* const Ys = (double2*)(sm + C::off_y) + warp * (NBT * 64) + lane;
  constexpr int DBT = C::DBT;
  float2* const Ds = (float2*)(sm + C::off_d) + warp * (DBT * 64) + lane;
  float* const Dp = (float*)(sm + C::off_d + W * DBT * 64 * 8) + (warp * (NBT - DBT) - DBT) * 64 + lane;
  auto sync = [&]() {
    if (W == 1) __syncwarp();
    else __syncthreads();
  };
  auto scale = [](double alpha, int n) { return alpha * __hiloint2double((n + 1023) << 20, 0); };  // alpha 2^n
  // the row groups this CTA never copies (a tile of fewer rows than the slot
  // has) are read by ldmatrix as absent rows: zero once
#pragma unroll 1
  for (int i = tid; i < C::total / 16; i += NT) ((uint4*)sm)[i] = make_uint4(0, 0, 0, 0);
  sync();

  // row groups rg0 .. rg0 + nrg, octets from o0 (at most mo) of an image with U-byte units
  auto rows = [&](uint32_t dst, int doct, const unsigned char* img, int head, int cols, int U, int rg0, int nrg, int o0) {
    const int oc = im_oct(cols), no = min(doct, oc - o0);
    im_copy<W>(dst, img + head + ((long long)rg0 * oc + o0) * U, no * (U / 16), nrg, oc * U, doct * U);
  };
  auto scales = [&](uint32_t dst, const unsigned char* img, int row, int groups) {
#pragma unroll 1
    for (int i = tid; i < 2 * groups; i += NT) cp16(dst + i * 16, img + (row + 4 * i) * 4);
  };
  // first-slot copy: A (or what stands in its place) and X for chunk (k0, l0)
  auto load1 = [&](const DgRec& r, int k0, int l0) {
    const int f = r.f & 3;
    if (f == 3) return;
    const unsigned char* ix = xi + (long long)r.x * 128;
    const unsigned char* ia = f == 1 ? ix : ops + (long long)r.a * 128;  // f == 1: P[a][k] = X^T, rows a of the vector image
    rows(sA, LO, ia, f == 1 ? im_xhead((arows + 15) / 16 * 16) : im_head(arows), f == 1 ? r.K : r.L, f == 1 ? IM_XUNIT : IM_UNIT, a0 >> 3, arg,
         (f ? k0 : l0) >> 3);
    scales(sEA, ia, a0, arg);
    if (f == 0) {
      const int kg = ((min(KM, r.K - k0) + 15) >> 4) * 2;
      const int kr = (r.K + 15) / 16 * 16;
      rows(sX, LO, ix, im_xhead(kr), r.L, IM_XUNIT, k0 >> 3, kg, l0 >> 3);
      scales(sEX, ix, k0, kg);
      scales(sXS, ix + im_head(kr), k0, kg);
    }
  };
  // second-slot copy: B (or the vector block in its place, without its last digit), columns from k0
  auto load2 = [&](const DgRec& r, int k0) {
    const bool v = (r.f & 3) == 2;
    const unsigned char* ib = v ? xi + (long long)r.x * 128 : ops + (long long)r.b * 128;
    if (v) {
      const int oc = im_oct(r.L), no = min(KO, oc - (k0 >> 3));
      const unsigned char* u = ib + im_xhead((brows + 15) / 16 * 16) + ((long long)(b0 >> 3) * oc + (k0 >> 3)) * IM_XUNIT;
#pragma unroll 1
      for (int g = 0; g < nbt; ++g)
        im_copy<W>(sB + g * KO * IM_UNIT, u + (long long)g * oc * IM_XUNIT, IM_UNIT / 16, no, IM_XUNIT, IM_UNIT);
    } else {
      rows(sB, KO, ib, im_head(brows), r.K, IM_UNIT, b0 >> 3, nbt, k0 >> 3);
    }
    scales(sEB, ib, b0, nbt);
  };

  DgRec rec;
  bool bad = false;      // an operand or a scale that this form cannot hold (alike in all threads of the CTA, or a lane's own)
  int ref = INT32_MIN;   // exponent that the certificate is kept relative to: of the first product that is not zero
  if (TL.t0 < TL.t1) {
    load1(recs[TL.t0], 0, 0);
    cp_commit();
  }
  for (int ti = TL.t0; ti < TL.t1; ++ti) {
    rec = recs[ti];
    const int ex = xsc[rec.xb];
    const bool more = ti + 1 < TL.t1;
    // the next record waits in L1 (in registers it would cost this product spills)
    if (more) asm volatile("prefetch.global.L1 [%0];" ::"l"(recs + ti + 1));
    const int f = rec.f & 3;
    const int ea = __double2hiint(rec.alpha) >> 20 & 0x7ff;
    if ((rec.f & 4) || ex == IM_SLOW || ea == 0x7ff || (ea == 0 && rec.alpha != 0.0)) {
      bad = true;
      break;
    }
    if (f == 3 || ex == IM_ZERO || ea == 0) {
      if (mine && ex != IM_ZERO && ea != 0) {  // Y += alpha X, as the FMA kernel does it
        const Task tk = tasks[ti];
        const double* pX = xv + (long long)vec * xs + (long long)(size_t)tk.X;
        const long long sa = bl ? tk.n : 1, sb = bl ? 1 : tk.n;
#pragma unroll 1
        for (int b = 0; b < nbt; ++b)
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            const int a = 16 * warp + g + 8 * h, c = 8 * b + 2 * t;
            const double* x = pX + (a0 + a) * sa + (b0 + c) * sb;
            double2 v = Ys[(2 * b + h) * 32];
            if (a < na && c < nb) v.x = fma(rec.alpha, x[0], v.x);
            if (a < na && c + 1 < nb) v.y = fma(rec.alpha, x[sb], v.y);
            Ys[(2 * b + h) * 32] = v;
          }
      }
      cp_wait();
      sync();
      if (more) load1(recs[ti + 1], 0, 0);
      cp_commit();
      continue;
    }
    if (ref == INT32_MIN) ref = ea + ex;
    // the certificate's weight of a row with scale e: 2^n times alpha's mantissa, n relative to ref; what lies too far
    // below counts with its errors alone
    const float am = __uint_as_float(0x3f800000u | (uint32_t)(__double2hiint(rec.alpha) & 0xfffff) << 3);
    const int atop = f == 1 ? ex : IM_ONE, btop = f == 2 ? ex : IM_ONE;
    auto weight = [&](int e) {
      const int n = ea + ex - ref + e - atop;
      if (e == im_none(atop)) return 0.f;
      if (n > 50) bad = true;
      return am * im_pow2(max(min(n, 50), -60));
    };
    auto far = [&](int e) { return e != 0 && e != im_none(atop) && ea + ex - ref + e - atop < -60; };  // 0: no such row
    // alpha 2^n, the scale of a row of sums; one that underflows (while its sums may not) is for the FMA kernel
    auto row_scale = [&](int e, int n) {
      if (e != 0 && ea - 1023 + n < -1000) bad = true;
      return scale(rec.alpha, n);
    };
    const int K = f == 2 ? rec.L : rec.K, L = rec.L;
    int hsh = 0;
#pragma unroll 1
    while ((32 << hsh) < L) ++hsh;
    // errors of a T entry beside A's last digits (1 per unit of X's row sum), in
    // units of 2^-56 of the scales: dropped pairs, X's last bit, the joined sums' roundings
    const float el = 0.01f + 0.033f * L + (float)((L + LK - 1) / LK) * (hsh ? 0.3f + 0.51f * (float)(1 << hsh) : 0.26f);
    // a sum may err by K + L units of 2^-53 of its magnitudes
    const float lim = fminf(DG_LIMIT * (float)(f == 0 ? K + L : K + 1), 4096.f);
    const float lim14 = lim * 0x1p-14f;
    for (int k0 = 0; k0 < K; k0 += KM) {
      const int kc = min(KM, K - k0);
      // T's digits; as f16, in units of 2^-59 of X's scale, what T may err by (lower bounds of sum |A||X|) and what it
      // errs by (upper bounds)
      uint32_t tf[KT / 2][IM_NX][4], mt[KT / 2][4], et[KT / 2][2];
      auto hide = [&](int e0, int e1) {  // no lower bounds for rows too far below
#pragma unroll
        for (int kk = 0; kk < KT / 2; ++kk)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (far(q & 1 ? e1 : e0)) mt[kk][q] = 0u;
      };
      double s0 = 0.0, s1 = 0.0;
      float ws0 = 0.f, ws1 = 0.f, wt0 = 0.f, wt1 = 0.f;
#pragma unroll
      for (int kk = 0; kk < KT / 2; ++kk) {
        et[kk][0] = et[kk][1] = 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) mt[kk][q] = 0u;
      }
      cp_wait();
      sync();  // the first slot is in, the second is free
      load2(rec, k0);
      cp_commit();
      if (f == 0) {
        long long T[KT][4];
#pragma unroll
        for (int b = 0; b < KT; ++b)
#pragma unroll
          for (int e = 0; e < 4; ++e) T[b][e] = 0;
        for (int l0 = 0; l0 < L; l0 += LK) {
          const int lc = min(LK, L - l0);
          if (l0) {
            sync();
            load1(rec, k0, l0);
            cp_commit();
            cp_wait();
            sync();
          }
          if (!mine) continue;
          uint32_t alow[LK / 16][4];
#pragma unroll
          for (int h = 0; h < LK / 16; ++h) {
            ldsm4(alow[h], sA + (uint32_t)(((2 * warp + (mj & 1)) * LO + 2 * h + (mj >> 1)) * IM_UNIT + mr16));
#pragma unroll
            for (int q = 0; q < 4; ++q) alow[h][q] = dg_low(alow[h][q]);
          }
          // 8 rows of X at a time: 16 would take the registers of another warp
#pragma unroll(C::GU)
          for (int q8 = 0; q8 < KT; ++q8) {
            if (8 * q8 >= ((kc + 15) & ~15)) break;
            float acc[DG_S][4], sa[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int h = 0; h < LK / 16; ++h) {
              if (h > 0 && 16 * h >= lc) break;
              uint32_t xf[IM_NX / 2][4];  // two digits each, in halves
              const uint32_t xa = sX + (uint32_t)((q8 * LO + 2 * h + (mj & 1)) * IM_XUNIT + (mj >> 1) * 128 + mr16);
#pragma unroll
              for (int j = 0; j < IM_NX / 2; ++j) ldsm4(xf[j], xa + j * 256);
              const uint32_t aa = sA + (uint32_t)(((2 * warp + (mj & 1)) * LO + 2 * h + (mj >> 1)) * IM_UNIT + mr16);
#pragma unroll
              for (int i = 0; i < DG_N; ++i) {
                uint32_t af[4];
                ldsm4(af, aa + i * 128);
#pragma unroll
                for (int j = 0; i + j < DG_S; ++j) {
                  const uint32_t x0 = xf[j / 2][2 * (j & 1)], x1 = xf[j / 2][2 * (j & 1) + 1];
                  if (h == 0 && i == 0) mma_first(acc[i + j], af, x0, x1);
                  else mma_acc(acc[i + j], af, x0, x1);
                }
              }
              mma_acc(sa, alow[h], dg_low(xf[0][0]), dg_low(xf[0][1]));  // the same sums of lower bounds
            }
            long long v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              v[e] = dg_join(acc[0][e], acc[1][e], acc[2][e], acc[3][e], acc[4][e], acc[5][e], acc[6][e], acc[7][e]);
              if (hsh) v[e] >>= hsh;
            }
            const int k = 8 * q8 + 2 * t;
            const int2 ek = *(const int2*)(eX + k);
            const float2 sk = *(const float2*)(xsum + k);
            auto down = [&](int e) { return __uint_as_float((uint32_t)max(124 - ex + e, 0) << 23); };  // 2^(-3 - distance)
            const float f0 = down(ek.x), f1 = down(ek.y), m0 = f0 * lim14, m1 = f1 * lim14;
            const uint32_t e2 = dg_pack(fmaf(sk.x, -1.015f, -el) * f0, fmaf(sk.y, -1.015f, -el) * f1);
            auto keep = [&](int b) {
#pragma unroll
              for (int e = 0; e < 4; ++e) T[b][e] += v[e];
              uint32_t &u0 = mt[b / 2][2 * (b & 1)], &u1 = mt[b / 2][2 * (b & 1) + 1];
              if (l0 == 0) {
                u0 = dg_pack(sa[0] * m0, sa[1] * m1);
                u1 = dg_pack(sa[2] * m0, sa[3] * m1);
                et[b / 2][b & 1] = e2;
              } else {
                u0 = dg_more(u0, sa[0] * m0, sa[1] * m1);
                u1 = dg_more(u1, sa[2] * m0, sa[3] * m1);
              }
            };
            if (q8 == 0) keep(0);
            else if (q8 == 1) keep(1);
            else if (KT == 4 && q8 == 2) keep(KT - 2);
            else if (KT == 4) keep(KT - 1);
          }
        }
        if (mine) {
          // normalise T per row over the chunk: row k lies eX[k] below the block's scale ex
          int m0 = 0, m1 = 0, dx[KT][2];
#pragma unroll
          for (int b = 0; b < KT; ++b) {
#pragma unroll
            for (int e = 0; e < 2; ++e) dx[b][e] = min(ex - eX[8 * b + 2 * t + e], 63);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int h = (int)(T[b][e] >> 32), ah = (h ^ (h >> 31)) >> min(dx[b][e & 1], 31);
              if (e < 2) m0 = max(m0, ah);
              else m1 = max(m1, ah);
            }
          }
#pragma unroll
          for (int s = 1; s < 4; s <<= 1) {
            m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, s));
            m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, s));
          }
          const int z0 = __clz(m0 + (m0 >> 7) + 1) - 1, z1 = __clz(m1 + (m1 >> 7) + 1) - 1;
          auto bias = [](long long v, int s) {  // v 2^s, 0x80 in every byte
            return (unsigned long long)((long long)((unsigned long long)v << max(s, 0)) >> max(-s, 0)) + 0x8080808080808080ull;
          };
#pragma unroll
          for (int kk = 0; kk < KT / 2; ++kk)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int b = 2 * kk + (q >> 1), e = 2 * (q & 1), z = q & 1 ? z1 : z0;
              const unsigned long long v0 = bias(T[b][e], z - dx[b][0]), v1 = bias(T[b][e + 1], z - dx[b][1]);
              const uint32_t h0 = (uint32_t)(v0 >> 32), l0_ = (uint32_t)v0, h1 = (uint32_t)(v1 >> 32), l1_ = (uint32_t)v1;
              tf[kk][0][q] = digit2<0>(h0, l0_, h1, l1_);
              tf[kk][1][q] = digit2<1>(h0, l0_, h1, l1_);
              tf[kk][2][q] = digit2<2>(h0, l0_, h1, l1_);
              tf[kk][3][q] = digit2<3>(h0, l0_, h1, l1_);
              tf[kk][4][q] = digit2<4>(h0, l0_, h1, l1_);
              tf[kk][5][q] = digit2<5>(h0, l0_, h1, l1_);
              tf[kk][6][q] = digit2<6>(h0, l0_, h1, l1_);
              tf[kk][7][q] = digit2<7>(h0, l0_, h1, l1_);
            }
          const int base = ex - 1022 - 1022 - 57 + 63 - 57 + hsh;  // scales of X and A, of T's sums, of Y's
          const int e0 = eA[16 * warp + g], e1 = eA[16 * warp + g + 8];
          s0 = row_scale(e0, e0 + base - z0);
          s1 = row_scale(e1, e1 + base - z1);
          ws0 = weight(e0);
          ws1 = weight(e1);
          wt0 = ws0 * im_pow2(6 + hsh - z0);  // T's scale after normalising
          wt1 = ws1 * im_pow2(6 + hsh - z1);
          if (far(e0) || far(e1)) hide(e0, e1);
          ws0 *= 0x1p-4f;  // 2^3 of down, 2^-7 of B's digit
          ws1 *= 0x1p-4f;
        }
      } else if (mine) {
#pragma unroll
        for (int kk = 0; kk < KT / 2; ++kk)
#pragma unroll
          for (int i = 0; i < IM_NX; ++i) {
            const uint32_t at = (uint32_t)(((2 * warp + (mj & 1)) * LO + 2 * kk + (mj >> 1)) * (f == 1 ? IM_XUNIT : IM_UNIT) + i * 128 + mr16);
            if (i < DG_N || f == 1) ldsm4(tf[kk][i], sA + at);
            else tf[kk][i][0] = tf[kk][i][1] = tf[kk][i][2] = tf[kk][i][3] = 0u;
          }
        const uint32_t lim7 = dg_pack(lim * 0x1p-7f, lim * 0x1p-7f);
#pragma unroll
        for (int kk = 0; kk < KT / 2; ++kk) {
#pragma unroll
          for (int q = 0; q < 4; ++q) mt[kk][q] = dg_mul(dg_low(tf[kk][0][q]), lim7);
          et[kk][0] = et[kk][1] = f == 2 ? dg_pack(-1.02f, -1.02f) : 0u;  // A's last digits against the magnitudes of B
        }
        const int e0 = eA[16 * warp + g], e1 = eA[16 * warp + g + 8];
        s0 = row_scale(e0, e0 - 1022 - 57);
        s1 = row_scale(e1, e1 - 1022 - 57);
        wt0 = weight(e0);
        wt1 = weight(e1);
        if (far(e0) || far(e1)) hide(e0, e1);
        ws0 = wt0 * 0x1p-7f;
        ws1 = wt1 * 0x1p-7f;
      }
      if (mine) {
        // B's last digits against T's magnitudes (its leading digits and the rest, at most half of one), T's last
        // bits, the dropped pairs and the joined sum's last bit
        float st[4] = {0.f, 0.f, 0.f, 0.f};
        const uint32_t one = dg_pack(1.f, 1.f);
        uint32_t a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = dg_abs(tf[0][0][q]);
        mma_acc(st, a, one, one);
        if (KT == 4 && kc > 16) {
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] = dg_abs(tf[KT / 2 - 1][0][q]);
          mma_acc(st, a, one, one);
        }
        const float rest = 0.05f * kc + 0.6f;
        wt0 *= -fmaf(st[0], 1.02f * 0x1p-7f, rest);
        wt1 *= -fmaf(st[2], 1.02f * 0x1p-7f, rest);
      }
      cp_wait();
      sync();  // the second slot is in, the first is free
      const bool on = k0 + KM < K;
      DgRec nx = rec;
      if (!on && more) nx = recs[ti + 1];
      if (on || more) load1(nx, on ? k0 + KM : 0, 0);
      cp_commit();
      if (!mine) continue;
#pragma unroll 1
      for (int b = 0; b < nbt; ++b) {
        float acc[DG_S][4];
        uint32_t bf[DG_N][KT];
        const uint32_t ba = sB + (uint32_t)((b * KO + (KT == 4 ? mj : (mj & 1))) * IM_UNIT + mr16);
#pragma unroll
        for (int j = 0; j < DG_N; j += KT == 4 ? 1 : 2) {
          uint32_t r[4];  // four octets of a digit, or two of two digits
          ldsm4(r, ba + (KT == 4 ? j : min(j + (mj >> 1), DG_N - 1)) * 128);
          bf[j][0] = r[0];
          bf[j][1] = r[1];
          if (KT == 4 || j + 1 < DG_N) {
            bf[KT == 4 ? j : j + 1][KT - 2] = r[2];
            bf[KT == 4 ? j : j + 1][KT - 1] = r[3];
          }
        }
#pragma unroll
        for (int i = 0; i < IM_NX; ++i)
#pragma unroll
          for (int j = 0; j < DG_N && i + j < DG_S; ++j) {
            if (i == 0 || (i == 1 && j == DG_N - 1)) mma_first(acc[i + j], tf[0][i], bf[j][0], bf[j][1]);
            else mma_acc(acc[i + j], tf[0][i], bf[j][0], bf[j][1]);
          }
        if (KT == 4 && kc > 16) {
#pragma unroll
          for (int i = 0; i < IM_NX; ++i)
#pragma unroll
            for (int j = 0; j < DG_N && i + j < DG_S; ++j) mma_acc(acc[i + j], tf[KT / 2 - 1][i], bf[j][KT - 2], bf[j][KT - 1]);
        }
        const int2 eb = *(const int2*)(eB + 8 * b + 2 * t);
        float sa[4] = {0.f, 0.f, 0.f, 0.f};  // what the sums may err by, less what they do
        {
          const uint32_t ea0[4] = {et[0][0], et[0][0], et[0][1], et[0][1]};
          mma_acc(sa, mt[0], dg_low(bf[0][0]), dg_low(bf[0][1]));
          mma_acc(sa, ea0, dg_high(bf[0][0]), dg_high(bf[0][1]));
          if (KT == 4 && kc > 16) {
            const uint32_t ea1[4] = {et[KT / 2 - 1][0], et[KT / 2 - 1][0], et[KT / 2 - 1][1], et[KT / 2 - 1][1]};
            mma_acc(sa, mt[KT / 2 - 1], dg_low(bf[0][KT - 2]), dg_low(bf[0][KT - 1]));
            mma_acc(sa, ea1, dg_high(bf[0][KT - 2]), dg_high(bf[0][KT - 1]));
          }
        }
        const float c0 = im_pow2(eb.x - btop), c1 = im_pow2(eb.y - btop);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float d0 = fmaf(h ? ws1 : ws0, sa[2 * h], h ? wt1 : wt0), d1 = fmaf(h ? ws1 : ws0, sa[2 * h + 1], h ? wt1 : wt0);
          if (DBT == NBT || b < DBT) {
            float2 v = Ds[(2 * b + h) * 32];
            v.x = fmaf(c0, d0, v.x);
            v.y = fmaf(c1, d1, v.y);
            Ds[(2 * b + h) * 32] = v;
          } else {  // the sum of the smaller of two is at most either's sum
            Dp[(2 * b + h) * 32] += 8 * b + 2 * t + 1 < nb ? fminf(c0 * d0, c1 * d1) : c0 * d0;
          }
          double2 v = Ys[(2 * b + h) * 32];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int e = 2 * h + c;
            const long long j = dg_join(acc[0][e], acc[1][e], acc[2][e], acc[3][e], acc[4][e], acc[5][e], acc[6][e], acc[7][e]);
            double& o = c ? v.y : v.x;
            o = fma(dg_double(j, (c ? eb.y : eb.x) + 63), h ? s1 : s0, o);
          }
          Ys[(2 * b + h) * 32] = v;
        }
      }
    }
  }
  cp_wait();

  // without a certificate the piece goes to the FMA kernel, which runs after this one
  if (mine && !bad)
#pragma unroll 1
    for (int b = 0; b < nbt; ++b)
#pragma unroll 1
      for (int h = 0; h < 2; ++h)
        if (16 * warp + g + 8 * h < na && 8 * b + 2 * t < nb) {
          const float2 d = DBT == NBT || b < DBT ? Ds[(2 * b + h) * 32] : make_float2(Dp[(2 * b + h) * 32], 0.f);
          if (!(d.x >= 0.f) || (8 * b + 2 * t + 1 < nb && !(d.y >= 0.f))) bad = true;
        }
  if (W == 1 ? __any_sync(0xffffffffu, bad) : __syncthreads_or(bad)) {
    if (tid == 0) failed[atomicAdd(nfailed, 1)] = blockIdx.x;
    return;
  }
  double* Y = yv + (long long)vec * ys + G.yoff;
  double* P = TL.poff >= 0 ? part + (long long)vec * psize + TL.poff : nullptr;  // split piece
  if (mine)
#pragma unroll 1
    for (int b = 0; b < nbt; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int a = 16 * warp + g + 8 * (e >> 1), c = 8 * b + 2 * t + (e & 1);
        if (a >= na || c >= nb) continue;
        const double2 v = Ys[(2 * b + (e >> 1)) * 32];
        const int i = bl ? a : c, j = bl ? c : a;
        if (P) P[i * TL.ncols + j] = e & 1 ? v.y : v.x;
        else Y[(long long)(TL.row0 + i) * G.r + TL.col0 + j] = e & 1 ? v.y : v.x;
      }
}

// residency: 12 CTAs of one warp (168 registers), 4 of two and 2 of four (shared
// memory: digits of both operands' chunks and the sums)
using ImS = ImCfg<1, 2, 2, 16, 16, 12>;
using ImM = ImCfg<2, 4, 3, 32, 32, 4>;
using ImL = ImCfg<4, 7, 7, 32, 32, 2>;

static_assert(ImS::CTAS == kDgClass[0].ctas && ImM::CTAS == kDgClass[1].ctas && ImL::CTAS == kDgClass[2].ctas &&
                  ImS::AR == kDgClass[0].a && ImM::AR == kDgClass[1].a && ImL::AR == kDgClass[2].a &&
                  ImS::BR == kDgClass[0].b && ImM::BR == kDgClass[1].b && ImL::BR == kDgClass[2].b &&
                  ImS::KM == kDgClass[0].km && ImM::KM == kDgClass[1].km && ImL::KM == kDgClass[2].km,
              "the classes the host plans with");

struct DgPlan {
  void* mem = nullptr;  // records, operator images, vector blocks and the images of the first call's vectors
  DgRec* recs = nullptr;
  unsigned char* ops = nullptr;
  DgXBlock* xblocks = nullptr;
  int nx = 0;
  unsigned char* x = nullptr;  // vector images, xbytes a vector, then their blocks' scales
  long long xbytes = 0;
  int* xscale = nullptr;  // nx a vector
  int x_nvec = 0;
  void* xmem = nullptr;   // images of more vectors
  long long vectors(int nvec) const { return (xbytes + 4LL * nx + 512) * nvec; }
  void set_vectors(unsigned char* p, int nvec) {
    x = p;
    xscale = (int*)(p + xbytes * nvec);
    x_nvec = nvec;
  }
};

template <class T>
T* carve(unsigned char*& p, long long n) {
  T* r = (T*)p;
  p += ((long long)sizeof(T) * n + 255) / 256 * 256;
  return r;
}

}  // namespace

void release_digit_plan(void* p) {
  DgPlan* P = (DgPlan*)p;
  if (!P) return;
  if (P->mem) dfree(P->mem);
  if (P->xmem) dfree(P->xmem);
  delete P;
}

// The plan of a list that is kept on the device: its images and records, made
// on the device in three launches.  Images are made only where they leave at
// least half of the memory that neither the step's own plan nor anything else
// has a claim to; without them the list stays with the FMA kernel.
bool prepare_digits(CudaBackend& be, const TaskList& tl, DevList& d, int nvec, long long length) {
  if (d.dg_none || !be.ok()) return false;
  DgPlan* P = (DgPlan*)d.dg;
  if (P && P->x_nvec >= nvec) return true;
  const long long avail = std::min(be.mem_limit() - be.mem_used(), be.mem_free()) - be.last_step_bytes;
  if (!P) {
    d.dg_none = true;  // until it is made
    const long long nt = (long long)tl.tasks.size(), ng = (long long)tl.groups.size();
    if (nt == 0 || ng == 0 || length <= 0) return false;
    P = new DgPlan();
    const int max_x = (int)(4 * ng + 4096);
    bool made = false;
    // a short list may have as many operators as products, in the table half as
    // many as slots; of a long one a quarter of the products' count holds them
    // many times over, and a larger table is tried if it does not
    for (long long want = nt <= (1 << 16) ? std::max(2 * nt, 4096LL) : nt / 4; !made; want *= 8) {
      unsigned cap = 4096;
      while (cap < want && cap < (1u << 30)) cap <<= 1;
      const int max_jobs = (int)(cap / 2);
      const long long bytes = 12LL * cap + (long long)sizeof(DgImage) * max_jobs + 8 * length +
                              (long long)sizeof(DgXBlock) * max_x + ng + 8192;
      if (bytes + nt * (long long)sizeof(DgRec) > avail / 2) break;
      // small tables stay for the next list, large ones go back
      const long long room = (bytes + (4LL << 20) - 1) >> 22 << 22;
      const bool keep = bytes <= (16LL << 20) && room <= avail / 2;
      unsigned char* tmp = nullptr;
      if (keep) tmp = (unsigned char*)be.scratch(room, 4);
      else if (dmalloc(&tmp, bytes) != cudaSuccess) cudaGetLastError();
      if (!tmp) break;
      unsigned char* p = tmp;
      DgPlanState* st = carve<DgPlanState>(p, 1);
      unsigned long long* keys = carve<unsigned long long>(p, cap);
      int* xtab = carve<int>(p, 2 * length);
      const size_t zero = p - tmp;
      int* slot = carve<int>(p, cap);
      DgImage* jobs = carve<DgImage>(p, max_jobs);
      DgXBlock* xb = carve<DgXBlock>(p, max_x);
      unsigned char* aside = carve<unsigned char>(p, ng);
      be.note(cudaMemsetAsync(tmp, 0, zero, be.stream()), "digit plan");
      be.note(cudaMemcpyAsync(aside, d.dg_aside.data(), ng, cudaMemcpyHostToDevice, be.stream()), "digit plan");
      k_dg_find<<<(unsigned)ng, 128, 0, be.stream()>>>(d.tasks, d.groups, aside, keys, slot, cap - 1, jobs, max_jobs, xtab,
                                                       2ull * length, xb, max_x, st);
      be.launches++;
      be.note(cudaGetLastError(), "k_dg_find");
      DgPlanState h{};
      auto state = [&]() {
        be.note(cudaMemcpyAsync(&h, st, sizeof(h), cudaMemcpyDeviceToHost, be.stream()), "digit plan");
        be.note(cudaStreamSynchronize(be.stream()), "digit plan");
        return be.ok() && !h.fail;
      };
      bool again = false;
      if (!state()) {
        again = be.ok() && want < 4 * nt;
      } else {
        // with the vectors of this call: an allocation takes a short list's product half as long as it runs
        P->nx = h.nx;
        P->xbytes = (long long)h.xunits * 128;
        const long long total = (long long)h.units * 128 + (long long)sizeof(DgRec) * nt +
                                (long long)sizeof(DgXBlock) * h.nx + P->vectors(nvec) + 1280;
        if (total <= avail / 2 && dmalloc(&P->mem, total) == cudaSuccess) {
          unsigned char* q = (unsigned char*)P->mem;
          P->ops = carve<unsigned char>(q, (long long)h.units * 128);
          P->recs = carve<DgRec>(q, nt);
          P->xblocks = carve<DgXBlock>(q, h.nx);
          P->set_vectors(carve<unsigned char>(q, P->vectors(nvec)), nvec);
          if (h.njobs > 0) k_dg_ops<<<(unsigned)h.njobs, 128, 0, be.stream()>>>(jobs, P->ops);
          k_dg_records<<<(unsigned)ng, 128, 0, be.stream()>>>(d.tasks, d.groups, aside, keys, slot, cap - 1, jobs, xtab, xb,
                                                              P->recs, st);
          be.launches += 2;
          be.note(cudaGetLastError(), "digit images");
          be.note(cudaMemcpyAsync(P->xblocks, xb, sizeof(DgXBlock) * h.nx, cudaMemcpyDeviceToDevice, be.stream()), "digit plan");
          made = state();
        } else {
          cudaGetLastError();
        }
      }
      if (!keep) dfree(tmp);
      if (!again) break;
    }
    if (!made) {
      release_digit_plan(P);
      return false;
    }
    d.dg = P;
    d.dg_none = false;
  }
  if (P->x_nvec >= nvec) return true;
  // images of more vectors, where they leave half of what is free; otherwise
  // the call runs on as many at a time as there are
  void* more = nullptr;
  if (P->vectors(nvec) > avail / 2 || dmalloc(&more, P->vectors(nvec)) != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  be.free_graphs(d);  // graphs captured with the smaller images would write through freed pointers
  cudaStreamSynchronize(be.stream());
  if (P->xmem) dfree(P->xmem);
  P->xmem = more;
  P->set_vectors((unsigned char*)more, nvec);
  return true;
}

int digit_vectors(const DevList& d) { return ((const DgPlan*)d.dg)->x_nvec; }

// the vectors' digits, ahead of the product kernels; clears the counts of failed pieces
void enqueue_digit_vectors(CudaBackend& be, const DevList& d, const double* xv, long long xs, int nvec, int* failed) {
  const DgPlan* P = (const DgPlan*)d.dg;
  k_dg_x<<<dim3(P->nx, nvec), 128, 0, be.stream()>>>(P->xblocks, P->nx, xv, xs, P->x, P->xbytes, P->xscale, failed);
  be.launches++;
  be.note(cudaGetLastError(), "k_dg_x");
}

// more than 48 KB of dynamic shared memory is asked for once, outside any capture
cudaError_t fp64_digits_init() {
  auto set = [](const void* f, int bytes) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  cudaError_t e = set((const void*)k_tasks_im<ImM>, ImM::total);
  if (e == cudaSuccess) e = set((const void*)k_tasks_im<ImL>, ImL::total);
  return e;
}

// one class of tiles; pieces without a certificate are listed in failed, their number in nfailed
void launch_fp64_digits(int cls, unsigned grid, cudaStream_t s, const void* plan, const Task* tasks,
                        const Group* groups, const Tile* tiles, int tile0, const double* xv, double* yv, long long xs,
                        long long ys, double* part, long long psize, int nv, int* nfailed, int* failed) {
  const DgPlan* P = (const DgPlan*)plan;
  auto go = [&](auto kernel, int nt, int smem) {
    kernel<<<grid, nt, smem, s>>>(P->recs, tasks, groups, tiles, tile0, P->ops, P->x, P->xbytes, P->xscale, P->nx, xv, yv,
                                  xs, ys, part, psize, nv, nfailed, failed);
  };
  if (cls == 0) go(k_tasks_im<ImS>, ImS::NT, ImS::total);
  else if (cls == 1) go(k_tasks_im<ImM>, ImM::NT, ImM::total);
  else go(k_tasks_im<ImL>, ImL::NT, ImL::total);
}

}  // namespace tns
