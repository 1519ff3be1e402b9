// Grouped complex FP64 block GEMM on the half-precision tensor pipe:
// C (M x N) = alpha * sum_terms op(A) op(B) (+ C), FP64 in and out.
//
// This part's FP64 pipe does 2 multiply-adds per clock and SM (1.7 measured,
// DMMA m8n8k4 the same), its f16 mma.sync pipe 1024.  So every operand is cut
// into OZ_S integer slices of 9 bits (the splitting of Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59, 2012) and the products of slices run on the
// f16 pipe, where they are exact:
//   * each row of op(A) and each column of op(B) of one K group (at most 32
//     complex) is scaled by the power of two above its largest real or
//     imaginary part, x = X 2^E with |X| < 1, and written as
//       X = sum_p d_p 2^-(8 + 9 p),  p = 0 .. 6,  |d_p| <= 256 integer
//     (62 fractional bits; an FP64 number within 2^9 of the row's largest
//     enters unrounded);
//   * the integer products d_p e_q with p + q = s are added into one FP32
//     accumulator per s = 0 .. 6.  |d e| <= 2^16 and at most 64 real K and s + 1
//     pairs give at most (s + 1) 2^22, so the sums are exact (<= 2^24) for s <= 3;
//     from s = 4 on (units of 2^-52 and less of row times column scale) they could
//     reach 7 2^22 and round to the next even integer, if all digits of all
//     products were near 256 and of one sign.  Dropped are s >= 7, at most 0.75
//     2^-60 per real product, and the operands' bits below 2^-62, 0.5 2^-60;
//   * the seven sums of an output become one 64-bit integer, that one an
//     FP64 number, and only the sum over K groups and terms is FP64
//     arithmetic (one addition per group).
// These errors are relative to the row's largest element times the column's.  An
// output whose own products are all far below that, as in a state whose bonds
// are not balanced, is added up on the FP64 pipe instead (OZ_LEAD below), so
// that the error is that of FP64 sums everywhere.
// A complex product takes the real 2x2 form: one k16 MMA step holds 8 complex
// k of op(A) as (re, im) pairs; complex column n of op(B) is stored as the real
// columns 2n, (br, -bi) pairs, and 2n + 1, (bi, br) pairs.
//
// Tile of at most 64 x 24 complex, 8 warps; a warp owns up to three of the
// 4 x 6 MMA subtiles (m16 x 4 complex columns), dead subtiles are skipped.
// Blocks are ragged (K of 8-60, one side <= 36), so mma.sync with its 16 x 4
// grain wastes less than tcgen05's 128 rows; the slices are also made where
// they are used.
//
// What bounds it: latency.  Two CTAs of 8 warps per SM (shared memory) go through
// load, slice and multiply phases with a barrier after each: 40% of the issue
// slots and 24% of the warps are busy, the tensor pipe about 10%.  Measured
// on <psi|H|phi> at L = 16, D = 256 (32 launches, 7.2 GFLOP): 4.4 ms, where the
// FP64 pipe's kernel took 9.7 ms (4.1 without the FP64 pipe for single outputs,
// whose results were wrong there); the same with bonds rescaled by 2^+-20, where
// everything goes to the FP64 pipe: 11.3 ms; the error against 64 bits of the
// adjoint energy gradient at L = 12, D = 128 is 0.96e-14, the mean over 24 states
// (FP64 pipe: 1.13e-14).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "kernels.hpp"

namespace tdmps {

namespace {

constexpr int OZ_M = 64;        // most rows of an output tile (complex)
constexpr int OZ_N = 24;        // most columns of an output tile
constexpr int OZ_SUB = 3;       // MMA subtiles of a warp
constexpr int OZ_S = 7;         // slices per operand
constexpr int OZ_STAGE = 8;     // complex K per MMA step; the unit of split-K
constexpr int OZ_KC = 32;       // complex K per group
constexpr int OZ_THREADS = 256;
constexpr int OZ_WA = OZ_M * OZ_KC, OZ_WB = 2 * OZ_N * OZ_KC;   // half2 words of one slice
constexpr int OZ_SMEM = OZ_S * (OZ_WA + OZ_WB) * 4;          // A and B slices
constexpr int OZ_LD = OZ_KC + 1;   // complex FP64 row in shared memory (OzFrag::stage)
static_assert((OZ_M + OZ_N) * OZ_LD * 16 <= OZ_SMEM, "staged numbers take the slices' place");
constexpr int OZ_INF = 0x7ff;

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ void zfma(double2& c, double2 a, double2 b) {
  c.x = fma(a.x, b.x, fma(-a.y, b.y, c.x));
  c.y = fma(a.x, b.y, fma(a.y, b.x, c.y));
}

__device__ __forceinline__ void mma_f16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},"
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// four 8 x 8 half matrices, one 16-byte row address per lane
__device__ __forceinline__ void ldmatrix4(uint32_t* r, uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr));
}
__device__ __forceinline__ void ldmatrix2(uint32_t* r, uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(saddr));
}
// a b + c in 64 bits
__device__ __forceinline__ long long madwide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// word of (row, complex k) in one slice: the XOR spreads the eight 16-byte
// rows that one ldmatrix phase reads over all banks
__device__ __forceinline__ int oz_word(int row, int k) { return row * OZ_KC + (k ^ ((row & 7) << 2)); }

// size of a number as an integer that orders like it (0 only for zero); the
// upper bits are the exponent field
__device__ __forceinline__ int oz_key(double x) {
  return (__double2hiint(x) & 0x7FFFFFFF) | (int)min((unsigned)__double2loint(x), 1u);
}
__device__ __forceinline__ int oz_exp(int key) { return max(key >> 20, 1); }

// x 2^(1022 - E) as a 62-bit fraction plus the digit bias: sum_j 256 512^j, so
// that every 9-bit field holds digit + 256
__device__ __forceinline__ unsigned long long oz_fixed(double x, int E) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & OZ_INF;
  const unsigned int mh = (hi & 0xFFFFF) | (e ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32) | (unsigned int)__double2loint(x);
  const int sh = E - (e ? e : 1);
  unsigned long long f = sh < 62 ? (m << 9) >> sh : 0ull;
  if (hi < 0) f = 0ull - f;
  constexpr unsigned long long bias =
      256ull * ((1ull << 54) + (1ull << 45) + (1ull << 36) + (1ull << 27) + (1ull << 18) +
                (1ull << 9) + 1ull);
  return f + bias;
}

// the seven digit pairs of one element: row r of A, or real columns 2r and
// 2r + 1 of B
template <bool IS_B>
__device__ __forceinline__ void oz_store(uint32_t* s, int r, int k, double2 v, int E) {
  const unsigned long long fr = oz_fixed(v.x, E), fi = oz_fixed(v.y, E);
  const uint32_t rl = (uint32_t)fr, rh = (uint32_t)(fr >> 32), il = (uint32_t)fi, ih = (uint32_t)(fi >> 32);
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6500));   // 1280
  const int w0 = oz_word(IS_B ? 2 * r : r, k), w1 = oz_word(2 * r + 1, k);
#pragma unroll
  for (int p = 0; p < OZ_S; ++p) {
    const int b = 9 * (OZ_S - 1 - p);
    const uint32_t x = b >= 32 ? rh >> (b & 31) : __funnelshift_r(rl, rh, b);
    const uint32_t y = b >= 32 ? ih >> (b & 31) : __funnelshift_r(il, ih, b);
    // 0x6400 | f is the half 1024 + f; the top field reaches 512
    const uint32_t w = (__byte_perm(x, y, 0x5410) & (p == 0 ? 0x03FF03FFu : 0x01FF01FFu)) | 0x64006400u;
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&w), off);
    const uint32_t u = *reinterpret_cast<const uint32_t*>(&d);
    if (IS_B) {
      s[p * OZ_WB + w0] = u ^ 0x80000000u;
      s[p * OZ_WB + w1] = __byte_perm(u, u, 0x1032);
    } else {
      s[p * OZ_WA + w0] = u;
    }
  }
}

// One operand of a K group, R rows of at most OZ_KC complex k.  With k
// contiguous in memory (row_op: the operand's row is the stored row; A with
// OP_N / OP_J, B with OP_T / OP_C) a warp takes one row at a time (lane = k),
// otherwise lane = row; either way a warp reads consecutive addresses.
// Thread element j is row oz_row(j), complex k oz_k(j).
template <int R>
struct OzFrag {
  static constexpr int RB = (R + 31) / 32, N = 4 * RB;   // row blocks of 32, elements per thread
  double2 v[N];
  static __device__ __forceinline__ int row(int j, bool row_op) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    return row_op ? warp + 8 * j : lane + 32 * (j % RB);
  }
  static __device__ __forceinline__ int k(int j, bool row_op) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    return row_op ? lane : warp + 8 * (j / RB);
  }
  // loads the group (scaled by sc when `scaled`); a segmented operand has one
  // block per segment of its rows (sg, so non-null)
  __device__ __forceinline__ void load(const void* base, int ld, const GemmSeg* sg,
                                       const SegOps* so, int op, int row0, int rows, int k0, int nk,
                                       bool row_op, bool scaled, double2 sc) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int r = row(j, row_op), kk = k(j, row_op);
      v[j] = make_double2(0.0, 0.0);
      if (r < rows && kk < nk) {
        const double2* P = (const double2*)base;
        int x = row0 + r, l = ld;
        if (sg) {
          const int s = (x >= sg->off[1]) + (x >= sg->off[2]) + (x >= sg->off[3]);
          P = (const double2*)so->p[s];
          l = so->ld[s];
          x -= sg->off[s];
        }
        if (P) v[j] = P[row_op ? (size_t)x * l + k0 + kk : (size_t)(k0 + kk) * l + x];
      }
    }
    if (op == OP_C || op == OP_J) {
#pragma unroll
      for (int j = 0; j < N; ++j) v[j].y = -v[j].y;
    }
    if (scaled) {
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] = zmul(sc, v[j]);
    }
  }
  // leaves the size (oz_key) of the largest part of each row in key[row], and
  // those of the largest real and imaginary part of all rows in key[part],
  // key[part + 1] (all zeroed before)
  __device__ __forceinline__ void sizes(int rows, bool row_op, int* key, int part) const {
    int re = 0, im = 0;
    if (row_op) {
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int r = row(j, true);
        if (r >= rows) break;   // the same for every lane
        const int x = oz_key(v[j].x), y = oz_key(v[j].y);
        re = max(re, x);
        im = max(im, y);
        const int e = __reduce_max_sync(0xffffffffu, max(x, y));
        if ((threadIdx.x & 31) == 0) key[r] = e;
      }
    } else {
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        int xb = 0, yb = 0;
#pragma unroll
        for (int j = b; j < N; j += RB) {
          xb = max(xb, oz_key(v[j].x));
          yb = max(yb, oz_key(v[j].y));
        }
        const int e = max(xb, yb);
        if (e) atomicMax(&key[row(b, false)], e);
        re = max(re, xb);
        im = max(im, yb);
      }
    }
    re = __reduce_max_sync(0xffffffffu, re);
    im = __reduce_max_sync(0xffffffffu, im);
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&key[part], re);
      atomicMax(&key[part + 1], im);
    }
  }
  // the slices; rows past the block only reach outputs that are never stored,
  // k is zero-filled to the MMA step
  template <bool IS_B>
  __device__ __forceinline__ void slice(uint32_t* s, int rows, int nk8, bool row_op,
                                        const int* key) const {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int r = row(j, row_op), kk = k(j, row_op);
      if (r < rows && kk < nk8) oz_store<IS_B>(s, r, kk, v[j], oz_exp(key[r]));
    }
  }
  // the numbers themselves, [row][k]
  __device__ __forceinline__ void stage(double2* s, int rows, bool row_op) const {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int r = row(j, row_op);
      if (r < rows) s[r * OZ_LD + k(j, row_op)] = v[j];
    }
  }
};

// t 2^k as an FP64 number, on the integer ALU (the conversion instruction runs
// on the FP64 pipe)
__device__ __forceinline__ double oz_double(long long t, int k) {
  if (t == 0) return 0.0;
  const unsigned long long a = (unsigned long long)(t < 0 ? -t : t);
  const int lz = __clzll((long long)a);
  const unsigned long long n = a << lz;             // leading one at bit 63
  const int e = 1023 + 63 - lz + k;
  // 53 bits rounded to nearest; the leading one adds 1 to the exponent field
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1);
  const unsigned long long sign = (unsigned long long)t & (1ull << 63);
  if (e > 0 && e < OZ_INF - 1)
    return __longlong_as_double((long long)(sign | (((unsigned long long)(e - 1) << 52) + m)));
  return scalbn(__longlong_as_double((long long)(sign | ((1022ull << 52) + m))), e - 1023);
}

// the value of one output from its seven sums, times 2^k (k: scale of row and column)
__device__ __forceinline__ double oz_value(const float (&acc)[OZ_S][4], int c, int k) {
  int g[OZ_S];
#pragma unroll
  for (int s = 0; s < OZ_S; ++s) g[s] = __float2int_rn(acc[s][c]);
  // sum_s g_s 512^(6 - s) = 2^27 h + l, |h| < 2^50, |l| < 2^43, in units small
  // enough that the 64-bit sum keeps at least 60 bits of it (a row and a
  // column whose large elements do not meet leave h small)
  const long long h = madwide(g[0], 1 << 27, madwide(g[1], 1 << 18, madwide(g[2], 1 << 9, (long long)g[3])));
  const long long l = madwide(g[4], 1 << 18, madwide(g[5], 1 << 9, (long long)g[6]));
  const int hh = (int)(h >> 32);
  const int drop = max(0, 29 - __clz(hh ^ (hh >> 31)));   // |h| < 2^(35 + drop), drop <= 15
  const long long t = (h << (27 - drop)) + (l >> drop);
  return oz_double(t, k - 70 + drop);
}

// What the slices of a group cannot give as accurately as FP64 arithmetic is
// added up on the FP64 pipe.  The error of the slices is at most 1.25 2^-60 per
// real product (truncation of both operands, dropped digit products), in units
// of the row's largest element times the column's; that of FP64 arithmetic is
// 2^-53 of the product itself.  So
//   * sum |a| |b| of an output has to reach 1.25 2^-7 of these units.  It does not
//     where large elements of A only meet small ones of B.  The sum of the
//     products of the leading digits' magnitudes, over both parts, is at most
//     4 times it in units of 2^-16 (a leading digit of 1 may stand for a half,
//     and the parts count a product up to twice);
//   * each part's scale over the group has to be within 2^-7 of that of both, unless the
//     part is zero throughout: the imaginary part of nearly real data.
// Of the outputs of the performance cases 0 to 0.1% fail the first, fewer the
// second.  A few outputs of a CTA: the warp for each (oz_direct); more than
// OZ_FEW threads with such outputs: from the numbers in shared memory, and
// without slices for the rest of the CTA's work once half of the threads have
// some.  Always from shared memory: the energy gradient above 4.64 ms, with the
// line at 16 threads 4.55; all from single lanes and global memory: the rescaled
// <psi|H|phi> 30 ms in all, now 14.8.
constexpr int OZ_FEW = 16;
constexpr float OZ_LEAD = 2560.f;   // 4 x 1.25 x 2^-7 x 2^16
constexpr int OZ_PART = 7;
// the parts that fail the second rule (bit 0 real, bit 1 imaginary), from the
// sizes of the largest real and imaginary part of A and of B
__device__ __forceinline__ int oz_weak_parts(const int* a, const int* b) {
  constexpr int none = -8192;
  const int ax = a[0] ? a[0] >> 20 : none, ay = a[1] ? a[1] >> 20 : none;
  const int bx = b[0] ? b[0] >> 20 : none, by = b[1] ? b[1] >> 20 : none;
  const int line = max(ax, ay) + max(bx, by) - OZ_PART;
  const int re = max(ax + bx, ay + by), im = max(ax + by, ay + bx);
  return (re >= 0 && re < line ? 1 : 0) | (im >= 0 && im < line ? 2 : 0);
}

enum : int { OZ_ROW_A = 1, OZ_ROW_B = 2, OZ_CONJ_A = 4, OZ_CONJ_B = 8 };

// element (x, k0) of an operand and the stride of its k
__device__ __forceinline__ void oz_operand(const void* base, int ld, const GemmSeg* sg, const SegOps* so,
                                           int x, int k0, bool row_op, const double2*& p, size_t& step) {
  p = (const double2*)base;
  if (sg) {
    const int s = (x >= sg->off[1]) + (x >= sg->off[2]) + (x >= sg->off[3]);
    p = (const double2*)so->p[s];
    ld = so->ld[s];
    x -= sg->off[s];
  }
  p += row_op ? (size_t)x * ld + k0 : (size_t)k0 * ld + x;
  step = row_op ? 1 : ld;
}

// For each lane of a warp with `weak`: the sum of its output (r, c) over the
// kn <= 32 complex k of one group from k0 on the FP64 pipe, k per lane: a launch
// waits for the last of them (59 launches of the energy gradient above: 2.65 ms
// so, 2.88 with all k on one lane).
__device__ __forceinline__ double2 oz_direct(const GemmTerm& tr, const GemmSeg* sgA, const GemmSeg* sgB,
                                             const SegOps* so, int mode, double2 sc, bool scaled, int r,
                                             int c, int k0, int kn, bool weak) {
  const int lane = threadIdx.x & 31;
  double2 mine = make_double2(0.0, 0.0);
  for (unsigned todo = __ballot_sync(0xffffffffu, weak); todo; todo &= todo - 1) {
    const int o = __ffs((int)todo) - 1;
    const double2 *a, *b;
    size_t sa, sb;
    oz_operand(tr.A, tr.lda, sgA, so, __shfl_sync(0xffffffffu, r, o), k0, mode & OZ_ROW_A, a, sa);
    oz_operand(tr.B, tr.ldb, sgB, so, __shfl_sync(0xffffffffu, c, o), k0, mode & OZ_ROW_B, b, sb);
    double2 s = make_double2(0.0, 0.0);
    if (lane < kn) {
      double2 x = a[lane * sa], y = b[lane * sb];
      if (mode & OZ_CONJ_A) x.y = -x.y;
      if (mode & OZ_CONJ_B) y.y = -y.y;
      if (scaled) x = zmul(sc, x);
      s = zmul(x, y);
    }
#pragma unroll
    for (int w = 1; w < 32; w <<= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, w);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, w);
    }
    if (lane == o) mine = s;
  }
  return mine;
}

// tiles of one dimension: as few as fit, of equal size rounded up to the
// subtile's
__host__ __device__ inline int oz_tiles(int n, int most) { return (n + most - 1) / most; }
__host__ __device__ inline int oz_edge(int n, int most, int grain) {
  const int c = oz_tiles(n, most);
  return ((n + c - 1) / c + grain - 1) / grain * grain;
}

// element (r, c) of a task's result (or of its split's slice)
__device__ __forceinline__ void f64_store(const GemmTask& t, const GemmSeg* sg, int split, int r, int c,
                                          double2 v) {
  if (t.splits > 1) {
    ((double2*)t.part)[((size_t)split * t.M + r) * t.N + c] = v;
    return;
  }
  double2* p;
  if (sg) {
    const int x = sg->dim == 0 ? r : c;
    const int s = (x >= sg->off[1]) + (x >= sg->off[2]) + (x >= sg->off[3]);
    const int y = x - sg->off[s];
    p = (double2*)sg->C[s] + (sg->dim == 0 ? (size_t)y * sg->ldc[s] + c : (size_t)r * sg->ldc[s] + y);
  } else {
    p = (double2*)t.C + (t.ct ? (size_t)c * t.ldc + r : (size_t)r * t.ldc + c);
  }
  if (t.beta) { v.x += p->x; v.y += p->y; }
  *p = v;
}

__global__ void __launch_bounds__(OZ_THREADS, 2) k_gemm(const GemmTask* __restrict__ tasks,
                                                        const GemmTerm* __restrict__ terms,
                                                        const GemmSeg* __restrict__ segs,
                                                        const SegOps* __restrict__ segops,
                                                        const int* __restrict__ tile_task) {
  extern __shared__ __align__(16) uint32_t oz_sh[];
  uint32_t* sA = oz_sh;
  uint32_t* sB = oz_sh + OZ_S * OZ_WA;
  // sizes of the rows of A, the columns of B, then of their parts (OzFrag::load)
  __shared__ int keyA[2][OZ_M + 2], keyB[2][32 + 2];
  const GemmTask& t = tasks[tile_task[blockIdx.x]];
  const unsigned local = blockIdx.x - t.tile_base, splits = t.splits;
  unsigned split = 0, rest = local;
  if (splits > 1) {
    split = local % splits;
    rest = local / splits;
  }
  const int M = t.M, N = t.N, walk = t.walk;
  const int tm = oz_edge(M, OZ_M, 16), tn = oz_edge(N, OZ_N, 4);
  const unsigned ny = rest / (unsigned)t.tiles_m;
  const int m0 = (int)(rest - ny * t.tiles_m) * tm;
  const int rows = min(tm, M - m0);
  const int opA = t.opA, opB = t.opB, tbeg = t.term_begin, tend = t.term_end;
  const bool rowA = opA == OP_N || opA == OP_J, rowB = opB == OP_T || opB == OP_C;
  const GemmSeg* sg = t.seg1 ? segs + (t.seg1 - 1) : nullptr;
  const GemmSeg *sgA = nullptr, *sgB = nullptr;
  if (sg) (sg->dim == 0 ? sgA : sgB) = sg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, q = lane & 3;
  // ldmatrix row of this lane: of A, 8-row halves then 4-word k halves; of B,
  // the k halves
  const int lr = lane & 7, la = ((lane >> 3) & 1) * 8 + lr, ka = (lane >> 4) * 4,
            kb = ((lane >> 3) & 1) * 4;
  const uint32_t aA = (uint32_t)__cvta_generic_to_shared(sA), aB = (uint32_t)__cvta_generic_to_shared(sB);
  // this split's share of the task's K steps (OZ_STAGE each, over all terms)
  int lo = 0, hi = 0x7fffffff;
  if (splits > 1) {
    unsigned S = 0;
    for (int e = tbeg; e < tend; ++e) S += (terms[e].K + OZ_STAGE - 1) / OZ_STAGE;
    lo = (int)(split * S / splits);
    hi = (int)((split + 1) * S / splits);
  }
  double2 alpha = t.alpha;
  if (t.alpha_ptr) alpha = zmul(alpha, *t.alpha_ptr);
  if (t.alpha_div) {
    const double2 b = *t.alpha_div;
    const double d = b.x * b.x + b.y * b.y;
    alpha = make_double2((alpha.x * b.x + alpha.y * b.y) / d, (alpha.y * b.x - alpha.x * b.y) / d);
  }
  const bool unit = alpha.x == 1.0 && alpha.y == 0.0;
  if (threadIdx.x < OZ_M + 2) keyA[0][threadIdx.x] = 0;
  if (threadIdx.x < 32 + 2) keyB[0][threadIdx.x] = 0;
  __syncthreads();
  int bufA = 0, bufB = 0;
  bool sliced_a = false, plain = false;   // the same in all threads
  double2* xA = (double2*)oz_sh;
  double2* xB = xA + OZ_M * OZ_LD;
  const int nsm = (rows + 15) >> 4;
  const int mode = (rowA ? OZ_ROW_A : 0) | (rowB ? OZ_ROW_B : 0) |
                   (opA == OP_C || opA == OP_J ? OZ_CONJ_A : 0) |
                   (opB == OP_C || opB == OP_J ? OZ_CONJ_B : 0);
  // the column tiles of this CTA: one, or (walk > 1: a task of one K group)
  // several that share the slices of A
  for (int w = 0; w < walk; ++w) {
    const int n0 = (int)(ny * walk + w) * tn;
    if (n0 >= N) break;
    const int cols = min(tn, N - n0);
    // live subtiles, dealt to the warps in turn
    const int nsub = nsm * ((cols + 3) >> 2);
    auto sub_col = [&](int i) {   // first column of subtile warp + 8 i
      const int sub = warp + 8 * i;
      return 4 * (nsm == 4 ? sub >> 2 : nsm == 2 ? sub >> 1 : nsm == 1 ? sub : sub / 3);
    };
    auto sub_row = [&](int i, int col) { return (warp + 8 * i - (col >> 2) * nsm) * 16; };
    double2 out[OZ_SUB][2];   // [subtile][row half]: rows g and g + 8, complex column q
#pragma unroll
    for (int i = 0; i < OZ_SUB; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) out[i][j] = make_double2(0.0, 0.0);
    int idx = 0;
    bool first = true;
    for (int e = tbeg; e < tend && idx < hi; ++e) {
      const GemmTerm& tr = terms[e];
      const int K = tr.K, nk = (K + OZ_STAGE - 1) / OZ_STAGE;
      if (idx + nk <= lo) { idx += nk; continue; }
      double2 sc = tr.scale;
      if (tr.scale_ptr) sc = zmul(sc, *tr.scale_ptr);
      const bool scaled = sc.x != 1.0 || sc.y != 0.0;
      const SegOps* so = sg ? segops + tr.pad : nullptr;
      const int c0 = max(lo - idx, 0), c1 = min(hi - idx, nk);
      idx += nk;
      // groups of at most OZ_KC, of equal size
      const unsigned ng = (unsigned)(c1 - c0 + OZ_KC / OZ_STAGE - 1) / (OZ_KC / OZ_STAGE);
      for (unsigned gi = 0; gi < ng; ++gi) {
        const int s0 = c0 + (int)(gi * (unsigned)(c1 - c0) / ng);
        const int s1 = c0 + (int)((gi + 1) * (unsigned)(c1 - c0) / ng);
        const int k0 = s0 * OZ_STAGE, kn8 = (s1 - s0) * OZ_STAGE, kn = min(K - k0, kn8);
        unsigned todo = ~0u;      // two bits per output: the parts for the FP64 pipe
        int nweak = OZ_THREADS;   // threads that have some
        if (!plain) {
          const int *ra = keyA[bufA], *rb = keyB[bufB];
          const bool fresh = w == 0 || !sliced_a;
          {
            OzFrag<OZ_N> fb;
            fb.load(tr.B, tr.ldb, sgB, so, opB, n0, cols, k0, kn, rowB, false, sc);
            fb.sizes(cols, rowB, keyB[bufB], 32);
            if (fresh) {
              OzFrag<OZ_M> fa;
              fa.load(tr.A, tr.lda, sgA, so, opA, m0, rows, k0, kn, rowA, scaled, sc);
              fa.sizes(rows, rowA, keyA[bufA], OZ_M);
              __syncthreads();
              fa.slice<false>(sA, rows, kn8, rowA, ra);
              bufA ^= 1;
            } else {
              __syncthreads();
            }
            fb.slice<true>(sB, cols, kn8, rowB, rb);
            bufB ^= 1;
          }
          if (fresh && threadIdx.x < OZ_M + 2) keyA[bufA][threadIdx.x] = 0;
          if (threadIdx.x < 32 + 2) keyB[bufB][threadIdx.x] = 0;
          if (!fresh) ra = keyA[bufA ^ 1];   // what the slices were made with
          sliced_a = true;
          todo = 0;
          __syncthreads();
          const int weak_parts = oz_weak_parts(ra + OZ_M, rb + 32);
#pragma unroll
          for (int i = 0; i < OZ_SUB; ++i) {
            if (warp + 8 * i < nsub) {
              const int nc = sub_col(i), mr = sub_row(i, nc);
              float acc[OZ_S][4];
#pragma unroll
              for (int s = 0; s < OZ_S; ++s)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[s][c] = 0.f;
              float lead[4] = {0.f, 0.f, 0.f, 0.f};
              for (int ks = 0; ks < kn8; ks += OZ_STAGE) {
                const uint32_t wa = aA + 4 * oz_word(mr + la, ks + ka);
                const uint32_t wb = aB + 4 * oz_word(2 * nc + lr, ks + kb);
                uint32_t bf[OZ_S][2];
#pragma unroll
                for (int p = 0; p < OZ_S; ++p) ldmatrix2(bf[p], wb + p * OZ_WB * 4);
#pragma unroll
                for (int p = 0; p < OZ_S; ++p) {
                  uint32_t af[4];
                  ldmatrix4(af, wa + p * OZ_WA * 4);
#pragma unroll
                  for (int r = 0; r + p < OZ_S; ++r) mma_f16(acc[p + r], af, bf[r][0], bf[r][1]);
                  if (p == 0) {   // the leading digits without their signs
                    constexpr uint32_t mag = 0x7FFF7FFFu;
#pragma unroll
                    for (int j = 0; j < 4; ++j) af[j] &= mag;
                    mma_f16(lead, af, bf[0][0] & mag, bf[0][1] & mag);
                  }
                }
              }
              // accumulators 0, 1: row g, complex column q; 2, 3: row g + 8
              const int eb = oz_exp(rb[nc + q]);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int mh = mr + g + 8 * h;
                const int ea = oz_exp(ra[mh]);
                const int k = ea + eb - 2 * 1022;
                double2 v = make_double2(oz_value(acc, 2 * h, k), oz_value(acc, 2 * h + 1, k));
                // a zero row or column needs nothing
                const int weak = ra[mh] == 0 || rb[nc + q] == 0          ? 0
                                 : lead[2 * h] + lead[2 * h + 1] < OZ_LEAD ? 3
                                                                          : weak_parts;
                if (weak & 1) v.x = 0.0;
                if (weak & 2) v.y = 0.0;
                todo |= (unsigned)weak << (2 * (2 * i + h));
                // an infinity or NaN in the row or the column
                if (ea == OZ_INF || eb == OZ_INF) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
                // the first group needs no addition (out is zero): a real branch,
                // so that the FP64 pipe is left alone
                if (!first) {
                  asm volatile("");
                  v.x += out[i][h].x;
                  v.y += out[i][h].y;
                }
                out[i][h] = v;
              }
            }
          }
          nweak = __syncthreads_count(todo != 0);
        }
        first = false;
        if (nweak == 0) continue;
        const bool stage = nweak > OZ_FEW;
        if (stage) {
          OzFrag<OZ_M> fa;
          fa.load(tr.A, tr.lda, sgA, so, opA, m0, rows, k0, kn, rowA, scaled, sc);
          fa.stage(xA, rows, rowA);
          OzFrag<OZ_N> fb;
          fb.load(tr.B, tr.ldb, sgB, so, opB, n0, cols, k0, kn, rowB, false, sc);
          fb.stage(xB, cols, rowB);
          sliced_a = false;
          plain = nweak > OZ_THREADS / 2;
          __syncthreads();
        }
#pragma unroll 1
        for (int o = 0; o < 2 * OZ_SUB; ++o) {
          const int weak = warp + 8 * (o >> 1) < nsub ? (int)(todo >> (2 * o)) & 3 : 0;
          if (!__any_sync(0xffffffffu, weak)) continue;
          const int nc = sub_col(o >> 1), mr = sub_row(o >> 1, nc) + g + 8 * (o & 1);
          double2 d = make_double2(0.0, 0.0);
          if (stage) {
            const double2 *a = xA + mr * OZ_LD, *b = xB + (nc + q) * OZ_LD;
            for (int x = 0; x < kn; ++x) zfma(d, a[x], b[x]);
          } else {
            d = oz_direct(tr, sgA, sgB, so, mode, sc, scaled, m0 + mr, n0 + nc + q, k0, kn, weak);
          }
#pragma unroll
          for (int i = 0; i < 2 * OZ_SUB; ++i)
            if (o == i) {
              if (weak & 1) out[i >> 1][i & 1].x += d.x;
              if (weak & 2) out[i >> 1][i & 1].y += d.y;
            }
        }
        if (stage) __syncthreads();
      }
    }
#pragma unroll
    for (int i = 0; i < OZ_SUB; ++i) {
      if (warp + 8 * i >= nsub) continue;
      const int nc = sub_col(i), mr = sub_row(i, nc);
      const int c = n0 + nc + q;
      if (c >= n0 + cols) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int rl = mr + g + 8 * h, r = m0 + rl;
        if (rl >= rows) continue;
        double2 v = out[i][h];
        if (!unit) {
          asm volatile("");
          v = zmul(alpha, v);
        }
        f64_store(t, sg, (int)split, r, c, v);
      }
    }
  }
}

// ------------------------------------------------------------------ small launches

// The same GEMM (no segments) on the FP64 pipe, for launches whose tiles are a
// few thousand multiply-adds each: there the sliced kernel's fixed cost (three
// dependent phases and about 3,000 instructions per warp) is longer than the
// arithmetic, and what counts is the length of the dependent chain.  Tile
// 16 x 16; each of four groups of 64 threads walks a quarter of the K steps (8
// each, over all terms) without block barriers, and their sums are added in
// group order at the end; the terms come in batches of 32, one load deep.
// Measured against one 32 x 32 tile per CTA with split-K and a reduction launch:
// a small overlap (L = 8, D = 32) 286 -> 230 us, a five-term sum at L = 12,
// D = 128 4.70 -> 4.24 ms.
constexpr int ST = 16, SK = 8, SG = 4, STERMS = 32;

__global__ void __launch_bounds__(64 * SG) k_gemm_small(const GemmTask* __restrict__ tasks,
                                                        const GemmTerm* __restrict__ terms,
                                                        const int* __restrict__ tile_task) {
  struct Term {
    const double2 *A, *B;
    int lda, ldb, K, s0;   // s0: first K step
    double2 sc;
    bool scaled;
  };
  // operand chunks of the groups, then their sums
  __shared__ double2 sh[2 * SG * SK * (ST + 1)];
  __shared__ Term tm[STERMS];
  __shared__ int batch_steps;
  static_assert(SG * ST * ST <= 2 * SG * SK * (ST + 1), "the sums take the chunks' place");
  const GemmTask& t = tasks[tile_task[blockIdx.x]];
  const int tid = threadIdx.x, grp = tid >> 6, lt = tid & 63;
  double2(*As)[ST + 1] = (double2(*)[ST + 1])(sh + grp * SK * (ST + 1));
  double2(*Bs)[ST + 1] = (double2(*)[ST + 1])(sh + (SG + grp) * SK * (ST + 1));
  const int local = blockIdx.x - t.tile_base, splits = t.splits, tiles_m = t.tiles_m;
  const int split = splits > 1 ? local % splits : 0, rest = splits > 1 ? local / splits : local;
  const int m0 = (rest % tiles_m) * ST, n0 = (rest / tiles_m) * ST;
  const int M = t.M, N = t.N, opA = t.opA, opB = t.opB, tend = t.term_end;
  const bool tA = opA == OP_T || opA == OP_C, tB = opB == OP_N || opB == OP_J;   // rows contiguous
  const bool cA = opA == OP_C || opA == OP_J, cB = opB == OP_C || opB == OP_J;
  const int tx = lt & 7, ty = lt >> 3;
  // rows past the block edge do no arithmetic (a warp covers 8 rows)
  const bool rows_live = m0 + 2 * ty < M;
  int lo = 0, hi = 0x7fffffff;
  if (splits > 1) {
    int S = 0;
    for (int e = t.term_begin; e < tend; ++e) S += (terms[e].K + SK - 1) / SK;
    lo = (int)((long long)split * S / splits);
    hi = (int)((long long)(split + 1) * S / splits);
  }
  auto barrier = [&]() { asm volatile("bar.sync %0, 64;" : : "r"(1 + grp) : "memory"); };
  // rows [r0, R) x k [k0, K) of an operand into a chunk: k contiguous in
  // memory: 8 rows x 8 k per pass, else 16 rows x 4 k
  auto load = [&](double2(*S)[ST + 1], const double2* P, int ld, bool rows_contig, bool conj, int r0,
                  int R, int k0, int K, bool scaled, double2 sc) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = rows_contig ? lt & 15 : (lt >> 3) + 8 * j, k = rows_contig ? (lt >> 4) + 4 * j : lt & 7;
      double2 v = make_double2(0.0, 0.0);
      if (r0 + r < R && k0 + k < K) {
        v = P[rows_contig ? (size_t)(k0 + k) * ld + r0 + r : (size_t)(r0 + r) * ld + k0 + k];
        if (conj) v.y = -v.y;
        if (scaled) v = zmul(sc, v);
      }
      S[k][r] = v;
    }
  };
  double2 acc[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = make_double2(0.0, 0.0);
  int base = 0;   // steps before this batch of terms
  for (int b0 = t.term_begin; b0 < tend && base < hi; b0 += STERMS) {
    const int nb = min(STERMS, tend - b0);
    if (tid < 32) {
      int nk = 0;
      if (tid < nb) {
        const GemmTerm& g = terms[b0 + tid];
        Term& x = tm[tid];
        x.A = (const double2*)g.A;
        x.B = (const double2*)g.B;
        x.lda = g.lda;
        x.ldb = g.ldb;
        x.K = g.K;
        nk = (g.K + SK - 1) / SK;
        double2 sc = g.scale;
        if (g.scale_ptr) sc = zmul(sc, *g.scale_ptr);
        x.sc = sc;
        x.scaled = sc.x != 1.0 || sc.y != 0.0;
      }
      int sum = nk;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, sum, o);
        if (tid >= o) sum += y;
      }
      if (tid < nb) tm[tid].s0 = base + sum - nk;
      if (tid == 31) batch_steps = sum;
    }
    __syncthreads();
    const int end = min(hi, base + batch_steps);
    int i = 0;
    // this group's run of them
    const int s0 = max(lo, base), ns = max(0, end - s0);
    const int sb = s0 + grp * ns / SG, se = s0 + (grp + 1) * ns / SG;
    for (int s = sb; s < se; ++s) {
      while (i + 1 < nb && tm[i + 1].s0 <= s) ++i;
      const Term& g = tm[i];
      const int K = g.K, k0 = (s - g.s0) * SK;
      load(As, g.A, g.lda, tA, cA, m0, M, k0, K, g.scaled, g.sc);
      load(Bs, g.B, g.ldb, tB, cB, n0, N, k0, K, false, g.sc);
      barrier();
      if (rows_live) {
        const int kl = min(SK, K - k0);
        for (int k = 0; k < kl; ++k) {
          const double2 a0 = As[k][ty * 2], a1 = As[k][ty * 2 + 1];
          const double2 c0 = Bs[k][tx * 2], c1 = Bs[k][tx * 2 + 1];
          zfma(acc[0][0], a0, c0);
          zfma(acc[0][1], a0, c1);
          zfma(acc[1][0], a1, c0);
          zfma(acc[1][1], a1, c1);
        }
      }
      barrier();
    }
    base += batch_steps;
    __syncthreads();
  }
  double2* red = sh;   // [group][row][column]
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) red[(grp * ST + ty * 2 + i) * ST + tx * 2 + j] = acc[i][j];
  __syncthreads();
  const int r = m0 + tid / ST, c = n0 + tid % ST;
  if (r >= M || c >= N) return;
  double2 v = red[tid];
#pragma unroll
  for (int g = 1; g < SG; ++g) {
    v.x += red[g * ST * ST + tid].x;
    v.y += red[g * ST * ST + tid].y;
  }
  double2 alpha = t.alpha;
  if (t.alpha_ptr) alpha = zmul(alpha, *t.alpha_ptr);
  if (t.alpha_div) {
    const double2 b = *t.alpha_div;
    const double d = b.x * b.x + b.y * b.y;
    alpha = make_double2((alpha.x * b.x + alpha.y * b.y) / d, (alpha.y * b.x - alpha.x * b.y) / d);
  }
  if (alpha.x != 1.0 || alpha.y != 0.0) {
    asm volatile("");
    v = zmul(alpha, v);
  }
  f64_store(t, nullptr, split, r, c, v);
}

}  // namespace

int f64_tiles_m(int M, bool small) { return oz_tiles(M, small ? ST : OZ_M); }
int f64_tiles_n(int N, bool small, int walk) {
  return small ? oz_tiles(N, ST) : oz_tiles(oz_tiles(N, OZ_N), walk);
}
// At most 4 column tiles share the slices of A: with 1 / 2 / 4 / 8 the GEMM of
// <psi|H|phi> at L = 16, D = 256 takes 4.53 / 4.37 / 4.40 / 4.40 ms, of the energy
// gradient at L = 12, D = 128 2.63 / 2.65 / 2.68 / 2.68 ms (fewer CTAs).
int f64_walk(int N, int nterms, int K) {
  return nterms == 1 && K <= OZ_KC ? std::min(4, std::max(1, oz_tiles(N, OZ_N))) : 1;
}
int f64_stage_k() { return OZ_STAGE; }   // = SK

void launch_gemm(const GemmTask* d_tasks, const GemmTerm* d_terms, const GemmSeg* d_segs,
                 const SegOps* d_segops, const int* d_tile_task, int ntiles, bool small,
                 cudaStream_t st) {
  if (ntiles <= 0) return;
  if (small) {
    k_gemm_small<<<ntiles, 64 * SG, 0, st>>>(d_tasks, d_terms, d_tile_task);
    return;
  }
  set_smem_limit((const void*)k_gemm, OZ_SMEM);
  k_gemm<<<ntiles, OZ_THREADS, OZ_SMEM, st>>>(d_tasks, d_terms, d_segs, d_segops, d_tile_task);
}

}  // namespace tdmps
