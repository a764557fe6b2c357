// Binary64 contractions on the 5th-generation tensor cores.
//
// GB300 runs binary64 FMAs at 1.26 TF/s and fp16 MMAs at nearly 2,000, so a
// binary64 product made of exact fp16 products pays off: the error-free
// transformation of matrix products of Ozaki, Ogita, Oishi & Rump (Numer.
// Algorithms 59, 2012; on tensor cores: Mukunoki, Ozaki, Ogita & Imamura 2020).
//
// Scheme.  Each vector of the contraction (a column of the block within a
// cell, a row of the cell matrix, ...) shares one power-of-two scale, set by
// its largest entry: x = 2^(E - 1084) I with an integer |I| < 2^62.  I is kept
// as a 64-bit word of balanced base-256 digits, I = sum_i d_i 2^(56 - 8 i),
// i = 0..7, |d_0| <= 64, |d_i| <= 128 (byte 7 - i of the word is d_i + 128),
// and every digit is an exact fp16 number.  The M operand enters with digits
// 0..6 (54 bits, rounded to nearest), the N operand with all eight.  The
// products d_i e_j of equal i + j = g are summed by the tensor core into one
// FP32 accumulator of group g = 0..7 (35 MMAs per 16-deep step; the pairs
// beyond g = 7 lie below 2^-64 of the largest product and are dropped).  The
// sums are integers: over a segment of at most 192 terms the bounds are 2^20
// for g = 0 and 192 g 2^14 < 2^24 for g <= 5, so FP32 accumulation is exact in
// any order (g = 6, 7 can round at 2^-60 of the largest product).  After a
// segment the groups are combined in 64-bit integers, V = sum_g I_g 2^(41 - 8 g),
// and V is rounded once to binary64 when the contraction ends (or every 960
// terms, so that |V| < 2^63).  The cell products cancel (||H~|| is hundreds of
// times the low eigenvalues), so their sums keep four more bits, 2^(45 - 8 g):
// the scale of a row of the cell matrix is raised where its first digits would
// add up to more than 2^11.
// The error is normwise: an entry 2^k below the largest of its vector enters with
// 54 - k (M) or 62 - k (N) bits, so K terms are off by K 2^-53 max|a| max|b| at most
// besides the rounding of the sums, where binary64 FMAs are off by K 2^-53 sum |a||b|:
// less in the norm, more in an entry that only small values make up
// (chfsi_set_fp64_products chooses).
//
//  ex_kernel<CELL>  R_e = H~_e Y_e for every cell (M: columns of Y, N: rows of
//                   the cell matrix)
//  ex_kernel<GRAM>  partial sums of A^T B over row splits (M: columns of A,
//                   N: columns of B)
//  ex_kernel<TALL>  X U (M: rows of X, N: columns of U)
// each preceded by a pass that turns the binary64 operands into words, laid
// out K-major (consecutive threads take consecutive M or N indices).
//
// One persistent CTA per SM works through 128 x 48 output tiles.  TMEM holds
// the eight 48-column accumulators (384 columns) and two buffers of the M
// operand's seven digit planes (2 x 56 columns): with both operands in shared
// memory an MMA of this shape would read 5.5 KB of it (44 cycles at 128 B/clk)
// for 24 cycles of math, with the M operand in TMEM it reads 1.5 KB (12).
// Warps 0-7 drain the accumulators, 8-15 load and expand the M words and store
// them to TMEM (two sets of four, alternating chunks), 16-18 expand the N words
// into a ring in shared memory, 19 issues the MMAs.  The groups are drained one
// after another while the MMAs of the later groups, and then of the next
// segment, go on.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include <cuda_fp16.h>

#include "digits.cuh"
#include "ex.h"
#include "tc_ptx.cuh"

namespace chfsi {

using namespace ptx;

namespace {

constexpr int NA = 7, NB = 8;               // digits of the M and the N operand
constexpr int NG = 8;                       // accumulator groups
constexpr int KC = 16;                      // K per chunk (one MMA step)
constexpr int BM = 128, BN = 48;            // output tile
constexpr int HN = BN / 2;                  // columns per drain warp
constexpr int PLANE = BN * KC * 2;          // bytes of one digit plane of the N operand
constexpr int B_STAGE = NB * PLANE;         // 12,288 B
constexpr int STAGES = 8;
constexpr int A_DEP = 3, B_DEP = 4;         // chunks of words in flight per producer warp
constexpr int A_WORDS = KC * 32 * 8;        // bytes of one warp's chunk: 16 x 32 M words,
constexpr int B_WORDS = KC * 16 * 8;        //   16 x 16 N words
constexpr int TA = NG * BN;                 // first TMEM column of the M operand
constexpr int TA_BUF = NA * KC / 2;         // 56 columns per buffer
constexpr int SEG = 12;                     // chunks per segment at most (192 terms) unless shown to be safe
constexpr int FLUSH = 5;                    // segments per integer accumulation (960 terms)
constexpr int EX_THREADS = 640;
constexpr int EX_SMEM = STAGES * B_STAGE + 8 * A_DEP * A_WORDS + 3 * B_DEP * B_WORDS + 512;
constexpr int kNonFinite = 1 << 20;         // scale mark of a vector holding an infinity or a NaN
constexpr int kNoScale = -(1 << 20);        // scale of a vector of zeros
// Scratch of one launch's words: the operands are processed in slices of at
// most this size (cells, or rows of the block).
constexpr size_t kWordBytes = (size_t)512 << 20;

enum ExMode { EX_CELL = 0, EX_GRAM = 1, EX_TALL = 2 };

struct ExParams {
  int64_t nitems;
  const uint64_t* A;        // M words
  const uint64_t* B;        // N words
  int64_t sa, sb;           // their K strides
  // CELL: cells of this launch, from cell e0
  int64_t e0;
  const int16_t* hexp;      // per cell row (all cells)
  const int* hsum;          // bound of the FP32 sums over a whole cell row (ex_h_scale_kernel)
  const int16_t* cexp;      // per (cell of this launch, column)
  int ne, ncol;
  // GRAM: rows of this launch, in splits of rps rows
  int64_t M, rps;
  int n1, n2;
  const int* aexp;          // column scales
  const int* bexp;
  int ntile, lower;
  // TALL: rows r0 .. r0 + M
  int64_t r0;
  const int* rexp;          // row scales (relative to the column scales), all rows
  const int* uexp;          // scales of U's columns (with X's folded in)
  int upper;
  double* C;                // R / partial / C
  int64_t ldc;
  ExWatch watch;
};

__device__ __forceinline__ int elem_off(int r, int k) {   // 16-bit elements, K-major core matrices
  return (r >> 3) * 128 + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

// fp16 pair (bytes picked by sel from x, minus 128): PRMT makes 1024 + byte.
__device__ __forceinline__ uint32_t half_pair(uint32_t x, uint32_t sel) {
  const uint32_t t = __byte_perm(x, 0x64646464u, sel);
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t), __half2half2(__float2half_rn(1152.f)));
  return *reinterpret_cast<const uint32_t*>(&h);
}
// The first ND digits of two words as fp16 pairs, digit d to out[d * stride].
template <int ND>
__device__ __forceinline__ void expand_pair(uint64_t w0, uint64_t w1, uint32_t* out, int stride) {
  const uint32_t h0 = (uint32_t)(w0 >> 32), h1 = (uint32_t)(w1 >> 32), l0 = (uint32_t)w0, l1 = (uint32_t)w1;
  const uint32_t ht = __byte_perm(h0, h1, 0x7362), hb = __byte_perm(h0, h1, 0x5140);
  const uint32_t lt = __byte_perm(l0, l1, 0x7362), lb = __byte_perm(l0, l1, 0x5140);
  out[0] = half_pair(ht, 0x4342);
  out[stride] = half_pair(ht, 0x4140);
  out[2 * stride] = half_pair(hb, 0x4342);
  out[3 * stride] = half_pair(hb, 0x4140);
  out[4 * stride] = half_pair(lt, 0x4342);
  out[5 * stride] = half_pair(lt, 0x4140);
  out[6 * stride] = half_pair(lb, 0x4342);
  if (ND == 8) out[7 * stride] = half_pair(lb, 0x4140);
}

// V += I_g 2^(SH - 8 g) for a drained group sum f = I_g, plus a constant per
// segment (group_offset over the eight groups).  The sums of at most 2^22 (g =
// 0, 1) and those that may be rounded (g = 6, 7: to units of V) are converted by
// adding 1.5 2^23, whose low mantissa bits then hold the integer: the conversion
// instruction runs at an eighth of the rate of the adds and, used for all
// groups, bounds the drain.
constexpr float kMagic = 12582912.f;
constexpr uint64_t kMagicBits = 0x4B400000u;
template <int SH>
__device__ constexpr uint64_t group_offset() {
  return (kMagicBits << SH) + (kMagicBits << (SH - 8)) + 2 * kMagicBits;
}
template <int SH>
__device__ __forceinline__ void add_group(int64_t& V, float f, int g) {
  if (g < 2) {
    const uint32_t b = __float_as_uint(f + kMagic);
    V += (int64_t)((uint64_t)(b << (SH - 32 - 8 * g)) << 32);
  } else if (g < 6) {
    V += (int64_t)__float2int_rn(f) * (1ll << (SH - 8 * (g < 6 ? g : 5)));
  } else {
    V += (int64_t)(uint64_t)__float_as_uint(fmaf(f, 1.f / (float)(1 << (g < 6 ? 0 : 8 * g - SH)), kMagic));
  }
}

// V 2^(ex - 2056 - SH) rounded to binary64 (ex: sum of the two scales); integer
// arithmetic only, since the conversion and the scaling would take two
// binary64-pipe operations per output.  LOW: results below the normal numbers are
// rounded to units of 2^-1074, else they are zeros.
template <int SH, bool LOW>
__device__ __forceinline__ double compose(int64_t v, int ex) {
  if (v == 0) return 0.0;
  const uint64_t a = v < 0 ? (uint64_t)(-v) : (uint64_t)v;
  const int lz = __clzll((long long)a);
  const uint64_t t = a << lz;                        // top bit set
  uint64_t m = t >> 11;
  m += ((t & 0x7ff) + (m & 1)) > 0x400;              // to nearest, ties to even
  const int f = 63 - lz + ex - 1033 - SH;                 // exponent field
  const uint64_t sg = v < 0 ? 0x8000000000000000ull : 0ull;
  if (!LOW && f <= 0) return __longlong_as_double((long long)sg);
  if (f <= 0) {                                      // units of 2^-1074
    const int sh = 12 - f;
    if (sh > 64) return __longlong_as_double((long long)sg);
    const uint64_t q = sh > 63 ? 0 : t >> sh, h = 1ull << (sh - 1), r = t & (h | (h - 1));
    return __longlong_as_double((long long)(sg | (q + (r > h || (r == h && (q & 1))))));
  }
  if (f >= 2047) return __longlong_as_double((long long)(sg | 0x7ff0000000000000ull));
  return __longlong_as_double((long long)(sg | (((uint64_t)f << 52) + (m - (1ull << 52)))));
}
__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// One output tile of the launch.
struct Item {
  const uint64_t *a, *b;   // words of (M or N index 0 of the tile, k = 0); rows of words start on 16 bytes
  int mv, nv;              // valid M and N indices
  int nk, kmax;            // chunks, K
  int m0, n0;              // first M / N index (CELL: column, cell row; GRAM: columns of A, B; TALL: -, column)
  int64_t row;             // CELL: cell of the launch; GRAM: split of the launch; TALL: first row of the launch
};
template <int MODE>
__device__ __forceinline__ Item decode(const ExParams& P, int64_t it) {
  Item r;
  if (MODE == EX_CELL) {
    const int nrt = (P.ne + BN - 1) / BN, nct = (P.ncol + BM - 1) / BM;
    const int rt = (int)(it % nrt);
    const int64_t q = it / nrt;
    r.row = q / nct;
    r.m0 = (int)(q % nct) * BM;
    r.n0 = rt * BN;
    r.kmax = P.ne;
    r.a = P.A + r.row * ((P.ne + KC - 1) / KC * KC) * P.sa + r.m0;
    r.b = P.B + (P.e0 + r.row) * P.ne * P.sb + r.n0;
    r.mv = P.ncol - r.m0;
    r.nv = P.ne - r.n0;
  } else if (MODE == EX_GRAM) {
    const int t1 = (P.n1 + BM - 1) / BM;
    r.row = it / P.ntile;
    int t = (int)(it % P.ntile), tj, ti;
    if (P.lower) {   // tiles with some i >= j: (ti + 1) 128 > tj 48
      tj = 0;
      for (;; ++tj) {
        const int c = t1 - tj * BN / BM;
        if (t < c) break;
        t -= c;
      }
      ti = t + tj * BN / BM;
    } else {
      tj = t / t1;
      ti = t % t1;
    }
    const int64_t k0 = r.row * P.rps;
    r.m0 = ti * BM;
    r.n0 = tj * BN;
    r.kmax = (int)min(P.rps, P.M - k0);
    r.a = P.A + k0 * P.sa + r.m0;
    r.b = P.B + k0 * P.sb + r.n0;
    r.mv = P.n1 - r.m0;
    r.nv = P.n2 - r.n0;
  } else {
    const int t2 = (P.n2 + BN - 1) / BN;
    const int64_t rt = it / t2;
    r.n0 = (int)(it % t2) * BN;
    r.m0 = 0;
    r.row = rt * BM;
    r.kmax = P.upper ? min(P.n1, r.n0 + BN) : P.n1;
    r.a = P.A + rt * ((P.n1 + KC - 1) / KC * KC) * BM;
    r.b = P.B + r.n0;
    r.mv = (int)min((int64_t)BM, P.M - r.row);
    r.nv = P.n2 - r.n0;
  }
  r.nk = (r.kmax + KC - 1) / KC;
  return r;
}

// Every `step`-th chunk of the CTA's items, from chunk `first` on.
template <int MODE>
struct Chunks {
  int64_t it;
  int i;
  Item I;
  __device__ __forceinline__ void settle(const ExParams& P) {
    while (it < P.nitems && i >= I.nk) {
      i -= I.nk;
      it += gridDim.x;
      if (it < P.nitems) I = decode<MODE>(P, it);
    }
  }
  __device__ __forceinline__ Chunks(const ExParams& P, int first) : it(blockIdx.x), i(first) {
    if (it < P.nitems) I = decode<MODE>(P, it);
    settle(P);
  }
  __device__ __forceinline__ bool valid(const ExParams& P) const { return it < P.nitems; }
  __device__ __forceinline__ void next(const ExParams& P, int step) {
    i += step;
    settle(P);
  }
};

template <int MODE>
__global__ void __launch_bounds__(EX_THREADS, 1) ex_kernel(const __grid_constant__ ExParams P) {
  constexpr int SH = MODE == EX_CELL ? 45 : 41;   // units of the integer sums
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* wordsA = smem + STAGES * B_STAGE;
  unsigned char* wordsB = wordsA + 8 * A_DEP * A_WORDS;
  uint64_t* bars = reinterpret_cast<uint64_t*>(wordsB + 3 * B_DEP * B_WORDS);
  constexpr int NBAR = 4 + 2 * STAGES + 2 * NG + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NBAR);
  const uint32_t bar0 = smem_u32(bars);
  auto fa = [&](int s) { return bar0 + 8 * s; };                        // M buffer full
  auto ea = [&](int s) { return bar0 + 8 * (2 + s); };                  // M buffer free
  auto fb = [&](int s) { return bar0 + 8 * (4 + s); };                  // N stage full
  auto eb = [&](int s) { return bar0 + 8 * (4 + STAGES + s); };         // N stage free
  auto gf = [&](int g) { return bar0 + 8 * (4 + 2 * STAGES + g); };     // group complete
  auto ge = [&](int g) { return bar0 + 8 * (4 + 2 * STAGES + NG + g); };   // group drained
  const uint32_t done = bar0 + 8 * (NBAR - 1);
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(fa(s), P.watch.withhold && blockIdx.x == 0 ? 5 : 4);   // 5: never full (test hook)
      mbar_init(ea(s), 1);
    }
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(fb(s), 3);
      mbar_init(eb(s), 1);
    }
    for (int g = 0; g < NG; ++g) {
      mbar_init(gf(g), 1);
      mbar_init(ge(g), 8);
    }
    mbar_init(done, 1);
    fence_mbar_init();
  }
  if (warp == 19) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int seg = MODE == EX_CELL && *P.hsum <= (1 << 24) - (1 << 18) ? 1 << 20 : SEG;   // chunks per segment
  // A role whose wait gives up records it and leaves; the waits of the roles
  // that depend on it then run out in turn, so that every warp reaches the end.
  auto give_up = [&](int site) { report_timeout(P.watch.status, site); };

  if (warp < 8) {
    // ---- drain: lane quarter warp % 4, N columns HN (warp / 4) ..
    const int q = warp & 3, half = warp >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + half * HN;
    int sc = 0;   // segments so far
    for (int64_t it = blockIdx.x; it < P.nitems; it += gridDim.x) {
      const Item I = decode<MODE>(P, it);
      const int nseg = (I.nk + seg - 1) / seg;
      int64_t V[HN];
#pragma unroll
      for (int j = 0; j < HN; ++j) V[j] = 0;
      bool first = true, ok = true;
      for (int sg = 0; sg < nseg; ++sg, ++sc) {
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          ok = __all_sync(0xffffffffu, ok && mbar_wait(gf(g), sc & 1));
          if (!ok) break;
          tc_fence_after();
          float f[HN];
#pragma unroll
          for (int b = 0; b < HN; b += 8) tmem_ld8(tbase + g * BN + b, f + b);
          tmem_wait_ld();
          tc_fence_before();       // the group's columns may be overwritten
          __syncwarp();
          if (lane == 0) mbar_arrive(ge(g));
#pragma unroll
          for (int j = 0; j < HN; ++j) add_group<SH>(V[j], f[j], g);
        }
        if (!ok) break;
        if (sg % FLUSH != FLUSH - 1 && sg != nseg - 1) continue;
        // ---- round to binary64 and write (later flushes add to the first)
        const int j0 = half * HN;
        const int m = q * 32 + lane;
        int en = 0, em = 0;            // scales: N index j0 + lane, M index m
        double* out;
        int64_t so;                    // stride between N indices
        if (MODE == EX_CELL) {
          if (j0 + lane < I.nv) en = P.hexp[(P.e0 + I.row) * P.ne + I.n0 + j0 + lane];
          if (m < I.mv) em = P.cexp[I.row * P.ncol + I.m0 + m];
          out = P.C + ((P.e0 + I.row) * P.ne + I.n0 + j0) * P.ldc + I.m0 + m;
          so = P.ldc;
        } else if (MODE == EX_GRAM) {
          if (j0 + lane < I.nv) en = P.bexp[I.n0 + j0 + lane];
          if (m < I.mv) em = P.aexp[I.m0 + m];
          out = P.C + I.row * (int64_t)P.n1 * P.n2 + (int64_t)(I.n0 + j0) * P.n1 + I.m0 + m;
          so = P.n1;
        } else {
          if (j0 + lane < I.nv) en = P.uexp[I.n0 + j0 + lane];
          if (m < I.mv) em = P.rexp[P.r0 + I.row + m];
          out = P.C + (P.r0 + I.row + m) * P.ldc + I.n0 + j0;
          so = 1;
        }
        const int64_t off = (int64_t)(group_offset<SH>() * (uint64_t)(sg % FLUSH + 1));   // segments in V
        constexpr int bad = MODE == EX_TALL ? kNonFinite : 2047;
        // tiles that may hold results below 2^-1022 (the smallest sum of their scales
        // with a single unit of V) are written by a loop of their own: with the tests
        // of that case in the one loop 8^3 cells, p = 6, 220 columns take 49.37 ms for
        // 40 steps, 48.97 this way and as without them
        auto write = [&](auto low) {
#pragma unroll
          for (int j = 0; j < HN; ++j) {
            const int e = __shfl_sync(0xffffffffu, en, j);
            if (j0 + j < I.nv && m < I.mv) {
              double v;
              if (e == bad || em == bad) v = quiet_nan();
              else v = compose<SH, decltype(low)::value>(V[j] - off, e + em);     // a vector of zeros has V = 0
              if (!first) v += *out;
              *out = v;
            }
            out += so;
            V[j] = 0;
          }
        };
        const int mn = __reduce_min_sync(0xffffffffu, j0 + lane < I.nv && lane < HN ? en : 1 << 20);
        if (__any_sync(0xffffffffu, m < I.mv && em + mn <= 1033 + SH)) write(std::true_type());
        else write(std::false_type());
        first = false;
      }
      if (!ok) {
        give_up(91);
        break;
      }
    }
  } else if (warp < 16) {
    // ---- M operand: set (warp - 8) / 4 takes the chunks of its parity.  Each
    // warp copies the words of its 32 rows A_DEP chunks ahead (16-byte pieces of
    // two rows; pieces past the edge are not copied: any word is a finite number
    // and their results are not stored; K is padded with zero words).
    const int q = warp & 3, set = (warp - 8) >> 2;
    const uint32_t tdst = tmem + ((uint32_t)(q * 32) << 16) + TA + set * TA_BUF;
    unsigned char* stage = wordsA + (warp - 8) * A_DEP * A_WORDS;
    Chunks<MODE> L(P, set);
    int issued = 0;
    auto issue = [&] {
      if (L.valid(P)) {
        const int piece = lane & 15, k0 = lane >> 4;
        const int r = q * 32 + piece * 2;
        const uint64_t* src = L.I.a + ((int64_t)L.i * KC + k0) * P.sa + r;
        const uint32_t dst = smem_u32(stage + issued % A_DEP * A_WORDS) + k0 * 256 + piece * 16;
        if (r < L.I.mv) {
#pragma unroll
          for (int k = 0; k < KC; k += 2) cp_async16(dst + k * 256, src + (int64_t)k * P.sa);
        }
        ++issued;
        L.next(P, 2);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int d = 0; d < A_DEP; ++d) issue();
    bool ok = true;
    int ph = 1;
    for (int n = 0; n < issued; ++n) {
      cp_async_wait<A_DEP - 1>();
      __syncwarp();
      const uint64_t* w = reinterpret_cast<const uint64_t*>(stage + n % A_DEP * A_WORDS) + lane;
      uint32_t o[NA * 8];
#pragma unroll
      for (int k = 0; k < KC; k += 2) expand_pair<NA>(w[k * 32], w[k * 32 + 32], o + k / 2, 8);
      __syncwarp();
      issue();
      ok = __all_sync(0xffffffffu, mbar_wait(ea(set), ph));
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int d = 0; d < NA; ++d) tmem_st8(tdst + d * 8, o + d * 8);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(fa(set));
      ph ^= 1;
    }
    cp_async_wait<0>();
    if (!ok) give_up(92);
  } else if (warp < 19) {
    // ---- N operand: 16 rows x 2 halves of K per warp, copied likewise
    const int bw = warp - 16;
    const int rl = lane & 15, h = lane >> 4;
    unsigned char* stage = wordsB + bw * B_DEP * B_WORDS;
    unsigned char* base = smem + elem_off(bw * 16 + rl, h * 8) * 2;
    Chunks<MODE> L(P, 0);
    int issued = 0;
    auto issue = [&] {
      if (L.valid(P)) {
        const int piece = lane & 7, k0 = lane >> 3;
        const int r = bw * 16 + piece * 2;
        const uint32_t dst = smem_u32(stage + issued % B_DEP * B_WORDS) + k0 * 128 + piece * 16;
        if (r < L.I.nv) {
#pragma unroll
          for (int k = 0; k < KC; k += 4) {
            const int kk = min(L.i * KC + k0 + k, L.I.kmax - 1);
            cp_async16(dst + k * 128, L.I.b + (int64_t)kk * P.sb + r);
          }
        }
        ++issued;
        L.next(P, 1);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int d = 0; d < B_DEP; ++d) issue();
    int st = 0, ph = 1;
    bool ok = true;
    for (int n = 0; n < issued; ++n) {
      cp_async_wait<B_DEP - 1>();
      __syncwarp();
      const uint64_t* w = reinterpret_cast<const uint64_t*>(stage + n % B_DEP * B_WORDS) + h * 8 * 16 + rl;
      uint32_t o[NB * 4];
#pragma unroll
      for (int k = 0; k < 8; k += 2) expand_pair<NB>(w[k * 16], w[k * 16 + 16], o + k / 2, 4);
      __syncwarp();
      issue();
      ok = __all_sync(0xffffffffu, mbar_wait(eb(st), ph));
      if (!ok) break;
#pragma unroll
      for (int d = 0; d < NB; ++d)
        *reinterpret_cast<uint4*>(base + st * B_STAGE + d * PLANE) =
            make_uint4(o[4 * d], o[4 * d + 1], o[4 * d + 2], o[4 * d + 3]);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(fb(st));
      if (++st == STAGES) st = 0, ph ^= 1;
    }
    cp_async_wait<0>();
    if (!ok) give_up(93);
  } else if (elect_one()) {
    int st = 0, ph = 0, sc = 0;
    int ab = 0, pa = 0;            // M buffer and its phase
    bool ok = true;
    for (int64_t it = blockIdx.x; it < P.nitems && ok; it += gridDim.x) {
      const Item I = decode<MODE>(P, it);
      const int nseg = (I.nk + seg - 1) / seg;
      for (int sg = 0; sg < nseg && ok; ++sg, ++sc) {
        // segments of nearly equal length
        const int i0 = (int)((int64_t)I.nk * sg / nseg), i1 = (int)((int64_t)I.nk * (sg + 1) / nseg);
        for (int i = i0; i < i1; ++i) {
          ok = mbar_wait(fb(st), ph) && mbar_wait(fa(ab), pa);
          if (!ok) break;
          tc_fence_after();
          const uint32_t ta = tmem + TA + ab * TA_BUF;
          const uint64_t b0 = umma_desc(smem_u32(smem + st * B_STAGE), 128, 256);
          // M digit d times the N digits 0 .. 7 - d at once: their planes lie one
          // after another along N, as the accumulators of the groups d .. 7 do, so
          // one MMA of up to 256 columns takes up to five of the products (10
          // MMAs per chunk; 35 single ones are bound by their issue)
#pragma unroll
          for (int d = 0; d < NA; ++d) {
            constexpr int NMAX = 256 / BN;
            const int n1 = NG - d <= NMAX ? NG - d : (NG - d + 1) / 2;
            if (d == 0 && i == i0) {   // the accumulators of the previous segment have been read
#pragma unroll
              for (int g = 0; g < n1; ++g) ok = ok && mbar_wait(ge(g), (sc & 1) ^ 1);
              tc_fence_after();
            }
            if (ok) mma_f16_ts(tmem + d * BN, ta + d * 8, b0, idesc_f16(BM, n1 * BN), i > i0 || d > 0);
            if (n1 < NG - d) {
              if (d == 0 && i == i0) {
#pragma unroll
                for (int g = n1; g < NG; ++g) ok = ok && mbar_wait(ge(g), (sc & 1) ^ 1);
                tc_fence_after();
              }
              if (ok)
                mma_f16_ts(tmem + (d + n1) * BN, ta + d * 8, b0 + (uint64_t)(n1 * (PLANE / 16)),
                           idesc_f16(BM, (NG - d - n1) * BN), i > i0 || d > 0);
            }
            if (ok && i == i1 - 1) {
              umma_commit(gf(d));
              if (d == NA - 1) umma_commit(gf(d + 1));
            }
          }
          if (!ok) break;
          umma_commit(eb(st));
          umma_commit(ea(ab));
          if (++st == STAGES) st = 0, ph ^= 1;
          if ((ab ^= 1) == 0) pa ^= 1;
        }
      }
    }
    if (!ok) give_up(94);
    umma_commit(done);           // every MMA issued has completed before TMEM is freed
    mbar_wait(done, 0);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 19) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------- words
// The block's rows of every cell as words (K-major, rows padded to a multiple of
// 16 with zero words, row stride ldw) and the
// scales of the (cell, column) pairs: block (32, 8) per (cell, 32 columns),
// one pass for the largest entry, one (out of L1 / L2) for the words.
__global__ void __launch_bounds__(256) ex_cell_words_kernel(const int32_t* __restrict__ dofmap, int64_t e0, int ne,
                                                            const double* __restrict__ Y, int64_t ldy, int ncol,
                                                            int16_t* __restrict__ cexp, uint64_t* __restrict__ W,
                                                            int ldw) {
  const int64_t e = blockIdx.x;
  const int nep = (ne + KC - 1) / KC * KC;
  const int c = blockIdx.y * 32 + threadIdx.x;
  const int32_t* dm = dofmap + (e0 + e) * ne;
  int m = 0;
  if (c < ncol) {
#pragma unroll 8
    for (int l = threadIdx.y; l < ne; l += 8) {
      const int g = __ldg(dm + l);
      if (g >= 0) m = max(m, __double2hiint(__ldg(Y + (int64_t)g * ldy + c)) & 0x7fffffff);
    }
  }
  __shared__ int red[8][32];
  red[threadIdx.y][threadIdx.x] = m;
  __syncthreads();
  if (c >= ncol) return;
#pragma unroll
  for (int w = 0; w < 8; ++w) m = max(m, red[w][threadIdx.x]);
  m = max(m >> 20, 1);
  if (threadIdx.y == 0) cexp[e * ncol + c] = (int16_t)m;
#pragma unroll 8
  for (int l = threadIdx.y; l < nep; l += 8) {
    const int g = l < ne ? __ldg(dm + l) : -1;
    uint64_t w = kZeroWord;
    if (g >= 0) {
      const double v = __ldg(Y + (int64_t)g * ldy + c);
      w = word_of(v, m - expo(v));
    }
    W[(e * nep + l) * ldw + c] = w;
  }
}

// Exponent field of the largest entry of every column of X (M x n); out zeroed
// by the caller.  finite: entries that are infinities or NaN do not count.
__global__ void __launch_bounds__(256) ex_col_scale_kernel(const double* __restrict__ X, int64_t ldx, int64_t M,
                                                           int n, int finite, int* __restrict__ out) {
  const int c = blockIdx.x * 32 + threadIdx.x;
  int m = 0;
  if (c < n) {
#pragma unroll 8
    for (int64_t r = (int64_t)blockIdx.y * 8 + threadIdx.y; r < M; r += (int64_t)gridDim.y * 8) {
      const int e = expo(__ldg(X + r * ldx + c));
      m = max(m, finite && e == 2047 ? 1 : e);
    }
  }
  __shared__ int red[8][32];
  red[threadIdx.y][threadIdx.x] = m;
  __syncthreads();
  if (threadIdx.y == 0 && c < n) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, red[w][threadIdx.x]);
    atomicMax(out + c, m);
  }
}

// Words of rows [0, M) of X under its column scales (row stride ldw), padded to a
// multiple of 16 rows with zero words.
__global__ void __launch_bounds__(256) ex_col_words_kernel(const double* __restrict__ X, int64_t ldx, int64_t M,
                                                           int n, const int* __restrict__ cexp,
                                                           uint64_t* __restrict__ W, int ldw) {
  const int c = blockIdx.x * 32 + threadIdx.x;
  if (c >= n) return;
  const int m = cexp[c];
  const int64_t mp = (M + KC - 1) / KC * KC;
#pragma unroll 8
  for (int64_t r = (int64_t)blockIdx.y * 8 + threadIdx.y; r < mp; r += (int64_t)gridDim.y * 8) {
    const double v = r < M ? __ldg(X + r * ldx + c) : 0.0;
    W[r * ldw + c] = word_of(v, m - expo(v));
  }
}

// Row scales of X relative to its column scales: max_k (exponent(x_rk) - ecol[k]).
__global__ void __launch_bounds__(256) ex_row_scale_kernel(const double* __restrict__ X, int64_t ldx, int64_t M,
                                                           int n, const int* __restrict__ ecol,
                                                           int* __restrict__ rexp) {
  const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= M) return;
  int m = kNoScale;
#pragma unroll 4
  for (int k = lane; k < n; k += 32) {
    const double v = __ldg(X + r * ldx + k);
    const int e = expo(v);
    if (nonzero(v)) m = max(m, e == 2047 ? kNonFinite : e - __ldg(ecol + k));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) rexp[r] = m;
}

// Words of X under its row scales, transposed tile by tile: W[tile][k][128 rows],
// k padded to a multiple of 16 with zero words.  Block (32, 8): 32 rows x 32 columns.
__global__ void __launch_bounds__(256) ex_row_words_kernel(const double* __restrict__ X, int64_t ldx, int64_t M,
                                                           int n, const int* __restrict__ ecol,
                                                           const int* __restrict__ rexp, uint64_t* __restrict__ W) {
  __shared__ uint64_t t[32][33];
  const int64_t r0 = (int64_t)blockIdx.x * 32;
  const int k0 = blockIdx.y * 32;
  const int k = k0 + threadIdx.x;
  const int ek = k < n ? ecol[k] : 0;
#pragma unroll
  for (int i = 0; i < 32; i += 8) {
    const int64_t r = r0 + threadIdx.y + i;
    uint64_t w = kZeroWord;
    if (r < M && k < n) {
      const double v = __ldg(X + r * ldx + k);
      w = word_of(v, rexp[r] - expo(v) + ek);
    }
    t[threadIdx.y + i][threadIdx.x] = w;
  }
  __syncthreads();
  const int64_t tile = r0 / BM;
  const int rr = (int)(r0 % BM) + threadIdx.x, np = (n + KC - 1) / KC * KC;
#pragma unroll
  for (int i = 0; i < 32; i += 8) {
    const int kk = k0 + threadIdx.y + i;
    if (kk < np) W[(tile * np + kk) * BM + rr] = t[threadIdx.x][threadIdx.y + i];
  }
}

// Scales of U's columns with the column scales of X folded in, one warp per column.
__global__ void __launch_bounds__(256) ex_u_scale_kernel(const double* __restrict__ U, int64_t ldu, int n1, int n2,
                                                         int upper, int trans, const int* __restrict__ ecol,
                                                         int* __restrict__ uexp) {
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (j >= n2) return;
  int m = kNoScale;
  const int kend = upper ? min(n1, j + 1) : n1;
  for (int k = lane; k < kend; k += 32) {
    const double v = trans ? U[j + (int64_t)k * ldu] : U[k + (int64_t)j * ldu];
    const int e = expo(v);
    if (nonzero(v)) m = max(m, e == 2047 ? kNonFinite : e + ecol[k]);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) uexp[j] = m;
}

// Words of U, K-major (row stride ldw).
__global__ void __launch_bounds__(256) ex_u_words_kernel(const double* __restrict__ U, int64_t ldu, int n1, int n2,
                                                         int upper, int trans, const int* __restrict__ ecol,
                                                         const int* __restrict__ uexp, uint64_t* __restrict__ W,
                                                         int ldw) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n1 * n2) return;
  const int j = (int)(idx % n2), k = (int)(idx / n2);
  uint64_t w = kZeroWord;
  if (!upper || k <= j) {
    const double x = trans ? U[j + (int64_t)k * ldu] : U[k + (int64_t)j * ldu];
    w = word_of(x, uexp[j] - expo(x) - ecol[k]);
  }
  W[(int64_t)k * ldw + j] = w;
}

// Scales of the cell matrices' rows, one warp per row (the exponent of the
// largest entry, raised until the first digits add up to at most 2,040), and the largest over all
// rows (atomicMax into hsum, zeroed by the caller) of the bounds of their group
// sums g <= 5: the sums of |digits| of the row against the largest digits any M
// vector can have (64 for the first, else 128).  Up to 2^24 one FP32 segment
// over the whole row is exact.
__global__ void __launch_bounds__(256) ex_h_scale_kernel(const double* __restrict__ Ht, int64_t rows, int ne,
                                                         int16_t* __restrict__ hexp, int* __restrict__ hsum) {
  const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  int m = 0;
  for (int k = lane; k < ne; k += 32)
    if (nonzero(Ht[r * ne + k])) m = max(m, expo(Ht[r * ne + k]));
  m = __reduce_max_sync(0xffffffffu, m);
  if (m == 0) m = 1023;   // the row of an eliminated node: any scale, not one that looks like tiny results
  int a[6];
  for (int up = 0;; ++up) {
#pragma unroll
    for (int d = 0; d < 6; ++d) a[d] = 0;
    for (int k = lane; k < ne; k += 32) {
      const double v = Ht[r * ne + k];
      const uint64_t w = word_of(v, m - expo(v));
#pragma unroll
      for (int d = 0; d < 6; ++d) a[d] += abs((int)((w >> (56 - 8 * d)) & 0xff) - 128);
    }
#pragma unroll
    for (int d = 0; d < 6; ++d) a[d] = __reduce_add_sync(0xffffffffu, a[d]);
    if (a[0] <= 2040 || m >= 2040 || up == 8) break;   // |V| <= 64 a[0] 2^45 + ... < 2^63
    ++m;
  }
  int bound = 0, below = 0;
#pragma unroll
  for (int g = 0; g < 6; ++g) {
    bound = max(bound, (64 * a[g] + 128 * below) * (g < 2 ? 4 : 1));
    below += a[g];
  }
  if (lane == 0) {
    hexp[r] = (int16_t)m;
    atomicMax(hsum, bound);
  }
}

// ---------------------------------------------------------------- assembly, reduction
// Each thread: one unknown, two columns (pairs of a row in consecutive threads).
// Sums the cell rows holding the unknown in ascending cell order, adds the
// projector term, applies the three-term update.  Y_out may alias Y_prev, not Y_in.
__global__ void __launch_bounds__(256) ex_assemble_kernel(const __grid_constant__ ExAssembleArgs P, int vio) {
  const uint32_t np = (uint32_t)(P.ncol + 1) / 2;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int64_t j = idx >> 32 ? idx / np : (int64_t)((uint32_t)idx / np);
  const int c = (int)(idx - j * np) * 2;
  if (j >= P.M || c >= P.ncol) return;
  const bool two = c + 1 < P.ncol;
  const int k0 = __ldg(P.node_ptr + j), n = __ldg(P.node_ptr + j + 1) - k0;
  // the rows of Y first, then the rows of R two at a time (an unknown lies in 1,
  // 2, 4 or 8 cells)
  double y0 = 0.0, y1 = 0.0, p0 = 0.0, p1 = 0.0;
  double* out = P.Yout + j * P.ld_out + c;
  if (vio && two) {
    if (P.shift != 0.0) {
      const double2 t = *reinterpret_cast<const double2*>(P.Yin + j * P.ld_in + c);
      y0 = t.x;
      y1 = t.y;
    }
    if (P.Yprev) {
      const double2 t = *reinterpret_cast<const double2*>(P.Yprev + j * P.ld_prev + c);
      p0 = t.x;
      p1 = t.y;
    }
  } else {
    if (P.shift != 0.0) {
      y0 = P.Yin[j * P.ld_in + c];
      if (two) y1 = P.Yin[j * P.ld_in + c + 1];
    }
    if (P.Yprev) {
      p0 = P.Yprev[j * P.ld_prev + c];
      if (two) p1 = P.Yprev[j * P.ld_prev + c + 1];
    }
  }
  double s0 = 0.0, s1 = 0.0;                   // rows of R are padded to an even length
  int k = k0;
  if (n & 1) {
    const double2 r = __ldg(reinterpret_cast<const double2*>(P.R + (int64_t)__ldg(P.node_ent + k) * P.ldr + c));
    s0 = r.x;
    s1 = r.y;
    ++k;
  }
#pragma unroll 1
  for (; k < k0 + n; k += 2) {
    const int e0 = __ldg(P.node_ent + k), e1 = __ldg(P.node_ent + k + 1);
    const double2 r = __ldg(reinterpret_cast<const double2*>(P.R + (int64_t)e0 * P.ldr + c));
    const double2 t = __ldg(reinterpret_cast<const double2*>(P.R + (int64_t)e1 * P.ldr + c));
    s0 += r.x;
    s1 += r.y;
    s0 += t.x;
    s1 += t.y;
  }
  if (P.NL) {
    s0 += P.NL[j * P.ld_nl + c];
    if (two) s1 += P.NL[j * P.ld_nl + c + 1];
  }
  // alpha (s - shift y) + beta y_prev in three operations: the kernel moves 37
  // bytes per value and a binary64 operation per value costs as much time as 11
  double o0 = P.alpha * s0, o1 = P.alpha * s1;
  if (P.shift != 0.0) {
    const double as = -P.alpha * P.shift;
    o0 = fma(as, y0, o0);
    o1 = fma(as, y1, o1);
  }
  if (P.Yprev) {
    o0 = fma(P.beta, p0, o0);
    o1 = fma(P.beta, p1, o1);
  }
  if (vio && two) {
    *reinterpret_cast<double2*>(out) = make_double2(o0, o1);
  } else {
    out[0] = o0;
    if (two) out[1] = o1;
  }
}

// C = (C with add, else 0) + the row splits, in ascending order.
__global__ void ex_reduce_kernel(const double* __restrict__ partial, int nsplit, int n1, int n2,
                                 double* __restrict__ C, int64_t ldc, int lower, int add) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n1 * n2) return;
  const int i = (int)(idx % n1), j = (int)(idx / n1);
  if (lower && i / BM < j / BN * BN / BM) return;    // tile not computed
  double s = add ? C[i + (int64_t)j * ldc] : 0.0;
  for (int z = 0; z < nsplit; ++z) s += partial[(int64_t)z * n1 * n2 + idx];
  C[i + (int64_t)j * ldc] = s;
}

int sm_count() {
  static int n = 0;
  static std::once_flag f;
  std::call_once(f, [] {
    int d = 0;
    cudaGetDevice(&d);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d) != cudaSuccess || n < 1) n = 152;
  });
  return n;
}

template <int MODE>
cudaError_t launch(const ExParams& P, cudaStream_t s) {
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(ex_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, EX_SMEM);
  });
  if (P.nitems <= 0) return cudaSuccess;
  note_launch();
  ex_kernel<MODE><<<(unsigned)std::min<int64_t>(P.nitems, sm_count()), EX_THREADS, EX_SMEM, s>>>(P);
  return cudaGetLastError();
}

int pad2(int n) { return (n + 1) & ~1; }       // 16-byte rows of words
int64_t padk(int64_t k) { return (k + KC - 1) / KC * KC; }
size_t align256(size_t b) { return (b + 255) / 256 * 256; }

// Row blocks of the column-wise passes: about 8 thread blocks per SM.
unsigned row_blocks(int64_t M, int n) {
  const int64_t xs = (n + 31) / 32;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((M + 63) / 64, (8 * 152 + xs - 1) / xs));
}
cudaError_t col_scale(const double* X, int64_t ldx, int64_t M, int n, int finite, int* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, (size_t)n * sizeof(int), s);
  if (e != cudaSuccess) return e;
  note_launch();
  ex_col_scale_kernel<<<dim3((n + 31) / 32, row_blocks(M, n)), dim3(32, 8), 0, s>>>(X, ldx, M, n, finite, out);
  return cudaGetLastError();
}

int gram_tiles(int n1, int n2, int lower) {
  const int t1 = (n1 + BM - 1) / BM, t2 = (n2 + BN - 1) / BN;
  if (!lower) return t1 * t2;
  int n = 0;
  for (int tj = 0; tj < t2; ++tj) n += std::max(0, t1 - tj * BN / BM);
  return n;
}
// Plan of a Gram product: rows in `slices` launches of `srows` rows, each in
// `nsplit` splits of `rps` rows (the last launch may have fewer).
struct GramPlan {
  int64_t srows, slices, rps, nsplit;
};
GramPlan gram_plan(int64_t M, int n1, int n2, int lower, bool same) {
  GramPlan g;
  const int64_t per_row = 8 * (int64_t)(same ? n1 : n1 + n2);
  g.srows = std::max<int64_t>(KC, (int64_t)kWordBytes / per_row / KC * KC);
  g.slices = (M + g.srows - 1) / g.srows;
  g.srows = ((M + g.slices - 1) / g.slices + KC - 1) / KC * KC;      // even slices
  g.slices = (M + g.srows - 1) / g.srows;
  // splits of a slice: the count whose last wave of tiles is fullest, up to eight
  // or as many as write 64 MB of partial sums over all slices (each is written and
  // read again).  The sums of one slice are added to C before the next one's: kept
  // for all of them they would take 25 GB at 2.7 million rows and 3,000 columns.
  const int64_t tiles = std::max(1, gram_tiles(n1, n2, lower));
  const int64_t cap = std::max<int64_t>(8, ((int64_t)64 << 20) / ((int64_t)n1 * n2 * 8) / g.slices);
  const int nsm = sm_count();
  double bestc = 1e300;
  int64_t best = 1;
  for (int64_t z = 1; z <= std::min<int64_t>(cap, (g.srows + 255) / 256); ++z) {
    const int64_t r = ((g.srows + z - 1) / z + KC - 1) / KC * KC;
    const int64_t waves = (tiles * z + nsm - 1) / nsm;
    // rows per SM plus a fixed cost per tile (pipeline fill and drain, about 100 rows)
    const double c = (double)waves * (double)(r + 100);
    if (c < bestc * 0.995) bestc = c, best = z;
  }
  g.rps = ((g.srows + best - 1) / best + KC - 1) / KC * KC;
  g.nsplit = (g.srows + g.rps - 1) / g.rps;
  return g;
}

// Rows per launch of a rotation (whole 128-row tiles).
int64_t tall_rows(int64_t M, int n1) {
  const int64_t tiles = (M + BM - 1) / BM;
  const int64_t fit = std::max<int64_t>(1, (int64_t)kWordBytes / (8ll * BM * n1));
  const int64_t slices = (tiles + fit - 1) / fit;
  return (tiles + slices - 1) / slices * BM;
}
// Cells per launch.
int64_t cell_slice(int64_t ncells, int ne, int ncol) {
  const int64_t fit = std::max<int64_t>(1, (int64_t)kWordBytes / (8ll * ne * ncol));
  const int64_t slices = (ncells + fit - 1) / fit;
  return (ncells + slices - 1) / slices;
}

}  // namespace

int64_t ex_cell_tiles(int64_t ncells, int ne, int ncol) {
  return ncells * ((ne + BN - 1) / BN) * ((ncol + BM - 1) / BM);
}

void ex_cell_bytes(int64_t ncells, int ne, size_t* words, size_t* ex) {
  *words = (size_t)ncells * ne * pad2(ne) * sizeof(uint64_t);
  *ex = 16 + (size_t)ncells * ne * sizeof(int16_t);
}

cudaError_t ex_pack_cells(const ExCellData& d, const CellMatArgs& m, int ne, cudaStream_t s) {
  const int64_t rows = m.ncells * ne;
  cudaError_t e = cudaMemsetAsync(d.hsum, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  note_launch();
  ex_h_scale_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(m.Ht, rows, ne, d.hexp(), d.hsum);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return launch_cell_words(m, d.hexp(), d.words, pad2(ne), s);
}

size_t ex_cell_work_bytes(int64_t ncells, int ne, int ncol) {
  const size_t c = (size_t)cell_slice(ncells, ne, ncol);
  return align256(c * ncol * sizeof(int16_t)) + c * padk(ne) * pad2(ncol) * sizeof(uint64_t);
}

cudaError_t ex_cell_launch(const ExCellData& d, const ExCellArgs& a, const ExWatch& w, cudaStream_t s) {
  if (a.ncells <= 0 || a.ncol <= 0) return cudaSuccess;
  const int64_t slice = cell_slice(a.ncells, a.ne, a.ncol);
  int16_t* cexp = (int16_t*)a.work;
  uint64_t* W = (uint64_t*)((char*)a.work + align256((size_t)slice * a.ncol * sizeof(int16_t)));
  for (int64_t e0 = 0; e0 < a.ncells; e0 += slice) {
    const int64_t n = std::min(slice, a.ncells - e0);
    note_launch();
    ex_cell_words_kernel<<<dim3((unsigned)n, (a.ncol + 31) / 32), dim3(32, 8), 0, s>>>(
        a.dofmap, e0, a.ne, a.Y, a.ldy, a.ncol, cexp, W, pad2(a.ncol));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ExParams P{};
    P.A = W;
    P.sa = pad2(a.ncol);
    P.B = d.words;
    P.sb = pad2(a.ne);
    P.e0 = e0;
    P.hexp = d.hexp();
    P.hsum = d.hsum;
    P.cexp = cexp;
    P.ne = a.ne;
    P.ncol = a.ncol;
    P.C = a.R;
    P.ldc = a.ldr;
    P.nitems = ex_cell_tiles(n, a.ne, a.ncol);
    P.watch = w;
    if ((e = launch<EX_CELL>(P, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t ex_assemble_launch(const ExAssembleArgs& a, cudaStream_t s) {
  if (a.M <= 0 || a.ncol <= 0) return cudaSuccess;
  auto al = [](const void* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 1) == 0; };
  const int vio = al(a.Yin, a.ld_in) && al(a.Yout, a.ld_out) && (!a.Yprev || al(a.Yprev, a.ld_prev));
  note_launch();
  ex_assemble_kernel<<<(unsigned)((a.M * ((a.ncol + 1) / 2) + 255) / 256), 256, 0, s>>>(a, vio);
  return cudaGetLastError();
}

static size_t gram_bytes(const GramPlan& g, int n1, int n2, bool same) {
  return align256((size_t)(n1 + n2) * sizeof(int)) + align256((size_t)g.nsplit * n1 * n2 * sizeof(double)) +
         (size_t)g.srows * (same ? pad2(n1) : pad2(n1) + pad2(n2)) * sizeof(uint64_t);
}
size_t ex_gram_work_bytes(int64_t M, int n1, int n2, int lower) {
  return std::max(gram_bytes(gram_plan(M, n1, n2, lower, false), n1, n2, false),
                  gram_bytes(gram_plan(M, n1, n2, lower, true), n1, n2, true));
}

cudaError_t ex_gram(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t M, int n1, int n2,
                    double* C, int64_t ldc, int lower, void* work, size_t work_bytes, const ExWatch& w,
                    cudaStream_t s) {
  if (n1 <= 0 || n2 <= 0) return cudaSuccess;
  const bool same = B == A && ldb == lda && n2 <= n1;
  const GramPlan g = gram_plan(M, n1, n2, lower, same);
  if (work_bytes < gram_bytes(g, n1, n2, same)) return cudaErrorInvalidValue;
  int* aexp = (int*)work;
  int* bexp = same ? aexp : aexp + n1;
  double* partial = (double*)((char*)work + align256((size_t)(n1 + n2) * sizeof(int)));
  uint64_t* WA = (uint64_t*)((char*)partial + align256((size_t)g.nsplit * n1 * n2 * sizeof(double)));
  uint64_t* WB = same ? WA : WA + (size_t)g.srows * pad2(n1);
  cudaError_t e = col_scale(A, lda, M, n1, 0, aexp, s);
  if (e != cudaSuccess) return e;
  if (!same && (e = col_scale(B, ldb, M, n2, 0, bexp, s)) != cudaSuccess) return e;
  for (int64_t i = 0; i < g.slices; ++i) {
    const int64_t r0 = i * g.srows, rows = std::min(g.srows, M - r0);
    note_launch();
    ex_col_words_kernel<<<dim3((n1 + 31) / 32, row_blocks(rows, n1)), dim3(32, 8), 0, s>>>(A + r0 * lda, lda, rows, n1,
                                                                                           aexp, WA, pad2(n1));
    if (!same) {
      note_launch();
      ex_col_words_kernel<<<dim3((n2 + 31) / 32, row_blocks(rows, n2)), dim3(32, 8), 0, s>>>(B + r0 * ldb, ldb, rows,
                                                                                             n2, bexp, WB, pad2(n2));
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ExParams P{};
    P.A = WA;
    P.sa = pad2(n1);
    P.B = WB;
    P.sb = pad2(same ? n1 : n2);
    P.M = rows;
    P.rps = g.rps;
    P.n1 = n1;
    P.n2 = n2;
    P.aexp = aexp;
    P.bexp = bexp;
    P.lower = lower;
    P.ntile = gram_tiles(n1, n2, lower);
    P.C = partial;
    const int64_t nsplit = (rows + g.rps - 1) / g.rps, tot = (int64_t)n1 * n2;
    P.nitems = P.ntile * nsplit;
    P.watch = w;
    if ((e = launch<EX_GRAM>(P, s)) != cudaSuccess) return e;
    note_launch();
    ex_reduce_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(partial, (int)nsplit, n1, n2, C, ldc, lower, i > 0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t ex_tall_work_bytes(int64_t M, int n1, int n2) {
  return align256((size_t)M * 4) + align256((size_t)(n1 + n2) * 4) + align256((size_t)n1 * pad2(n2) * 8) +
         (size_t)tall_rows(M, n1) * padk(n1) * 8;
}

cudaError_t ex_tall(const double* A, int64_t lda, const double* U, int64_t ldu, int64_t M, int n1, int n2,
                    double* C, int64_t ldc, int upper, int trans, void* work, const ExWatch& w, cudaStream_t s) {
  if (M <= 0 || n1 <= 0 || n2 <= 0) return cudaSuccess;
  int* rexp = (int*)work;
  int* ecol = (int*)((char*)work + align256((size_t)M * 4));
  int* uexp = ecol + n1;
  uint64_t* WU = (uint64_t*)((char*)ecol + align256((size_t)(n1 + n2) * 4));
  uint64_t* WX = (uint64_t*)((char*)WU + align256((size_t)n1 * pad2(n2) * 8));
  cudaError_t e = col_scale(A, lda, M, n1, 1, ecol, s);
  if (e != cudaSuccess) return e;
  note_launch();
  ex_row_scale_kernel<<<(unsigned)((M + 7) / 8), 256, 0, s>>>(A, lda, M, n1, ecol, rexp);
  note_launch();
  ex_u_scale_kernel<<<(n2 + 7) / 8, 256, 0, s>>>(U, ldu, n1, n2, upper, trans, ecol, uexp);
  const int64_t tot = (int64_t)n1 * n2;
  note_launch();
  ex_u_words_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(U, ldu, n1, n2, upper, trans, ecol, uexp, WU,
                                                                  pad2(n2));
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int64_t slice = tall_rows(M, n1);
  for (int64_t r0 = 0; r0 < M; r0 += slice) {
    const int64_t rows = std::min(slice, M - r0);
    note_launch();
    ex_row_words_kernel<<<dim3((unsigned)((rows + 31) / 32), (n1 + 31) / 32), dim3(32, 8), 0, s>>>(
        A + r0 * lda, lda, rows, n1, ecol, rexp + r0, WX);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ExParams P{};
    P.A = WX;
    P.sa = BM;
    P.B = WU;
    P.sb = pad2(n2);
    P.M = rows;
    P.r0 = r0;
    P.n1 = n1;
    P.n2 = n2;
    P.rexp = rexp;
    P.uexp = uexp;
    P.upper = upper;
    P.C = C;
    P.ldc = ldc;
    P.nitems = (rows + BM - 1) / BM * ((n2 + BN - 1) / BN);
    P.watch = w;
    if ((e = launch<EX_TALL>(P, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace chfsi
