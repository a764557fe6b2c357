// Cholesky factor S = L L^T and L^{-1} of CholGS in one sweep, binary64.
//
// Right-looking over blocks of 32 columns.  After block column k of L is known,
// one launch subtracts its products from the trailing lower tiles,
// S_ij -= L_ik L_jk^T, and from the right-hand sides of the inverse,
// X_ic -= L_ik X_kc (c <= k < i): T^2/2 tiles or so at every step (T = n / 32), so
// the chip stays full to the end, where the factor alone thins out as (T - k)^2 / 2.
// Its first block takes the next diagonal tile and factors it, so that the serial
// part (32 pivots) runs beside the other tiles.
//
// Bound by the binary64 ALU (2 FMA per clock and SM; 2 n^3 / 3 operations, 0.7
// ms at n = 1,100) and, with few tiles, by the chain of 32 pivots and the two
// launches of a step.  n = 1,100: 1.4 ms, where cuSOLVER's potrf took 4.0 and a
// forward substitution per column of the inverse 1.1.  A whole CholGS of 64,000
// rows (mixed precision) before and now: n = 36 0.45 -> 0.36 ms, 550 3.2 -> 1.6,
// 1,100 6.8 -> 3.1, 3,300 34.5 -> 30.3, 5,000 116 -> 91: one path for every n.
#include <algorithm>
#include <mutex>

#include "internal.h"

namespace chfsi {
namespace {

constexpr int NB = 32;                // tile
constexpr int GROUP = 128;            // threads per tile
constexpr int GROUPS = 4;             // tiles in flight per SM
struct GroupSmem {
  double A[NB][NB + 1];               // [contracted][row]
  double B[NB][NB + 2];               // [contracted][column]
};
// More than half of an SM's shared memory: the pivots of the first thread block,
// a serial chain, share the binary64 units of their SM with no other block
// (n = 1,100: 36 us per step, 59 with blocks of one tile each, three to an SM).
constexpr int UPDATE_SMEM = 120 * 1024;
static_assert(GROUPS * sizeof(GroupSmem) <= UPDATE_SMEM, "tiles in flight");

__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(GROUP) : "memory");
}

// v / d by a third-order Newton step on the binary32 reciprocal of d's
// significand (relative error 2^-22; its cube lies below rounding).  Four
// binary64 operations of 64 clocks each, a division takes as long as 5.5 more;
// it is left to pivots whose reciprocal is out of range (columns of norm below
// 2^-511 have such squares).
__device__ __forceinline__ double quotient(double v, double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const int e = (hi >> 20) & 0x7ff;
  if (e < 2 || e > 2044) return v / d;
  const double m = __hiloint2double((int)((hi & 0xfffff) | 0x3ff00000), (int)lo);
  const uint32_t f = __float_as_uint(__fdividef(1.f, __uint_as_float(0x3f800000 | (hi & 0xfffff) << 3 | lo >> 29)));
  const double y = __hiloint2double((int)(((f >> 23) + 896) << 20 | (f >> 3 & 0xfffff)), (int)(f << 29));
  const double r = fma(-m, y, 1.0);
  const double z = fma(y, fma(r, r, r), y);
  return v * __hiloint2double((__double2hiint(z) - ((e - 1023) << 20)) | (int)(hi & 0x80000000u), __double2loint(z));
}

// The diagonal tile at o (nv columns): S minus the products with the 32 columns
// in P ([contracted][row], null for the first tile), then L_kk and L_kk^{-1}; rows
// and columns from nv on are those of the unit matrix.  Elimination without
// square roots, A = E^{-1} D E^{-T}, with E built in the places that the eliminated
// columns leave: step j adds multiples of row j, of A right of column j and of E
// left of it, to the rows below.  V[j] keeps column j of E^{-1} D from j on and
// row j of E before.  A binary64 instruction takes a warp 64 clocks whatever its
// active lanes, so the lower triangle is packed: the elements of the rows in
// descending order over the 128 threads, five at most per thread, of which step
// j needs a prefix (3.2 on average, 8 for a 32 x 32 square).  One barrier per step.
__device__ void factor_tile(const double (*P)[NB + 1], double (*V)[NB + 1], double* __restrict__ S,
                            double* __restrict__ X, int64_t ld, int o, int nv, int* __restrict__ info) {
  constexpr int SLOTS = (NB * (NB + 1) / 2 + GROUP - 1) / GROUP;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double a[SLOTS];
  int er[SLOTS], ec[SLOTS], top[SLOTS];                      // row, column, the warp's largest row
#pragma unroll
  for (int i = 0; i < SLOTS; ++i) {
    int c = i * GROUP + threadIdx.x, r = NB - 1;
    while (r >= 0 && c > r) c -= r + 1, --r;
    er[i] = r;                                               // -1: no element
    ec[i] = r < 0 ? 0 : c;
    top[i] = __shfl_sync(0xffffffffu, r, 0);
    a[i] = r >= 0 && r < nv ? S[o + r + (int64_t)(o + c) * ld] : (r == c ? 1.0 : 0.0);
    if (P && top[i] >= 0) {
      const int rr = max(r, 0);
#pragma unroll 8
      for (int k = 0; k < NB; ++k) a[i] = fma(-P[k][rr], P[k][ec[i]], a[i]);
    }
  }
#pragma unroll 1
  for (int j = 0; j < NB; ++j) {
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
      if (ec[i] == j && er[i] >= j) V[j][er[i]] = a[i];
      if (er[i] == j) V[j][ec[i]] = a[i];
    }
    group_sync(0);
    if (top[0] <= j) continue;                               // this warp's rows are finished
    const double s = quotient(-V[j][lane], V[j][j]);
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
      if (top[i] > j) {
        const double t = __shfl_sync(0xffffffffu, s, max(er[i], 0));
        if (er[i] > j) a[i] = ec[i] == j ? t : fma(t, V[j][ec[i]], a[i]);
      }
    }
  }
  const double d = V[lane][lane], rs = rsqrt(d);
  if (w == 0) {
    const uint32_t bad = __ballot_sync(0xffffffffu, lane < nv && (!(d > 0.0) || isinf(d)));
    if (lane == 0 && bad && *info == 0) *info = o + __ffs(bad);
  }
#pragma unroll
  for (int u = 0; u < NB / 4; ++u) {                         // row lane, column c
    const int c = w * (NB / 4) + u;
    const double rc = __shfl_sync(0xffffffffu, rs, c);
    if (c <= lane && lane < nv) {
      S[o + lane + (int64_t)(o + c) * ld] = V[c][lane] * rc;
      X[o + lane + (int64_t)(o + c) * ld] = c == lane ? rs : V[lane][c] * rs;
    }
  }
}

// Step k: tiles of the trailing matrix and of the inverse's right-hand sides
// minus the products with block column k; the first thread block takes the next
// diagonal tile and factors it.  k = -1: only that.  Each group of four warps of
// the other blocks works through tiles: warp w has columns 8 w .. 8 w + 7, lane =
// row.  One block per SM.
__global__ void __launch_bounds__(GROUP * GROUPS, 1) chol_update_kernel(double* __restrict__ S, int n, int k, int ntile,
                                                                       double* __restrict__ X, int* __restrict__ info) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int g = threadIdx.x / GROUP;
  GroupSmem& sm = reinterpret_cast<GroupSmem*>(smem)[g];
  const int T = (n + NB - 1) / NB;
  const int lane = threadIdx.x & 31, c0 = (threadIdx.x % GROUP >> 5) * 8;
  const int k0 = k * NB;
  if (blockIdx.x == 0) {
    if (g > 0) return;
    const int o = k0 + NB;
    if (k >= 0) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        sm.A[c0 + u][lane] = o + lane < n ? S[o + lane + (int64_t)(k0 + c0 + u) * n] : 0.0;
      group_sync(0);
    }
    factor_tile(k >= 0 ? sm.A : nullptr, reinterpret_cast<GroupSmem*>(smem)[1].A, S, X, n, o, min(NB, n - o), info);
    return;
  }
  // tiles: lower tiles (i, j) with k < j <= i first, diagonal after diagonal
  // (the first is that of the first block), then (i, c) of the inverse, c <= k < i
  const int m = T - 1 - k, tri = m * (m + 1) / 2;
  for (int t = 1 + g * (gridDim.x - 1) + blockIdx.x - 1; t < ntile; t += GROUPS * (gridDim.x - 1)) {
    int i, j, b = t;
    const bool inv = b >= tri;
    if (!inv) {
      int w = m;
      for (i = 0; b >= w; --w) b -= w, ++i;         // i: distance from the diagonal
      j = k + 1 + b;
      i += j;
    } else {
      b -= tri;
      i = k + 1 + b / (k + 1);
      j = b % (k + 1);
    }
    const int r0 = i * NB, j0 = j * NB;
    double* C = (inv ? X : S) + r0 + lane + (int64_t)(j0 + c0) * n;
    const bool row = r0 + lane < n;
    double acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int kk = c0 + u;                        // block column k is a full one
      acc[u] = row && j0 + c0 + u < n ? C[(int64_t)u * n] : 0.0;
      sm.A[kk][lane] = row ? S[r0 + lane + (int64_t)(k0 + kk) * n] : 0.0;
      if (inv) sm.B[lane][kk] = X[k0 + lane + (int64_t)(j0 + kk) * n];
      else sm.B[kk][lane] = j0 + lane < n ? S[j0 + lane + (int64_t)(k0 + kk) * n] : 0.0;
    }
    group_sync(g);
#pragma unroll 4
    for (int kk = 0; kk < NB; ++kk) {
      const double x = -sm.A[kk][lane];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        const double2 y = *reinterpret_cast<const double2*>(&sm.B[kk][c0 + u]);
        acc[u] = fma(x, y.x, acc[u]);
        acc[u + 1] = fma(x, y.y, acc[u + 1]);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (row && j0 + c0 + u < n) C[(int64_t)u * n] = acc[u];
    group_sync(g);
  }
}

// Block column k of L below its diagonal tile, L_ik = S_ik L_kk^{-T}, and block row
// k of the inverse left of it, X_kc = L_kk^{-1} X_kc: eight rows (columns) of a
// tile per thread block, in place.  Thread: row (column) t % 8, its entries g and
// 31 - g, g = t / 8, 33 products together (the inverse is triangular).
__global__ void __launch_bounds__(GROUP) chol_panel_kernel(double* __restrict__ S, int n, int k,
                                                                  double* __restrict__ X) {
  __shared__ double B[NB][NB + 1], A[NB][9];       // L_kk^{-1} [column][row], [contracted][row of the tile]
  const int T = (n + NB - 1) / NB, below = T - 1 - k;
  const int o = k * NB, nv = min(NB, n - o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x >> 2;
  const bool inv = b >= below;
  const int b0 = (inv ? b - below : k + 1 + b) * NB + (blockIdx.x & 3) * 8;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int c = w * 8 + u;
    B[c][lane] = lane < nv && c < nv ? X[o + lane + (int64_t)(o + c) * n] : 0.0;
  }
  if (!inv) {
    const int r = threadIdx.x & 7, c = threadIdx.x >> 3;
    A[c][r] = b0 + r < n ? S[b0 + r + (int64_t)(o + c) * n] : 0.0;
    A[c + 16][r] = b0 + r < n ? S[b0 + r + (int64_t)(o + c + 16) * n] : 0.0;
  } else {
    A[lane][w] = lane < nv ? X[o + lane + (int64_t)(b0 + w) * n] : 0.0;
    A[lane][w + 4] = lane < nv ? X[o + lane + (int64_t)(b0 + w + 4) * n] : 0.0;
  }
  __syncthreads();
  const int r = threadIdx.x & 7, g = threadIdx.x >> 3;
  const int h = NB - 1 - g;
  double x0 = 0.0, x1 = 0.0, y0 = 0.0, y1 = 0.0;
  const int kx = 4 * w + 3, ky = NB - 1 - 4 * w;    // the warp's longest rows of each kind
#pragma unroll 4
  for (int kk = 0; kk <= kx; kk += 2) {
    x0 = fma(A[kk][r], B[kk][g], x0);
    x1 = fma(A[kk + 1][r], B[kk + 1][g], x1);
  }
#pragma unroll 4
  for (int kk = 0; kk <= ky; kk += 2) {
    y0 = fma(A[kk][r], B[kk][h], y0);
    y1 = fma(A[kk + 1][r], B[kk + 1][h], y1);
  }
  __syncthreads();
  A[g][r] = x0 + x1;
  A[h][r] = y0 + y1;
  __syncthreads();
  if (!inv) {
    const int c = threadIdx.x >> 3;
    if (b0 + r < n) {
      S[b0 + r + (int64_t)(o + c) * n] = A[c][r];
      S[b0 + r + (int64_t)(o + c + 16) * n] = A[c + 16][r];
    }
  } else if (lane < nv) {
    X[o + lane + (int64_t)(b0 + w) * n] = A[lane][w];
    X[o + lane + (int64_t)(b0 + w + 4) * n] = A[lane][w + 4];
  }
}

}  // namespace

cudaError_t launch_chol_inverse(double* S, int n, double* X, int* info, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  static std::once_flag once;
  static int sms = 0;
  std::call_once(once, [] {
    int d = 0;
    cudaGetDevice(&d);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d) != cudaSuccess || sms < 2) sms = 152;
    cudaFuncSetAttribute(chol_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, UPDATE_SMEM);
  });
  cudaError_t e = cudaMemsetAsync(info, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(X, 0, (size_t)n * n * sizeof(double), s);
  if (e != cudaSuccess) return e;
  const int T = (n + NB - 1) / NB;
  for (int k = -1; k < T; ++k) {
    if (k >= 0 && T > 1) {
      note_launch();
      chol_panel_kernel<<<4 * (T - 1), GROUP, 0, s>>>(S, n, k, X);
    }
    if (k == T - 1) break;
    const int m = T - 1 - k, ntile = k < 0 ? 1 : m * (m + 1) / 2 + m * (k + 1);
    note_launch();
    chol_update_kernel<<<std::min(ntile, sms), GROUP * GROUPS, UPDATE_SMEM, s>>>(S, n, k, ntile, X, info);
  }
  return cudaGetLastError();
}

}  // namespace chfsi
