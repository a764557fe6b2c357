// The cell matrices on the device: H~_e = D_e^{-1/2} (1/2 K + V_e) D_e^{-1/2}
// (Eq. discreteHam scaled as in Eq. hep) in binary64 for all cells, and the
// potential factor w V jac at the Gauss points that the matrix-free apply takes.
//
//  potential_kernel   V = wells (each summed over its image shifts) + given
//                     values, times the weights, one block per cell.  A Gaussian
//                     is a product over the axes, so a well costs 3 q
//                     exponentials and 2 q^3 / q + q^3 products per cell instead
//                     of q^3 exponentials.
//  cell_matrix_kernel V_e by sum factorisation over the unordered node pairs of
//                     each axis: B_ai B_al is symmetric in (i, l), so the three
//                     contractions run over n1 (n1 + 1) / 2 pairs per axis
//                     (n1 = 7: 28^3 q products for the last one instead of 49^3 q)
//                     and every value serves up to eight entries.  The scaling
//                     D_e^{-1/2} is a product over the axes (the assembled GLL
//                     mass of a uniform mesh), the same in every cell, and goes
//                     into the 1-D factors and the shared kinetic matrix: one
//                     addition per entry is left.
// Both are bound by the binary64 ALU rate (2 FMA per clock and SM; 1.06 ms for the
// matrices below).  12^3 cells, p = 6, 108 wells: 0.25 and 1.25 ms (0.43 and 2.0
// with a barrier per well, one z pair per round and the loads of K one by one; on
// 16 host threads, with the upload: 185).  The digit words take no binary64
// operation beyond the contractions.
#include <algorithm>
#include <mutex>

#include "digits.cuh"
#include "internal.h"

namespace chfsi {

namespace {

constexpr int PT = 256;

// wells: n x 5 (centre, depth, 1 / (2 w^2)), images as explicit centres; a well
// whose largest value in the cell is below e^-41.5 (1e-18) of its depth is
// left out.  Sums in the order of the list.
__global__ void __launch_bounds__(PT) potential_kernel(CellMatArgs P, int pw) {
  extern __shared__ double sm[];
  const int q = P.q, q2 = q * q, nq = q2 * q;
  double* g = sm;                                     // pw x 3 x q
  double* yz = g + pw * 3 * q;                        // pw x q^2: D g_y g_z
  double* v = yz + pw * q2;                           // q^3
  __shared__ int list[PT];
  __shared__ int cnt[PT / 32];
  const int64_t e = blockIdx.x;
  const int c3[3] = {(int)(e % P.n[0]), (int)((e / P.n[0]) % P.n[1]), (int)(e / ((int64_t)P.n[0] * P.n[1]))};
  double lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = c3[a] * P.h[a];
    hi[a] = lo[a] + P.h[a];
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int t = tid; t < nq; t += PT) v[t] = 0.0;
  for (int w0 = 0; w0 < P.nwell; w0 += PT) {
    // ordered list of the chunk's wells in range
    bool in = false;
    if (w0 + tid < P.nwell) {
      const double* w = P.wells + 5 * (int64_t)(w0 + tid);
      double r2 = 0.0;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double d = w[a] < lo[a] ? lo[a] - w[a] : (w[a] > hi[a] ? w[a] - hi[a] : 0.0);
        r2 += d * d;
      }
      in = !(r2 * w[4] > 41.5);
    }
    const unsigned b = __ballot_sync(0xffffffffu, in);
    __syncthreads();
    if (lane == 0) cnt[warp] = __popc(b);
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int k = 0; k < PT / 32; ++k) {
      if (k < warp) base += cnt[k];
      total += cnt[k];
    }
    if (in) list[base + __popc(b & ((1u << lane) - 1))] = w0 + tid;
    __syncthreads();
    for (int l0 = 0; l0 < total; l0 += pw) {
      const int nl = min(pw, total - l0);
      for (int t = tid; t < nl * 3 * q; t += PT) {
        const int k = t / (3 * q), a = t / q % 3, i = t % q;
        const double* w = P.wells + 5 * (int64_t)list[l0 + k];
        const double d = lo[a] + (P.gx[i] + 1.0) * P.h[a] / 2.0 - w[a];
        g[t] = exp(-d * d * w[4]);
      }
      __syncthreads();
      for (int t = tid; t < nl * q2; t += PT) {
        const int k = t / q2, i = t % q2;
        const double* gk = g + k * 3 * q;
        yz[t] = P.wells[5 * (int64_t)list[l0 + k] + 3] * gk[q + i % q] * gk[2 * q + i / q];
      }
      __syncthreads();
      for (int t = tid; t < nq; t += PT) {
        const int i = t / q, a = t % q;
        double s = v[t];
        for (int k = 0; k < nl; ++k) s = fma(-yz[k * q2 + i], g[k * 3 * q + a], s);
        v[t] = s;
      }
      __syncthreads();
    }
  }
  for (int t = tid; t < nq; t += PT) {
    const int a = t % q, b = t / q % q, c = t / q2;
    const double s = (v[t] + (P.vqp ? P.vqp[e * nq + t] : 0.0)) * P.jac;
    P.wv[e * nq + t] = s * P.gw[a] * P.gw[b] * P.gw[c];
  }
}

__device__ __forceinline__ int pair_index(int i, int l) {   // unordered pairs, i >= l first
  const int a = max(i, l), b = min(i, l);
  return a * (a + 1) / 2 + b;
}
// The first index of an unordered pair.
__device__ __forceinline__ int pair_first(int u) {
  int i = 0;
  while ((i + 1) * (i + 2) / 2 <= u) ++i;
  return i;
}
// fixed_of for a term that may exceed the scale (s < 0) in a sum that does not:
// modulo 2^64.
__device__ __forceinline__ uint64_t fixed_term(double v, int s) {
  return s >= 0 ? (uint64_t)fixed_of(v, s) : s > -64 ? (uint64_t)fixed_of(v, 0) << -s : 0;
}
// Threads per cell: shared memory admits one block per SM for p >= 7, two for p =
// 5, 6 (p = 7: 1.35 ms with 512 threads, 1.16 with 1,024; p = 6: 1.53 and 1.89).
__host__ __device__ constexpr int cell_threads(int n1) { return n1 >= 8 ? 1024 : n1 >= 6 ? 512 : 256; }
constexpr int ZB = 2;                     // z pairs per round

// WORDS: digit words instead of the binary64 entries: entry (l, k) under the
// scale of row l at W[(e NE + k) ldw + l], the sum of the kinetic part (twice the
// precision of binary64) and the potential part in integers.
template <int N1, bool WORDS>
__global__ void __launch_bounds__(cell_threads(N1)) cell_matrix_kernel(CellMatArgs P, int jb, const int16_t* __restrict__ hexp,
                                                          uint64_t* __restrict__ W, int ldw) {
  constexpr int NU = N1 * (N1 + 1) / 2, NN = N1 * N1, NE = NN * N1, N4 = NN * NN;
  constexpr int NT = cell_threads(N1);
  extern __shared__ double sm[];
  const int q = P.q, q2 = q * q, nq = q2 * q;
  double* bb = sm;                        // 3 x q x NU: s_i B_ai B_al s_l per axis
  double* t1 = bb + 3 * q * NU;           // q^2 x NU
  double* slab = t1 + q2 * NU;            // ZB x jb x NU
  double* t2 = slab + ZB * jb * NU;       // q x jb x NU; first w V jac, q^3
  uint16_t* idx = reinterpret_cast<uint16_t*>(t2 + max(q * jb * NU, nq));   // N4: (row, column) -> (jm, il)
  __shared__ bool live[NE];               // nodes that are not eliminated
  const int64_t e = blockIdx.x;
  for (int t = threadIdx.x; t < 3 * q * NU; t += NT) {
    const int ax = t / (q * NU), a = t / NU % q, u = t % NU;
    const int i = pair_first(u), l = u - i * (i + 1) / 2;
    bb[t] = P.B[a * N1 + i] * P.B[a * N1 + l] * (P.s1[ax * N1 + i] * P.s1[ax * N1 + l]);
  }
  const double* by = bb + q * NU;
  const double* bz = by + q * NU;
  for (int t = threadIdx.x; t < nq; t += NT) t2[t] = P.wv[e * nq + t];
  int dead = 0;
  for (int l = threadIdx.x; l < NE; l += NT) {
    live[l] = P.dofmap[e * NE + l] >= 0;
    dead |= !live[l];
  }
  for (int t = threadIdx.x; t < N4; t += NT) {
    const int r = t / NN, c = t % NN;
    idx[t] = (uint16_t)(pair_index(r / N1, c / N1) * NU + pair_index(r % N1, c % N1));
  }
  dead = __syncthreads_or(dead);
  for (int t = threadIdx.x; t < q2 * NU; t += NT) {      // x: (c b a) -> (c b il)
    const int u = t % NU, cb = t / NU;
    double s = 0.0;
    for (int a = 0; a < q; ++a) s = fma(bb[a * NU + u], t2[cb * q + a], s);
    t1[t] = s;
  }
  for (int j0 = 0; j0 < NU; j0 += jb) {                   // y pairs, jb at a time
    const int nj = min(jb, NU - j0), nt = nj * NU;
    __syncthreads();
    for (int t = threadIdx.x; t < q * nt; t += NT) {     // y: (c b il) -> (c jm il)
      const int u = t % NU, w = t / NU % nj, c = t / nt;
      double s = 0.0;
      for (int b = 0; b < q; ++b) s = fma(by[b * NU + j0 + w], t1[(c * q + b) * NU + u], s);
      t2[t] = s;
    }
    for (int z0 = 0; z0 < NU; z0 += ZB) {                 // z: -> ZB slabs (jm il)
      const int nz = min(ZB, NU - z0);
      __syncthreads();
      for (int t = threadIdx.x; t < nz * nt; t += NT) {
        const int zz = t / nt, w = t - zz * nt;
        double s = 0.0;
        for (int c = 0; c < q; ++c) s = fma(bz[c * NU + z0 + zz], t2[c * nt + w], s);
        slab[t] = s;
      }
      __syncthreads();
      // pair z = (k, nk): entries (i j k), (l m nk), and for nk < k the
      // transposed block
      for (int zz = 0; zz < nz; ++zz) {
        const int kf = pair_first(z0 + zz), ks = z0 + zz - kf * (kf + 1) / 2;
        const double* x = slab + zz * nt;
        for (int side = 0; side < (ks < kf ? 2 : 1); ++side) {
          const int kr = side ? ks : kf, kc = side ? kf : ks;
          // U entries per thread at a time: the loads of K come from L2
          constexpr int U = (N4 + NT - 1) / NT < 5 ? (N4 + NT - 1) / NT : 5;
          for (int t0 = threadIdx.x; t0 < N4; t0 += NT * U) {
            int id[U];
            double k0[U], k1[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int t = t0 + NT * u, r = t / NN, c = t % NN;
              id[u] = t < N4 ? (int)idx[t] - j0 * NU : -1;
              if (id[u] >= nt) id[u] = -1;
              if (id[u] >= 0) {
                const int64_t o = (int64_t)(r + NN * kr) * NE + c + NN * kc;
                k0[u] = __ldg(P.K + o);
                if (WORDS) k1[u] = __ldg(P.K + NE * NE + o);
              }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              if (id[u] < 0) continue;
              const int t = t0 + NT * u, r = t / NN, c = t % NN;
              const int row = r + NN * kr, col = c + NN * kc;
              const bool on = !dead || (live[row] && live[col]);
              if (!WORDS) {
                P.Ht[(e * NE + row) * NE + col] = on ? k0[u] + x[id[u]] : 0.0;
              } else {   // the matrix is symmetric: col is the word's row
                const double v = x[id[u]];
                const int ex = hexp[e * NE + col];
                W[(e * NE + row) * ldw + col] = on ? fixed_term(k0[u], ex - expo(k0[u])) + fixed_term(k1[u], ex - expo(k1[u])) +
                                                         fixed_term(v, ex - expo(v)) + kZeroWord
                                                   : kZeroWord;
              }
            }
          }
        }
      }
    }
  }
}

template <int N1, bool WORDS>
cudaError_t launch_n(const CellMatArgs& P, const int16_t* hexp, uint64_t* W, int ldw, cudaStream_t s) {
  constexpr int NU = N1 * (N1 + 1) / 2, NN = N1 * N1;
  const int q = P.q;
  auto bytes = [q](int jb) {
    return sizeof(double) * ((size_t)3 * q * NU + q * q * NU + ZB * jb * NU + std::max((size_t)q * jb * NU, (size_t)q * q * q)) +
           sizeof(uint16_t) * NN * NN;
  };
  int jb = NU;                       // all y pairs at once unless they don't fit (p = 8 and the finest rules)
  while (bytes(jb) > 226 * 1024) jb = (jb + 1) / 2;
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(cell_matrix_kernel<N1, WORDS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  });
  note_launch();
  cell_matrix_kernel<N1, WORDS><<<(unsigned)P.ncells, cell_threads(N1), bytes(jb), s>>>(P, jb, hexp, W, ldw);
  return cudaGetLastError();
}
template <bool WORDS>
cudaError_t launch_any(const CellMatArgs& P, const int16_t* hexp, uint64_t* W, int ldw, cudaStream_t s) {
  switch (P.n1) {
    case 2: return launch_n<2, WORDS>(P, hexp, W, ldw, s);
    case 3: return launch_n<3, WORDS>(P, hexp, W, ldw, s);
    case 4: return launch_n<4, WORDS>(P, hexp, W, ldw, s);
    case 5: return launch_n<5, WORDS>(P, hexp, W, ldw, s);
    case 6: return launch_n<6, WORDS>(P, hexp, W, ldw, s);
    case 7: return launch_n<7, WORDS>(P, hexp, W, ldw, s);
    case 8: return launch_n<8, WORDS>(P, hexp, W, ldw, s);
    default: return launch_n<9, WORDS>(P, hexp, W, ldw, s);
  }
}

}  // namespace

cudaError_t launch_cell_matrices(const CellMatArgs& P, cudaStream_t s) {
  const int q = P.q;
  // wells per batch: as fit in the 48 KB that need no opt-in (q = 7: 32)
  const size_t per = sizeof(double) * (3 * q + q * q), base = sizeof(double) * q * q * q;
  const int pw = (int)std::min<size_t>(32, std::max<size_t>(1, (46 * 1024 - std::min<size_t>(base, 46 * 1024)) / per));
  note_launch();
  potential_kernel<<<(unsigned)P.ncells, PT, base + pw * per, s>>>(P, pw);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_any<false>(P, nullptr, nullptr, 0, s);
}

cudaError_t launch_cell_words(const CellMatArgs& P, const int16_t* hexp, uint64_t* W, int ldw, cudaStream_t s) {
  return launch_any<true>(P, hexp, W, ldw, s);
}

}  // namespace chfsi
