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
// Both are bound by the binary64 ALU rate (2 FMA per clock and SM).  12^3 cells,
// p = 6, 108 wells: 0.43 and 2.0 ms (on 16 host threads, with the upload: 185 ms).
#include <algorithm>
#include <mutex>

#include "digits.cuh"
#include "internal.h"

namespace chfsi {

namespace {

constexpr int PW = 32;       // wells per batch of 1-D factors
constexpr int PT = 256;

// wells: n x 5 (centre, depth, 1 / (2 w^2)), images as explicit centres; a well
// whose largest value in the cell is below e^-41.5 (1e-18) of its depth is
// left out.  Sums in the order of the list.
__global__ void __launch_bounds__(PT) potential_kernel(CellMatArgs P) {
  extern __shared__ double sm[];
  const int q = P.q, q2 = q * q, nq = q2 * q;
  double* g = sm;                                     // PW x 3 x q
  double* yz = g + PW * 3 * q;                        // q^2: D g_y g_z of one well
  double* v = yz + q2;                                // q^3
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
    for (int l0 = 0; l0 < total; l0 += PW) {
      const int nl = min(PW, total - l0);
      for (int t = tid; t < nl * 3 * q; t += PT) {
        const int k = t / (3 * q), a = t / q % 3, i = t % q;
        const double* w = P.wells + 5 * (int64_t)list[l0 + k];
        const double d = lo[a] + (P.gx[i] + 1.0) * P.h[a] / 2.0 - w[a];
        g[t] = exp(-d * d * w[4]);
      }
      __syncthreads();
      for (int k = 0; k < nl; ++k) {
        const double* gk = g + k * 3 * q;
        const double dep = P.wells[5 * (int64_t)list[l0 + k] + 3];
        for (int t = tid; t < q2; t += PT) yz[t] = dep * gk[q + t % q] * gk[2 * q + t / q];
        __syncthreads();
        for (int t = tid; t < nq; t += PT) v[t] = fma(-yz[t / q], gk[t % q], v[t]);
        __syncthreads();
      }
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

// WORDS: digit words instead of the binary64 entries: entry (l, k) under the
// scale of row l at W[(e NE + k) ldw + l].
template <int N1, bool WORDS>
__global__ void __launch_bounds__(256) cell_matrix_kernel(CellMatArgs P, int jb, const int16_t* __restrict__ hexp,
                                                          uint64_t* __restrict__ W, int ldw) {
  constexpr int NU = N1 * (N1 + 1) / 2, NN = N1 * N1, NE = NN * N1;
  extern __shared__ double sm[];
  const int q = P.q, q2 = q * q, nq = q2 * q;
  double* bb = sm;                        // 3 x q x NU: s_i B_ai B_al s_l per axis
  double* t1 = bb + 3 * q * NU;           // q^2 x NU
  double* slab = t1 + q2 * NU;            // jb x NU
  double* t2 = slab + jb * NU;            // q x jb x NU; first w V jac, q^3
  __shared__ bool live[NE];               // nodes that are not eliminated
  const int64_t e = blockIdx.x;
  for (int t = threadIdx.x; t < 3 * q * NU; t += 256) {
    const int ax = t / (q * NU), a = t / NU % q, u = t % NU;
    int i = 0;
    while ((i + 1) * (i + 2) / 2 <= u) ++i;
    const int l = u - i * (i + 1) / 2;
    bb[t] = P.B[a * N1 + i] * P.B[a * N1 + l] * (P.s1[ax * N1 + i] * P.s1[ax * N1 + l]);
  }
  const double* by = bb + q * NU;
  const double* bz = by + q * NU;
  for (int t = threadIdx.x; t < nq; t += 256) t2[t] = P.wv[e * nq + t];
  for (int l = threadIdx.x; l < NE; l += 256) live[l] = P.dofmap[e * NE + l] >= 0;
  __syncthreads();
  for (int t = threadIdx.x; t < q2 * NU; t += 256) {      // x: (c b a) -> (c b il)
    const int u = t % NU, cb = t / NU;
    double s = 0.0;
    for (int a = 0; a < q; ++a) s = fma(bb[a * NU + u], t2[cb * q + a], s);
    t1[t] = s;
  }
  for (int j0 = 0; j0 < NU; j0 += jb) {                   // y pairs, jb at a time
    const int nj = min(jb, NU - j0);
    __syncthreads();
    for (int t = threadIdx.x; t < q * nj * NU; t += 256) {   // y: (c b il) -> (c jm il)
      const int u = t % NU, w = t / NU % nj, c = t / (nj * NU);
      double s = 0.0;
      for (int b = 0; b < q; ++b) s = fma(by[b * NU + j0 + w], t1[(c * q + b) * NU + u], s);
      t2[t] = s;
    }
    for (int k = 0; k < N1; ++k)
      for (int nk = 0; nk <= k; ++nk) {
        const int z = k * (k + 1) / 2 + nk;
        __syncthreads();
        for (int t = threadIdx.x; t < nj * NU; t += 256) {
          double s = 0.0;
          for (int c = 0; c < q; ++c) s = fma(bz[c * NU + z], t2[c * nj * NU + t], s);
          slab[t] = s;
        }
        __syncthreads();
        // entries (i j k), (l m nk), and for nk < k the transposed block
        for (int side = 0; side < (nk < k ? 2 : 1); ++side) {
          const int kr = side ? nk : k, kc = side ? k : nk;
          for (int t = threadIdx.x; t < NN * NN; t += 256) {
            const int r = t / NN, c = t % NN;
            const int jm = pair_index(r / N1, c / N1) - j0;
            if (jm < 0 || jm >= nj) continue;
            const int row = r + NN * kr, col = c + NN * kc;
            const double x = slab[jm * NU + pair_index(r % N1, c % N1)];
            const bool on = live[row] && live[col];
            const double kin = P.K[(int64_t)row * NE + col];
            if (!WORDS) {
              P.Ht[(e * NE + row) * NE + col] = on ? kin + x : 0.0;
            } else {   // kin + x exactly, plus the kinetic remainder (the matrix is symmetric: col is the word's row)
              const double h = kin + x, t = h - kin;
              const double lo = ((kin - (h - t)) + (x - t)) + P.K[(int64_t)(NE + row) * NE + col];
              const int ex = hexp[e * NE + col];
              W[(e * NE + row) * ldw + col] =
                  on ? fixed_of(h, ex - expo(h)) + fixed_of(lo, ex - expo(lo)) + kZeroWord : kZeroWord;
            }
          }
        }
      }
  }
}

template <int N1, bool WORDS>
cudaError_t launch_n(const CellMatArgs& P, const int16_t* hexp, uint64_t* W, int ldw, cudaStream_t s) {
  constexpr int NU = N1 * (N1 + 1) / 2;
  const int q = P.q;
  auto bytes = [q](int jb) {
    return sizeof(double) * ((size_t)3 * q * NU + q * q * NU + jb * NU +
                             std::max((size_t)q * jb * NU, (size_t)q * q * q));
  };
  int jb = NU;                       // all y pairs at once but for the largest rules (p = 8, q > 10)
  while (bytes(jb) > 226 * 1024) jb = (jb + 1) / 2;
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(cell_matrix_kernel<N1, WORDS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  });
  note_launch();
  cell_matrix_kernel<N1, WORDS><<<(unsigned)P.ncells, 256, bytes(jb), s>>>(P, jb, hexp, W, ldw);
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
  const size_t smem = sizeof(double) * ((size_t)PW * 3 * q + q * q + q * q * q);
  note_launch();
  potential_kernel<<<(unsigned)P.ncells, PT, smem, s>>>(P);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_any<false>(P, nullptr, nullptr, 0, s);
}

cudaError_t launch_cell_words(const CellMatArgs& P, const int16_t* hexp, uint64_t* W, int ldw, cudaStream_t s) {
  return launch_any<true>(P, hexp, W, ldw, s);
}

}  // namespace chfsi
