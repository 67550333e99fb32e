// Reverse mode of the Poisson element tensors with respect to the vertex coordinates.
//
// Forward (Section 3.3, test case 2): A^K_i = sum_alpha A0[i][alpha] G[alpha] with
// G = s K K^T, s = |det J|, K = J^{-1}, J = [x_1 - x_0, ..., x_d - x_0].
// Given the upstream gradient dA[e][i] = dL/dA^K_i:
//   Gbar[alpha] = sum_i A0[i][alpha] dA[e][i]                      (transposed contraction)
//   c           = Gbar : (K K^T)
//   dL/dJ       = s (c K^T - K^T (Gbar + Gbar^T) K K^T)
// which follows from d s = s tr(K dJ) and dK = -K dJ K. Column c of J is
// x_{c+1} - x_0, so dL/dx_{c+1} += dL/dJ[:, c] and dL/dx_0 -= sum_c dL/dJ[:, c]; the
// vertex gradients are accumulated with FP64 atomic adds.
//
// Only the symmetric part of Gbar enters, and A0 is symmetric in (i1, i2) (a symmetric
// form, Section 3.5): with the d(d+1)/2 columns (a,a) and (a,b) + (b,a) of the kernels'
// layout, gp[k] = sum_{i1 <= i2} A0[i1][i2][k] (dA[i1][i2] + dA[i2][i1]). That contraction
// runs in fixed point (fixed_point.cuh): in FP64 its n^2 d(d+1)/2 multiply-adds held the
// FP64 pipe at 95% (P2 tetrahedra: 300 of the 381 SM clocks a cell took).
//
// Every warp works by itself (no CTA barrier after the start, so the load, integer and FP64
// phases of different warps overlap) on tiles of up to 32 cells:
//   load         the dA of 32/L cells at a time, asynchronously into shared memory, rows
//                padded to an odd number of doubles;
//   contraction  L lanes per cell: the cell's largest exponent first, then each pair i1 <= i2
//                rounded to 57 or 58 bits, its two halves added as integers, times the
//                fixed-point A0 of the pair; the L partial sums are added as integers;
//   chain rule   one lane per cell of the tile: FP64 J^-1, |det J| and the formula above, and
//                FP64 atomics to the d+1 vertices.
// Bound by the FP64 geometry and chain rule (pipe 49% busy) and the integer instructions
// (issue 44%) at 20 resident warps. Backward pass, FP64 multiply-adds -> here: P2 on 1.05 M
// tetrahedra 1390 -> 510 us (730-890 us with CTA-wide phases and a barrier between them),
// P3 on 82,944 501 -> 175, P4 on 24,576 586 -> 165, P1 on 663,552 320 -> 219 us.
//
// A column's sum is held in units of 2^-B of (largest A0 of the column) (largest |dA| of the
// cell), so it keeps the digits that FP64 multiply-adds keep only while its own sum of |terms| is
// not far below those scales: with one large dA entry on which a column does not depend, or a dA
// of few entries, it is. The contraction therefore also sums |A0||f| of each column in half
// precision (three packed multiply-adds beside 18 integer ones) and takes a cell only where every
// column's sum reaches THETA; there the worst error over dA of independent, rank-one, diagonal and
// widely spread entries is 1e-16 to 8e-16 of the sum of |terms|, as with FP64 multiply-adds (2e-16
// to 1e-15). P1's columns have three or four terms, and 3% of the cells of a rank-one dA would fail,
// more than half of the warps: there dA is held in wide parts (fixed_point.cuh), and a cell is
// taken where its nonzero entries are within 2^28 of one another. Other cells, and those whose dA
// is not finite or lies outside [2^-900, 2^900] (P1: [2^-700, 2^900]), take FP64 multiply-adds
// over all n^2 entries, L lanes per cell.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "ffc_internal.h"
#include "fixed_point.cuh"
#include "geometry.cuh"

namespace ffc {
namespace {

template <int D, int Q>
struct AdjCfg {
  static constexpr int N = nscalar(D, Q);
  static constexpr int NN = N * N;
  static constexpr int NP = D * (D + 1) / 2;
  static constexpr int NE = N * (N + 1) / 2;
  // lanes per cell: 4-10 KB of staged dA per warp
  static constexpr int L = NN <= 16 ? 1 : (NN <= 64 ? 2 : (NN <= 128 ? 4 : (NN <= 256 ? 8 : (NN <= 512 ? 16 : 32))));
  static constexpr int CW = 32 / L;      // cells of a batch
  static constexpr int STRIDE = NN | 1;  // doubles of a staged row: odd, no bank conflicts over cells
  // warps per CTA: 16 in one CTA where the reference tensor takes 30 KB (P4 tetrahedra)
  static constexpr int WARPS = NE * NP > 2000 ? 16 : 4;
  static constexpr int MIN_BLOCKS = WARPS > 4 ? 1 : (NE > 200 ? 5 : 6);  // (P3 tetrahedra: 45 KB a CTA)
  static constexpr bool WIDE = Q == 1;
  // bits of a factor: the products of high parts h <= 2^(BITS - 29) of a lane's pairs, and of a
  // cell's where its lanes' sums are added in one piece, stay within 63 bits
  static constexpr int BITS = NE > 21 && NE <= 55 ? 57 : 58;
  static constexpr bool SPLIT = NE > 55;
  static constexpr int SUMMED = SPLIT ? (NE + L - 1) / L : NE;
  static_assert(double(SUMMED) * double(1ull << (2 * (BITS - 29))) < 9.0e18, "the sums must fit in 63 bits");
  // smallest sum of |A0||f| of a column, in units of 2^(its exponents): the errors of NE random
  // roundings of 2^-BITS against 2^-53 of it
  [[maybe_unused]] static constexpr int THETA = BITS - 52 - (NE > 100 ? 2 : 0) - (NE > 500 ? 2 : 0);
  static constexpr int NH = (NP + 1) / 2;  // half2 words of a pair's |A0|
  static constexpr int ROWS = CW * STRIDE;  // doubles of a warp's staged rows
  static constexpr int WBUF = ROWS + 32 * NP;  // and its cells' sums
  static constexpr size_t HB = WIDE ? 0 : (size_t(NE) * NH * 4 + 7) / 8 * 8;
  static constexpr size_t SMEM =
      HB + size_t(WARPS) * WBUF * 8 + size_t(NE) * NP * 8 + size_t(NE) * 4 + size_t(NP) * 4;
};

// the geometry chain rule of one cell and its atomics; S = Gbar + Gbar^T
//   dL/dJ = s (c I - P) K^T,  P = K^T S K,  c = tr(P) / 2
// (the formula above with K taken out on the right: 90 FP64 operations instead of 120)
template <int D>
__device__ __forceinline__ void adjoint_chain(const double K[D][D], double s, const double S[D][D], const int* id,
                                              double* dvert) {
  double W[D][D], P[D][D], c = 0.0;
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int r = 0; r < D; ++r) {
      double t = 0.0;
#pragma unroll
      for (int b = 0; b < D; ++b) t = fma(S[a][b], K[b][r], t);
      W[a][r] = t;
    }
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int m = r; m < D; ++m) {
      double t = 0.0;
#pragma unroll
      for (int a = 0; a < D; ++a) t = fma(K[a][r], W[a][m], t);
      P[r][m] = P[m][r] = t;
    }
#pragma unroll
  for (int r = 0; r < D; ++r) c += P[r][r];
  c *= 0.5 * s;
  double Qm[D][D];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int m = r; m < D; ++m) Qm[r][m] = Qm[m][r] = r == m ? fma(-s, P[r][r], c) : -s * P[r][m];
#pragma unroll
  for (int r = 0; r < D; ++r) {
    double sum = 0.0;
#pragma unroll
    for (int col = 0; col < D; ++col) {
      double t = 0.0;
#pragma unroll
      for (int m = 0; m < D; ++m) t = fma(Qm[r][m], K[col][m], t);
      atomicAdd(dvert + (long long)id[col + 1] * D + r, t);
      sum += t;
    }
    atomicAdd(dvert + (long long)id[0] * D + r, -sum);
  }
}

__device__ __forceinline__ void adj_copy8(double* dst, const double* src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}

// `tile_cells`: cells of a warp's tile, a multiple of CW, at most 32
template <int D, int Q>
__global__ void __launch_bounds__(AdjCfg<D, Q>::WARPS * 32, AdjCfg<D, Q>::MIN_BLOCKS)
    poisson_adjoint_kernel(const int32_t* __restrict__ cells, const double* __restrict__ vertices, long long n_vert,
                           const double* __restrict__ a0t, const double* __restrict__ dA, double* dvert,
                           long long n_elem, int tile_cells, unsigned* status) {
  using C = AdjCfg<D, Q>;
  constexpr int N = C::N, NN = C::NN, NP = C::NP, NE = C::NE, L = C::L, NT = C::WARPS * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __half2* ah = reinterpret_cast<__half2*>(smem_raw);                // [NE][NH] |A0| 2^-(column's exponent)
  int2* as = reinterpret_cast<int2*>(smem_raw + C::HB);              // [NE][NP] A0, fixed point
  double* wbuf = reinterpret_cast<double*>(as + NE * NP);            // [WARPS][WBUF]
  unsigned* pairs = reinterpret_cast<unsigned*>(wbuf + C::WARPS * C::WBUF);  // [NE] positions of (i1, i2), (i2, i1)
  int* ae = reinterpret_cast<int*>(pairs + NE);                      // [NP] exponents of A0's columns
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t < NP) ae[t] = -1022;
  for (int u = t; u < NE; u += NT) {
    int i1 = 0, v = u;
    while (v >= N - i1) v -= N - i1++;  // row i1 holds the pairs (i1, i1 .. N-1)
    pairs[u] = unsigned(i1 * N + i1 + v) | (unsigned((i1 + v) * N + i1) << 16);
  }
  __syncthreads();
  for (int w = t; w < NE * NP; w += NT)
    atomicMax(ae + w % NP, fix_exponent(__ldg(a0t + (w % NP) * NN + (pairs[w / NP] & 0xffffu))));
  __syncthreads();
  for (int w = t; w < NE * NP; w += NT)
    as[w] = fix_parts<C::BITS>(__ldg(a0t + (w % NP) * NN + (pairs[w / NP] & 0xffffu)), ae[w % NP]);
  if constexpr (!C::WIDE) {
    for (int w = t; w < NE * C::NH; w += NT) {
      const int u = w / C::NH, k = 2 * (w % C::NH), p = int(pairs[u] & 0xffffu);
      const float x = k < NP ? float(ldexp(fabs(__ldg(a0t + k * NN + p)), -ae[k])) : 0.f;
      const float y = k + 1 < NP ? float(ldexp(fabs(__ldg(a0t + (k + 1) * NN + p)), -ae[k + 1])) : 0.f;
      ah[w] = __floats2half2_rn(x, y);
    }
  }
  __syncthreads();
  double* rows = wbuf + warp * C::WBUF;  // [CW][STRIDE] dA of the batch
  double* gp = rows + C::ROWS;           // [32][NP] Gbar + Gbar^T of the tile's cells
  const int bc = lane / L, l = lane % L;
  const unsigned mask = L == 32 ? 0xffffffffu : ((1u << (L % 32)) - 1u) << (bc * L);
  const long long n_tiles = (n_elem + tile_cells - 1) / tile_cells;
  for (long long tile = (long long)blockIdx.x * C::WARPS + warp; tile < n_tiles;
       tile += (long long)gridDim.x * C::WARPS) {
    const long long e0 = tile * tile_cells;
    const int nc = int(n_elem - e0 < tile_cells ? n_elem - e0 : tile_cells);
    for (int b = 0; b < nc; b += C::CW) {
      const int nb = min(C::CW, nc - b);
      if (bc < nb) {  // each cell's lanes copy its row: 8 L contiguous bytes a row and step
        const double* src = dA + (e0 + b + bc) * NN;
#pragma unroll 5
        for (int k = l; k < NN; k += L) adj_copy8(rows + bc * C::STRIDE + k, src + k);
      }
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      __syncwarp();
      if (bc < nb) {
        const double* x = rows + bc * C::STRIDE;
        int top = -1022;
#pragma unroll 5
        for (int k = l; k < NN; k += L) top = max(top, fix_exponent(x[k]));
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(mask, top, o));
        double* g = gp + (b + bc) * NP;
        bool done = false;
        if constexpr (C::WIDE) {
          static_assert(L == 1 && NE <= 10, "a lane has the whole cell; sums of up to 10 terms");
          int low = 1025;  // of the nonzero entries
#pragma unroll
          for (int k = 0; k < NN; ++k) low = min(low, fix_exponent_or(x[k], 1025));
          if (low == 1025 && top == -1022) {
#pragma unroll
            for (int k = 0; k < NP; ++k) g[k] = 0.0;
            done = true;
          } else if (top <= 900 && low >= FIX_CELL_MIN_WIDE && top - low <= 28) {
            FixAccWide acc[NP];
#pragma unroll 2
            for (int u = 0; u < NE; ++u) {
              const unsigned pq = pairs[u];
              const int p1 = int(pq & 0xffffu), p2 = int(pq >> 16);
              int4 f = fix_parts_wide<C::BITS>(x[p1], top + 1);
              if (p1 != p2) {
                const int4 f2 = fix_parts_wide<C::BITS>(x[p2], top + 1);
                f.x += f2.x, f.y += f2.y, f.z += f2.z;
              }
              const int2* a = as + u * NP;
#pragma unroll
              for (int k = 0; k < NP; ++k) acc[k].add(a[k], f);
            }
#pragma unroll
            for (int k = 0; k < NP; ++k)
              g[k] = fix_to_double(acc[k], (ae[k] + top + 1 + 58 - 2 * C::BITS + (k < D ? 1 : 0)) * (1 << 20));
            done = true;
          }
        } else {
          if (top == -1022) {  // all zero (the gradients of local functionals mostly are) or denormal
            int any = 0;
            for (int k = l; k < NN; k += L) any |= x[k] != 0.0;
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) any |= __shfl_xor_sync(mask, any, o);
            if (any == 0) {
              for (int k = l; k < NP; k += L) g[k] = 0.0;
              done = true;
            }
          } else if (top <= 900 && top >= FIX_CELL_MIN) {
            FixAcc acc[NP];
            __half2 mass[C::NH];  // sums of |A0||f| of two columns each
#pragma unroll
            for (int k = 0; k < C::NH; ++k) mass[k] = __float2half2_rn(0.f);
#pragma unroll 2
            for (int u = l; u < NE; u += L) {
              const unsigned pq = pairs[u];
              const int p1 = int(pq & 0xffffu), p2 = int(pq >> 16);
              long long f = fix_round<C::BITS>(x[p1], top + 1);
              if (p1 != p2) f += fix_round<C::BITS>(x[p2], top + 1);
              const int2 fs = fix_split(f);
              const int2* a = as + u * NP;
#pragma unroll
              for (int k = 0; k < NP; ++k) acc[k].add(a[k], fs);
              const __half2 m = __float2half2_rn(float(abs(fs.x)) * (1.f / float(1 << (C::BITS - 29))));
#pragma unroll
              for (int k = 0; 2 * k < NP; ++k) mass[k] = __hfma2(ah[u * C::NH + k], m, mass[k]);
            }
            float least = 1.f;
#pragma unroll
            for (int k = 0; 2 * k < NP; ++k) {
#pragma unroll
              for (int o = L / 2; o > 0; o >>= 1) mass[k] = __hadd2(mass[k], __shfl_xor_sync(mask, mass[k], o));
              const float2 m = __half22float2(mass[k]);
              least = fminf(least, m.x);
              if (2 * k + 1 < NP) least = fminf(least, m.y);
            }
            done = least >= 1.f / float(1 << C::THETA);
            if (done) {
#pragma unroll
              for (int k = 0; k < NP; ++k) {
                long long v = acc[k].sum();
                // a diagonal entry of Gbar + Gbar^T is twice Gbar's
                int e = ae[k] + top + 1 + 58 - 2 * C::BITS + (k < D ? 1 : 0);
                if constexpr (C::SPLIT) {
                  int low = int(v) & 0xfffff;
                  v >>= 20;
#pragma unroll
                  for (int o = L / 2; o > 0; o >>= 1) {
                    v += __shfl_xor_sync(mask, v, o);
                    low += __shfl_xor_sync(mask, low, o);
                  }
                  v += low >> 20;
                  low &= 0xfffff;
                  if (v < (1ll << 42) && v >= -(1ll << 42)) {
                    v = v * (1ll << 20) + low;
                  } else {
                    v = v * (1ll << 14) + (low >> 6);
                    e += 6;
                  }
                } else {
#pragma unroll
                  for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
                }
                if (l == 0) g[k] = fix_to_double(v, e * (1 << 20));
              }
            }
          }
        }
        if (!done) {  // the cell's lanes agree
          double v[NP];
#pragma unroll
          for (int k = 0; k < NP; ++k) v[k] = 0.0;
#pragma unroll 2
          for (int i = l; i < NN; i += L) {
#pragma unroll
            for (int k = 0; k < NP; ++k) v[k] = fma(__ldg(a0t + k * NN + i), x[i], v[k]);
          }
#pragma unroll
          for (int k = 0; k < NP; ++k) {
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) v[k] += __shfl_xor_sync(mask, v[k], o);
            if (l == 0) g[k] = k < D ? 2.0 * v[k] : v[k];
          }
        }
      }
      __syncwarp();  // the rows are overwritten next; the sums are read below
    }
    if (lane < nc) {
      const long long e = e0 + lane;
      double K[D][D], s, S[D][D];
      bool degenerate, bad_index;
      cell_geometry<D>(cells, vertices, n_vert, e, K, s, degenerate, bad_index);
      if (degenerate) atomicOr(status, FFC_FLAG_DEGENERATE);
      if (bad_index) {
        atomicOr(status, FFC_FLAG_BOUNDS);
      } else {
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int b = 0; b < D; ++b) S[a][b] = gp[lane * NP + sym_pair_index<D>(a < b ? a : b, a < b ? b : a)];
        int id[D + 1];
#pragma unroll
        for (int j = 0; j <= D; ++j) id[j] = __ldg(cells + e * (D + 1) + j);
        adjoint_chain<D>(K, s, S, id, dvert);
      }
    }
    __syncwarp();  // the next tile's sums overwrite gp
  }
}

template <int D, int Q>
int run(const LaunchArgs& a, const double* dA, double* dvert) {
  using C = AdjCfg<D, Q>;
  auto kern = poisson_adjoint_kernel<D, Q>;
  constexpr int NT = C::WARPS * 32;
  int sms = 0, per_sm = 1;
  if (launch_config(reinterpret_cast<const void*>(kern), NT, C::SMEM, 100, &sms, &per_sm) != FFC_OK)
    return FFC_ECUDA;
  // tiles of 32 cells keep every lane in the chain rule; meshes of fewer cells than that per
  // resident warp take fewer (whole batches), so that the batches spread over the warps
  const long long warps = (long long)sms * per_sm * C::WARPS;
  long long tile = (a.n_elem + warps - 1) / warps;
  tile = tile >= 32 ? 32 : (tile + C::CW - 1) / C::CW * C::CW;
  long long grid = (long long)sms * per_sm;
  const long long need = (a.n_elem + tile * C::WARPS - 1) / (tile * C::WARPS);
  if (grid > need) grid = need;
  kern<<<unsigned(grid), NT, C::SMEM, static_cast<cudaStream_t>(a.stream)>>>(
      a.cells, a.vertices, a.n_vert, a.t->a0t_f64, dA, dvert, a.n_elem, int(tile), a.status);
  return cudaPeekAtLastError() == cudaSuccess ? FFC_OK : FFC_ECUDA;
}

}  // namespace

int launch_adjoint(const LaunchArgs& a, const double* dA, double* dvert) {
  if (a.f->kind != FFC_POISSON) return FFC_EUNSUPPORTED;
  if (a.f->d == 3) {
    switch (a.f->q) {
      case 1: return run<3, 1>(a, dA, dvert);
      case 2: return run<3, 2>(a, dA, dvert);
      case 3: return run<3, 3>(a, dA, dvert);
      case 4: return run<3, 4>(a, dA, dvert);
    }
  } else {
    switch (a.f->q) {
      case 1: return run<2, 1>(a, dA, dvert);
      case 2: return run<2, 2>(a, dA, dvert);
      case 3: return run<2, 3>(a, dA, dvert);
      case 4: return run<2, 4>(a, dA, dvert);
    }
  }
  return FFC_EUNSUPPORTED;
}

}  // namespace ffc
