// FP64 element tensors of the Poisson form (P1..P4, triangles and tetrahedra) and their
// fused assembly, with the contraction A^K_i = sum_alpha A0[i][alpha] G_K[alpha]
// (Section 3.2, Section 3.3 test case 2) in fixed point (fixed_point.cuh).
//
// What bounds it: with FP64 multiply-adds the contraction held the FP64 pipe at 87-92%
// with the issue slots at 11-19%. In fixed point only the per-cell geometry is left on
// that pipe, and an entry is 18 wide integer multiply-adds (0.72 SM clocks, a quarter of
// the 6 FP64 ones) and about 25 other integer instructions. Now the latency of a chunk
// (28% of the warps resident, issue 44%) and, for P1 and P2, the FP64 geometry bound the
// tabulation (P4 0.59 of HBM), FP64 atomics the assembly. Measured, FP64 multiply-adds ->
// fixed point: P4 tabulate of 384,000 tets 2645 -> 932 us, P3 assembly of 178,746 tets
// (with zeroing) 546 -> 324 us, P2 tabulate of 1.05 M tets 790 -> 327 us; cells that take the
// FP64 multiply-adds (stretched 1:64) P4 of 196,608 tets 1354 -> 745 us, P2 of 384,000 283 -> 161.
//
// One CTA takes tiles of E consecutive cells (persistent grid-stride loop):
//   geometry  one thread per cell: FP64 J, K = J^-1, |det J| and the symmetric G_K
//             (d(d+1)/2 values), stored as fixed-point parts with the cell's exponent;
//   chunks    CELLS cells at a time: thread t owns the entries i1 <= i2 (Section 3.5: a
//             symmetric form needs fewer operations) u = t mod NTI + r NTI of the cells of
//             its group and writes each result at (i1, i2) and (i2, i1) of the chunk's
//             element tensors in shared memory, two buffers deep;
//   epilogue  tabulate: one thread writes the chunk to A_K with a bulk copy, so the
//             transposed halves leave the SM as whole lines; assembly: the threads walk
//             the chunk in row-major order (coalesced slot loads, made before the
//             contraction) and add each value at csr_val[slot] with an FP64 atomic.
//
// The fixed point needs the diagonal entries of G_K within 2^6 of one another (edge-length
// ratios up to about 8, measured by the gradients' lengths) and each off-diagonal entry either
// zero or with terms within 2^6 of the largest entry, the terms of G_ab = det sum_c K_ac K_bc
// taken with those of the cofactors behind K: the error, below 2^-57 of the largest G_K entry
// times the row's largest A0 entry, is then below the rounding that an entry of G_K carries from
// its own terms. (A tensor entry can hang on one off-diagonal entry alone. On nearly
// axis-aligned corners, K = I plus a shear s, that is s, computed to 2^-53 s: held in units of
// 2^-59 it would keep 27 of its bits for s = 2^-32. Cells whose rows of K cancel, jittered or
// structured meshes among them, pass: their G_ab carries the error of the larger terms.) Other
// cells, and cells whose G_K is not finite or lies outside [2^-900, 2^900], take the FP64
// multiply-adds with A0 from global memory.
#include <cuda_runtime.h>

#include <cfloat>

#include "ffc_internal.h"
#include "fixed_point.cuh"
#include "geometry.cuh"
#include "simt_block.cuh"

namespace ffc {
namespace {

constexpr int FIX_BITS = 59;   // |alpha| <= 6 terms
constexpr int FIX_SPREAD = 6;  // of a cell's G_K entries, as a power of two

template <int D, int Q>
struct FixedCfg {
  static constexpr int N = nscalar(D, Q);
  static constexpr int NN = N * N;
  static constexpr int NP = D * (D + 1) / 2;
  static constexpr int NE = N * (N + 1) / 2;            // entries contracted per cell
  static constexpr int R = NE > 320 ? 2 : 1;            // entries per thread
  static constexpr int NTI = (NE + R - 1) / R;
  static constexpr int EG = NTI >= 256 ? 1 : 256 / NTI;  // thread groups
  static constexpr int NT = (NTI * EG + 31) / 32 * 32;
  // cells per chunk: 20 or 40 KB of staged element tensors per buffer (P4 with 20 KB, two
  // cells a chunk: 589 against 554 us; P2 with 40 KB, two CTAs: 297 against 205 us), whole
  // rounds of the groups, an even number (bulk copies move multiples of 16 bytes)
  static constexpr int STEP = EG % 2 ? 2 * EG : EG;
  static constexpr int CELLS_T = (R > 1 ? 40000 : 20000) / (NN * 8) / STEP * STEP;
  static constexpr int CELLS = CELLS_T < STEP ? STEP : (CELLS_T > 128 ? 128 / STEP * STEP : CELLS_T);
  // cells per tile: about 96, whole chunks
  static constexpr int E = CELLS >= 96 ? CELLS : 96 / CELLS * CELLS;
  static constexpr int BUF = CELLS * NN;                   // doubles of one staging buffer
  static constexpr int SLOTS = (BUF + NT - 1) / NT;        // assembly: values per thread and chunk
  static constexpr size_t SMEM = size_t(2) * BUF * 8 + size_t(E) * NP * 8 + size_t(E) * 4;
  // resident CTAs: two of 320 threads with two entries each (one entry and 640 threads:
  // 607 against 554 us for 196,608 P4 tets), else four (P3 at 384,000 tets 396 us, three 409,
  // five and six spill: 412, 482)
  static constexpr int MIN_BLOCKS = R > 1 ? 2 : 4;
};

struct FixedParams {
  const int32_t* cells;
  const double* vertices;
  long long n_vert;
  const double* a0t;  // [NP][NN] reference tensor, symmetric layout, transposed
  double* out;        // A_K [n_elem][NN] (tabulate)
  const int32_t* slot;
  double* csr_val;
  long long nnz;
  long long n_elem;
  unsigned* status;
};

// Sentinel exponent of a cell that takes the FP64 multiply-adds (an exponent is stored
// shifted into a double's exponent field, a multiple of 2^20).
constexpr int FIX_NONE = 1;

// The cell's G_K: fixed-point parts and the exponent, or doubles and FIX_NONE.
template <int D, int Q>
__device__ __forceinline__ void fixed_geometry(const FixedParams& p, long long e, int2* g, int* expo) {
  constexpr int NP = FixedCfg<D, Q>::NP;
  double J[D][D], K[D][D], det, G[NP];
  bool degenerate, bad_index;
  cell_jacobian<D>(p.cells, p.vertices, p.n_vert, e, J, bad_index);
  invert_jacobian<D>(J, K, det, degenerate);
  geometry_tensor_k<D, FFC_POISSON, Q>(K, det, nullptr, 0.0, 0.0, [&](int a, double v) { G[a] = v; });
  if (degenerate) atomicOr(p.status, FFC_FLAG_DEGENERATE);
  if (bad_index) atomicOr(p.status, FFC_FLAG_BOUNDS);
  int hi = fix_exponent(G[0]), lo = hi;  // exponents of the diagonal entries (slots 0 .. D-1)
#pragma unroll
  for (int a = 1; a < D; ++a) {
    const int x = fix_exponent(G[a]);
    hi = max(hi, x);
    lo = min(lo, x);
  }
  int top = hi;
#pragma unroll
  for (int a = D; a < NP; ++a) top = max(top, fix_exponent(G[a]));
  bool fixed = top <= 900 && lo >= FIX_CELL_MIN && hi - lo <= FIX_SPREAD;
  // FP32 holds the off-diagonal entries' terms for cells of 1e-18 to 1e18; elsewhere they over-
  // or underflow, which fails the comparison
  float U[D][D], Ka[D][D];
  cofactor_terms<D>(J, U);
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int c = 0; c < D; ++c) Ka[a][c] = magnitude_f32(K[a][c]);
  const float least = top > -100 && top < 120 ? __int_as_float((top - FIX_SPREAD + 127) << 23) : INFINITY;
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = a + 1; b < D; ++b) {
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < D; ++c) s = fmaf(U[a][c], Ka[b][c], fmaf(Ka[a][c], U[b][c], s));
      fixed = fixed && ((s >= least && s <= FLT_MAX) || !fix_nonzero(G[sym_pair_index<D>(a, b)]));
    }
  *expo = fixed ? top * (1 << 20) : FIX_NONE;
#pragma unroll
  for (int a = 0; a < NP; ++a)
    g[a] = fixed ? fix_parts<FIX_BITS>(G[a], top) : make_int2(__double2hiint(G[a]), __double2loint(G[a]));
}

template <int D, int Q, bool ASSEMBLE>
__global__ void __launch_bounds__(FixedCfg<D, Q>::NT, FixedCfg<D, Q>::MIN_BLOCKS)
    poisson_fixed_kernel(FixedParams p) {
  using C = FixedCfg<D, Q>;
  constexpr int N = C::N, NN = C::NN, NP = C::NP, R = C::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* stage = reinterpret_cast<double*>(smem_raw);         // [2][BUF]
  int2* gs = reinterpret_cast<int2*>(stage + 2 * C::BUF);      // [E][NP]
  int* ge = reinterpret_cast<int*>(gs + size_t(C::E) * NP);    // [E]
  const int t = threadIdx.x;
  const int ti = t % C::NTI, eg = t / C::NTI;
  // the thread's entries: positions and the reference tensor rows in fixed point
  int pos1[R], pos2[R], ea[R];
  int2 a[R][NP];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int u = ti + r * C::NTI;
    const bool live = u < C::NE && eg < C::EG;
    int i1 = 0, v = live ? u : 0;
    while (v >= N - i1) v -= N - i1++;  // row i1 holds the entries (i1, i1 .. N-1)
    pos1[r] = live ? i1 * N + i1 + v : -1;
    pos2[r] = (i1 + v) * N + i1;
    double x[NP];
    ea[r] = FIX_ROW_MIN;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      x[k] = live ? __ldg(p.a0t + size_t(k) * NN + pos1[r]) : 0.0;
      ea[r] = max(ea[r], fix_exponent(x[k]));
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) a[r][k] = fix_parts<FIX_BITS>(x[k], ea[r]);
    ea[r] = (ea[r] + 58 - 2 * FIX_BITS) * (1 << 20);
  }
  int buf_of = 0;       // staging buffer of the next chunk
  const long long n_tiles = (p.n_elem + C::E - 1) / C::E;
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const long long e0 = tile * C::E;
    const int nc = int(p.n_elem - e0 < C::E ? p.n_elem - e0 : C::E);
    for (int el = t; el < nc; el += C::NT) fixed_geometry<D, Q>(p, e0 + el, gs + el * NP, ge + el);
    __syncthreads();
    for (int c0 = 0; c0 < nc; c0 += C::CELLS) {
      const int ncc = min(C::CELLS, nc - c0), nv = ncc * NN;
      double* buf = stage + buf_of * C::BUF;
      const long long o0 = (e0 + c0) * NN;  // the chunk's first value
      int sl[ASSEMBLE ? C::SLOTS : 1];
      if constexpr (ASSEMBLE) {
#pragma unroll
        for (int j = 0; j < C::SLOTS; ++j) {
          const int k = t + j * C::NT;
          sl[j] = k < nv ? __ldg(p.slot + o0 + k) : -1;
        }
      }
      if (eg < C::EG) {
#pragma unroll 1
        for (int el = eg; el < ncc; el += C::EG) {
          const int2* g = gs + (c0 + el) * NP;
          const int eG = ge[c0 + el];
          double* cell = buf + el * NN;
          double v[R];
          if (eG != FIX_NONE) {
            FixAcc acc[R];
#pragma unroll
            for (int k = 0; k < NP; ++k) {
              const int2 gk = g[k];
#pragma unroll
              for (int r = 0; r < R; ++r) acc[r].add(a[r][k], gk);
            }
#pragma unroll
            for (int r = 0; r < R; ++r)  // one of two entries on each pipe (P4: 554 -> 533 us)
              v[r] = r == 0 ? fix_to_double(acc[r].sum(), ea[r] + eG) : fix_to_double_fp64(acc[r].sum(), ea[r] + eG);
          } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              v[r] = 0.0;
#pragma unroll 1
              for (int k = 0; k < NP; ++k)
                v[r] = fma(__hiloint2double(g[k].x, g[k].y), __ldg(p.a0t + size_t(k) * NN + max(pos1[r], 0)), v[r]);
            }
          }
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (pos1[r] < 0) continue;
            cell[pos1[r]] = v[r];
            cell[pos2[r]] = v[r];
          }
        }
      }
      if constexpr (ASSEMBLE) {
        // the other buffer's readers are past this barrier's predecessor: one barrier a chunk
        __syncthreads();
#pragma unroll
        for (int j = 0; j < C::SLOTS; ++j) {
          const int k = t + j * C::NT;
          if (k < nv) {
            if (sl[j] >= 0 && sl[j] < p.nnz) atomicAdd(p.csr_val + sl[j], buf[k]);
            else atomicOr(p.status, FFC_FLAG_BOUNDS);
          }
        }
      } else {
        fence_async_smem();
        if (t == 0) bulk_wait_read<0>();  // the previous copy has read the other buffer
        __syncthreads();
        if (t == 0) {
          bulk_s2g(p.out + o0, buf, unsigned(nv * 8) & ~15u);
          bulk_commit();
          if (nv & 1) p.out[o0 + nv - 1] = buf[nv - 1];
        }
      }
      buf_of ^= 1;
    }
    __syncthreads();  // the tile's G_K is overwritten next
  }
  if constexpr (!ASSEMBLE) {
    if (t == 0) bulk_wait_all();  // shared memory stays valid until the copies are done
  }
}

template <int D, int Q, bool ASSEMBLE>
int run(const LaunchArgs& a) {
  using C = FixedCfg<D, Q>;
  static_assert(C::E % C::CELLS == 0 && C::CELLS % 2 == 0, "chunks of whole 16-byte groups");
  auto kern = poisson_fixed_kernel<D, Q, ASSEMBLE>;
  int sms = 0, per_sm = 1;
  if (launch_config(reinterpret_cast<const void*>(kern), C::NT, C::SMEM, 100, &sms, &per_sm) != FFC_OK)
    return FFC_ECUDA;
  FixedParams p{a.cells, a.vertices, a.n_vert, a.t->a0t_f64, static_cast<double*>(a.out), a.slot, a.csr_val,
                a.nnz, a.n_elem, a.status};
  const long long n_tiles = (a.n_elem + C::E - 1) / C::E;
  long long grid = (long long)sms * per_sm;
  if (grid > n_tiles) grid = n_tiles;
  kern<<<unsigned(grid), C::NT, C::SMEM, static_cast<cudaStream_t>(a.stream)>>>(p);
  return cudaPeekAtLastError() == cudaSuccess ? FFC_OK : FFC_ECUDA;
}

template <int D>
int by_degree(const LaunchArgs& a, bool assemble) {
  switch (a.f->q) {
    case 1: return assemble ? run<D, 1, true>(a) : run<D, 1, false>(a);
    case 2: return assemble ? run<D, 2, true>(a) : run<D, 2, false>(a);
    case 3: return assemble ? run<D, 3, true>(a) : run<D, 3, false>(a);
    case 4: return assemble ? run<D, 4, true>(a) : run<D, 4, false>(a);
  }
  return FFC_EUNSUPPORTED;
}

}  // namespace

int launch_poisson_fixed(const LaunchArgs& a, bool assemble) {
  if (a.f->kind != FFC_POISSON) return FFC_EUNSUPPORTED;
  return a.f->d == 2 ? by_degree<2>(a, assemble) : by_degree<3>(a, assemble);
}

}  // namespace ffc
