// Structured contraction of the vector forms on CUDA cores (tile body and kernel).
//
// For a component-blocked Cartesian vector basis (phi_i = psi_s e_c), the reference
// tensors of the convection and elasticity forms are block structured (Section 3.5
// proposes exploiting exactly this): the element tensor decomposes into n_s x n_s
// blocks indexed by the components (c1, c2),
//
//   A_K[(c1,s1),(c2,s2)] = sum_k R[(s1,s2)][k] * Gb_K[b(c1,c2)][k],
//
// with a reduced reference tensor R and nb reduced geometry blocks per cell:
//   convection  R[(s1,s2)][(t,a)] = int psi_s1 psi_t d_a psi_s2 (k = t*d + a, n_s*d values),
//               one block H[(t,a)] = |det J| sum_c K[a][c] w_{c,t}, used on the diagonal
//               blocks c1 = c2 (off-diagonal blocks are structurally zero);
//   elasticity  R = scalar stiffness int d_a1 psi_s1 d_a2 psi_s2 (k = a1*d + a2, d*d values),
//               nine blocks Gb[(c1,c2)][(a1,a2)] = |det J| (mu delta(c1,c2) (K K^T)[a1][a2]
//               + mu K[a1][c2] K[a2][c1] + lambda K[a1][c1] K[a2][c2]).
// This is the same value as the dense A0 : G_K contraction (identical sums), with
// 27x (convection) and 9x (elasticity) fewer multiply-adds and a reference tensor small
// enough for registers.
//
// The FP64 contraction runs in fixed point (fixed_point.cuh): with FP64 multiply-adds it
// held the FP64 pipe at 94% with the issue slots at 9%. Now the wide integer multiply-adds
// (convection P2: 90 per value, 360 SM clocks a cell against 306 for its A_K at the HBM
// rate), their latency at two resident CTAs and the geometry phase bound it. FP64
// multiply-adds -> fixed point: tabulate convection P2 on 384,000 tets 2309 -> 836 us, P1
// 237 -> 181; elasticity, whose parts are wider (45 wide multiply-adds per value, 53 of the 69
// SM clocks a warp's P3 values take), P3 on 48,000 tets 3183 -> 1297, P2 on 162,000 2607 -> 1221,
// P1 on 384,000 1182 -> 630; assembly of 82,944 tets, convection P2 570 -> 272, elasticity P2
// 1508 -> 702 us.
//
// Thread layouts. Elasticity, "row slots": a slot is (s1, c2, s2), numbered with s2
// fastest, then c2, then s1, so consecutive slots are consecutive entries of element
// tensor row (c1, s1) for every c1; the slot keeps R[(s1,s2)] in registers and per cell
// contracts it with the block (c1, c2) for each c1: a warp's store (or atomic) instruction
// covers a contiguous run of one row (one CSR row in assembly). Convection, "pair major":
// a slot is a pair (s1, s2); its one block is contracted once per cell and written to the
// d diagonal positions, zeros elsewhere (tabulate) or nothing (assembly); row slots would
// repeat that contraction d times. Earlier single layouts for both: "entry major" (each
// thread an entry of the row-major element tensor; convection P2 1.57 ms) and pair major
// for elasticity too (runs of n_s entries per store: elasticity P3 0.66 ms, batched 17.2
// ms, against 0.56 and 15.1 ms with row slots).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "ffc_internal.h"
#include "fixed_point.cuh"
#include "geometry.cuh"
#include "simt_kernels.cuh"

namespace ffc {

// BLOCK = 0: thread count from the number of pairs; BLOCK > 0: fixed block size shared
// with other forms (batched kernel). KE_T > 0: cells per thread group and tile (tiles
// are capped at 128 cells); 0 = 128 cells per tile.
template <int D, int FORM, int Q, typename T, int BLOCK = 0, int KE_T = 0>
struct BlockCfg {
  static constexpr int NS = nscalar(D, Q);
  static constexpr int N = D * NS;
  static constexpr int NN = N * N;
  static constexpr int KR = FORM == FFC_NS_CONVECTION ? NS * D : D * D;
  static constexpr int NB = FORM == FFC_NS_CONVECTION ? 1 : D * D;
  // FP64 elasticity keeps its geometry entries as wide fixed-point parts, 16 bytes each
  static constexpr bool WIDE = sizeof(T) == 8 && FORM == FFC_ELASTICITY;
  static constexpr int GW = WIDE ? 2 : 1;  // entries of type T a geometry entry takes
  static constexpr int VEC = WIDE ? 1 : 16 / int(sizeof(T));
  static constexpr int KRP = (KR + VEC - 1) / VEC * VEC;
  static constexpr bool DIAG = FORM == FFC_NS_CONVECTION;  // one block, on the diagonal
  static constexpr int NP2 = NS * NS;                      // pairs (s1, s2): rows of R
  static constexpr int NSL = DIAG ? NP2 : D * NS * NS;     // slots: pairs, or row slots (s1, c2, s2)
  // about 256 threads: whole groups of NSL slots, or up to 512 threads with several
  // slots each, rounded up to whole warps
  // (FP32 with 512 or more slots: 416 threads, two resident CTAs; see MIN_BLOCKS)
  static constexpr int NT0 = NSL >= 256 ? (NSL < 512 ? NSL : (sizeof(T) == 4 ? 416 : 512)) : NSL * (256 / NSL);
  static constexpr int NT = BLOCK > 0 ? BLOCK : (NT0 + 31) / 32 * 32;
  static constexpr int GRP = NT >= NSL ? NT / NSL : 1;  // thread groups; a tile's cells are dealt to them
  static constexpr int PPT = (NSL + NT - 1) / NT;       // slots per thread
  static constexpr bool REG_R = PPT * KR * int(sizeof(T)) / 4 <= 64;
  static constexpr int E_DEF = sizeof(T) == 8 ? 64 : 128;
  static constexpr int E = KE_T > 0 ? (KE_T * GRP < 128 ? KE_T * GRP : 128) : E_DEF;  // cells per tile
  static constexpr int NCOEF = FORM == FFC_NS_CONVECTION ? N : 0;
  static constexpr size_t G_BYTES = size_t(E) * NB * KRP * GW * sizeof(T);
  static constexpr size_t R_BYTES = REG_R ? 0 : size_t(NP2) * KRP * sizeof(T);
  static constexpr size_t W_BYTES = size_t(E) * NCOEF * sizeof(double);
  // FP64 contracts in fixed point (fixed_point.cuh): the geometry blocks and the reduced
  // rows are kept as fixed-point parts, with an exponent per cell and per slot
  static constexpr bool FIX = sizeof(T) == 8;
  static constexpr int BITS = 58;       // KR <= 31 terms (wide: 9)
  // FP64 scratch per cell: J^-1, |det J| and, for elasticity, |det J| mu K K^T (symmetric)
  static constexpr int XD = D * D + 1 + (DIAG ? 0 : D * (D + 1) / 2);
  static constexpr size_t X_BYTES = FIX ? size_t(E) * (XD * sizeof(double) + 4 * sizeof(int)) : 0;
  // FP64 convection: RowMasks and the exponents of K's entries
  static constexpr size_t M_BYTES =
      FIX && DIAG ? (size_t(NP2) * 16 + 4 + size_t(E) * (D * D + KR) * sizeof(int) + 15) / 16 * 16 : 0;
  static constexpr size_t SMEM = G_BYTES + R_BYTES + W_BYTES + X_BYTES + M_BYTES;
  // register budget of the single-form FP32 kernel: two resident CTAs of 257..511 threads
  // (up to 78 registers), three of up to 256; FP64 keeps its reduced rows in registers
  // without spills: three CTAs for convection P1 (two: 215 against 181 us), two of up to 320
  // threads (convection P2 with one: 1122 against 810 us, with three and spills 986 us;
  // elasticity P2 with one 1453 against 1221 us), one of more (elasticity P3 with two and
  // narrower parts: 1262 against 945 us)
  static constexpr int MIN_BLOCKS = sizeof(T) == 8 ? (DIAG && KR <= 12 ? 3 : (NT <= 320 ? 2 : 1))
                                                   : (NT >= 512 ? 1 : (NT > 256 ? 2 : 3));
};

template <class C, typename T>
struct BlockRows {
  using V = typename std::conditional<C::FIX, int2, T>::type;
  V rr[C::REG_R ? C::PPT : 1][C::REG_R ? C::KR : 1];  // reduced rows of the thread's slots
  int expo[C::FIX ? C::PPT : 1];                      // FP64: exponents of the results (<< 20)
};

// Sentinel exponent of a cell whose geometry blocks stay doubles (exponents are stored
// shifted into a double's exponent field, multiples of 2^20).
constexpr int BLOCK_FIX_NONE = 1;

// Tabulate of the single-form convection kernels: the element tensors of CELLS cells
// at a time are put together in shared memory (the off-diagonal blocks, always zero, are
// written there once), then one thread writes them to A_K with a TMA bulk copy, two
// buffers deep, so A_K leaves the SM as whole contiguous lines instead of runs of n_s
// floats. Convection P2 on 384,000 cells: 0.362 ms with direct stores; 0.297 ms staged
// with 4-cell chunks and 128-cell tiles, against 0.31-0.34 ms for 2-, 6- or 8-cell chunks
// or 64-cell tiles. Elasticity, whose row-slot stores are already contiguous runs of a
// row, writes directly (staged in 2-cell chunks its P3 tabulate went 0.513 -> 0.608 ms).
template <class C, typename T, bool ASSEMBLE>
struct BlockStaging {
  static constexpr bool ON = !ASSEMBLE && C::DIAG;
  static constexpr int CELLS = C::GRP > 4 ? C::GRP : 4;  // at least one cell per thread group
  static constexpr size_t BUF = size_t(CELLS) * C::NN * sizeof(T);  // a multiple of 16 bytes
  static constexpr size_t BYTES = ON ? 2 * BUF : 0;
};

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
// shared -> global bulk copy (addresses 16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_s2g(void* gdst, const void* ssrc, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(gdst), "r"(smem_u32(ssrc)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(PENDING) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// The thread's slots: slot j is q = t mod NSL (NT >= NSL, group t / NSL) or q = t + j*NT
// (NT < NSL, one group); -1: none. Slot q is (s1, c2, s2) with s2 fastest.
template <class C>
__device__ __forceinline__ int slot_of(int t, int j) {
  if constexpr (C::NT >= C::NSL) return (j == 0 && t < C::GRP * C::NSL) ? t % C::NSL : -1;
  else return (t + j * C::NT < C::NSL) ? t + j * C::NT : -1;
}
template <class C>
__device__ __forceinline__ int pair_of_slot(int q) {  // the row (s1, s2) of R a slot uses
  if constexpr (C::DIAG) return q;
  const int s2 = q % C::NS, s1 = q / (C::NS * (C::N / C::NS));
  return s1 * C::NS + s2;
}

// Bit masks of R's rows (FP64 convection), in shared memory: bit k of `large` for the entries
// within 2^2 of the row's largest, of `live` for the nonzero ones, and the `n_least` rows
// `least` (both masks) whose large mask holds no other row's (P2: 22 of 100): a cell whose large
// entries meet every one of these meets every row's.
template <class C>
struct RowMasks {
  uint2* least;
  unsigned *large, *live;
  int* n_least;
  int* k_expo;  // [E][D D] exponents of the cells' K, FIX_ZERO for zero
  int* terms;   // [E][KR] exponents of det sum_c |K_ac||w_ct|
  __device__ __forceinline__ explicit RowMasks(unsigned char* smem) {
    least = reinterpret_cast<uint2*>(smem + C::SMEM - C::M_BYTES);
    large = reinterpret_cast<unsigned*>(least + C::NP2);
    live = large + C::NP2;
    n_least = reinterpret_cast<int*>(live + C::NP2);
    k_expo = n_least + 1;
    terms = k_expo + C::E * (C::N / C::NS) * (C::N / C::NS);
  }
};
constexpr int FIX_ZERO = -5000;  // exponent of a zero factor: below that of any product

// The reduced reference tensor rows (registers, or shared memory behind the geometry
// blocks; the first barrier of block_tile orders those stores).
template <class C, int D, int FORM, typename T>
__device__ __forceinline__ void block_rows_init(const void* r, BlockRows<C, T>& b, unsigned char* smem) {
  const int t = threadIdx.x;
  const T* Rg = static_cast<const T*>(r);
  if constexpr (C::REG_R) {
#pragma unroll
    for (int j = 0; j < C::PPT; ++j) {
      const int q = slot_of<C>(t, j);
      const int pp = q >= 0 ? pair_of_slot<C>(q) : 0;
      if constexpr (C::FIX) {
        int e = FIX_ROW_MIN;
        for (int k = 0; k < C::KR; ++k) e = max(e, fix_exponent(Rg[size_t(pp) * C::KR + k]));
#pragma unroll
        for (int k = 0; k < C::KR; ++k) b.rr[j][k] = fix_parts<C::BITS>(Rg[size_t(pp) * C::KR + k], e);
        b.expo[j] = (e + 58 - 2 * C::BITS) * (1 << 20);
        if constexpr (C::DIAG) {
          static_assert(C::KR < 32 && C::NT >= C::NSL, "a bit per entry, and one to spare; a row per thread");
          const RowMasks<C> rm(smem);
          unsigned large = 0u, live = 0u;
          for (int k = 0; k < C::KR; ++k) {
            const double x = Rg[size_t(pp) * C::KR + k];
            if (fix_exponent(x) >= e - 2) large |= 1u << k;
            if (fix_nonzero(x)) live |= 1u << k;
          }
          if (t < C::NP2) {  // the first group's
            rm.large[t] = large;
            rm.live[t] = live;
          }
          if (t == 0) *rm.n_least = 0;
          __syncthreads();
          if (t < C::NP2) {
            bool keep = true;
            for (int r = 0; r < C::NP2; ++r)
              keep = keep && ((rm.large[r] & ~large) != 0u || (rm.large[r] == large && r >= t));
            if (keep) rm.least[atomicAdd(rm.n_least, 1)] = make_uint2(large, live);
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < C::KR; ++k) b.rr[j][k] = q >= 0 ? Rg[size_t(pp) * C::KR + k] : T(0);
      }
    }
  } else {
    T* Rs = reinterpret_cast<T*>(smem + C::G_BYTES);
    for (int k = t; k < C::NP2 * C::KRP; k += C::NT) {
      const int rw = k / C::KRP, kk = k % C::KRP;
      Rs[k] = kk < C::KR ? Rg[size_t(rw) * C::KR + kk] : T(0);
    }
  }
}

// FP64: the geometry blocks of a tile's cells in fixed point. One thread per cell forms
// J^-1 and |det J|; then the whole CTA forms the blocks, one (cell, node) or (cell, c1, c2)
// part at a time, with the cell's largest exponent in shared memory, and rewrites them in
// place as fixed-point parts. (One thread per cell for all of it left five of seven warps
// waiting: convection P2 881 against 816 us.)
//
// Convection takes the fixed point where every entry of the tensor has a term R H of which R is
// within 2^2 of its row's largest entry and H, taken as det sum_c |K_ac||w_ct|, within 2^3 of
// the cell's largest: an entry then errs by no more of the sum of its |terms| than FP64
// multiply-adds (worst of random, aligned, stretched, one-sided and widely spread inputs 5.4e-16
// against 5.0e-16 for P1, 4.3e-16 against 1.0e-15 for P2; with 2^4 1.7e-15). That fails for a cell whose coefficients or rows of K
// differ by more (a component 1e-4 of the others on an aligned cell, a single nonzero node):
// its entries that hang on the small ones would keep 58 bits less the difference. The threads
// of each slot test their rows' masks against the cell's. An entry with no term passes (w = 0).
// Elasticity: a block entry is a product of two entries of K, det and mu or lambda, and a tensor
// entry can hang on a single one (P1: one of 9 wherever s1 and s2 are not vertex 0), on cells
// with rows along the axes a small one. So its parts are wide, 87 bits below the cell's largest
// entry, and the cell is taken where the product of the two smallest entries of K (those that
// are zero but for rounding counted by the size of their cofactor's products), det and the
// smaller of |mu| and |lambda| is within 2^28 of that.
//
// All finite and far from the ends of the range. Other cells keep doubles and BLOCK_FIX_NONE.
// The exponents of the two smallest nonzero entries of K = J^-1, added. An entry below 2^-50 of
// its cofactor's products has no digit right and counts by those.
template <int D>
__device__ __forceinline__ int smallest_product(const double J[D][D], const double K[D][D], double det) {
  float U[D][D];
  cofactor_terms<D>(J, U);
  const float inv = 1.f / float(det);
  int k1 = 1025, k2 = 1025;
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const float u = U[a][c] * inv;
      int x = fix_exponent_or(K[a][c], 1025);
      if (u >= 1e-30f && u <= 1e30f && magnitude_f32(K[a][c]) < u * 0x1p-50f)
        x = int(__float_as_uint(u) >> 23) - 126;
      k2 = min(k2, max(k1, x));
      k1 = min(k1, x);
    }
  return k1 + k2;
}

template <class C, int D, int FORM>
__device__ __forceinline__ void block_geometry_fixed(const SimtParams& p, long long e0, double* Gs, const double* Ws,
                                                     double* Ks, int* Xs, unsigned char* smem) {
  constexpr bool CONV = FORM == FFC_NS_CONVECTION;
  constexpr int PARTS = CONV ? C::NS : D * D;      // parts of a cell's blocks
  constexpr int PLEN = CONV ? D : C::KRP;          // stored entries of a part
  constexpr int PUSED = CONV ? D : D * D;          // entries used
  constexpr int GW = C::GW;                        // doubles an entry takes
  const int t = threadIdx.x;
  const int nc = int(p.n_elem - e0 < C::E ? p.n_elem - e0 : C::E);
  int* Ts = Xs + C::E;      // [E] largest exponent of the blocks
  int* Ls = Xs + 2 * C::E;  // [E] elasticity: smallest exponent allowed for
  unsigned* Ms = reinterpret_cast<unsigned*>(Ls);  // [E] convection: bit k for the large entries of H
  unsigned* Zs = Ms + C::E;                        // [E] and for the nonzero ones; bit 31: H has a denormal
  [[maybe_unused]] const RowMasks<C> rm(smem);
  for (int el = t; el < nc; el += C::NT) {
    double J[D][D], K[D][D], det;
    bool degenerate, bad_index;
    cell_jacobian<D>(p.cells, p.vertices, p.n_vert, e0 + el, J, bad_index);
    invert_jacobian<D>(J, K, det, degenerate);
    if (degenerate) atomicOr(p.status, FFC_FLAG_DEGENERATE);
    if (bad_index) atomicOr(p.status, FFC_FLAG_BOUNDS);
    double* k = Ks + el * C::XD;
#pragma unroll
    for (int a = 0; a < D; ++a) {
#pragma unroll
      for (int b = 0; b < D; ++b) k[a * D + b] = K[a][b];
      if constexpr (!CONV) {
#pragma unroll
        for (int b = a; b < D; ++b) {
          double s = 0.0;
#pragma unroll
          for (int c = 0; c < D; ++c) s = fma(K[a][c], K[b][c], s);
          k[D * D + 1 + sym_pair_index<D>(a, b)] = s * (det * p.mu);
        }
      }
    }
    k[D * D] = det;
    Ts[el] = -1022;
    if constexpr (CONV) {
      Ms[el] = Zs[el] = 0u;
      Xs[el] = 0;
#pragma unroll
      for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) rm.k_expo[el * D * D + a * D + b] = fix_exponent_or(K[a][b], FIX_ZERO);
    } else {
      Ls[el] = smallest_product<D>(J, K, det) + fix_exponent(det) +
               min(fix_exponent_or(p.mu, 1025), fix_exponent_or(p.lambda, 1025));
    }
  }
  __syncthreads();
  for (int w = t; w < nc * PARTS; w += C::NT) {
    const int el = w / PARTS, part = w - el * PARTS;
    const double* K = Ks + el * C::XD;
    const double det = K[D * D];
    double* g = Gs + (size_t(el) * C::NB * C::KRP + part * PLEN) * GW;
    int top = -1022;
    if constexpr (CONV) {
      double wc[D];
      int we[D];
#pragma unroll
      for (int c = 0; c < D; ++c) {
        wc[c] = Ws[el * C::NCOEF + c * C::NS + part];
        we[c] = fix_exponent_or(wc[c], FIX_ZERO);
      }
      const int de = fix_exponent(det);
      unsigned denormal = 0u;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        double h = 0.0;
        int x = 2 * FIX_ZERO;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          h = fma(K[a * D + c], wc[c], h);
          x = max(x, rm.k_expo[el * D * D + a * D + c] + we[c]);
        }
        rm.terms[w * D + a] = x + de;
        g[a] = det * h;
        top = max(top, fix_exponent(g[a]));
        if (fix_exponent(g[a]) == -1022 && fix_nonzero(g[a])) denormal = 1u << 31;
      }
      if (denormal) atomicOr(Zs + el, denormal);
    } else {
      const int c1 = part / D, c2 = part - c1 * D;
      const double dm = det * p.mu, dl = det * p.lambda;
#pragma unroll
      for (int a1 = 0; a1 < D; ++a1) {
        const double m1 = dm * K[a1 * D + c2], l1 = dl * K[a1 * D + c1];
#pragma unroll
        for (int a2 = 0; a2 < D; ++a2) {
          const int ab = sym_pair_index<D>(a1 < a2 ? a1 : a2, a1 < a2 ? a2 : a1);
          double v = c1 == c2 ? K[D * D + 1 + ab] : 0.0;
          v = fma(l1, K[a2 * D + c2], fma(m1, K[a2 * D + c1], v));
          g[(a1 * D + a2) * GW] = v;
          top = max(top, fix_exponent(v));
        }
      }
    }
    atomicMax(Ts + el, top);
  }
  __syncthreads();
  if constexpr (CONV) {
    for (int w = t; w < nc * PARTS; w += C::NT) {  // the masks of the thread's parts
      const int el = w / PARTS, part = w - el * PARTS, least = Ts[el] - 3;
      unsigned large = 0u, live = 0u;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        large |= unsigned(rm.terms[w * D + a] >= least) << a;
        live |= unsigned(rm.terms[w * D + a] > FIX_ZERO / 2) << a;
      }
      atomicOr(Ms + el, large << (part * D));
      atomicOr(Zs + el, live << (part * D));
    }
    __syncthreads();
    // every cell against the least masks, a lane per cell; those that miss one whose row has
    // no term at all (few) against every row. Xs: bit 0 multiply-adds, bit 1 undecided
    static_assert(C::NT >= C::E, "a thread or more per cell");
    bool undecided = false;
    const int el0 = t % C::E;
    if (t < C::NT / C::E * C::E && el0 < nc) {
      const unsigned large = Ms[el0], live = Zs[el0];
      bool failed = false;
      for (int i = t / C::E; i < *rm.n_least; i += C::NT / C::E) {
        const uint2 r = rm.least[i];
        if ((r.x & large) == 0u) {
          if (r.y & live) failed = true;
          else undecided = true;
        }
      }
      if (failed || undecided) atomicOr(Xs + el0, failed ? BLOCK_FIX_NONE : 2);
      undecided = undecided && !failed;
    }
    if (__syncthreads_or(undecided)) {
      const int q = slot_of<C>(t, 0);
      if (q >= 0) {
        const unsigned large = rm.large[q], live = rm.live[q];
        for (int el = t / C::NSL; el < nc; el += C::GRP)
          if (Xs[el] == 2 && (large & Ms[el]) == 0u && (live & Zs[el]) != 0u) atomicOr(Xs + el, BLOCK_FIX_NONE);
      }
      __syncthreads();
    }
  }
  for (int w = t; w < nc * PARTS; w += C::NT) {  // each thread its own parts again
    const int el = w / PARTS, part = w - el * PARTS;
    int top = Ts[el];
    bool fixed = top <= 900 && top >= (C::WIDE ? FIX_CELL_MIN_WIDE : FIX_CELL_MIN);
    if constexpr (CONV) {
      if (top == -1022 && !(Zs[el] >> 31)) {  // H = 0: its parts are zero
        fixed = true;
        top = FIX_CELL_MIN;
      }
      fixed = fixed && !(Xs[el] & BLOCK_FIX_NONE);
    } else {
      fixed = fixed && top - Ls[el] <= 28;
    }
    if (part == 0) Xs[el] = fixed ? top * (1 << 20) : BLOCK_FIX_NONE;
    if (!fixed) continue;
    double* g = Gs + (size_t(el) * C::NB * C::KRP + part * PLEN) * GW;
#pragma unroll
    for (int k = 0; k < PUSED; ++k) {
      if constexpr (C::WIDE) reinterpret_cast<int4*>(g)[k] = fix_parts_wide<C::BITS>(g[k * GW], top);
      else reinterpret_cast<int2*>(g)[k] = fix_parts<C::BITS>(g[k], top);
    }
  }
}

// One tile of E cells: reduced geometry blocks into shared memory, then each thread
// contracts its pairs with every block of the group's cells. Contains block barriers.
template <class C, int D, int FORM, int Q, typename T, bool ASSEMBLE>
__device__ __forceinline__ void block_tile(const SimtParams& p, long long tile, unsigned char* smem,
                                           const BlockRows<C, T>& br, int* staged_chunks = nullptr) {
  T* Gs = reinterpret_cast<T*>(smem);                                       // [E][NB][KRP]
  const T* Rs = reinterpret_cast<const T*>(smem + C::G_BYTES);              // [NP2][KRP]
  double* Ws = reinterpret_cast<double*>(smem + C::G_BYTES + C::R_BYTES);   // [E][NCOEF]
  double* Ks = reinterpret_cast<double*>(smem + C::G_BYTES + C::R_BYTES + C::W_BYTES);  // FP64: [E][XD]
  int* Xs = reinterpret_cast<int*>(Ks + (C::FIX ? C::E * C::XD : 0));                    // FP64: [E] exponents
  const int t = threadIdx.x;
  const long long e0 = tile * C::E;
  if constexpr (C::NCOEF > 0) {
    const long long lim = (p.n_elem - e0) * C::NCOEF;
    const double* src = p.coeffs + e0 * C::NCOEF;
    for (int k = t; k < C::E * C::NCOEF; k += C::NT) Ws[k] = (k < lim) ? __ldg(src + k) : 0.0;
  }
  __syncthreads();
  // ---- reduced geometry blocks of the tile's cells
  if constexpr (C::FIX) block_geometry_fixed<C, D, FORM>(p, e0, Gs, Ws, Ks, Xs, smem);
  else for (int el = t; el < C::E; el += C::NT) {
    const long long e = e0 + el;
    T* g = Gs + size_t(el) * C::NB * C::KRP;
    // J^{-1} and det J in FP64 (measured: forming J^{-1} in FP32 from the FP64 adjugate,
    // as the dense kernels do, made this tile slower); the reduced geometry blocks, their
    // products with the coefficients, in the contraction's type (rounded to it anyway)
    double K[D][D] = {}, det = 0.0;
    bool live = e < p.n_elem;
    if (live) {
      bool degenerate, bad_index;
      cell_geometry<D>(p.cells, p.vertices, p.n_vert, e, K, det, degenerate, bad_index);
      if (degenerate) atomicOr(p.status, FFC_FLAG_DEGENERATE);
      if (bad_index) atomicOr(p.status, FFC_FLAG_BOUNDS);
    }
    using GT = T;
    GT Kt[D][D], dett = GT(det);
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int b = 0; b < D; ++b) Kt[a][b] = GT(K[a][b]);
    if constexpr (FORM == FFC_NS_CONVECTION) {
      const double* w = Ws + el * C::NCOEF;
#pragma unroll
      for (int st = 0; st < C::NS; ++st) {
        GT wc[D];
#pragma unroll
        for (int c = 0; c < D; ++c) wc[c] = GT(w[c * C::NS + st]);
#pragma unroll
        for (int a = 0; a < D; ++a) {
          GT h = GT(0);
#pragma unroll
          for (int c = 0; c < D; ++c) h = fma(Kt[a][c], wc[c], h);
          g[st * D + a] = live ? dett * h : T(0);
        }
      }
    } else {
      GT KK[D][D];
#pragma unroll
      for (int a1 = 0; a1 < D; ++a1)
#pragma unroll
        for (int a2 = 0; a2 < D; ++a2) {
          GT sum = GT(0);
#pragma unroll
          for (int b = 0; b < D; ++b) sum = fma(Kt[a1][b], Kt[a2][b], sum);
          KK[a1][a2] = sum;
        }
      const GT mu = GT(p.mu), lambda = GT(p.lambda);
#pragma unroll
      for (int c1 = 0; c1 < D; ++c1)
#pragma unroll
        for (int c2 = 0; c2 < D; ++c2)
#pragma unroll
          for (int a1 = 0; a1 < D; ++a1)
#pragma unroll
            for (int a2 = 0; a2 < D; ++a2) {
              GT v = mu * Kt[a1][c2] * Kt[a2][c1] + lambda * Kt[a1][c1] * Kt[a2][c2];
              if (c1 == c2) v += mu * KK[a1][a2];
              g[(c1 * D + c2) * C::KRP + a1 * D + a2] = live ? dett * v : T(0);
            }
    }
#pragma unroll
    for (int b = 0; b < C::NB; ++b)
      for (int k = C::KR; k < C::KRP; ++k) g[b * C::KRP + k] = T(0);
  }
  __syncthreads();
  // ---- contraction: the thread's slots x the group's cells
  constexpr bool DIAG = C::DIAG;
  constexpr int NPOS = DIAG ? D * D : D;  // element-tensor entries a slot writes per cell
  const int grp = C::NT >= C::NSL ? t / C::NSL : 0;
  const long long left = p.n_elem - e0;
  const int nc = int(left < C::E ? left : C::E);
  // R[(s1,s2)] . block of cell el
  auto contract = [&](const T* gblk, int el, int j, const T* rrow, int row) {
    if constexpr (C::FIX) {
      const int eG = Xs[el];
      if (eG == BLOCK_FIX_NONE) {
        const double* R = static_cast<const double*>(p.a0) + size_t(row) * C::KR;
        double acc = 0.0;
        if constexpr (C::KR % 2 == 0) {  // rows of whole 16-byte pairs
#pragma unroll 3
          for (int k = 0; k < C::KR; k += 2) {
            const double2 r = __ldg(reinterpret_cast<const double2*>(R + k));
            acc = fma(gblk[k], r.x, acc);
            acc = fma(gblk[k + 1], r.y, acc);
          }
        } else {
          for (int k = 0; k < C::KR; ++k) acc = fma(gblk[k * C::GW], __ldg(R + k), acc);
        }
        return acc;
      }
      const int4* gv = reinterpret_cast<const int4*>(gblk);
      const int e20 = br.expo[j] + eG;
      if constexpr (C::WIDE) {
        FixAccWide acc;
#pragma unroll
        for (int k = 0; k < C::KR; ++k) acc.add(br.rr[j][k], gv[k]);
        return fix_to_double(acc, e20);
      } else {
        FixAcc acc;
#pragma unroll
        for (int k = 0; k < C::KR; k += 2) {
          const int4 x = gv[k / 2];
          acc.add(br.rr[j][k], make_int2(x.x, x.y));
          if (k + 1 < C::KR) acc.add(br.rr[j][k + 1 < C::KR ? k + 1 : k], make_int2(x.z, x.w));
        }
        return fix_to_double_fp64(acc.sum(), e20);
      }
    } else {
      const float4* gv = reinterpret_cast<const float4*>(gblk);
      T acc = T(0);
#pragma unroll
      for (int kv = 0; kv < C::KRP / C::VEC; ++kv) {
        const float4 x = gv[kv];
        const T xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int m = 0; m < C::VEC; ++m) {
          const int k = kv * C::VEC + m;
          if (k < C::KR) {
            if constexpr (C::REG_R) acc = fma(xs[m], br.rr[j][k < C::KR ? k : 0], acc);
            else acc = fma(xs[m], rrow[k], acc);
          }
        }
      }
      return acc;
    }
  };
  using SG = BlockStaging<C, T, ASSEMBLE>;
  if constexpr (SG::ON) {
    // chunks of SG::CELLS cells; within a chunk the groups take cells grp, grp + GRP, ...
    T* stage = reinterpret_cast<T*>(smem + C::SMEM);
    for (int c0 = 0; c0 < nc; c0 += SG::CELLS) {
      const int b = *staged_chunks & 1;
      T* buf = stage + b * (SG::BUF / sizeof(T));
      if (*staged_chunks >= 2 && t == 0) bulk_wait_read<1>();  // the copy that last read buf is done
      __syncthreads();
      const int ncc = nc - c0 < SG::CELLS ? nc - c0 : SG::CELLS;
#pragma unroll
      for (int j = 0; j < C::PPT; ++j) {
        const int q = slot_of<C>(t, j);
        if (q < 0) continue;
        const int s2 = q % C::NS, s1 = q / C::NS;
        const T* rrow = Rs + size_t(q) * C::KRP;
        for (int el = c0 + grp; el < c0 + ncc; el += C::GRP) {
          const T* gcell = Gs + size_t(el) * C::NB * C::KRP * C::GW;
          T* cb = buf + size_t(el - c0) * C::NN;
          const T v = contract(gcell, el, j, rrow, q);  // one value on the d diagonal positions
#pragma unroll
          for (int c = 0; c < D; ++c) cb[(c * C::NS + s1) * C::N + c * C::NS + s2] = v;
        }
      }
      fence_async_smem();
      __syncthreads();
      if (t == 0) {
        bulk_s2g(static_cast<T*>(p.out) + (e0 + c0) * C::NN, buf, unsigned(ncc * C::NN * sizeof(T)));
        bulk_commit();
      }
      ++*staged_chunks;
    }
  } else {
#pragma unroll
    for (int j = 0; j < C::PPT; ++j) {
      const int q = slot_of<C>(t, j);
      if (q < 0) continue;
      int s1, s2, c2 = 0;
      if constexpr (DIAG) {
        s1 = q / C::NS;
        s2 = q % C::NS;
      } else {
        s2 = q % C::NS;
        c2 = (q / C::NS) % D;
        s1 = q / (C::NS * D);
      }
      const T* rrow = Rs + size_t(s1 * C::NS + s2) * C::KRP;
      // positions of the slot's entries: all d*d blocks (c1, c2) of the pair (convection),
      // or the d entries ((c1,s1),(c2,s2)) of the row slot (elasticity)
      int pos[NPOS];
      bool live_pos[NPOS];  // assembly: structural zeros add nothing
#pragma unroll
      for (int m = 0; m < NPOS; ++m) {
        const int c1 = DIAG ? m / D : m;
        const int cc2 = DIAG ? m % D : c2;
        pos[m] = (c1 * C::NS + s1) * C::N + cc2 * C::NS + s2;
        live_pos[m] = !DIAG || c1 == cc2;
      }
      // assembly: the slots of the next cell are loaded while this cell's atomics issue
      int sl_next[ASSEMBLE ? NPOS : 1];
      if constexpr (ASSEMBLE) {
#pragma unroll
        for (int m = 0; m < NPOS; ++m)
          sl_next[m] = (grp < nc && live_pos[m]) ? __ldg(p.slot + (e0 + grp) * C::NN + pos[m]) : -1;
      }
#pragma unroll 1
      for (int el = grp; el < nc; el += C::GRP) {
        const long long e = e0 + el;
        int sl[ASSEMBLE ? NPOS : 1];
        if constexpr (ASSEMBLE) {
          const int en = el + C::GRP;
#pragma unroll
          for (int m = 0; m < NPOS; ++m) {
            sl[m] = sl_next[m];
            sl_next[m] = (en < nc && live_pos[m]) ? __ldg(p.slot + (e0 + en) * C::NN + pos[m]) : -1;
          }
        }
        const T* gcell = Gs + size_t(el) * C::NB * C::KRP * C::GW;
        T vdiag = T(0);
        if constexpr (DIAG) vdiag = contract(gcell, el, j, rrow, s1 * C::NS + s2);
#pragma unroll
        for (int m = 0; m < NPOS; ++m) {
          if (ASSEMBLE && !live_pos[m]) continue;
          const T v = DIAG ? (live_pos[m] ? vdiag : T(0))
                           : contract(gcell + (m * D + c2) * C::KRP * C::GW, el, j, rrow, s1 * C::NS + s2);
          if constexpr (ASSEMBLE) {
            const int sv = sl[m];
            if (sv >= 0 && sv < p.nnz) atomicAdd(p.csr_val + sv, double(v));
            else atomicOr(p.status, FFC_FLAG_BOUNDS);
          } else {
            __stcs(static_cast<T*>(p.out) + e * C::NN + pos[m], v);
          }
        }
      }
    }
  }
  __syncthreads();
}

template <int D, int FORM, int Q, typename T, bool ASSEMBLE>
__global__ void __launch_bounds__(BlockCfg<D, FORM, Q, T>::NT, BlockCfg<D, FORM, Q, T>::MIN_BLOCKS)
    simt_block_kernel(SimtParams p) {
  using C = BlockCfg<D, FORM, Q, T>;
  using SG = BlockStaging<C, T, ASSEMBLE>;
  extern __shared__ __align__(16) unsigned char smem[];
  BlockRows<C, T> rows;
  block_rows_init<C, D, FORM, T>(p.a0, rows, smem);
  if constexpr (SG::ON) {  // the zero blocks of both staging buffers, written once
    T* stage = reinterpret_cast<T*>(smem + C::SMEM);
    for (size_t k = threadIdx.x; k < SG::BYTES / sizeof(T); k += C::NT) stage[k] = T(0);
  }
  int staged_chunks = 0;
  const long long n_tiles = (p.n_elem + C::E - 1) / C::E;
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x)
    block_tile<C, D, FORM, Q, T, ASSEMBLE>(p, tile, smem, rows, &staged_chunks);
  if constexpr (SG::ON) {
    if (threadIdx.x == 0) bulk_wait_all();  // shared memory stays valid until the copies are done
  }
}

}  // namespace ffc
