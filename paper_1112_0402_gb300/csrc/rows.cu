// Row-owner assembly: Algorithm 2 (Section 2.2) with its loops ordered by global row.
//
// Algorithm 2 adds each element tensor into the global matrix, A[iota(i1), iota(i2)] +=
// A^K[i1][i2]; done cell by cell on a GPU, every addition is a global FP64 atomic and the
// matrix must be zeroed first. Here the same sums are taken row by row instead: the
// entries of global row r receive exactly the rows A^K[i1][:] of the cells K that hold r
// as local dof i1 (the "pairs" (K, i1) of row r). The rows are cut into chunks of
// consecutive rows (at most 4096 values and 320 pairs each); a CTA sums one chunk at a
// time in shared memory, computing every element-tensor entry on the fly from a per-cell
// geometry tensor G_K (A^K[i1][i2] = sum_alpha A0[i1][i2][alpha] G_K[alpha], Section
// 3.2), and then writes the chunk's CSR values once, in order: no global atomics, no
// zeroing pass, every value written exactly once.
//
// Work layout inside a chunk. The plan stores each chunk's pairs grouped by local index
// i1 (a "class"; within a class the pairs of different rows alternate), the class runs, the
// run in which each of 32 equal shares of the pairs begins, and per pair the chunk-relative
// positions of its columns i2 = 0..n-1. Every warp sums one share: the reference-tensor
// entries A0[i1][i2][.] its lanes need stay in registers for a class run, each pair's G_K is
// a shared-memory broadcast, and one warp instruction adds the contributions of one
// element-tensor row (or of a few rows of different global rows), whose positions are
// distinct: the shared-memory atomics meet no same-address conflicts and few bank conflicts.
// For n >= 32 lane l takes column l of every pair (and the columns beyond 32 are packed over
// the lanes of separate steps); for n < 32 a warp takes 32 / n pairs side by side. Later
// chunks' plan data and geometry tensors are staged in shared memory with cp.async while the
// current chunk is summed and the previous one written out.
//
// What bounds it: the L1 / shared-memory data pipe (71% busy for P4: bank conflicts of the
// atomics, 2.7 cycles each, plan copies, write-out) and instruction issue (65%). Measured,
// a queue of warp tasks with in-loop bounds and 64-bit conversions -> equal shares: mass +
// Poisson pair, P3 on 215,622 tets 496 -> 354 us, P4 on 663,552 tets 3493 -> 2953 us (0.43
// of HBM on 8.68 GB), P2 on 384,000 tets 347 -> 252 us, P4 on 180,000 triangles 564 -> 184 us.
//
// Fixed-point accumulation. The sums are kept in fixed point with one unit per chunk and
// form, where 2^(eb-1) bounds every partial sum of every entry of the chunk (the largest
// |contribution| bound of a pair, a0max[i1] * sum|G_K|, times the largest number of pairs
// of one row). An FP32 contribution x is one 31-bit digit, x 2^(31-eb) rounded to the
// nearest integer (u = 2^(eb-31)): the scaling is exact and the sums stay within 2^30 u,
// so one 32-bit shared-memory atomic per contribution adds it, whatever the number of
// contributions. An FP64 contribution is split into three signed 21-bit digits on the
// grids 2^(eb-20), 2^(eb-41), 2^(eb-62) (u = 2^(eb-62)), each added with a 32-bit atomic
// into its own array (a digit sum of up to 1023 contributions cannot overflow 32 bits):
// 32-bit shared atomics run about seven times faster than 64-bit ones on this GPU.
// Chunks whose bound lies outside the range of the FP32 scale, and FP64 contributions,
// take an integer conversion instead (truncation, error < u). The value of an entry is
// the digit sums' value in units u, rounded once to FP64 in integer arithmetic. Integer
// addition is exact and associative, so the result does not depend on the order of the additions:
// per entry |result - exact sum of the contributions| <= m u / 2 + an ulp of the result
// (m contributions; u / 2 < 2^-30 B for FP32, 2^-61 B for FP64, B the chunk's bound), and
// the matrix is reproducible bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "ffc_internal.h"
#include "geometry.cuh"

namespace ffc {
namespace {

constexpr int ROWS_VMAX = 4096;           // values of one chunk (shared-memory accumulators)
constexpr int ROWS_VSTRIDE = ROWS_VMAX + 4;  // ints of one digit array: a chunk's values, shifted by 0 or 1
constexpr int ROWS_PMAX = 320;            // pairs of one chunk (a multiple of 32)
constexpr int ROWS_MAX_INCIDENCE = 1023;  // digit sums of 21-bit digits stay within 32 bits
constexpr int ROWS_MAX_LOCAL = 64;        // local dofs per cell the plan carries
constexpr int ROWS_GEOM = 8;              // doubles of geometry scratch per cell (RowsGeo::GS, FP64)

constexpr int ROWS_WARPS = 32;            // equal shares of a chunk's pairs the plan prepares

// Class runs of a chunk of P pairs: at most one per local index i1.
__host__ __device__ constexpr int region_runs(int n, long long P) { return int(n < P ? n : P); }

// A chunk's region of plan data (16-byte aligned, a multiple of 16 bytes):
//   uint8  first[ROWS_WARPS]  the run that holds pair P w / ROWS_WARPS, the first of share w
//   uint32 run[region_runs]   i1 | k0 << 7 | k1 << 19: pairs [k0, k1) are class i1, in order
//   int32  pr[P]              the pairs e * n + i1, grouped by class
//   uint16 pos[P][n]          chunk-relative value index of column i2 of each pair
__host__ __device__ constexpr long long region_pr_offset(int n, long long P) {
  return ROWS_WARPS + 4ll * region_runs(n, P);
}
__host__ __device__ constexpr long long region_bytes(int n, long long P) {
  return (region_pr_offset(n, P) + 4 * P + 2 * P * n + 15) / 16 * 16;
}

}  // namespace
}  // namespace ffc

struct ffc_row_plan {
  int device = 0;
  int64_t n_elem = 0;
  int n_local = 0;
  int64_t n_dof = 0;
  int64_t nnz = 0;
  int max_row = 0;
  int max_incidence = 0;
  int vmax = 0;                     // values of the largest chunk
  int max_pairs = 0;                // pairs of the largest chunk
  int max_region = 0;               // bytes of the largest chunk region
  int64_t n_chunks = 0;
  int64_t region_total = 0;         // bytes of all regions
  int64_t* row_ptr = nullptr;       // [n_dof + 1] copy of the pattern's row offsets
  int32_t* chunk_row = nullptr;     // [n_chunks + 1] first row of each chunk
  int32_t* chunk_pair = nullptr;    // [n_chunks + 1] first pair of each chunk (row order)
  int64_t* chunk_off = nullptr;     // [n_chunks + 1] byte offset of each chunk's region
  int64_t* chunk_val = nullptr;     // [n_chunks + 1] first CSR value of each chunk
  int32_t* chunk_inc = nullptr;     // [n_chunks] most pairs of one row in the chunk
  unsigned char* region = nullptr;  // [region_total] chunk regions (see region_bytes)
  void* geom = nullptr;             // per-cell geometry scratch, [n_elem][ROWS_GEOM] doubles
  int2* chunk_eb = nullptr;         // [n_chunks] scratch: the chunk's bound exponents (two forms)
};

namespace ffc {
namespace {

constexpr unsigned PLAN_BAD_DOF = 1u, PLAN_MISSING = 2u, PLAN_BAD_ROW_PTR = 8u;

int cuda_fail(cudaError_t e, const char* what) {
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? FFC_ENOMEM : FFC_ECUDA;
}

// ---------------------------------------------------------------- plan construction

__global__ void plan_count(const int32_t* __restrict__ dofmap, long long total, long long n_dof,
                           int32_t* __restrict__ cnt, unsigned* err) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int r = dofmap[t];
    if (r < 0 || r >= n_dof) {
      atomicOr(err, PLAN_BAD_DOF);
      continue;
    }
    atomicAdd(cnt + r, 1);
  }
}

constexpr int SCAN_T = 1024, SCAN_V = 4, SCAN_CHUNK = SCAN_T * SCAN_V;

// Exclusive scan of one value per thread over a block of SCAN_T threads; `total` gets
// the block's sum. Uses `tot` (32 ints of shared memory); ends with a barrier.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t s, int32_t* tot, int32_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) tot[w] = x;
  __syncthreads();
  if (w == 0) {
    int32_t t = tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    tot[lane] = t;
  }
  __syncthreads();
  const int32_t ex = x - s + (w > 0 ? tot[w - 1] : 0);
  total = tot[31];
  __syncthreads();
  return ex;
}

// exclusive scan of a[0, n) in chunks of SCAN_CHUNK, each chunk's total to sums[chunk]
__global__ void __launch_bounds__(SCAN_T) scan_chunks(int32_t* __restrict__ a, long long n,
                                                      int32_t* __restrict__ sums) {
  __shared__ int32_t tot[32];
  const long long base = blockIdx.x * (long long)SCAN_CHUNK + threadIdx.x * SCAN_V;
  int32_t v[SCAN_V], s = 0;
#pragma unroll
  for (int j = 0; j < SCAN_V; ++j) {
    v[j] = base + j < n ? a[base + j] : 0;
    s += v[j];
  }
  int32_t total;
  int32_t ex = block_exclusive_scan(s, tot, total);
#pragma unroll
  for (int j = 0; j < SCAN_V; ++j) {
    if (base + j < n) a[base + j] = ex;
    ex += v[j];
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// exclusive scan of the chunk totals in place (one block, sequential over SCAN_T pieces)
__global__ void __launch_bounds__(SCAN_T) scan_sums(int32_t* __restrict__ sums, int nb) {
  __shared__ int32_t tot[32];
  int32_t carry = 0;
  for (int b0 = 0; b0 < nb; b0 += SCAN_T) {
    const int i = b0 + threadIdx.x;
    const int32_t s = i < nb ? sums[i] : 0;
    int32_t total;
    const int32_t ex = block_exclusive_scan(s, tot, total);
    if (i < nb) sums[i] = carry + ex;
    carry += total;
  }
}

__global__ void __launch_bounds__(SCAN_T) scan_add(int32_t* __restrict__ a, long long n,
                                                   const int32_t* __restrict__ sums) {
  const long long base = blockIdx.x * (long long)SCAN_CHUNK;
  const int32_t off = sums[blockIdx.x];
  for (int j = threadIdx.x; j < SCAN_CHUNK; j += SCAN_T)
    if (base + j < n) a[base + j] += off;
}

// the pairs (e, i1) of each row, grouped by row (order within a row: arbitrary)
__global__ void plan_fill(const int32_t* __restrict__ dofmap, long long total, long long n_dof,
                          const int32_t* __restrict__ inc_ptr, int32_t* __restrict__ fill,
                          int32_t* __restrict__ inc_tmp) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int r = dofmap[t];
    if (r < 0 || r >= n_dof) continue;
    const int j = atomicAdd(fill + r, 1);
    inc_tmp[inc_ptr[r] + j] = int32_t(t);
  }
}

// One thread per chunk: the chunk's pairs grouped by class i1; within a class ordered by
// (rank of the pair among the class's pairs of its row, row, cell), so consecutive pairs
// of a class belong to different rows where the class has several. Writes the ordered
// pairs, the class runs and the first run of each share into the chunk's region. `key` is
// scratch [total].
__global__ void plan_sort(const int32_t* __restrict__ dofmap, const int32_t* __restrict__ chunk_row,
                          const int32_t* __restrict__ chunk_pair, const int64_t* __restrict__ chunk_off,
                          long long n_chunks, int n, const int32_t* __restrict__ inc_tmp,
                          unsigned long long* __restrict__ key, unsigned char* __restrict__ region) {
  constexpr unsigned long long E_MASK = (1ull << 30) - 1;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_chunks;
       c += (long long)gridDim.x * blockDim.x) {
    const int r0 = chunk_row[c];
    const int p0 = chunk_pair[c], P = chunk_pair[c + 1] - p0;
    unsigned char* reg = region + chunk_off[c];
    uint32_t* run_of = reinterpret_cast<uint32_t*>(reg + ROWS_WARPS);
    int32_t* pr = reinterpret_cast<int32_t*>(reg + region_pr_offset(n, P));
    unsigned long long* kk = key + p0;
    // key (i1, row - r0, e) of each pair (i1 < 64, row - r0 < 2^16, e < 2^30), by insertion
    for (int j = 0; j < P; ++j) {
      const int t = inc_tmp[p0 + j];
      const unsigned long long kv = (static_cast<unsigned long long>(t % n) << 58) |
                                    (static_cast<unsigned long long>(dofmap[t] - r0) << 30) |
                                    static_cast<unsigned long long>(t / n);
      int q = j;
      while (q > 0 && kk[q - 1] > kv) {
        kk[q] = kk[q - 1];
        --q;
      }
      kk[q] = kv;
    }
    // each class: its pairs (the pairs of a row get ranks 0, 1, ..., emitted by (rank,
    // row, e)) and its run
    int a = 0, n_runs = 0, share = 0;
    for (int i = 0; i < n; ++i) {
      int b = a;
      while (b < P && int(kk[b] >> 58) == i) ++b;
      int out = a;
      for (int rank = 0; out < b; ++rank) {
        int rr = -1, run = 0;
        for (int j = a; j < b; ++j) {
          const int row = int((kk[j] >> 30) & 0xFFFFull);
          run = (row == rr) ? run + 1 : 0;
          rr = row;
          if (run == rank) pr[out++] = int32_t((kk[j] & E_MASK) * n + i);
        }
      }
      if (b > a) {
        for (; share < ROWS_WARPS && P * share / ROWS_WARPS < b; ++share) reg[share] = (unsigned char)n_runs;
        run_of[n_runs++] = uint32_t(i) | (uint32_t(a) << 7) | (uint32_t(b) << 19);
      }
      a = b;
    }
  }
}

// One CTA per chunk: the chunk-relative position of every contribution (pair k, column
// i2): binary search of column dofmap[e][i2] in the sorted columns of row dofmap[e][i1].
__global__ void plan_positions(const int32_t* __restrict__ dofmap, int n, const int64_t* __restrict__ row_ptr,
                               const int32_t* __restrict__ col, const int32_t* __restrict__ chunk_row,
                               const int32_t* __restrict__ chunk_pair, const int64_t* __restrict__ chunk_off,
                               long long n_chunks, unsigned char* __restrict__ region, unsigned* err) {
  for (long long c = blockIdx.x; c < n_chunks; c += gridDim.x) {
    const int r0 = chunk_row[c], r1 = chunk_row[c + 1];
    const int P = chunk_pair[c + 1] - chunk_pair[c];
    const long long base = row_ptr[r0];
    unsigned char* reg = region + chunk_off[c];
    const int32_t* pr = reinterpret_cast<const int32_t*>(reg + region_pr_offset(n, P));
    uint16_t* pos = reinterpret_cast<uint16_t*>(reg + region_pr_offset(n, P) + 4ll * P);
    for (int w = threadIdx.x; w < P * n; w += blockDim.x) {
      const int k = w / n, i2 = w - k * n;
      const int t = pr[k];
      const int e = t / n, i1 = t - e * n;
      const int r = dofmap[(long long)e * n + i1];
      const int cj = dofmap[(long long)e * n + i2];
      uint16_t q = 0;
      if (r < r0 || r >= r1) {
        atomicOr(err, PLAN_MISSING);
      } else {
        long long lo = row_ptr[r], hi = row_ptr[r + 1];
        const long long end = hi;
        while (lo < hi) {
          const long long mid = (lo + hi) >> 1;
          if (col[mid] < cj) lo = mid + 1;
          else hi = mid;
        }
        if (lo < end && col[lo] == cj) q = uint16_t(lo - base);
        else atomicOr(err, PLAN_MISSING);
      }
      pos[w] = q;
    }
  }
}

// ---------------------------------------------------------------- fixed point

// smallest eb with 2^(eb-1) >= b for a bound b >= 0 (zero and denormal bounds give the
// smallest exponent of the type)
__device__ __forceinline__ int bound_exponent(float b) { return int((__float_as_uint(b) >> 23) & 0xffu) - 125; }
__device__ __forceinline__ int bound_exponent(double b) {
  return int((static_cast<unsigned long long>(__double_as_longlong(b)) >> 52) & 0x7ffull) - 1021;
}

// x / 2^ulog truncated toward zero, for |x| / 2^ulog < 2^62 (integer arithmetic only)
__device__ __forceinline__ long long to_fixed(float x, int ulog) {
  const unsigned b = __float_as_uint(x);
  const int ex = int((b >> 23) & 0xffu);
  unsigned m = b & 0x7fffffu;
  int ee = 1;
  if (ex) {
    m |= 0x800000u;
    ee = ex;
  }
  const int sh = ee - 150 - ulog;  // x = m 2^(ee - 150)
  unsigned long long f;
  if (sh >= 0) f = static_cast<unsigned long long>(m) << (sh < 63 ? sh : 63);
  else f = -sh < 32 ? static_cast<unsigned long long>(m >> -sh) : 0ull;
  return (b >> 31) ? -static_cast<long long>(f) : static_cast<long long>(f);
}

__device__ __forceinline__ long long to_fixed(double x, int ulog) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ex = int((b >> 52) & 0x7ffull);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  int ee = 1;
  if (ex) {
    m |= 1ull << 52;
    ee = ex;
  }
  const int sh = ee - 1075 - ulog;  // x = m 2^(ee - 1075)
  unsigned long long f;
  if (sh >= 0) f = m << (sh < 63 ? sh : 63);
  else f = -sh < 64 ? (m >> -sh) : 0ull;
  return (b >> 63) ? -static_cast<long long>(f) : static_cast<long long>(f);
}

__device__ __noinline__ double scaled_to_double(long long v, int ulog) { return scalbn(static_cast<double>(v), ulog); }

// v * 2^ulog rounded to the nearest double (ties to even), in integer arithmetic (the
// hardware int64 -> FP64 conversion runs on GB300's narrow FP64 pipe): the magnitude is
// normalised to a leading one at bit 63, its top 53 bits are added to (exponent - 1) << 52
// (the leading one completes the exponent field, and a carry out of the significand on
// rounding moves the value to the next binade by itself). Zero is a select; results
// outside the normal range (bounds far from 1) take a called slow path, so the common
// path never issues FP64 instructions.
__device__ __forceinline__ double fixed_to_double(long long v, int ulog) {
  const unsigned long long sign = static_cast<unsigned long long>(v) & (1ull << 63);
  unsigned long long m = sign ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
  const int lz = __clzll(static_cast<long long>(m));
  m <<= (lz & 63);
  const int e = 63 - lz + ulog + 1023;
  const unsigned long long sig = m >> 11, rb = m & 0x7ffull;
  const unsigned long long up = (rb > 0x400ull) | ((rb == 0x400ull) & sig & 1ull);
  unsigned long long bits = sign | ((static_cast<unsigned long long>(e - 1) << 52) + sig + up);
  if (m == 0) bits = sign;
  if (m != 0 && (e <= 0 || e >= 2047)) return scaled_to_double(v, ulog);
  return __longlong_as_double(static_cast<long long>(bits));
}

// v * 2^ulog for |v| < 2^53, which a double holds exactly: the magnitude's leading one is
// placed at bit 52 and (exponent - 1) << 52 added (the leading one completes the exponent
// field); no rounding step. Zero is a select; results outside the normal range take the
// called slow path.
__device__ __forceinline__ double fixed_to_double_exact(long long v, int ulog) {
  const unsigned long long sign = static_cast<unsigned long long>(v) & (1ull << 63);
  unsigned long long m = sign ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
  const int lz = __clzll(static_cast<long long>(m));  // >= 11
  const int e = 63 - lz + ulog + 1023;
  m <<= ((lz - 11) & 63);
  unsigned long long bits = sign | ((static_cast<unsigned long long>(e - 1) << 52) + m);
  if (m == 0) bits = sign;
  if (m != 0 && (e <= 0 || e >= 2047)) return scaled_to_double(v, ulog);
  return __longlong_as_double(static_cast<long long>(bits));
}

// Digits of the fixed-point sums: one 31-bit digit for FP32 contributions, three 21-bit
// digits (63 bits) for FP64 ones.
template <typename T>
__host__ __device__ constexpr int rows_ndig() { return sizeof(T) == 4 ? 1 : 3; }

// The digits of one contribution for |x| <= 2^(eb-1): NDIG = 3 on the grids 2^(eb-20),
// 2^(eb-41), 2^(eb-62) (unit u = 2^(eb-62)); NDIG = 1 one digit on the grid 2^(eb-31)
// (u = 2^(eb-31): a chunk's sums stay within 2^30 u, so one 32-bit integer holds them
// whatever the number of contributions). `magic`: the FP32 scale 2^(31 - eb) is a normal
// float; otherwise the integer conversion.
template <int NDIG>
struct Digits {
  static_assert(NDIG == 1 || NDIG == 3, "31 bits for FP32, 63 for FP64");
  float scale;
  int ulog;
  bool magic;
  __device__ __forceinline__ void init(int eb) {
    magic = NDIG == 1 && eb >= -96 && eb <= 157;
    scale = __int_as_float((31 - (magic ? eb : 0) + 127) << 23);
    ulog = eb - (NDIG == 1 ? 31 : 62);
  }
  // MAGIC: x 2^(31 - eb) rounded to the nearest integer (the scaling is exact; valid when
  // `magic`); |x| <= 2^(eb-1) keeps it within 2^30. Otherwise the integer conversion
  template <bool MAGIC>
  __device__ __forceinline__ void split(float x, int (&d)[NDIG]) const {
    if constexpr (MAGIC) d[0] = __float2int_rn(x * scale);
    else d[0] = int(to_fixed(x, ulog));
  }
  template <bool MAGIC>
  __device__ __forceinline__ void split(double x, int (&d)[NDIG]) const {
    const long long f = to_fixed(x, ulog);
    d[2] = int(f & 0x1FFFFFll);
    d[1] = int((f >> 21) & 0x1FFFFFll);
    d[0] = int(f >> 42);
  }
  // whether every nonzero one-digit result stays normal
  __device__ __forceinline__ bool stays_normal() const { return ulog >= -1022 && ulog <= 980; }
  // a one-digit sum s * 2^ulog whose result stays normal, in 32-bit integer instructions: the
  // magnitude is normalised to a leading one at bit 31, which completes the exponent field;
  // exact, zero is a select
  __device__ __forceinline__ double value_int(int s) const {
    const unsigned m = unsigned(abs(s));
    unsigned sh;  // leading zeros; 2^32 - 1 for zero, whose shift gives zero
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(sh) : "r"(m));
    unsigned n;
    asm("shl.b32 %0, %1, %2;" : "=r"(n) : "r"(m), "r"(sh));
    const unsigned hi = (n >> 11) + (unsigned(1053 + ulog) << 20) - (sh << 20);
    return __hiloint2double(s == 0 ? 0 : int(hi | (unsigned(s) & 0x80000000u)), int(n << 21));
  }
  // the entry's value from its digit sums, rounded once to FP64
  __device__ __forceinline__ double value(const int (&s)[NDIG]) const {
    if constexpr (NDIG == 1) {  // |v| < 2^31: exact in a double
      return fixed_to_double_exact(static_cast<long long>(s[0]), ulog);
    } else {
      const long long v =
          static_cast<long long>(s[0]) * (1ll << 42) + static_cast<long long>(s[1]) * (1ll << 21) + s[2];
      return fixed_to_double(v, ulog);
    }
  }
};

// ---------------------------------------------------------------- geometry

// The three launches of a call are a chain (geometry, bounds, rows); each kernel lets the next
// one be placed while it runs and waits for the one before where it first needs its results,
// which takes the launch gaps out of small calls.
__device__ __forceinline__ void grid_let_next() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void grid_wait_before() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Form codes of the row kernels: FFC_MASS, FFC_POISSON, or the (mass, Poisson) pair.
constexpr int ROWS_PAIR = FFC_PAIR_MASS_POISSON;

template <int D, int FORM>
struct RowsGeo {
  static constexpr int NF = FORM == ROWS_PAIR ? 2 : 1;        // matrices
  static constexpr int NP = D * (D + 1) / 2;                  // symmetric Poisson G_K entries
  // stored per cell: mass [|det|, |det|]; Poisson [G (NP), pad, sum|G| in slot 7]; pair [G (NP),
  // pad, |det| in slot 6, sum|G| in slot 7]
  static constexpr int GS = FORM == FFC_MASS ? 2 : 8;
  static_assert(GS <= ROWS_GEOM, "the plan's scratch");
  static constexpr int DET = FORM == ROWS_PAIR ? 6 : 0;
  // G_K slots of the contribution bounds' sums: |G| of a single form, and for the pair the
  // mass's |det J| and the Poisson sum|G|, side by side for one load
  static constexpr int SUM_A = FORM == ROWS_PAIR ? DET : (FORM == FFC_POISSON ? 7 : 1);
};

// One thread per cell: G_K exactly as the fused CUDA-core element-tensor kernels form it
// (FP32: mass |det J| from the FP64 determinant; Poisson the FP64 adjugate and
// determinant, K and the symmetric G in FP32; FP64: everything in FP64), and the sums
// of |G_K| for the bounds.
template <int D, int FORM, typename T>
__global__ void __launch_bounds__(256) rows_geometry(const int32_t* __restrict__ cells,
                                                     const double* __restrict__ vertices, long long n_vert,
                                                     long long n_elem, T* __restrict__ G, unsigned* status) {
  using C = RowsGeo<D, FORM>;
  grid_let_next();
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n_elem;
       e += (long long)gridDim.x * blockDim.x) {
    T g[C::GS];
#pragma unroll
    for (int a = 0; a < C::GS; ++a) g[a] = T(0);
    bool degenerate = false, bad_index = false;
    if constexpr (FORM == FFC_MASS) {
      double det;
      cell_det<D>(cells, vertices, n_vert, e, det, degenerate, bad_index);
      g[0] = T(det);
      g[1] = fabs(g[0]);
    }
    if constexpr (FORM == FFC_POISSON || FORM == ROWS_PAIR) {
      bool dg, bi;
      if constexpr (sizeof(T) == 4) {
        float K[D][D], det;
        cell_geometry_f32<D>(cells, vertices, n_vert, e, K, det, dg, bi);
        if constexpr (FORM == ROWS_PAIR) g[C::DET] = det;  // the mass's |det J|, as cell_det rounds it
        geometry_tensor_f32<D, FFC_POISSON, 1, true>(K, det, nullptr, 0.0, 0.0, reinterpret_cast<float*>(g));
      } else {
        double K[D][D], det;
        cell_geometry<D>(cells, vertices, n_vert, e, K, det, dg, bi);
        geometry_tensor_k<D, FFC_POISSON, 1>(K, det, nullptr, 0.0, 0.0, [&](int a, double v) { g[a] = T(v); });
      }
      T s = T(0);
#pragma unroll
      for (int a = 0; a < C::NP; ++a) s += fabs(g[a]);
      g[7] = s;
      degenerate |= dg;
      bad_index |= bi;
    }
    T* dst = G + e * C::GS;
#pragma unroll
    for (int a = 0; a < C::GS; ++a) dst[a] = g[a];
    if (degenerate) atomicOr(status, FFC_FLAG_DEGENERATE);
    if (bad_index) atomicOr(status, FFC_FLAG_BOUNDS);
  }
}

// ---------------------------------------------------------------- assembly

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Reference tensors in T, and the largest |A0| entry of each row i1 (the bounds' factor).
struct RowsTensors {
  const void* a;  // mass or single form (layouts: load_a0)
  const void* b;  // pair: Poisson
  const void* max_a;
  const void* max_b;
};

struct RowsParams {
  const int64_t* chunk_off;
  const int32_t* chunk_pair;
  const int64_t* chunk_val;
  const int32_t* chunk_inc;
  int2* chunk_eb;  // bound exponents of the chunk's forms (ROWS_NO_BOUND: not finite)
  const unsigned char* region;
  const void* G;
  RowsTensors a0;
  double* out_a;
  double* out_b;
  long long n_chunks;
  int meta_off;  // byte offset of the chunk-extent ring in shared memory
  int pmax;   // pairs of the largest chunk
  int rmax;   // bytes of the largest chunk region
  unsigned* status;
};

template <int D, int FORM, int Q>
struct RowsCfg {
  static constexpr int N = nscalar(D, Q);
  static constexpr bool MAIN = N >= 32;          // lane l takes column l of every pair
  static constexpr int W = MAIN ? N - 32 : 0;    // columns beyond the first 32, spread over the lanes
  static constexpr int PP = MAIN ? 1 : 32 / N;   // pairs a warp takes side by side, N lanes each
  static constexpr int TP = W > 0 ? 32 / W : 1;  // pairs of a column tail's step
  static constexpr int NP = D * (D + 1) / 2;
  static constexpr int NA = FORM == ROWS_PAIR ? 1 + NP : (FORM == FFC_POISSON ? NP : 1);  // A0 values per entry
  static constexpr int NG = FORM == FFC_MASS ? 1 : 8;  // G_K values read per pair (vector loads)
};

// A0 entry (i1, i2) of the kernel's form(s), in the order the contraction uses: mass and FP64
// from the [i1][alpha][i2] copies (lanes of consecutive i2 read consecutive words), FP32
// Poisson from the padded rows [i1][i2][alpha], in two vector loads instead of six
template <int FORM, int N, int NA, int NP, typename T>
__device__ __forceinline__ void load_a0(const T* __restrict__ A0a, const T* __restrict__ A0b, int i1, int i2,
                                        T (&a)[NA]) {
  if constexpr (FORM == FFC_MASS) {
    a[0] = __ldg(A0a + i1 * N + i2);
  } else {
    constexpr int o = FORM == ROWS_PAIR ? 1 : 0;
    if constexpr (o) a[0] = __ldg(A0a + i1 * N + i2);
    const T* A0p = o ? A0b : A0a;
    if constexpr (sizeof(T) == 4) {  // [i1][i2][NP padded to 16 bytes]
      const float4* r = reinterpret_cast<const float4*>(A0p) + (i1 * N + i2) * ((NP + 3) / 4);
      const float4 x = __ldg(r);
      a[o] = x.x, a[o + 1] = x.y, a[o + 2] = x.z;
      if constexpr (NP > 3) {
        const float2 y = __ldg(reinterpret_cast<const float2*>(r + 1));
        a[o + 3] = x.w, a[o + 4] = y.x, a[o + 5] = y.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NP; ++j) a[o + j] = __ldg(A0p + (i1 * NP + j) * N + i2);
    }
  }
}

// the first NG values of a pair's G_K from shared memory (16-byte aligned rows for NG = 8)
template <int NG, typename T>
__device__ __forceinline__ void load_gk(const T* gs, T (&g)[NG]) {
  if constexpr (NG == 1) {
    g[0] = gs[0];
  } else if constexpr (sizeof(T) == 4) {
    const float4 x = reinterpret_cast<const float4*>(gs)[0], y = reinterpret_cast<const float4*>(gs)[1];
    g[0] = x.x, g[1] = x.y, g[2] = x.z, g[3] = x.w, g[4] = y.x, g[5] = y.y, g[6] = y.z, g[7] = y.w;
  } else {
#pragma unroll
    for (int j = 0; j < NG / 2; ++j) {
      const double2 x = reinterpret_cast<const double2*>(gs)[j];
      g[2 * j] = x.x;
      g[2 * j + 1] = x.y;
    }
  }
}

// the contributions of one element-tensor entry: sum_alpha G_K[alpha] A0[i1][i2][alpha]
// (FMA order as in the fused element-tensor kernels, so FP32 values agree bit for bit)
template <int FORM, int NA, int NG, int NF, typename T>
__device__ __forceinline__ void contract(const T (&g)[NG], const T (&a)[NA], T (&v)[NF]) {
  if constexpr (FORM == ROWS_PAIR) {
    v[0] = fma(g[6], a[0], T(0));  // |det J| sits in slot 6
    T s = T(0);
#pragma unroll
    for (int j = 1; j < NA; ++j) s = fma(g[j - 1], a[j], s);
    v[1] = s;
  } else {
    T s = T(0);
#pragma unroll
    for (int j = 0; j < NA; ++j) s = fma(g[j], a[j], s);
    v[0] = s;
  }
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Adds one entry's contributions (digits) at chunk position q; base[f] is form f's first
// digit array (the arrays of one form ROWS_VSTRIDE ints apart).
template <bool MAGIC, int NF, int NDIG, typename T>
__device__ __forceinline__ void add_digits(int* const (&base)[NF], const Digits<NDIG> (&dig)[NF], const T (&v)[NF],
                                           int q) {
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    int d[NDIG];
    dig[f].template split<MAGIC>(v[f], d);
    int* a = base[f] + q;
#pragma unroll
    for (int j = 0; j < NDIG; ++j) atomicAdd(a + j * ROWS_VSTRIDE, d[j]);
  }
}

// Positions come from a validated plan (every (row, col) pair was found in the pattern when
// the plan was built, so q < V); the mask only keeps a shared-memory index in range.
__device__ __forceinline__ int rows_pos(int q) { return q & (ROWS_VMAX - 1); }

// Pairs [k0, k1) of class i1 of a chunk, by one warp: for n >= 32 lane l takes column l of
// every pair, for n < 32 the warp takes 32 / n pairs side by side, n lanes each; the lane's
// A0 column stays in registers. (With the (pair, column) items packed over all 32 lanes
// each step divided by n and a lane held the A0 columns of lcm(32, n) / 32 steps: P4
// triangles 628 against 220 us on 180,000 cells.)
template <class K, int FORM, int NF, int GS, bool MAGIC, int NDIG, typename T>
__device__ __forceinline__ void run_pairs(int i1, int k0, int k1, const T* gs, const uint16_t* pos,
                                          int* const (&base)[NF], const Digits<NDIG> (&dig)[NF], const T* A0a,
                                          const T* A0b) {
  constexpr int N = K::N, NA = K::NA, NG = K::NG;
  const int lane = threadIdx.x & 31;
  const int sub = K::MAIN ? 0 : lane / N, i2 = K::MAIN ? lane : lane - sub * N;
  if (sub >= K::PP) return;
  T am[NA];
  load_a0<FORM, N, NA, K::NP, T>(A0a, A0b, i1, i2, am);
  const uint16_t* pl = pos + i2;
#pragma unroll 3
  for (int k = k0 + sub; k < k1; k += K::PP) {
    T g[NG];
    load_gk<NG, T>(gs + k * GS, g);
    const int q = rows_pos(pl[k * N]);
    T v[NF];
    contract<FORM, NA, NG, NF, T>(g, am, v);
    add_digits<MAGIC, NF, NDIG, T>(base, dig, v, q);
  }
}

// One warp's share [k0, k1) of a chunk's pairs: the class runs it meets, from run r on.
template <class K, int FORM, int NF, int GS, bool MAGIC, int NDIG, typename T>
__device__ __forceinline__ void share_task(int r, int k0, int k1, const unsigned* run, const int32_t* pr, const T* gs,
                                           const uint16_t* pos,
                                            int* const (&base)[NF], const Digits<NDIG> (&dig)[NF], const T* A0a,
                                           const T* A0b) {
  if constexpr (sizeof(T) == 8 && !K::MAIN && K::PP * K::N < 28) {
    // the FP64 pipe takes as long for 20 lanes as for 32 (P3 tetrahedra): the share's
    // (pair, column) items packed over all lanes, A0 from the L1 cache
    constexpr int N = K::N, NA = K::NA, NG = K::NG;
#pragma unroll 1
    for (int f = threadIdx.x & 31; f < (k1 - k0) * N; f += 32) {
      const int k = k0 + f / N, i2 = f % N;
      T a[NA], g[NG];
      load_a0<FORM, N, NA, K::NP, T>(A0a, A0b, pr[k] % N, i2, a);
      load_gk<NG, T>(gs + k * GS, g);
      const int q = rows_pos(pos[k * N + i2]);
      T v[NF];
      contract<FORM, NA, NG, NF, T>(g, a, v);
      add_digits<MAGIC, NF, NDIG, T>(base, dig, v, q);
    }
    return;
  }
  for (int k = k0; k < k1; ++r) {
    const unsigned ud = run[r];
    const int end = min(k1, int(ud >> 19));
    run_pairs<K, FORM, NF, GS, MAGIC, NDIG, T>(int(ud & 127u), k, end, gs, pos, base, dig, A0a, A0b);
    k = end;
  }
}

// The columns beyond the first 32 (n > 32) of pairs [step TP, (step + 1) TP) of a chunk,
// packed over the lanes, W to a pair.
template <class K, int FORM, int NF, int GS, bool MAGIC, int NDIG, typename T>
__device__ __forceinline__ void tail_step(int step, int P, const int32_t* pr, const T* gs, const uint16_t* pos,
                                          int* const (&base)[NF], const Digits<NDIG> (&dig)[NF], const T* A0a,
                                          const T* A0b) {
  constexpr int N = K::N, NA = K::NA, NG = K::NG, TP = K::TP;
  const int lane = threadIdx.x & 31, sub = lane / K::W, i2 = 32 + lane - sub * K::W;
  const int k = step * TP + sub;
  if (sub >= TP || k >= P) return;
  T a[NA], g[NG];
  load_a0<FORM, N, NA, K::NP, T>(A0a, A0b, pr[k] % N, i2, a);
  load_gk<NG, T>(gs + k * GS, g);
  const int q = rows_pos(pos[k * N + i2]);
  T v[NF];
  contract<FORM, NA, NG, NF, T>(g, a, v);
  add_digits<MAGIC, NF, NDIG, T>(base, dig, v, q);
}

// The bound exponents of every chunk, before the rows: a warp per chunk takes the largest
// contribution bound of its pairs (max|A0[i1][.][.]| sum|G_K|) times the most pairs of a row,
// and 2^(eb-1) is that or the next power of two. In rows_assemble one warp did this for a
// later chunk in every iteration and its chain of loads and shuffles was the iteration's
// shortest possible time (235 of 443 us for P4 pair rows of 82,944 tets with no other work);
// here all chunks run side by side.
constexpr int ROWS_NO_BOUND = INT_MAX;  // the bound is not finite

template <int D, int FORM, int Q, typename T>
__global__ void __launch_bounds__(256) rows_bounds(RowsParams p) {
  using C = RowsGeo<D, FORM>;
  using K = RowsCfg<D, FORM, Q>;
  constexpr int N = K::N, NF = C::NF;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const T big = sizeof(T) == 4 ? T(FLT_MAX) : T(DBL_MAX);
  const T* M[2] = {static_cast<const T*>(p.a0.max_a), static_cast<const T*>(p.a0.max_b)};
  grid_let_next();
  const T* G = static_cast<const T*>(p.G);
  bool waited = false;
  for (long long c = blockIdx.x * 8ll + w; c < p.n_chunks; c += gridDim.x * 8ll) {
    // the plan's part first, all of the lane's pairs at once: only the geometry has to wait
    const int P = p.chunk_pair[c + 1] - p.chunk_pair[c];
    const int32_t* pr = reinterpret_cast<const int32_t*>(p.region + p.chunk_off[c] + region_pr_offset(N, P));
    constexpr int PL = ROWS_PMAX / 32;
    int t[PL];
#pragma unroll
    for (int j = 0; j < PL; ++j) t[j] = lane + 32 * j < P ? __ldg(pr + lane + 32 * j) : -1;
    if (!waited) grid_wait_before();
    waited = true;
    T pb[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) pb[f] = T(0);
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      if (t[j] < 0) continue;
      const int e = t[j] / N, i1 = t[j] - e * N;
      const T* g = G + (long long)e * C::GS + C::SUM_A;
      T s[NF];
      if constexpr (NF == 1) {
        s[0] = *g;
      } else {
        using V = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
        const V v = *reinterpret_cast<const V*>(g);
        s[0] = v.x, s[1] = v.y;
      }
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        const T x = __ldg(M[f] + i1) * fabs(s[f]);
        pb[f] = fmax(pb[f], x == x ? x : big * T(2));  // NaN -> inf
      }
    }
    int eb[2] = {0, 0};
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const T bnd = warp_max(pb[f]) * T(p.chunk_inc[c]);
      eb[f] = bnd <= big ? bound_exponent(bnd) : ROWS_NO_BOUND;
    }
    if (lane == 0) p.chunk_eb[c] = make_int2(eb[0], eb[1]);
  }
}

// State of one chunk, prepared some iterations ahead by one warp and read with 16-byte loads.
struct __align__(16) RowsForm {  // of one form
  double* out;                   // output of digit index 0: the chunk's first value - shift
  int eb;                        // bound exponent (ROWS_NO_BOUND: not finite)
  int shift;                     // chunk position q sits at digit index q + shift: index 0 is
                                 // then at a 16-byte aligned output address
};
struct __align__(16) RowsChunk {
  RowsForm form[2];
  long long region;  // byte offset of its region
  int P, V;          // pairs, CSR values
  int bytes, pad[3]; // of the region
};
__device__ __forceinline__ RowsForm rows_form(const RowsChunk& c, int f) {
  const int4 v = *reinterpret_cast<const int4*>(&c.form[f]);
  RowsForm r;
  r.out = reinterpret_cast<double*>(static_cast<unsigned long long>(unsigned(v.y)) << 32 | unsigned(v.x));
  r.eb = v.z;
  r.shift = v.w;
  return r;
}

// mbarrier helpers of the staging copies: cp.async issued by one warp, tracked by an
// mbarrier of arrival count 32 (each lane arrives when its own copies have landed)
__device__ __forceinline__ uint32_t rows_smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void rows_bar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(rows_smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void rows_cp_async_arrive(unsigned long long* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(rows_smem_u32(bar)) : "memory");
}
// Bounded wait for the completion of the phase of parity `parity`: false after ~2^22 polls.
__device__ __forceinline__ bool rows_bar_wait(unsigned long long* bar, unsigned parity) {
  const uint32_t addr = rows_smem_u32(bar);
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// The chunks of this CTA are c_i = blockIdx.x + i * gridDim.x. In iteration i every warp sums
// its equal share of chunk i's pairs (into accumulator buffer i % 2) and writes its blocks of
// chunk i - 1's values (from the other buffer, which it clears); odd warps write first, so
// the warps of a scheduler mix the shared-memory atomics of one with the conversions of the
// other. Staging runs beside it: warps 0-7 copy chunk i + 3's plan region, warps 8-15 gather
// the G_K of chunk i + 2's pairs (its region was asked for an iteration earlier) and warp 16
// prepares the state of chunk i + 5. The copies are cp.async, tracked by mbarriers that
// their readers wait for an iteration or two later, so no warp waits for memory. One
// CTA-wide barrier closes each iteration. (A queue of warp tasks instead, units of up to 16
// pairs and 128-value blocks handed out by a shared counter, took 1.65 us an iteration on
// fetching and staging alone.) Staging depths: regions 4 buffers (i .. i + 3), geometry 3
// (i .. i + 2), chunk states a ring of 8 (i - 1 .. i + 5). A wait that gives up sets
// FFC_FLAG_TIMEOUT and ends the CTA's work after the iteration.
// One CTA per SM: 32 warps for FP32 (64 registers a thread), 16 for FP64.
template <int D, int FORM, int Q, typename T>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 1024 : 512, 1) rows_assemble(RowsParams p) {
  using C = RowsGeo<D, FORM>;
  using K = RowsCfg<D, FORM, Q>;
  constexpr int N = K::N, NF = C::NF, GS = C::GS, TH = sizeof(T) == 4 ? 1024 : 512;
  constexpr int NDIG = rows_ndig<T>();  // digits: 31-bit fixed point for FP32, 63-bit for FP64
  constexpr int ACC = NF * NDIG * ROWS_VSTRIDE;  // ints of one accumulator buffer
  constexpr int NW = TH / 32, SW = NW / 4;  // warps; of one staging job
  extern __shared__ __align__(16) unsigned char smem[];
  int* acc = reinterpret_cast<int*>(smem);                                   // [2][NF][NDIG][ROWS_VSTRIDE]
  unsigned char* rbuf = smem + size_t(2) * ACC * 4;                          // [4][rmax] plan regions
  T* gbuf = reinterpret_cast<T*>(rbuf + 4 * size_t(p.rmax));                 // [3][pmax][GS]
  RowsChunk* ring = reinterpret_cast<RowsChunk*>(smem + p.meta_off);          // [8] chunk states
  unsigned long long* rbar = reinterpret_cast<unsigned long long*>(ring + 8);  // [4] region copies
  unsigned long long* gbar = rbar + 4;                                          // [3] geometry copies
  const T* A0a = static_cast<const T*>(p.a0.a);
  const T* A0b = static_cast<const T*>(p.a0.b);
  const T* Gall = static_cast<const T*>(p.G);
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int G1 = int(gridDim.x);
  const int n_iter = blockIdx.x < p.n_chunks ? int((p.n_chunks - blockIdx.x + G1 - 1) / G1) : 0;
  for (int i = 4 * t; i < 2 * ACC; i += 4 * TH) *reinterpret_cast<int4*>(acc + i) = make_int4(0, 0, 0, 0);
  if (t < 7) rows_bar_init(rbar + t, 32 * SW);
  bool failed = false;  // a wait of this warp gave up
  auto give_up = [&]() {
    if (lane == 0) atomicOr(p.status, FFC_FLAG_TIMEOUT);
    failed = true;
  };
  auto chunk_at = [&](int i) -> RowsChunk& { return ring[i & 7]; };
  // the state of iteration i's chunk into ring slot i % 8, by one warp: lanes 0-6 load its
  // extents and exponents, lanes 0 and 1 derive each form's part
  auto chunk_load = [&](int i) {
    long long v = 0;
    if (i < n_iter) {
      const long long c = blockIdx.x + (long long)i * G1;
      if (lane < 2) v = p.chunk_pair[c + lane];
      else if (lane < 4) v = p.chunk_off[c + lane - 2];
      else if (lane < 6) v = p.chunk_val[c + lane - 4];
      else if (lane < 7) v = reinterpret_cast<const long long*>(p.chunk_eb)[c];
    }
    return v;
  };
  auto chunk_store = [&](int i, long long v) {
    auto from = [&](int l) { return __shfl_sync(0xffffffffu, v, l); };
    const int P = int(from(1) - from(0));
    const long long r0 = from(2), r1 = from(3), v0 = from(4), v1 = from(5), ebs = from(6);
    RowsChunk& ch = chunk_at(i);
    if (lane < NF) {
      const int eb = int(lane == 0 ? ebs : ebs >> 32);
      double* out = (lane == 0 ? p.out_a : p.out_b) + v0;
      const int sh = int((reinterpret_cast<uintptr_t>(out) >> 3) & 1);
      ch.form[lane].out = out - sh;
      ch.form[lane].eb = eb;
      ch.form[lane].shift = sh;
    }
    if (lane == 2) {
      ch.region = r0;
      ch.bytes = int(r1 - r0);
      ch.P = P;
      ch.V = int(v1 - v0);
    }
  };
  auto region_at = [&](int i) { return rbuf + (i & 3) * p.rmax; };
  auto geom_at = [&](unsigned i3) { return gbuf + i3 * p.pmax * GS; };  // i3 = i % 3
  // the plan region of chunk i (a multiple of 16 bytes, at most rmax) into buffer i % 4
  auto region_task = [&](int i, int part) {  // part of SW warps
    const unsigned char* src = p.region + chunk_at(i).region;
    unsigned char* dst = region_at(i);
    const int nb = chunk_at(i).bytes;
    for (int o = 16 * (part * 32 + lane); o < nb; o += 512 * SW) cp_async16(dst + o, src + o);
    rows_cp_async_arrive(rbar + (i & 3));
  };
  // the G_K of chunk i's pairs into buffer i % 3 (once the region has landed)
  auto geometry_task = [&](int i, int part) {  // part of SW warps
    if (!rows_bar_wait(rbar + (i & 3), unsigned(i >> 2) & 1u)) {
      give_up();
      return;
    }
    const int P = chunk_at(i).P;
    const int32_t* pr = reinterpret_cast<const int32_t*>(region_at(i) + region_pr_offset(N, P));
    T* gs = geom_at(unsigned(i) % 3u);
    for (int k = part * 32 + lane; k < P; k += 32 * SW) {
      const T* src = Gall + (long long)(pr[k] / N) * GS;
      if constexpr (GS * sizeof(T) == 8) {
        cp_async8(gs + k * GS, src);
      } else {
#pragma unroll
        for (int x = 0; x < int(GS * sizeof(T)) / 16; ++x)
          cp_async16(reinterpret_cast<unsigned char*>(gs + k * GS) + 16 * x,
                     reinterpret_cast<const unsigned char*>(src) + 16 * x);
      }
    }
    rows_cp_async_arrive(gbar + unsigned(i) % 3u);
  };
  // this warp's digit indices of chunk i, every NW-th 128, from accumulator buffer i % 2
  // (cleared): a lane converts two consecutive indices at a time and stores them together
  // (index x is output value x - shift, and output index 0 is 16-byte aligned), so a store
  // instruction covers 512 consecutive bytes. Two stores of a lane's four consecutive values,
  // each covering half of every line, cost the L1 data pipe twice the cycles (P4: 3123
  // against 2998 us); and half of the conversions on the FP64 pipe, 3034 us.
  auto write_task = [&](int i) {
    const RowsChunk& ch = chunk_at(i);
    const int V = ch.V;
    int* ab = acc + (i & 1) * ACC;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const RowsForm st = rows_form(ch, f);
      const int eb = st.eb, sh = st.shift;
      const bool fin = eb != ROWS_NO_BOUND;
      Digits<NDIG> dg;
      dg.init(fin ? eb : 0);
      const bool fast = NDIG == 1 && fin && dg.stays_normal();
      double* out = st.out;
      int* a = ab + f * NDIG * ROWS_VSTRIDE;
      const int hi = V + sh;
      for (int x0 = 128 * w + 2 * lane; x0 < hi; x0 += 128 * NW) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int x = x0 + 64 * h;
          if (x >= hi) break;
          int sd[2][NDIG];
#pragma unroll
          for (int d = 0; d < NDIG; ++d) {
            int2* src = reinterpret_cast<int2*>(a + d * ROWS_VSTRIDE + x);
            const int2 v = *src;
            *src = make_int2(0, 0);
            sd[0][d] = v.x;
            sd[1][d] = v.y;
          }
          double r[2];
          if (fast) {
            r[0] = dg.value_int(sd[0][0]);
            r[1] = dg.value_int(sd[1][0]);
          } else {
#pragma unroll
            for (int c = 0; c < 2; ++c) r[c] = fin ? dg.value(sd[c]) : __longlong_as_double(0x7ff8000000000000ll);
          }
          double* o = out + x;
          if (x >= sh && x + 1 < hi) {
            __stcs(reinterpret_cast<double2*>(o), make_double2(r[0], r[1]));
          } else {
            if (x >= sh) __stcs(o, r[0]);
            if (x + 1 >= sh && x + 1 < hi) __stcs(o + 1, r[1]);
          }
        }
      }
    }
  };
  grid_wait_before();
  // ---- prologue: states of chunks 0..4, regions of chunks 0..2, geometry of chunks 0..1
  if (w < 5) {
    const long long v = chunk_load(w);
    if (w < n_iter) chunk_store(w, v);
  }
  __syncthreads();
  if (w < 3 * SW && w / SW < n_iter) region_task(w / SW, w % SW);
  __syncthreads();
  if (w < 2 * SW && w / SW < n_iter) geometry_task(w / SW, w % SW);
  if (__syncthreads_or(failed)) {
    cp_async_commit();
    cp_async_wait_all();
    return;
  }
  unsigned i3 = 0, gpar = 0;  // i % 3, (i / 3) % 2
  for (int i = 0; i <= n_iter; ++i) {
    long long next = 0;
    if (w < SW) {
      if (i + 3 < n_iter) region_task(i + 3, w);
    } else if (w < 2 * SW) {
      if (i + 2 < n_iter) geometry_task(i + 2, w - SW);
    } else if (w == 2 * SW) {
      next = chunk_load(i + 5);
    }
    if (i >= 1 && (w & 1)) write_task(i - 1);
    if (i < n_iter) {
      if (rows_bar_wait(gbar + i3, gpar)) {  // chunk i's geometry; its region landed before that
        const RowsChunk& ch = chunk_at(i);
        const int P = ch.P;
        const unsigned char* reg = region_at(i);
        const unsigned* run = reinterpret_cast<const unsigned*>(reg + ROWS_WARPS);
        const int32_t* pr = reinterpret_cast<const int32_t*>(reg + region_pr_offset(N, P));
        const uint16_t* pos = reinterpret_cast<const uint16_t*>(reg + region_pr_offset(N, P) + 4 * P);
        const T* gs = geom_at(i3);
        Digits<NDIG> dig[NF];
        int* base[NF];
        bool magic = sizeof(T) == 4;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          const RowsForm st = rows_form(ch, f);
          dig[f].init(st.eb != ROWS_NO_BOUND ? st.eb : 0);
          magic = magic && dig[f].magic;
          base[f] = acc + (i & 1) * ACC + f * NDIG * ROWS_VSTRIDE + st.shift;
        }
        const int r = reg[w * (ROWS_WARPS / NW)], k0 = P * w / NW, k1 = P * (w + 1) / NW;
        auto sum = [&](auto m) {
          constexpr bool M = decltype(m)::value;
          share_task<K, FORM, NF, GS, M, NDIG, T>(r, k0, k1, run, pr, gs, pos, base, dig, A0a, A0b);
          // column tails go to the last warps, the first ones stage
          if constexpr (K::W > 0)
            for (int st = NW - 1 - w; st * K::TP < P; st += NW)
              tail_step<K, FORM, NF, GS, M, NDIG, T>(st, P, pr, gs, pos, base, dig, A0a, A0b);
        };
        if (magic) sum(std::true_type());
        else sum(std::false_type());
      } else {
        give_up();
      }
    }
    if (i >= 1 && !(w & 1)) write_task(i - 1);
    if (w == 2 * SW && i + 5 < n_iter) chunk_store(i + 5, next);
    if (i3 == 2) {
      i3 = 0;
      gpar ^= 1;
    } else {
      ++i3;
    }
    if (__syncthreads_or(failed)) break;
  }
  cp_async_commit();
  cp_async_wait_all();  // copies of chunks this CTA no longer needed (a wait that gave up)
}

template <int D, int FORM, int Q, typename T>
int launch_rows_t(const ffc_row_plan* plan, const RowsTensors& a0, double* out_a, double* out_b, unsigned* status,
                  cudaStream_t s) {
  using C = RowsGeo<D, FORM>;
  const int pmax = std::max(plan->max_pairs, 1);
  using K = RowsCfg<D, FORM, Q>;
  constexpr int NDIG = rows_ndig<T>();
  const int rmax = std::max(plan->max_region, 16);
  const size_t meta_off = (2 * size_t(C::NF) * NDIG * ROWS_VSTRIDE * 4 + 4 * size_t(rmax) +
                           3 * size_t(pmax) * C::GS * sizeof(T) + 15) / 16 * 16;
  const size_t smem = meta_off + 8 * sizeof(RowsChunk) + 7 * sizeof(unsigned long long);
  auto kern = rows_assemble<D, FORM, Q, T>;
  int dev = 0, smem_optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (smem > size_t(smem_optin)) return FFC_EUNSUPPORTED;  // the pair then runs as two single passes
  if (plan->n_chunks > (long long)INT_MAX) {  // iteration counters are 32-bit
    set_error("row-owner assembly: more than 2^31 - 1 chunks");
    return FFC_EINVAL;
  }
  int sms = 0, per_sm = 1;
  constexpr int TH = sizeof(T) == 4 ? 1024 : 512;
  if (launch_config(reinterpret_cast<const void*>(kern), TH, smem, -1, &sms, &per_sm) != FFC_OK)
    return FFC_ECUDA;
  long long blocks = (long long)sms * per_sm;
  if (blocks > plan->n_chunks) blocks = plan->n_chunks;
  if (blocks < 1) return FFC_OK;
  RowsParams prm{plan->chunk_off, plan->chunk_pair, plan->chunk_val, plan->chunk_inc, plan->chunk_eb, plan->region,
                 plan->geom, a0, out_a, out_b, (long long)plan->n_chunks, int(meta_off), pmax, rmax, status};
  const long long bound_blocks = std::min<long long>((plan->n_chunks + 7) / 8, (long long)sms * 8);
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(unsigned(bound_blocks));
  cfg.blockDim = dim3(256);
  cudaError_t e = cudaLaunchKernelEx(&cfg, rows_bounds<D, FORM, Q, T>, prm);
  if (e == cudaSuccess) {
    cfg.gridDim = dim3(unsigned(blocks));
    cfg.blockDim = dim3(TH);
    cfg.dynamicSmemBytes = smem;
    e = cudaLaunchKernelEx(&cfg, kern, prm);
  }
  return e == cudaSuccess ? FFC_OK : cuda_fail(e, "rows_assemble launch");
}

template <int D, int FORM, typename T>
int launch_rows_geometry(const ffc_row_plan* plan, const int32_t* cells, const double* vertices, int64_t n_vert,
                         unsigned* status, cudaStream_t s) {
  if (plan->n_elem == 0) return FFC_OK;
  int sms = 0;
  if (launch_config(reinterpret_cast<const void*>(rows_geometry<D, FORM, T>), 256, 0, -1, &sms, nullptr) != FFC_OK)
    return FFC_ECUDA;
  long long blocks = (plan->n_elem + 255) / 256;
  if (blocks > (long long)sms * 8) blocks = (long long)sms * 8;
  rows_geometry<D, FORM, T><<<unsigned(blocks), 256, 0, s>>>(cells, vertices, n_vert, plan->n_elem,
                                                              static_cast<T*>(plan->geom), status);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? FFC_OK : cuda_fail(e, "rows_geometry launch");
}

template <int D, int FORM, typename T>
int launch_rows_q(const ffc_row_plan* plan, int q, const int32_t* cells, const double* vertices, int64_t n_vert,
                  const RowsTensors& a0, double* out_a, double* out_b, unsigned* status, cudaStream_t s) {
  int rc = launch_rows_geometry<D, FORM, T>(plan, cells, vertices, n_vert, status, s);
  if (rc != FFC_OK) return rc;
  switch (q) {
    case 1: return launch_rows_t<D, FORM, 1, T>(plan, a0, out_a, out_b, status, s);
    case 2: return launch_rows_t<D, FORM, 2, T>(plan, a0, out_a, out_b, status, s);
    case 3: return launch_rows_t<D, FORM, 3, T>(plan, a0, out_a, out_b, status, s);
    case 4: return launch_rows_t<D, FORM, 4, T>(plan, a0, out_a, out_b, status, s);
    default: return FFC_EUNSUPPORTED;
  }
}

template <typename T>
int launch_rows_form(int form, int d, int q, const ffc_row_plan* plan, const int32_t* cells, const double* vertices,
                     int64_t n_vert, const RowsTensors& a0, double* out_a, double* out_b, unsigned* status,
                     cudaStream_t s) {
  if (d == 3) {
    if (form == FFC_MASS)
      return launch_rows_q<3, FFC_MASS, T>(plan, q, cells, vertices, n_vert, a0, out_a, out_b, status, s);
    if (form == FFC_POISSON)
      return launch_rows_q<3, FFC_POISSON, T>(plan, q, cells, vertices, n_vert, a0, out_a, out_b, status, s);
    if constexpr (sizeof(T) == 4)  // FP64 pairs are two single passes
      return launch_rows_q<3, ROWS_PAIR, T>(plan, q, cells, vertices, n_vert, a0, out_a, out_b, status, s);
    return FFC_EUNSUPPORTED;
  }
  if (form == FFC_MASS)
    return launch_rows_q<2, FFC_MASS, T>(plan, q, cells, vertices, n_vert, a0, out_a, out_b, status, s);
  if (form == FFC_POISSON)
    return launch_rows_q<2, FFC_POISSON, T>(plan, q, cells, vertices, n_vert, a0, out_a, out_b, status, s);
  if constexpr (sizeof(T) == 4)
    return launch_rows_q<2, ROWS_PAIR, T>(plan, q, cells, vertices, n_vert, a0, out_a, out_b, status, s);
  return FFC_EUNSUPPORTED;
}

void free_plan(ffc_row_plan* p) {
  if (!p) return;
  int cur = 0;
  cudaGetDevice(&cur);
  cudaSetDevice(p->device);
  cudaFree(p->row_ptr);
  cudaFree(p->chunk_row);
  cudaFree(p->chunk_pair);
  cudaFree(p->chunk_off);
  cudaFree(p->chunk_val);
  cudaFree(p->chunk_inc);
  cudaFree(p->region);
  cudaFree(p->geom);
  cudaFree(p->chunk_eb);
  cudaSetDevice(cur);
  delete p;
}

template <typename T>
int dev_alloc(T** p, size_t count) {
  const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), (count ? count : 1) * sizeof(T));
  return e == cudaSuccess ? FFC_OK : cuda_fail(e, "cudaMalloc");
}

// Common checks of the row assemblies; fills the device tensors of the form(s).
int rows_checks(const char* who, const ffc_form* f, const ffc_row_plan* plan, const int32_t* cells,
                const double* vertices, int64_t n_vert, const double* out, int precision) {
  if (!f || !plan || n_vert < 0 || (precision != FFC_FP64 && precision != FFC_FP32)) {
    set_error(std::string(who) + ": invalid argument");
    return FFC_EINVAL;
  }
  if ((f->kind != FFC_MASS && f->kind != FFC_POISSON) || f->rank != 2) {
    set_error(std::string(who) + ": mass and Poisson forms only");
    return FFC_EUNSUPPORTED;
  }
  if (f->n != plan->n_local) {
    set_error(std::string(who) + ": the plan was built for another number of local dofs");
    return FFC_EINVAL;
  }
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != plan->device) {
    set_error(std::string(who) + ": the plan lives on another device");
    return FFC_EINVAL;
  }
  if (plan->nnz == 0) return FFC_OK;
  if (!out || (reinterpret_cast<uintptr_t>(out) & 7) ||
      (plan->n_elem > 0 && (!cells || !vertices || n_vert == 0 || (reinterpret_cast<uintptr_t>(cells) & 15) ||
                            (reinterpret_cast<uintptr_t>(vertices) & 7)))) {
    set_error(std::string(who) + ": null or misaligned pointer");
    return FFC_EINVAL;
  }
  return FFC_OK;
}

}  // namespace
}  // namespace ffc

using namespace ffc;

extern "C" {

int ffc_row_plan_create(int64_t n_elem, int n_local, const int32_t* dofmap, int64_t n_dof, const int64_t* row_ptr,
                        const int32_t* col, int64_t nnz, void* stream, ffc_row_plan** out) {
  if (!out || n_elem < 0 || n_local < 2 || n_local > ROWS_MAX_LOCAL || n_dof < 1 || n_dof >= INT32_MAX || nnz < 0 ||
      !row_ptr || (n_elem > 0 && !dofmap) || (nnz > 0 && !col)) {
    set_error("ffc_row_plan_create: invalid argument (2 <= n_local <= 64)");
    return FFC_EINVAL;
  }
  if (n_elem * (long long)n_local >= INT32_MAX) {
    set_error("ffc_row_plan_create: n_elem * n_local must be below 2^31");
    return FFC_EINVAL;
  }
  if ((reinterpret_cast<uintptr_t>(dofmap) & 3) || (reinterpret_cast<uintptr_t>(row_ptr) & 7) ||
      (reinterpret_cast<uintptr_t>(col) & 3)) {
    set_error("ffc_row_plan_create: misaligned pointer");
    return FFC_EINVAL;
  }
  *out = nullptr;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  ffc_row_plan* p = new ffc_row_plan();
  cudaGetDevice(&p->device);
  p->n_elem = n_elem;
  p->n_local = n_local;
  p->n_dof = n_dof;
  p->nnz = nnz;
  const long long total = n_elem * (long long)n_local;
  const long long nb = (n_dof + 1 + SCAN_CHUNK - 1) / SCAN_CHUNK;
  int32_t *inc_ptr = nullptr, *inc_tmp = nullptr, *fill = nullptr, *sums = nullptr;
  unsigned long long* key = nullptr;
  unsigned* err = nullptr;
  int rc = FFC_OK;
  cudaError_t e = cudaSuccess;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
  const unsigned grid = unsigned(sms > 0 ? sms * 8 : 1024);
  unsigned host_err = 0;
  std::vector<int64_t> h_row_ptr(size_t(n_dof) + 1);
  std::vector<int32_t> h_inc_ptr(size_t(n_dof) + 1);
  std::vector<int32_t> h_chunk_row, h_chunk_pair, h_chunk_inc;
  std::vector<int64_t> h_chunk_off, h_chunk_val;
  if ((rc = dev_alloc(&p->row_ptr, size_t(n_dof) + 1)) || (rc = dev_alloc(&inc_ptr, size_t(n_dof) + 1)) ||
      (rc = dev_alloc(&inc_tmp, size_t(total))) || (rc = dev_alloc(&fill, size_t(n_dof))) ||
      (rc = dev_alloc(&sums, size_t(nb))) || (rc = dev_alloc(&err, 1)) ||
      (rc = dev_alloc(reinterpret_cast<double**>(&p->geom), size_t(n_elem) * ROWS_GEOM)))
    goto fail;
  if ((e = cudaMemcpyAsync(p->row_ptr, row_ptr, (size_t(n_dof) + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice,
                           s)) != cudaSuccess ||
      (e = cudaMemsetAsync(inc_ptr, 0, (size_t(n_dof) + 1) * sizeof(int32_t), s)) != cudaSuccess ||
      (e = cudaMemsetAsync(fill, 0, size_t(n_dof) * sizeof(int32_t), s)) != cudaSuccess ||
      (e = cudaMemsetAsync(err, 0, sizeof(unsigned), s)) != cudaSuccess) {
    rc = cuda_fail(e, "ffc_row_plan_create: memset");
    goto fail;
  }
  if (total > 0) plan_count<<<grid, 256, 0, s>>>(dofmap, total, n_dof, inc_ptr, err);
  scan_chunks<<<unsigned(nb), SCAN_T, 0, s>>>(inc_ptr, n_dof + 1, sums);
  scan_sums<<<1, SCAN_T, 0, s>>>(sums, int(nb));
  scan_add<<<unsigned(nb), SCAN_T, 0, s>>>(inc_ptr, n_dof + 1, sums);
  if (total > 0) plan_fill<<<grid, 256, 0, s>>>(dofmap, total, n_dof, inc_ptr, fill, inc_tmp);
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (e = cudaMemcpyAsync(h_row_ptr.data(), row_ptr, h_row_ptr.size() * sizeof(int64_t), cudaMemcpyDeviceToHost,
                           s)) != cudaSuccess ||
      (e = cudaMemcpyAsync(h_inc_ptr.data(), inc_ptr, h_inc_ptr.size() * sizeof(int32_t), cudaMemcpyDeviceToHost,
                           s)) != cudaSuccess ||
      (e = cudaMemcpyAsync(&host_err, err, sizeof(unsigned), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaStreamSynchronize(s)) != cudaSuccess) {
    rc = cuda_fail(e, "ffc_row_plan_create");
    goto fail;
  }
  if (host_err & PLAN_BAD_DOF) {
    set_error("ffc_row_plan_create: dof id out of range");
    rc = FFC_EBOUNDS;
    goto fail;
  }
  {
    // rows -> chunks (host, one pass): consecutive rows while the chunk holds at most
    // ROWS_VMAX values, ROWS_PMAX pairs and 65536 rows
    if (h_row_ptr[0] != 0 || h_row_ptr[n_dof] != nnz) host_err |= PLAN_BAD_ROW_PTR;
    int32_t cur_v = 0, cur_p = 0, cur_inc = 0, r_start = 0;
    int64_t off = 0;
    auto close_chunk = [&](int64_t r) {
      const int64_t bytes = region_bytes(n_local, cur_p);
      off += bytes;
      h_chunk_inc.push_back(cur_inc);
      p->vmax = std::max(p->vmax, int(cur_v));
      p->max_pairs = std::max(p->max_pairs, int(cur_p));
      p->max_region = std::max(p->max_region, int(bytes));
      h_chunk_row.push_back(int32_t(r));
      h_chunk_pair.push_back(h_inc_ptr[r]);
      h_chunk_off.push_back(off);
      h_chunk_val.push_back(h_row_ptr[r]);
      cur_v = cur_p = cur_inc = 0;
      r_start = int32_t(r);
    };
    h_chunk_row.push_back(0);
    h_chunk_pair.push_back(0);
    h_chunk_off.push_back(0);
    h_chunk_val.push_back(0);
    for (int64_t r = 0; r < n_dof && !(host_err & PLAN_BAD_ROW_PTR); ++r) {
      const int64_t L = h_row_ptr[r + 1] - h_row_ptr[r];
      const int32_t c = h_inc_ptr[r + 1] - h_inc_ptr[r];
      if (L < 0 || h_row_ptr[r + 1] > nnz) {
        host_err |= PLAN_BAD_ROW_PTR;
        break;
      }
      if (L > ROWS_VMAX || c > ROWS_PMAX || c > ROWS_MAX_INCIDENCE) {
        set_error("ffc_row_plan_create: row " + std::to_string(r) + " has " + std::to_string(L) + " entries and " +
                  std::to_string(c) + " (cell, local dof) pairs; at most " + std::to_string(ROWS_VMAX) + " and " +
                  std::to_string(std::min(ROWS_PMAX, ROWS_MAX_INCIDENCE)) + " are supported");
        rc = FFC_EINVAL;
        goto fail;
      }
      if (r > r_start && (cur_v + L > ROWS_VMAX || cur_p + c > ROWS_PMAX || r - r_start >= 65536)) close_chunk(r);
      cur_v += int32_t(L);
      cur_p += c;
      cur_inc = std::max(cur_inc, c);
      p->max_row = std::max(p->max_row, int(L));
      p->max_incidence = std::max(p->max_incidence, int(c));
    }
    if (host_err & PLAN_BAD_ROW_PTR) {
      set_error("ffc_row_plan_create: row_ptr is not monotone within [0, nnz]");
      rc = FFC_EINVAL;
      goto fail;
    }
    close_chunk(n_dof);
    p->n_chunks = int64_t(h_chunk_inc.size());
    p->region_total = off;
  }
  if ((rc = dev_alloc(&p->chunk_row, h_chunk_row.size())) || (rc = dev_alloc(&p->chunk_pair, h_chunk_pair.size())) ||
      (rc = dev_alloc(&p->chunk_off, h_chunk_off.size())) || (rc = dev_alloc(&p->chunk_val, h_chunk_val.size())) ||
      (rc = dev_alloc(&p->chunk_inc, h_chunk_inc.size())) || (rc = dev_alloc(&p->chunk_eb, h_chunk_inc.size())) ||
      (rc = dev_alloc(&p->region, size_t(p->region_total) + 16)) ||
      (rc = dev_alloc(&key, size_t(total))))
    goto fail;
  if ((e = cudaMemcpyAsync(p->chunk_row, h_chunk_row.data(), h_chunk_row.size() * 4, cudaMemcpyHostToDevice, s)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(p->chunk_pair, h_chunk_pair.data(), h_chunk_pair.size() * 4, cudaMemcpyHostToDevice, s)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(p->chunk_off, h_chunk_off.data(), h_chunk_off.size() * 8, cudaMemcpyHostToDevice, s)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(p->chunk_val, h_chunk_val.data(), h_chunk_val.size() * 8, cudaMemcpyHostToDevice, s)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(p->chunk_inc, h_chunk_inc.data(), h_chunk_inc.size() * 4, cudaMemcpyHostToDevice, s)) !=
          cudaSuccess ||
      (e = cudaMemsetAsync(p->region, 0, size_t(p->region_total) + 16, s)) != cudaSuccess) {
    rc = cuda_fail(e, "ffc_row_plan_create: chunk table");
    goto fail;
  }
  plan_sort<<<unsigned((p->n_chunks + 127) / 128), 128, 0, s>>>(dofmap, p->chunk_row, p->chunk_pair, p->chunk_off,
                                                                p->n_chunks, n_local, inc_tmp, key, p->region);
  if (total > 0)
    plan_positions<<<grid, 256, 0, s>>>(dofmap, n_local, p->row_ptr, col, p->chunk_row, p->chunk_pair, p->chunk_off,
                                        p->n_chunks, p->region, err);
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (e = cudaMemcpyAsync(&host_err, err, sizeof(unsigned), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaStreamSynchronize(s)) != cudaSuccess) {
    rc = cuda_fail(e, "ffc_row_plan_create");
    goto fail;
  }
  if (host_err & PLAN_MISSING) {
    set_error("ffc_row_plan_create: a (row, col) pair of a cell is not in the pattern");
    rc = FFC_EBOUNDS;
    goto fail;
  }
  cudaFree(inc_ptr);
  cudaFree(inc_tmp);
  cudaFree(fill);
  cudaFree(sums);
  cudaFree(err);
  cudaFree(key);
  *out = p;
  return FFC_OK;
fail:
  cudaStreamSynchronize(s);
  cudaFree(inc_ptr);
  cudaFree(inc_tmp);
  cudaFree(fill);
  cudaFree(sums);
  cudaFree(err);
  cudaFree(key);
  free_plan(p);
  return rc;
}

int ffc_row_plan_info(const ffc_row_plan* p, int64_t* n_dof, int64_t* nnz, int* max_row, int* max_incidence) {
  if (!p) return FFC_EINVAL;
  if (n_dof) *n_dof = p->n_dof;
  if (nnz) *nnz = p->nnz;
  if (max_row) *max_row = p->max_row;
  if (max_incidence) *max_incidence = p->max_incidence;
  return FFC_OK;
}

int ffc_row_plan_layout(const ffc_row_plan* p, int64_t* n_chunks, int* max_chunk_values, int* max_chunk_pairs,
                        int* max_region_bytes, int64_t* device_bytes) {
  if (!p) return FFC_EINVAL;
  if (n_chunks) *n_chunks = p->n_chunks;
  if (max_chunk_values) *max_chunk_values = p->vmax;
  if (max_chunk_pairs) *max_chunk_pairs = p->max_pairs;
  if (max_region_bytes) *max_region_bytes = p->max_region;
  if (device_bytes)
    *device_bytes = (p->n_dof + 1) * 8 + (p->n_chunks + 1) * (4 + 4 + 8 + 8) + p->n_chunks * (4 + 8) +
                    p->region_total + 16 + p->n_elem * ROWS_GEOM * 8;
  return FFC_OK;
}

void ffc_row_plan_destroy(ffc_row_plan* p) { free_plan(p); }

int ffc_assemble_rows(const ffc_form* f, const ffc_row_plan* plan, const int32_t* cells, const double* vertices,
                      int64_t n_vert, double* csr_val, int precision, void* stream) {
  int rc = rows_checks("ffc_assemble_rows", f, plan, cells, vertices, n_vert, csr_val, precision);
  if (rc != FFC_OK || plan->nnz == 0) return rc;
  DeviceTensors* t = nullptr;
  if ((rc = ensure_device_tensors(const_cast<ffc_form*>(f), &t)) != FFC_OK) return rc;
  uint32_t* st = status_word();
  if (!st) {
    set_error("status word allocation failed");
    return FFC_ECUDA;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (precision == FFC_FP32) {
    const RowsTensors a0{f->kind == FFC_POISSON ? t->a0v_f32 : t->a0s_f32, nullptr, t->a0m_f32, nullptr};
    rc = launch_rows_form<float>(f->kind, f->d, f->q, plan, cells, vertices, n_vert, a0, csr_val, nullptr, st, s);
  } else {
    const RowsTensors a0{t->a0s_f64, nullptr, t->a0m_f64, nullptr};
    rc = launch_rows_form<double>(f->kind, f->d, f->q, plan, cells, vertices, n_vert, a0, csr_val, nullptr, st, s);
  }
  if (rc == FFC_EUNSUPPORTED) set_error("ffc_assemble_rows: the plan's chunks need more shared memory than a CTA has");
  return rc;
}

int ffc_assemble_rows_pair(const ffc_form* fa, const ffc_form* fb, const ffc_row_plan* plan, const int32_t* cells,
                           const double* vertices, int64_t n_vert, double* csr_val_a, double* csr_val_b,
                           int precision, void* stream) {
  int rc = rows_checks("ffc_assemble_rows_pair", fa, plan, cells, vertices, n_vert, csr_val_a, precision);
  if (rc != FFC_OK) return rc;
  if ((rc = rows_checks("ffc_assemble_rows_pair", fb, plan, cells, vertices, n_vert, csr_val_b, precision)) != FFC_OK)
    return rc;
  if (fa->d != fb->d || fa->q != fb->q || csr_val_a == csr_val_b) {
    set_error("ffc_assemble_rows_pair: two forms on one space, two distinct matrices");
    return FFC_EINVAL;
  }
  if (plan->nnz == 0) return FFC_OK;
  if (fa->kind == fb->kind) {  // not the (mass, Poisson) pair: two single passes
    if ((rc = ffc_assemble_rows(fa, plan, cells, vertices, n_vert, csr_val_a, precision, stream)) != FFC_OK) return rc;
    return ffc_assemble_rows(fb, plan, cells, vertices, n_vert, csr_val_b, precision, stream);
  }
  const ffc_form* fm = fa->kind == FFC_MASS ? fa : fb;
  const ffc_form* fp = fa->kind == FFC_MASS ? fb : fa;
  double* vm = fa->kind == FFC_MASS ? csr_val_a : csr_val_b;
  double* vp = fa->kind == FFC_MASS ? csr_val_b : csr_val_a;
  DeviceTensors *tm = nullptr, *tp = nullptr;
  if ((rc = ensure_device_tensors(const_cast<ffc_form*>(fm), &tm)) != FFC_OK ||
      (rc = ensure_device_tensors(const_cast<ffc_form*>(fp), &tp)) != FFC_OK)
    return rc;
  uint32_t* st = status_word();
  if (!st) {
    set_error("status word allocation failed");
    return FFC_ECUDA;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (precision == FFC_FP32) {
    const RowsTensors a0{tm->a0s_f32, tp->a0v_f32, tm->a0m_f32, tp->a0m_f32};
    rc = launch_rows_form<float>(ROWS_PAIR, fm->d, fm->q, plan, cells, vertices, n_vert, a0, vm, vp, st, s);
    if (rc != FFC_EUNSUPPORTED) return rc;
  }
  // FP64 (whose double-buffered 63-bit accumulators of two matrices exceed the shared
  // memory), and chunks too large for one pass: two single passes
  if ((rc = ffc_assemble_rows(fm, plan, cells, vertices, n_vert, vm, precision, stream)) != FFC_OK) return rc;
  return ffc_assemble_rows(fp, plan, cells, vertices, n_vert, vp, precision, stream);
}

}  // extern "C"
