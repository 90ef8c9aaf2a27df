// k_factor.cu -- factorisation of the element-Jacobi blocks (Section 2.4:
// power-of-two row and column equilibration, then Gauss-Jordan elimination
// with partial pivoting to the explicit inverse) with the block in registers.
//
// What bounds an in-place Gauss-Jordan step is not its 2 n^2 flops but how
// often each entry travels: with the block in shared memory every step reads
// and writes all n^2 entries there.  Here a thread holds R whole rows of C
// columns in registers for the whole elimination, and B pivots (a panel) are
// taken together:
//  1. panel: the threads owning the panel's columns eliminate within it, one
//     pivot search (warp reductions on the bit patterns, then one slot per
//     warp) and one barrier per pivot; the multipliers stay in registers;
//  2. the B pivot rows of all other columns go to shared memory once, where a
//     thread per column runs the B x B triangular recurrence on them;
//  3. every other entry takes its B updates in registers, one shared-memory
//     broadcast (16 bytes) feeding R * 4 FMAs.
// Each entry sees the operations of the column-by-column elimination in the
// same order, so the inverse is bit for bit that of the cluster kernel
// (k_factor_cluster.cu), which keeps its columns in shared memory.
//
// Registers are not indexed by a loop variable: the panel is always columns
// 0 .. B-1 of its owner, whose update writes column j to j - B and whose
// finished panel columns are appended, so after its C / B panels the order is
// the original one.  Rows are not moved either: pos[] holds each row's
// position under the interchanges, and the rows and columns of the inverse
// are permuted on the way out (column k of the eliminated matrix is column
// pivot_row[k] of the inverse).
//
// Layout by size: n <= 64 one warp per block (R = 2 rows a lane above 32), no
// CTA barrier, in FP64 two warps at n = 64 and for few blocks of 36 and 40; 100 to 144 one CTA, a row per
// thread, in FP64 split over two column groups; n = 320 a cluster of 5 CTAs
// (FP32, two clusters' CTAs per SM) or 4 (FP64), whose registers hold 64 or 80
// columns of every row; the panel's owner writes its multipliers into every
// CTA's shared memory, one cluster barrier per panel.  For n = 320 in FP32,
// clusters of 2, 4 and 5 measured 13.1, 13.6 and 11.1 ms on 1728 blocks: the
// wider split leaves room for a second block whose update covers the panel's
// latency (about 10,000 cycles per 8 pivots, the bound that is left); in FP64,
// where the pipe is the bound, 4 CTAs take 129 ms and 5 take 138 ms.
//
// Measured on one GB300 (ms; before: the block in shared memory, one pivot at
// a time), FP32 / FP64, with the fraction of the FP64 peak (152 SMs x 2 FMA x
// 2.07 GHz) where that is the bound:
//   4096 blocks of n =  64   1.44 -> 0.30    4.05 ->  2.32 (73%)
//   4096 blocks of n = 100   5.4  -> 0.95   14.8  -> 11.9  (55%)
//   1728 blocks of n = 135  10.0  -> 1.00   23.4  -> 10.9  (61%)
//   1728 blocks of n = 320  58    -> 11.1  216    -> 127   (71%)
//
// Equilibration works on exponent fields: the scales are powers of two, so a
// scaled entry is the entry with its exponent shifted (and, for FP32, the
// significand rounded to nearest even) by integer operations, none of which
// occupies the FP64 pipe (one warp instruction per 64 cycles and
// sub-partition).  Entries whose shift would leave the normal range, and
// non-finite ones, take the floating-point operations instead.
#include <cooperative_groups.h>

#include "pmg_internal.h"

namespace cg = cooperative_groups;

namespace pmg {

namespace {

__device__ __forceinline__ double pow2_inv_scale_r(double m) {
  // 2^-k with m * 2^-k in [0.5, 1); 1 for m == 0
  if (!(m > 0.0)) return 1.0;
  int ex;
  frexp(m, &ex);
  return ldexp(1.0, -ex);
}
// 2^s, -1074 <= s <= 1024 (inf): rows up to the largest number have subnormal scales, 2^-1023 and 2^-1024
__device__ __forceinline__ double pow2_d(int s) {
  return __longlong_as_double(s > -1023 ? (long long)(s + 1023) << 52 : 1ll << (s + 1074));
}
__device__ __forceinline__ int pow2_exp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff) - 1023; }

// d 2^s 2^t (applied in that order) in the working precision.
template <class T>
__device__ __forceinline__ T scaled_entry(double d, int s, int t) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned long long mag = b & 0x7fffffffffffffffull;
  const int e = (int)(mag >> 52), e1 = e + s, e2 = e1 + t;
  const bool normal = e >= 1 && e <= 2046 && e1 >= 1 && e1 <= 2046;
  if (sizeof(T) == 8) {
    if (normal && e2 >= 1 && e2 <= 2046) return (T)__longlong_as_double((long long)(b + ((unsigned long long)(long long)(s + t) << 52)));
  } else {
    if (normal && e2 >= 897 && e2 <= 1150) {
      const unsigned long long m2 = mag + ((unsigned long long)(long long)(s + t) << 52);
      const unsigned int f = (unsigned int)((m2 + 0x0fffffffull + ((m2 >> 29) & 1ull)) >> 29) - (896u << 23);
      return (T)__uint_as_float(f | ((unsigned int)(b >> 32) & 0x80000000u));
    }
  }
  if (mag == 0) return (b >> 63) ? (T)-0.0 : (T)0.0;
  // the products themselves, in a loop that keeps them behind a branch: as
  // straight-line code they are predicated, and predicated-off FP64
  // instructions still take their 64 cycles of the pipe on every entry
#pragma unroll 1
  for (int k = 0; k < 2; ++k) d *= pow2_d(k == 0 ? s : t);
  return (T)d;
}

// Pivot keys: |x| ordered as its bit pattern, 0 for NaN (never preferred).
template <class T> struct Key { using type = unsigned long long; };
template <> struct Key<float> { using type = unsigned int; };
__device__ __forceinline__ unsigned int pivot_key(float x) {
  const unsigned int b = __float_as_uint(x) & 0x7fffffffu;
  return b > 0x7f800000u ? 0u : b + 1u;
}
__device__ __forceinline__ unsigned long long pivot_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  return b > 0x7ff0000000000000ull ? 0ull : b + 1ull;
}
// Largest key of the warp and, among its holders, the smallest position.
__device__ __forceinline__ void warp_best(unsigned int& key, int& pos) {
  const unsigned int m = __reduce_max_sync(0xffffffffu, key);
  pos = __reduce_min_sync(0xffffffffu, key == m ? pos : 0x7fffffff);
  key = m;
}
__device__ __forceinline__ void warp_best(unsigned long long& key, int& pos) {
  const unsigned int full = 0xffffffffu;
  const unsigned int hi = (unsigned int)(key >> 32), mh = __reduce_max_sync(full, hi);
  const unsigned int lo = hi == mh ? (unsigned int)key : 0u, ml = __reduce_max_sync(full, lo);
  pos = __reduce_min_sync(full, hi == mh && lo == ml ? pos : 0x7fffffff);
  key = ((unsigned long long)mh << 32) | ml;
}
__device__ __forceinline__ bool bad_pivot(float x, int n) {
  return !(fabsf(x) > n * 1.1920928955078125e-07f) || isinf(x);
}
__device__ __forceinline__ bool bad_pivot(double x, int n) {   // on the bit pattern: no FP64 instruction
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return !(b > __double_as_longlong(n * 2.220446049250313e-16)) || b >= 0x7ff0000000000000ll;
}

template <class T> struct Vec;
template <> struct Vec<float> { using type = float4; static constexpr int n = 4; };
template <> struct Vec<double> { using type = double2; static constexpr int n = 2; };
__device__ __forceinline__ void unpack(float4 v, float o[4]) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
__device__ __forceinline__ void unpack(double2 v, double o[2]) { o[0] = v.x; o[1] = v.y; }

// Sizes and the shared-memory layout of one element.
template <class T, int N, int R, int G, int CL, int B>
struct Lay {
  static constexpr int TR = ((N + R - 1) / R + 31) / 32 * 32;   // threads per column group
  static constexpr int WR = TR / 32;
  static constexpr int NE = TR * G;                             // threads per element and CTA
  static constexpr int GT = G * CL;                             // column groups of an element
  static constexpr int C = ((N + GT - 1) / GT + B - 1) / B * B; // columns per group
  static constexpr int CC = C * G;                              // columns per CTA
  static constexpr int NP = (N + B - 1) / B;                    // panels with pivots
  static constexpr int RT = TR * R;
  static constexpr int SC = C + 1;                              // row stride of the staged block
  static constexpr size_t a16(size_t x) { return (x + 15) & ~(size_t)15; }
  static constexpr size_t oPhys = 0;                                          // int [N]
  static constexpr size_t oEr = a16(oPhys + 4 * N);                           // int [N] row exponents
  static constexpr size_t oEc = a16(oEr + 4 * N);                             // int [CC] column exponents
  static constexpr size_t oSt = a16(oEc + 4 * CC);                            // T [G][N][SC], then reused:
  static constexpr size_t oU = oSt;                                           // T [B][CC] pivot rows
  static constexpr size_t oF = a16(oU + sizeof(T) * B * CC);                  // T [2][B][RT] multipliers
  static constexpr size_t oFp = a16(oF + (GT > 1 ? sizeof(T) * 2 * B * RT : 0));   // T [2][B][B] of the pivot rows
  static constexpr size_t oIp = a16(oFp + sizeof(T) * 2 * B * B);             // T [2][B] pivot reciprocals
  static constexpr size_t oPv = a16(oIp + sizeof(T) * 2 * B);                 // int [2][2][B] pivot rows, positions
  static constexpr size_t oKey = a16(oPv + 4 * 4 * B);                        // u64 [2][WR]
  static constexpr size_t oSl = a16(oKey + 8 * 2 * WR);                       // T [2][WR][B] candidate rows
  static constexpr size_t oSp = a16(oSl + sizeof(T) * 2 * WR * B);            // int [2][WR][2] position, row
  static constexpr size_t end = a16(oSp + 4 * 4 * WR);
  static constexpr size_t st_end = a16(oSt + sizeof(T) * G * N * SC);
  static constexpr size_t bytes = end > st_end ? end : st_end;
};

}  // namespace

template <class T, class W, int N, int R, int G, int CL, int B, int EPC, int MINB>
__global__ void __launch_bounds__(Lay<T, N, R, G, CL, B>::NE* EPC, MINB)
    factor_reg_kernel(int E, const double* __restrict__ Din, W* __restrict__ Dinv, double* __restrict__ rs,
                      double* __restrict__ cs, int* __restrict__ flag, int flag_base) {
  using Y = Lay<T, N, R, G, CL, B>;
  constexpr int TR = Y::TR, WR = Y::WR, NE = Y::NE, GT = Y::GT, C = Y::C, CC = Y::CC, RT = Y::RT, SC = Y::SC;
  constexpr int VN = Vec<T>::n;
  using V = typename Vec<T>::type;
  static_assert(EPC == 1 || NE == 32, "several elements per CTA only with one warp each");
  static_assert(C % VN == 0 && B % 4 == 0, "vector widths");
  extern __shared__ __align__(16) unsigned char raw[];
  unsigned char* sm = raw + (EPC > 1 ? (threadIdx.x / NE) * Y::bytes : 0);
  T* U = reinterpret_cast<T*>(sm + Y::oU);
  T* sF = reinterpret_cast<T*>(sm + Y::oF);
  T* sFp = reinterpret_cast<T*>(sm + Y::oFp);
  T* sIp = reinterpret_cast<T*>(sm + Y::oIp);
  int* sPv = reinterpret_cast<int*>(sm + Y::oPv);
  typename Key<T>::type* sKey = reinterpret_cast<typename Key<T>::type*>(sm + Y::oKey);
  T* sSl = reinterpret_cast<T*>(sm + Y::oSl);
  int* sSp = reinterpret_cast<int*>(sm + Y::oSp);
  int* sPhys = reinterpret_cast<int*>(sm + Y::oPhys);
  int* sEr = reinterpret_cast<int*>(sm + Y::oEr);
  int* sEc = reinterpret_cast<int*>(sm + Y::oEc);
  const int tid = EPC > 1 ? threadIdx.x % NE : threadIdx.x;
  const int g = G > 1 ? tid / TR : 0, rt = G > 1 ? tid - g * TR : tid;
  const int lane = threadIdx.x & 31, wr = rt >> 5;
  int rank = 0;
  if (CL > 1) rank = (int)cg::this_cluster().block_rank();
  const int gid = rank * G + g;
  const int e = CL > 1 ? blockIdx.x / CL : EPC > 1 ? blockIdx.x * EPC + threadIdx.x / NE : blockIdx.x;
  if (EPC > 1 && e >= E) return;   // whole warps, which meet no CTA barrier
  T* sSt = reinterpret_cast<T*>(sm + Y::oSt) + (size_t)g * N * SC;
  const double* D = Din + (size_t)e * N * N;
  auto bar_elem = [&]() {   // all threads of the element in this CTA
    if (NE == 32) __syncwarp();
    else __syncthreads();
  };
  auto bar_group = [&]() {   // the threads of one column group
    if (TR == 32) __syncwarp();
    else if (G == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(TR) : "memory");
  };
  // row scales: exponent field of each row's largest entry, a warp per row,
  // about 32 loads in flight per lane (one warp covers an L2 round trip alone)
  constexpr int LPR = (N + 31) / 32, RB = 32 / LPR, NW = NE / 32;
  for (int i0 = (tid >> 5) * RB; i0 < N; i0 += NW * RB) {
    double v[RB][LPR];
#pragma unroll
    for (int b = 0; b < RB; ++b)
#pragma unroll
      for (int q = 0; q < LPR; ++q)
        v[b][q] = i0 + b < N && lane + 32 * q < N ? __ldg(D + (size_t)(i0 + b) * N + lane + 32 * q) : 0.0;
#pragma unroll
    for (int b = 0; b < RB; ++b) {
      int m = 0;
#pragma unroll
      for (int q = 0; q < LPR; ++q) m = max(m, (int)((__double_as_longlong(v[b][q]) >> 52) & 0x7ff));
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0 && i0 + b < N) sEr[i0 + b] = m;
    }
  }
  for (int j = tid; j < CC; j += NE) sEc[j] = -100000;
  bar_elem();
  for (int i = tid; i < N; i += NE) {
    int m = sEr[i];
    if (m == 0 || m == 0x7ff) {   // zero, subnormal or non-finite rows
      double mx = 0.0;
      for (int j = 0; j < N; ++j) mx = fmax(mx, fabs(__ldg(D + (size_t)i * N + j)));
      m = 1022 - pow2_exp(pow2_inv_scale_r(mx));
    }
    sEr[i] = 1022 - m;
  }
  bar_elem();
  // column scales of this CTA's columns: NE / CC (or 1) threads per column
  {
    constexpr int parts = NE / CC > 0 ? NE / CC : 1;
    for (int t = tid; t < CC * parts; t += NE) {
      const int jl = t % CC, part = t / CC, col = rank * CC + jl;
      if (col >= N) continue;
      int m = -100000;
      bool odd = false;
      for (int i0 = part; i0 < N; i0 += 32 * parts) {
        double v[32];
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = i0 + q * parts < N ? __ldg(D + (size_t)(i0 + q * parts) * N + col) : 0.0;
#pragma unroll
        for (int q = 0; q < 32; ++q) {
          const unsigned long long mag = (unsigned long long)__double_as_longlong(v[q]) & 0x7fffffffffffffffull;
          if (mag == 0) continue;
          const int f = (int)(mag >> 52), e1 = f + sEr[i0 + q * parts];
          odd = odd || f == 0 || f == 0x7ff || e1 < 1 || e1 > 2046;
          m = max(m, e1);
        }
      }
      if (odd) {   // entries that leave the normal range: the products themselves
        double mx = 0.0;
        for (int i = 0; i < N; ++i) mx = fmax(mx, fabs(__ldg(D + (size_t)i * N + col) * pow2_d(sEr[i])));
        m = 100000 - pow2_exp(pow2_inv_scale_r(mx));
      }
      atomicMax(&sEc[jl], m);
    }
  }
  bar_elem();
  for (int j = tid; j < CC; j += NE) {
    const int m = sEc[j];   // largest exponent field, or 100000 - t from the products
    const int t = m == -100000 ? 0 : m > 50000 ? 100000 - m : 1022 - m;
    sEc[j] = t;
    if (rank * CC + j < N) cs[(size_t)e * N + rank * CC + j] = pow2_d(t);
  }
  if (rank == 0)
    for (int i = tid; i < N; i += NE) rs[(size_t)e * N + i] = pow2_d(sEr[i]);
  bar_elem();
  // the equilibrated block into registers through shared memory (converted
  // row by row, taken by columns); the converting loop stays rolled, since
  // every instruction here runs once per block and has to be fetched for it
  T a[R][C];
  int pos[R];
#pragma unroll
  for (int r = 0; r < R; ++r) pos[r] = rt + r * TR < N ? rt + r * TR : -1;
  {
    constexpr int LB = 16;
#pragma unroll 1
    for (int t0 = rt; t0 < N * C; t0 += LB * TR) {
      double v[LB];
#pragma unroll
      for (int q = 0; q < LB; ++q) {
        const int t = t0 + q * TR, i = t / C, col = gid * C + t % C;
        v[q] = t < N * C && col < N ? __ldg(D + (size_t)i * N + col) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < LB; ++q) {
        const int t = t0 + q * TR, i = t / C, j = t % C;
        if (t < N * C) sSt[i * SC + j] = scaled_entry<T>(v[q], sEr[i], sEc[g * C + j]);
      }
    }
    bar_elem();
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int j = 0; j < C; ++j) a[r][j] = pos[r] >= 0 ? sSt[(rt + r * TR) * SC + j] : (T)0;
    bar_elem();
  }
  if (CL > 1) cg::this_cluster().sync();   // every CTA runs before the first remote write
  bool bad = false;
  for (int p = 0; p < Y::NP; ++p) {
    const int k0 = p * B, kb = min(B, N - k0), par = p & 1;
    const bool own = GT == 1 || k0 / C == gid;
    T F[R][B];   // multipliers of this thread's rows
    T pa[R][B];  // the panel's columns
    if (own) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < B; ++s) { pa[r][s] = a[r][s]; F[r][s] = (T)0; }
      // one pass per pivot, not unrolled: the panel and its multipliers turn by
      // one place instead, so that the pivot column is always the first
#pragma unroll 1
      for (int s = 0; s < B; ++s) {
        const int k = k0 + s;
        if (s >= kb) {   // the padding of the last panel
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const T t = pa[r][0];
#pragma unroll
            for (int j = 1; j < B; ++j) { pa[r][j - 1] = pa[r][j]; F[r][j - 1] = F[r][j]; }
            pa[r][B - 1] = t;
            F[r][B - 1] = (T)0;
          }
          continue;
        }
        typename Key<T>::type key = 0;
        int bp = 0x7fffffff;
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (pos[r] >= k) {
            const typename Key<T>::type kr = pivot_key(pa[r][0]);
            if (bp == 0x7fffffff || kr > key || (kr == key && pos[r] < bp)) { key = kr; bp = pos[r]; }
          }
        warp_best(key, bp);
        T u[B];
        int prow = 0;
        if (WR == 1) {
          bool mine = false;
#pragma unroll
          for (int j = 0; j < B; ++j) u[j] = pa[0][j];
          prow = rt;
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (pos[r] == bp) {
              mine = true;
              prow = rt + r * TR;
#pragma unroll
              for (int j = 0; j < B; ++j) u[j] = pa[r][j];
            }
          const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
#pragma unroll
          for (int j = 0; j < B; ++j) u[j] = __shfl_sync(0xffffffffu, u[j], src);
          prow = __shfl_sync(0xffffffffu, prow, src);
        } else {
          const int s0 = (s & 1) * WR, sl = s0 + wr;
          if (lane == 0) {
            sKey[sl] = key;
            sSp[2 * sl] = bp;
          }
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (pos[r] == bp) {
              sSp[2 * sl + 1] = rt + r * TR;
#pragma unroll
              for (int j = 0; j < B; ++j) sSl[sl * B + j] = pa[r][j];
            }
          bar_group();
          typename Key<T>::type wk = 0;
          int wp = 0x7fffffff;
          if (lane < WR) {
            wk = sKey[s0 + lane];
            wp = sSp[2 * (s0 + lane)];
          }
          const int own_p = wp;
          warp_best(wk, wp);
          bp = wp;
          const int w = __ffs(__ballot_sync(0xffffffffu, own_p == bp)) - 1;
          const int sw = s0 + w;
          prow = sSp[2 * sw + 1];
#pragma unroll
          for (int j = 0; j < B; ++j) u[j] = sSl[sw * B + j];
        }
        bad = bad || bad_pivot(u[0], N);
        const T ip = (T)1 / u[0];
#pragma unroll
        for (int j = 1; j < B; ++j) u[j] *= ip;
        if (rt == 0) {   // the panel's pivots for the other phases and CTAs
#pragma unroll
          for (int c = 0; c < CL; ++c) {
            T* dIp = sIp;
            int* dPv = sPv;
            if (CL > 1) {
              dIp = cg::this_cluster().map_shared_rank(sIp, c);
              dPv = cg::this_cluster().map_shared_rank(sPv, c);
            }
            dIp[par * B + s] = ip;
            dPv[(par * 2 + 0) * B + s] = prow;
            dPv[(par * 2 + 1) * B + s] = bp;
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const bool piv = pos[r] == bp;
          const T f = pa[r][0];
#pragma unroll
          for (int j = 1; j < B; ++j) {
            pa[r][j - 1] = piv ? u[j] : fma(-f, u[j], pa[r][j]);
            F[r][j - 1] = F[r][j];
          }
          pa[r][B - 1] = piv ? ip : -f * ip;
          F[r][B - 1] = f;
          if (piv) pos[r] = k;
          else if (pos[r] == k) pos[r] = bp;
        }
      }
      // multipliers of the pivot rows, and of all rows for the other groups
#pragma unroll
      for (int c = 0; c < CL; ++c) {
        T* dFp = sFp;
        T* dF = sF;
        if (CL > 1) {
          dFp = cg::this_cluster().map_shared_rank(sFp, c);
          dF = cg::this_cluster().map_shared_rank(sF, c);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (pos[r] >= k0 && pos[r] < k0 + kb)
#pragma unroll
            for (int s = 0; s < B; ++s) dFp[(par * B + pos[r] - k0) * B + s] = F[r][s];
          if (GT > 1)
#pragma unroll
            for (int s = 0; s < B; ++s) dF[(par * B + s) * RT + rt + r * TR] = F[r][s];
        }
      }
    }
    if (GT > 1) {
      if (CL > 1) cg::this_cluster().sync();
      else bar_elem();
      if (!own) {
#pragma unroll
        for (int s = 0; s < B; ++s)
          if (s < kb) {
            const int prow = sPv[(par * 2 + 0) * B + s], lp = sPv[(par * 2 + 1) * B + s];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              if (pos[r] < 0) continue;
              if (rt + r * TR == prow) pos[r] = k0 + s;
              else if (pos[r] == k0 + s) pos[r] = lp;
            }
          }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int s = 0; s < B; ++s) F[r][s] = sF[(par * B + s) * RT + rt + r * TR];
      }
    }
    // the pivot rows to shared memory; their own entries restart from the
    // finished row s (0 - (-1) u_s), then take the later updates
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int sp = pos[r] - k0;
      if (sp >= 0 && sp < kb) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
          U[sp * CC + g * C + j] = a[r][j];
          a[r][j] = (T)0;
        }
#pragma unroll
        for (int s = 0; s < B; ++s) F[r][s] = s < sp ? (T)0 : s == sp ? (T)-1 : F[r][s];
      }
    }
    bar_elem();
    if (tid < kb) sPhys[k0 + tid] = sPv[(par * 2 + 0) * B + tid];
    for (int j = tid; j < CC; j += NE) {
      T u[B];
#pragma unroll
      for (int s = 0; s < B; ++s) {
        u[s] = (T)0;
        if (s < kb) {
          u[s] = U[s * CC + j];
#pragma unroll
          for (int t = 0; t < B; ++t)
            if (t < s) u[s] = fma(-sFp[(par * B + s) * B + t], u[t], u[s]);
          u[s] *= sIp[par * B + s];
        }
        U[s * CC + j] = u[s];
      }
    }
    bar_elem();
    // the other columns, in registers; the owner's panel moves to its end
    const T* Ug = U + g * C;
    if (own) {
#pragma unroll
      for (int j = B; j < C; j += VN) {
        T t[R][VN];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int q = 0; q < VN; ++q) t[r][q] = a[r][j + q];
#pragma unroll
        for (int s = 0; s < B; ++s) {
          T u[VN];
          unpack(*reinterpret_cast<const V*>(Ug + s * CC + j), u);
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < VN; ++q) t[r][q] = fma(-F[r][s], u[q], t[r][q]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int q = 0; q < VN; ++q) a[r][j + q - B] = t[r][q];
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < B; ++s) a[r][C - B + s] = pa[r][s];
    } else if (GT > 1) {
#pragma unroll
      for (int j = 0; j < C; j += VN)
#pragma unroll
        for (int s = 0; s < B; ++s) {
          T u[VN];
          unpack(*reinterpret_cast<const V*>(Ug + s * CC + j), u);
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < VN; ++q) a[r][j + q] = fma(-F[r][s], u[q], a[r][j + q]);
        }
    }
    // One warp meets no barrier in the next panel before it writes U again, and
    // its votes and shuffles order no memory.
    if (NE == 32) __syncwarp();
  }
  // a last group whose final columns are all padding still owes their turns
  const int turns = max(0, min(C / B, Y::NP - gid * (C / B)));
  bar_elem();   // sPhys complete
  // column-major inverse: column pivot_row[k], row pos
  W* out = Dinv + (size_t)e * N * N;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    int jj = j + turns * B;   // place of register j among the group's columns
    if (jj >= C) jj -= C;
    const int col = gid * C + jj;
    if (col < N) {
      const size_t o = (size_t)sPhys[col] * N;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (pos[r] >= 0) out[o + pos[r]] = (W)a[r][j];
    }
  }
  if (rt == 0 && bad) atomicMax(flag, flag_base + e + 1);
}

namespace {

// One launch (or, with prepare, the opt-in to its shared memory).
template <class T, class W, int N, int R, int G, int CL, int B, int EPC, int MINB>
cudaError_t reg_call(bool prepare, int E, const double* D, W* Dinv, double* rs, double* cs, int* flag, int base,
                     cudaStream_t s) {
  using Y = Lay<T, N, R, G, CL, B>;
  auto* k = factor_reg_kernel<T, W, N, R, G, CL, B, EPC, MINB>;
  if (prepare) return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(Y::bytes * EPC));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL > 1 ? E * CL : (E + EPC - 1) / EPC);
  cfg.blockDim = dim3(Y::NE * EPC);
  cfg.dynamicSmemBytes = Y::bytes * EPC;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CL > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, E, D, Dinv, rs, cs, flag, base);
}

// The block sizes 4 (P+1)^2 (quadrilaterals, P <= 5) and 5 (P+1)^3
// (hexahedra, P <= 3).  FP64 elements are 64-bit registers: panels of 4 and
// half the columns per thread from n = 100 on.  `few`: at most four blocks per
// SM, where one block's latency is the time and two warps of one row a lane take
// n = 36 from 154 to 101 us and n = 40 from 187 to 114; beyond, one warp of two
// rows a lane issues less (1000 blocks of n = 40 in 285 against 335 us, 4096 of
// n = 36 in 801 against 877).
template <class W>
cudaError_t reg_size32(bool prep, int n, int E, const double* D, W* Di, double* rs, double* cs, int* fl, int b,
                       cudaStream_t s) {
  switch (n) {
    case 4: return reg_call<float, W, 4, 1, 1, 1, 4, 4, 8>(prep, E, D, Di, rs, cs, fl, b, s);
    case 5: return reg_call<float, W, 5, 1, 1, 1, 8, 4, 8>(prep, E, D, Di, rs, cs, fl, b, s);
    case 16: return reg_call<float, W, 16, 1, 1, 1, 8, 4, 8>(prep, E, D, Di, rs, cs, fl, b, s);
    case 36: return reg_call<float, W, 36, 2, 1, 1, 4, 4, 3>(prep, E, D, Di, rs, cs, fl, b, s);
    case 40: return reg_call<float, W, 40, 2, 1, 1, 8, 4, 3>(prep, E, D, Di, rs, cs, fl, b, s);
    case 64: return reg_call<float, W, 64, 2, 1, 1, 8, 4, 2>(prep, E, D, Di, rs, cs, fl, b, s);
    case 100: return reg_call<float, W, 100, 1, 1, 1, 8, 1, 3>(prep, E, D, Di, rs, cs, fl, b, s);
    case 135: return reg_call<float, W, 135, 1, 1, 1, 8, 1, 2>(prep, E, D, Di, rs, cs, fl, b, s);
    case 144: return reg_call<float, W, 144, 1, 1, 1, 8, 1, 2>(prep, E, D, Di, rs, cs, fl, b, s);
    default: return reg_call<float, W, 320, 1, 1, 5, 8, 1, 2>(prep, E, D, Di, rs, cs, fl, b, s);
  }
}
cudaError_t reg_size64(bool prep, int n, int E, bool few, const double* D, double* Di, double* rs, double* cs,
                       int* fl, int b, cudaStream_t s) {
  switch (n) {
    case 4: return reg_call<double, double, 4, 1, 1, 1, 4, 4, 8>(prep, E, D, Di, rs, cs, fl, b, s);
    case 5: return reg_call<double, double, 5, 1, 1, 1, 4, 4, 8>(prep, E, D, Di, rs, cs, fl, b, s);
    case 16: return reg_call<double, double, 16, 1, 1, 1, 4, 4, 4>(prep, E, D, Di, rs, cs, fl, b, s);
    case 36:
      return few ? reg_call<double, double, 36, 1, 1, 1, 4, 1, 6>(prep, E, D, Di, rs, cs, fl, b, s)
                 : reg_call<double, double, 36, 2, 1, 1, 4, 4, 2>(prep, E, D, Di, rs, cs, fl, b, s);
    case 40:
      return few ? reg_call<double, double, 40, 1, 1, 1, 4, 1, 6>(prep, E, D, Di, rs, cs, fl, b, s)
                 : reg_call<double, double, 40, 2, 1, 1, 4, 4, 2>(prep, E, D, Di, rs, cs, fl, b, s);
    case 64: return reg_call<double, double, 64, 1, 1, 1, 4, 1, 5>(prep, E, D, Di, rs, cs, fl, b, s);
    case 100: return reg_call<double, double, 100, 1, 2, 1, 4, 1, 1>(prep, E, D, Di, rs, cs, fl, b, s);
    case 135: return reg_call<double, double, 135, 1, 2, 1, 4, 1, 1>(prep, E, D, Di, rs, cs, fl, b, s);
    case 144: return reg_call<double, double, 144, 1, 2, 1, 4, 1, 1>(prep, E, D, Di, rs, cs, fl, b, s);
    default: return reg_call<double, double, 320, 1, 1, 4, 4, 1, 1>(prep, E, D, Di, rs, cs, fl, b, s);
  }
}

cudaError_t reg_prec(bool prep, int prec, int n, int E, int sms, const double* D, void* Di, double* rs, double* cs,
                     int* fl, int b, cudaStream_t s) {
  if (prec == PMG_PREC_FP64) return reg_size64(prep, n, E, E <= 4 * sms, D, (double*)Di, rs, cs, fl, b, s);
  if (prec == PMG_PREC_BF16R) return reg_size32<__nv_bfloat16>(prep, n, E, D, (__nv_bfloat16*)Di, rs, cs, fl, b, s);
  return reg_size32<float>(prep, n, E, D, (float*)Di, rs, cs, fl, b, s);
}

}  // namespace

void launch_factor(const Ctx& c, LevelDev& L, int level, int prec, int* flag, cudaStream_t s) {
  const int base = level * c.E;   // the flag holds 1 + level E + element of the highest bad block
  const int C = factor_cluster_size(L.n, prec);
  if (C > 0) {
    launch_factor_cluster(c, L, level, prec, C, flag, s);
    return;
  }
  reg_prec(false, prec, L.n, c.E, c.sms, L.Dfull, L.Dinv, L.rs, L.cs, flag, base, s);
}

// Opt the kernels of every level into the shared memory they need (once,
// outside any stream capture).
cudaError_t prepare_kernels(const Ctx& c) {
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    const int n = c.lev[l].n, C = factor_cluster_size(n, c.cfg.block_prec);
    const cudaError_t e = C > 0 ? prepare_factor_cluster(n, c.cfg.block_prec, C)
                                : reg_prec(true, c.cfg.block_prec, n, c.E, c.sms, nullptr, nullptr, nullptr, nullptr,
                                           nullptr, 0, nullptr);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pmg
