// k3_blocks.cu -- application of the element-Jacobi blocks on hexahedra
// (Section 2.4, eq. smoothing_element_jacobi, d = 3): x = cs .* (D^-1 (rs .* r))
// with the factored inverse (column-major); one thread per solution point forms
// its point's five rows, so the threads of an element read every column
// contiguously.  Bound by the stream of the inverses (n^2 entries per element,
// read once).  Loaded into registers inside the product loop, the columns in
// flight are what a thread can hold (ten), which leaves HBM half idle at
// n = 320; here KC columns of each element at a time go through a ring of S
// stages in shared memory with 16-byte asynchronous copies.  The columns are
// used in the order of the register loop (kept for inverses that L2 holds), so
// the sums are the same bit for bit.
// Measured on one GB300, FP32, us (before, columns in registers): 960 elements of
// n = 320 97.6 -> 68.4 (393 MB, 5.7 TB/s), 2304 of n = 135 42.9 -> 37.6.  Inside the residual-and-update
// kernel (k3_residual.cu) the ring takes the shared memory that its resident
// CTAs need (n = 320: 104 -> 158 us), so that keeps its columns in registers.
// Assembly and factorisation: k_assemble.cu, k_factor.cu.
#include "pmg_internal.h"

namespace pmg {

// One element's chunk of KC columns starts at any multiple of the entry size
// when its columns are not multiples of 16 bytes (n = 135): it is copied from
// the 16-byte boundary at or below its first entry, and pieces that would pass
// the array's end are read entry by entry.
static __device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
static __device__ __forceinline__ void async_wait() {   // all but the N newest groups have landed
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <class W, int n, int EPB, int KC, int S>
struct BlockStream {
  static constexpr int colB = n * (int)sizeof(W), chunkB = KC * colB, NC = (n + KC - 1) / KC;
  static constexpr bool aligned = chunkB % 16 == 0 && (n * colB) % 16 == 0;
  static constexpr int segB = (chunkB + (aligned ? 0 : 15) + 15) / 16 * 16;   // one element's chunk
  static constexpr int stageB = segB * EPB;
  static constexpr size_t bytes = (size_t)S * stageB;

  // Chunk c of the elements e0 .. e0 + ne - 1 into its stage (one group per
  // call, empty past the last chunk).
  static __device__ __forceinline__ void issue(unsigned char* ring, const W* __restrict__ Dinv, int E, int e0, int ne,
                                               int c) {
    if (c < NC) {
      constexpr int pieces = segB / 16;
      unsigned char* st = ring + (size_t)(c % S) * stageB;
      const size_t total = (size_t)E * n * colB;
      for (int t = threadIdx.x; t < ne * pieces; t += blockDim.x) {
        const int le = t / pieces, p = t - le * pieces;
        const size_t off = (size_t)(e0 + le) * n * colB + (size_t)c * chunkB;   // first byte of the chunk
        const size_t src = (aligned ? off : off & ~(size_t)15) + 16 * (size_t)p;
        const size_t end = off + (size_t)(c == NC - 1 ? (n - c * KC) * colB : chunkB);
        unsigned char* dst = st + le * segB + 16 * p;
        if (src >= end) continue;
        if (aligned || src + 16 <= total) {
          const unsigned int d = (unsigned int)__cvta_generic_to_shared(dst);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d),
                       "l"(reinterpret_cast<const unsigned char*>(Dinv) + src)
                       : "memory");
        } else {
          for (size_t b = src; b < total; b += sizeof(W))
            *reinterpret_cast<W*>(dst + (b - src)) = Dinv[b / sizeof(W)];
        }
      }
    }
    async_commit();
  }
  // Column 0 of chunk c of local element le.
  static __device__ __forceinline__ const W* columns(const unsigned char* ring, int e0, int le, int c) {
    const unsigned char* s = ring + (size_t)(c % S) * stageB + le * segB;
    if (!aligned) s += ((size_t)(e0 + le) * n * colB + (size_t)c * chunkB) & 15;
    return reinterpret_cast<const W*>(s);
  }
};

// Elements per CTA (one or two warps), columns per chunk and stages.
template <int P>
struct ApplyEPB3 {
  static constexpr int value = P == 0 ? 64 : P == 1 ? 8 : P == 2 ? 2 : 1;
};
constexpr int kStages3 = 4;
template <int P>
struct StreamCols3 {
  static constexpr int value = P == 1 ? 5 : 4;
};
template <class W, int P>
using Stream3 =
    BlockStream<W, 5 * (P + 1) * (P + 1) * (P + 1), ApplyEPB3<P>::value, StreamCols3<P>::value, kStages3>;
template <class W, int P>
constexpr size_t stream3_bytes() { return P == 0 ? 0 : Stream3<W, P>::bytes; }   // P = 0 has no ring

template <class W, int P, bool STREAM>
__global__ void __launch_bounds__(64) apply3_kernel(int E, const W* __restrict__ Dinv, const double* __restrict__ rs,
                                                    const double* __restrict__ cs, const double* __restrict__ r,
                                                    double* __restrict__ x, int accumulate) {
  constexpr int N = (P + 1) * (P + 1) * (P + 1), n = 5 * N;
  constexpr int EPB = ApplyEPB3<P>::value;
  using Acc = typename Blk<W>::acc;
  using Stream = Stream3<W, P>;
  extern __shared__ __align__(16) unsigned char ring[];
  const int e0 = blockIdx.x * EPB, ne = min(EPB, E - e0);
  if (STREAM)
    for (int c = 0; c < kStages3 - 1; ++c) Stream::issue(ring, Dinv, E, e0, ne, c);
  __shared__ Acc sr[EPB][n];
  const int le = threadIdx.x / N, pt = threadIdx.x - le * N;
  const int e = blockIdx.x * EPB + le;
  const bool active = (le < EPB) && (e < E);
  const size_t plane = (size_t)E * N;
  if (active) {
#pragma unroll
    for (int v = 0; v < 5; ++v)
      sr[le][v * N + pt] = scaled_in<W>(r[v * plane + (size_t)e * N + pt], rs[(size_t)e * n + v * N + pt]);
  }
  Acc acc[5] = {0, 0, 0, 0, 0};
  if (STREAM) {
#pragma unroll 1
    for (int c = 0; c < Stream::NC; ++c) {
      async_wait<kStages3 - 2>();
      __syncthreads();   // chunk c (and, the first time, sr) visible; the stage of chunk c - 1 free
      Stream::issue(ring, Dinv, E, e0, ne, c + kStages3 - 1);
      if (active) {
        const W* Dm = Stream::columns(ring, e0, le, c) + pt;
        const Acc* rk = sr[le] + c * StreamCols3<P>::value;
        const int nk = min(StreamCols3<P>::value, n - c * StreamCols3<P>::value);
#pragma unroll
        for (int kk = 0; kk < StreamCols3<P>::value; ++kk) {
          if (kk < nk) {
            const Acc rr = rk[kk];
#pragma unroll
            for (int v = 0; v < 5; ++v) acc[v] = fma(blk_val(Dm[kk * n + v * N]), rr, acc[v]);
          }
        }
      }
    }
    if (!active) return;
  } else {
    __syncthreads();
    if (!active) return;
    const W* Dm = Dinv + (size_t)e * n * n + pt;
#pragma unroll 10
    for (int k = 0; k < n; ++k) {
      const Acc rr = sr[le][k];
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] = fma(blk_val(__ldg(Dm + (size_t)k * n + v * N)), rr, acc[v]);
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double xv = scaled_out<W>(acc[v], cs[(size_t)e * n + v * N + pt]);
    const size_t o = v * plane + (size_t)e * N + pt;
    if (accumulate) x[o] += xv;
    else x[o] = xv;
  }
}

// The ring pays where the inverses do not stay in the 129 MB L2 and its CTAs, whose
// number on an SM the shared memory limits, run in one wave.  More waves cost FP64
// inverses more than the ring gains, FP32 ones as much until n = 320 fills one and
// a half; BF16 inverses, and those of n = 40 in FP32, win in any number.  Inverses
// that L2 holds, applied again and again: 73 MB (FP32, n = 135) 37 us through the
// ring and 34 through registers, 52 MB (FP64, n = 320) 120 and 86.  us from
// memory, ring / registers (number of waves above one):
//   FP64 n = 320: 124 / 215 (102 MB), 172 / 225 (597), 296 / 234 (819, 2), 529 / 491
//     (1884, 4); n = 135: 94 / 114 (146), 184 / 131 (400, 2), 433 / 365 (1312, 5);
//     n = 40: 59 / 57 (102, 2), 130 / 101 (346): never;
//   FP32 n = 320: 56 / 108 (140), 126 / 134 (614), 147 / 139 (655, 2), 187 / 199
//     (1065, 2), 271 / 304 (1638, 3); n = 135: 48 / 60 (126), 70 / 69 (219), 87 /
//     75 (255, 2), 145 / 144 (656, 3); n = 40: 41 / 41 (88, 2), 58 / 62 (173, 3);
//   BF16 n = 320: 56 / 97 (149), 167 / 220 (819, 2); n = 135: 46 / 57 (100), 99 /
//     113 (328, 2); n = 40: 42 / 55 (86, 2).
template <class W, int P>
constexpr bool has_ring() { return P > 1 || (P == 1 && sizeof(W) < 8); }

template <class W>
static void apply3_dispatch(const Ctx& c, const LevelDev& L, const double* r, double* x, int acc, cudaStream_t s) {
  const W* Dinv = (const W*)L.Dinv;
#define PMG_AP3(PP)                                                                                          \
  do {                                                                                                       \
    constexpr int N = (PP + 1) * (PP + 1) * (PP + 1), epb = ApplyEPB3<PP>::value;                            \
    const int threads = (epb * N + 31) / 32 * 32, blocks = (c.E + epb - 1) / epb;                            \
    if (has_ring<W, PP>() && L.ring)                                                                         \
      apply3_kernel<W, PP, has_ring<W, PP>()>                                                                \
          <<<blocks, threads, stream3_bytes<W, PP>(), s>>>(c.E, Dinv, L.rs, L.cs, r, x, acc);                \
    else                                                                                                     \
      apply3_kernel<W, PP, false><<<blocks, threads, 0, s>>>(c.E, Dinv, L.rs, L.cs, r, x, acc);              \
  } while (0)
  switch (L.P) {
    case 0: PMG_AP3(0); break;
    case 1: PMG_AP3(1); break;
    case 2: PMG_AP3(2); break;
    default: PMG_AP3(3); break;
  }
#undef PMG_AP3
}

// Shared memory of the ring and whether a level's apply uses it (above).
template <class W, int P>
static cudaError_t prepare_ring(const Ctx& c, LevelDev& L) {
  L.ring = false;
  if (!has_ring<W, P>()) return cudaSuccess;
  constexpr int N = (P + 1) * (P + 1) * (P + 1), epb = ApplyEPB3<P>::value;
  auto* k = apply3_kernel<W, P, has_ring<W, P>()>;
  constexpr size_t bytes = stream3_bytes<W, P>();
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  int resident = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k, (epb * N + 31) / 32 * 32, bytes);
  const long long blocks = (c.E + epb - 1) / epb, wave = (long long)resident * c.sms;
  const bool any = sizeof(W) == 2 || P == 1 || (sizeof(W) == 4 && P == 3 && 2 * blocks >= 3 * wave);
  L.ring = sizeof(W) * c.E * L.n * L.n > (size_t)80000000 && (blocks <= wave || any);
  return e;
}
template <class W>
static cudaError_t prepare3(const Ctx& c, LevelDev& L) {
  switch (L.P) {
    case 0: return prepare_ring<W, 0>(c, L);
    case 1: return prepare_ring<W, 1>(c, L);
    case 2: return prepare_ring<W, 2>(c, L);
    default: return prepare_ring<W, 3>(c, L);
  }
}
cudaError_t prepare_apply3(Ctx& c) {
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    const cudaError_t e = c.cfg.block_prec == PMG_PREC_FP64    ? prepare3<double>(c, c.lev[l])
                          : c.cfg.block_prec == PMG_PREC_BF16R ? prepare3<__nv_bfloat16>(c, c.lev[l])
                                                               : prepare3<float>(c, c.lev[l]);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_apply3(const Ctx& c, const LevelDev& L, int prec, const double* r, double* x, int accumulate,
                   cudaStream_t s) {
  if (prec == PMG_PREC_FP64) apply3_dispatch<double>(c, L, r, x, accumulate, s);
  else if (prec == PMG_PREC_BF16R) apply3_dispatch<__nv_bfloat16>(c, L, r, x, accumulate, s);
  else apply3_dispatch<float>(c, L, r, x, accumulate, s);
}

}  // namespace pmg
