// fwi_conv_tc.cu -- the 3x3x3 convolutions of the learned preconditioner on the
// fifth-generation tensor cores (tcgen05, sm_103a), as implicit GEMMs with BF16 operands
// and FP32 accumulators in tensor memory (TMEM):
//
//   forward         y[co][p]  = act(b[co] + sum_t sum_ci w[co][ci][t] x[ci][p + off(t)])
//   backward data   dx[ci][p] = sum_t sum_co w[co][ci][t] dy[co][p - off(t)]
//   weight gradient dw[co][ci][t] = sum_p dy[co][p] x[ci][p + off(t)], db[co] = sum_p dy[co][p]
//
// t one of the 27 taps (kz, ky, kx; kx fastest), out-of-grid taps reading zero. Products
// of BF16 values are exact; the FP32 gradients of the backward passes enter as three BF16
// parts (hi, lo, lo2 with hi + lo + lo2 = dy to 2^-24), so their products stay exact too.
//
// All three read their activations from a channel-group-major copy src[g][z][y][x][8]
// (groups of 8 channels, zero past the real ones): a TMA box of a tile of 8 (x) x 16 (y)
// voxels of a plane with its halo lands in shared memory as [g][18][10][8], zero outside
// the grid, and the 8 x-voxels of a row at any tap shift are one 128-byte core matrix of
// the no-swizzle canonical layouts (8 rows of 16 bytes stored contiguously; LBO is the
// byte stride between core matrices along K and SBO along M or N, in K-major and MN-major
// operands). So the taps are shifted views of the box: no thread gathers anything. One
// elected lane per warp issues tcgen05.mma and commits them to mbarriers, a warp per plane
// (forward, data) or per tap (weight gradient); another issues the copies; the epilogue reads
// the accumulators with tcgen05.ld.
//
// Every mbarrier wait is bounded (about a second). A block whose wait gives up waits
// (bounded) for what it issued, writes NaN to its outputs (so the caller's loss turns
// non-finite) and frees its TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "fwi_conv_tc.h"
#include "fwi_internal.h"  // kSms

namespace fwi_tc {
namespace {

using fwi::kSms;
constexpr int kM = 128;           // MMA M: the voxels of a tile, or the gradient rows of the weight gradient
constexpr int kMaxN = 256;        // output channels per block (MMA N <= 256)
constexpr int kSmPerSM = 233472;  // shared memory of an SM (228 KB); 1 KB more is reserved per block
constexpr int kSmBlock = 230400;  // dynamic shared memory a block can have beside 2 KB of static
constexpr int kTmemCols = 512;    // TMEM columns of an SM
constexpr long long kWaitCycles = 2000000000LL;  // about a second

constexpr int kTX = 8, kTY = 16;              // tile of one plane (x, y)
constexpr int kBX = kTX + 2, kBY = kTY + 2;   // staged box with the halo
constexpr int kRowBytes = kBX * 16;           // one staged row of a group: 160 bytes
constexpr int kGroupBytes = kRowBytes * kBY;  // one staged group of a plane: 2880 bytes

__device__ __forceinline__ unsigned su32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor, no swizzle: start, leading (K) and stride (M/N) byte
// offsets in 16-byte units, descriptor version 1 (bit 46). Shared addresses fit the 14-bit
// field, so a view at a byte offset is the descriptor plus offset / 16.
__device__ __forceinline__ uint64_t smem_desc(unsigned addr, unsigned lbo, unsigned sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}
// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and B
// (bits 7-9, 10-12 = 1), N / 8 at bit 17, M / 16 at bit 24; both operands K-major (a caller
// sets bit 15 for an MN-major A, bit 16 for an MN-major B)
__host__ __device__ constexpr uint32_t instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
}

__device__ __forceinline__ void bar_init(uint64_t *b, int count = 1) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t *b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_done(uint64_t *b, unsigned parity) {
  unsigned d;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(d)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return d != 0;
}
__device__ __forceinline__ bool bar_wait(uint64_t *b, unsigned parity) {
  if (bar_done(b, parity)) return true;
  const long long t0 = clock64();
  while (!bar_done(b, parity))
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}
// one thread of a converged warp, by a predicate the compiler knows to be single: MMAs issued
// under it take their descriptors from uniform registers (issued under threadIdx.x == 0 they
// cost about 45 clocks each, whatever their size)
__device__ __forceinline__ bool elect_one() {
  unsigned e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}
// D (TMEM columns at d) (+)= A B, A in shared memory (descriptor) or TMEM (column address). A
// descriptor comes as its two halves: a view at a byte offset differs in the low half only
// (start address field), so the issuing thread's arithmetic stays 32-bit.
__device__ __forceinline__ void mma_ss(unsigned d, unsigned alo, unsigned ahi, unsigned blo, unsigned bhi, uint32_t idesc,
                                       unsigned acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n\t}" ::"r"(d),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_ts(unsigned d, unsigned a, unsigned blo, unsigned bhi, uint32_t idesc, unsigned acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 b, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, p;\n\t}" ::"r"(d),
      "r"(a), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc)
      : "memory");
}
// the barrier completes when every MMA this thread issued so far has
__device__ __forceinline__ void mma_commit(uint64_t *b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void tmem_alloc(unsigned *slot, int cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(unsigned tmem, int cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t r[16], unsigned a) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(a));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// max(f, 0) that keeps a NaN (fmaxf would return 0, and a tile given up would look like zeros)
__device__ __forceinline__ float relu_nan(float f) {
  float r;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(f));
  return r;
}
// 16 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_st16(unsigned a, const uint4 v[4]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(a),
      "r"(v[0].x), "r"(v[0].y), "r"(v[0].z), "r"(v[0].w), "r"(v[1].x), "r"(v[1].y), "r"(v[1].z), "r"(v[1].w),
      "r"(v[2].x), "r"(v[2].y), "r"(v[2].z), "r"(v[2].w), "r"(v[3].x), "r"(v[3].y), "r"(v[3].z), "r"(v[3].w)
      : "memory");
}

// a plane's halo box of a tile: x and the 8 channels of a group form one row of 80 elements
// (the inner coordinate 8 (x0 - 1) is a multiple of 16 bytes), then y, z and the groups
__device__ __forceinline__ void tma_box(void *dst, const CUtensorMap *tm, int x0, int y0, int z, int g0, uint64_t *b) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(su32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(8 * (x0 - 1)), "r"(y0 - 1), "r"(z), "r"(g0), "r"(su32(b))
      : "memory");
}
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, uint64_t *b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   su32(dst)),
               "l"(src), "r"(bytes), "r"(su32(b))
               : "memory");
}

// the three BF16 parts of an FP32 value, and the pattern of its part s
__device__ __forceinline__ void split3(float v, uint16_t h[3]) {
#pragma unroll
  for (int s = 0; s < 3; s++) {
    h[s] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    v -= __uint_as_float((uint32_t)h[s] << 16);
  }
}
__device__ __forceinline__ uint4 pack8(const uint16_t h[8]) {
  return make_uint4((uint32_t)h[0] | (uint32_t)h[1] << 16, (uint32_t)h[2] | (uint32_t)h[3] << 16,
                    (uint32_t)h[4] | (uint32_t)h[5] << 16, (uint32_t)h[6] | (uint32_t)h[7] << 16);
}

// The copies that a convolution needs before its MMAs are one launch: its blocks share out the
// source's and the weights' (or the gradient's) part. At 17 x 33 x 33 voxels, where each of them
// takes 2 to 4 us, launches of their own took 8 % of a training sample (1000 against 920 us).

// src[g][p][e] = x[8 g + e][p] (zero for channels >= cin), g = block / nx
__device__ __forceinline__ void group_major_block(const uint16_t *__restrict__ x, int64_t nv, int cin,
                                                  uint16_t *__restrict__ src, int block, int nx) {
  const int g = block / nx;
  const int n = cin - 8 * g;
  for (int64_t p = (int64_t)(block - g * nx) * 256 + threadIdx.x; p < nv; p += (int64_t)nx * 256) {
    const uint16_t *q = x + 8 * g * nv + p;
    uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int e = 0; e < 8; e++)
      if (e < n) v[e >> 1] |= (uint32_t)__ldg(q + e * nv) << (16 * (e & 1));
    *reinterpret_cast<uint4 *>(src + ((int64_t)g * nv + p) * 8) = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

// the split gradient in group-major form: channel s cop + co of src is part s of dy[co], cop
// the channels rounded up to 8; zero for co >= cout and for groups past 3 cop / 8. A thread
// reads 8 channels of a voxel once and writes their three parts. g = block / nx of cop / 8.
__device__ __forceinline__ void split_group_block(const float *__restrict__ dy, int64_t nv, int cout, int cop, int G,
                                                  uint16_t *__restrict__ src, int block, int nx) {
  const int gq = cop / 8, g = block / nx;
  for (int64_t p = (int64_t)(block - g * nx) * 256 + threadIdx.x; p < nv; p += (int64_t)nx * 256) {
    uint16_t h[3][8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
      uint16_t t[3];
      split3(8 * g + e < cout ? __ldg(dy + (int64_t)(8 * g + e) * nv + p) : 0.f, t);
#pragma unroll
      for (int s = 0; s < 3; s++) h[s][e] = t[s];
    }
#pragma unroll
    for (int s = 0; s < 3; s++) *reinterpret_cast<uint4 *>(src + ((int64_t)(s * gq + g) * nv + p) * 8) = pack8(h[s]);
    if (g == 0)
      for (int z = 3 * gq; z < G; z++) *reinterpret_cast<uint4 *>(src + ((int64_t)z * nv + p) * 8) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime
using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_tiled() {
  static const EncodeTiled fn = []() -> EncodeTiled {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<EncodeTiled>(p);
  }();
  return fn;
}

// tensor map of a group-major copy as (x and 8 channels: 8 W, H, D, G) BF16; boxes of one
// plane, gbox groups: (80, 18, 1, gbox), zero outside the grid
cudaError_t box_map(CUtensorMap *tm, uint16_t *src, int D, int H, int W, int G, int gbox) {
  const EncodeTiled enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  std::memset(tm, 0, sizeof(*tm));
  const cuuint64_t dims[4] = {(cuuint64_t)W * 8, (cuuint64_t)H, (cuuint64_t)D, (cuuint64_t)G};
  const cuuint64_t pitch[3] = {(cuuint64_t)W * 16, (cuuint64_t)W * H * 16, (cuuint64_t)W * H * D * 16};
  const cuuint32_t box[4] = {kBX * 8, kBY, 1, (cuuint32_t)gbox};
  const cuuint32_t step[4] = {1, 1, 1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, src, dims, pitch, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

// ---- forward and backward data. A block owns `planes` consecutive planes of an 8 x 16 tile
// (one accumulator of M = 128 voxels x nt_n channels each) and up to 256 GEMM output channels.
// The reduction runs pass by pass over gp channel groups and, in a pass, tap by tap: per
// (pass, tap) the weights (nt_n x 8 gp BF16, K-major) stream, `taps` taps per copy, through a
// ring of buffers, and each pair of groups is one MMA per plane, on views of the planes' boxes.
//
// Issuing an MMA costs its thread 50 to 150 clocks of descriptor arithmetic and moves to
// uniform registers (measured), more than an MMA of N = 32 runs (40 clocks): so warp p issues
// the MMAs of plane p, and the four chains keep the tensor pipe fed. Warp 4 copies, warps 5 to 8 write the results.
//
// Bound: in the MMA phase the operands' shared-memory reads (M = 128, K = 16: 4 KB of A for
// any N); the epilogue's stores (8 voxels of a row per channel) overlap it across the blocks
// of an SM and, with two accumulator sets, beside the next tile's MMAs. Several planes share each weight copy and two of three halo planes: with
// one plane a block, 28 -> 28 channels moved 90 KB through L2 per 128 voxels, 27 KB now.
// Measured at 65 x 129 x 129 voxels, whole calls with their copies: forward 28 -> 28 262 -> 143
// us, backward data 28 -> 84 1600 -> 519 us (one thread issuing for one plane a block before).
// ncu at 32 -> 32, forward: 112 us, tensor pipe 27 % (11 % before), 36 M warp instructions (87 M).
constexpr int kTileThreads = 288;
constexpr int kRingB = 4;      // most weight copies in flight
constexpr int kMaxPlanes = 4;  // output planes of a block
constexpr int kMaxBox = 2;     // box buffers (passes in flight)
// blocks of 288 threads that an SM's registers hold, forward (85 registers a thread) and backward data
// (72; held to 66 by a launch bound of three blocks it is up to 2.5 % slower). With three assumed for
// the forward, a grid had 456 blocks of which 304 ran, then 152 alone with a third of the tiles: 8 -> 16
// channels at 65 x 129 x 129 voxels 193 us, 97 with two; 28 -> 2 at 33 x 65 x 65 36.9 and 31.3.
constexpr int kTileBlocks[2] = {2, 3};

struct TileShape {
  int nt_n, ntiles;  // GEMM output channels per block, N tiles
  int gp, npass, G;  // groups per pass, passes, groups of the source (even)
  int planes, nbox;  // output planes per block, box buffers
  int taps, ring;    // taps per weight copy (1, 3 or 9), weight buffers
  int nacc;          // accumulator sets (2: a tile's epilogue runs beside the next tile's MMAs)
  int cols, smem;    // TMEM columns, dynamic shared memory
  int64_t tiles;     // (x, y) tiles x plane chunks x N tiles
  int grid;          // blocks
};

// weight chunks: for N tile nt, pass ps, tap t: nt_n x (gp x 8) K-major, core (kg, ng) at
// kg * (nt_n / 8) * 128 + ng * 128, i.e. 16 bytes (8 source channels) per (kg, n) in order.
// Source channel c = 8 (ps gp + kg) + kk; forward: w[n][c][t]; backward: c = s cop + co, w[co][n][t]
template <bool BWD>
__device__ __forceinline__ void pack_block(const uint16_t *__restrict__ w, int n_rows, int n_red, int cop, const TileShape &ts,
                                           uint16_t *__restrict__ out, int block, int nblocks) {
  const int64_t total = (int64_t)ts.ntiles * ts.npass * 27 * ts.gp * ts.nt_n;
  for (int64_t i = (int64_t)block * 256 + threadIdx.x; i < total; i += (int64_t)nblocks * 256) {
    const int r = (int)(i / ts.nt_n), q = r / ts.gp;  // (tile, pass, tap, kg), (tile, pass, tap)
    const int kg = r - q * ts.gp, t = q % 27, ps = q / 27 % ts.npass, nt = q / 27 / ts.npass;
    const int n = nt * ts.nt_n + (int)(i - (int64_t)r * ts.nt_n), c0 = 8 * (ps * ts.gp + kg);
    uint16_t h[8];
#pragma unroll
    for (int kk = 0; kk < 8; kk++) {
      const int c = c0 + kk;
      if (!BWD) {
        h[kk] = n < n_rows && c < n_red ? __ldg(w + ((int64_t)n * n_red + c) * 27 + t) : (uint16_t)0;
      } else {
        const int part = c / cop, co = c - part * cop;
        h[kk] = n < n_rows && part < 3 && co < n_red ? __ldg(w + ((int64_t)co * n_rows + n) * 27 + t) : (uint16_t)0;
      }
    }
    *reinterpret_cast<uint4 *>(out + i * 8) = pack8(h);
  }
}

// the copies of a forward (x) or backward-data (dy) convolution: blocks below nsrc the source,
// the others the weights
template <bool BWD>
__global__ void __launch_bounds__(256) tile_prep_kernel(const void *__restrict__ in, int64_t nv, int n_red, int cop,
                                                        const uint16_t *__restrict__ w, int n_rows, TileShape ts,
                                                        uint16_t *__restrict__ src, uint16_t *__restrict__ wp, int nx,
                                                        int nsrc) {
  const int b = blockIdx.x;
  if (b >= nsrc) pack_block<BWD>(w, n_rows, n_red, cop, ts, wp, b - nsrc, gridDim.x - nsrc);
  else if (BWD) split_group_block(static_cast<const float *>(in), nv, n_red, cop, ts.G, src, b, nx);
  else group_major_block(static_cast<const uint16_t *>(in), nv, n_red, src, b, nx);
}

template <bool BWD>
__global__ void __launch_bounds__(kTileThreads, 2)
    tile_conv_kernel(const __grid_constant__ CUtensorMap tm, const uint16_t *__restrict__ wpack,
                     const float *__restrict__ bias, int n_out, TileShape ts, int D, int H, int W, int relu,
                     void *__restrict__ yout) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t loaded[kRingB], done[kRingB], box_full[kMaxBox][kMaxPlanes + 2], box_free[kMaxBox], acc_full[2],
      acc_free[2], fin;
  __shared__ unsigned tslot;
  __shared__ float sbias[kMaxN];
  const int nt_n = ts.nt_n, gp = ts.gp, P = ts.planes, nbox = ts.nbox, npass = ts.npass, nacc = ts.nacc;
  const int plane_bytes = kGroupBytes * gp, box_bytes = plane_bytes * (P + 2);
  const int t_bytes = nt_n * gp * 16;  // one tap's weights
  const int taps = ts.taps, ring = ts.ring, b_bytes = t_bytes * taps;
  unsigned char *sb = sm + nbox * box_bytes;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int ntx = (W + kTX - 1) / kTX, txy = ntx * ((H + kTY - 1) / kTY), nz = (D + P - 1) / P;
  const unsigned lbo_b = (unsigned)(nt_n / 8) * 128u;
  const int per = 27 / taps, nch = npass * per;  // weight copies per pass, in all
  // tile t of the grid: N tile, plane chunk, (x, y) tile
  struct Tile {
    int nt, z0, np, x0, y0;
  };
  auto tile_at = [&](int64_t t) {
    const int xy = (int)(t % txy), zc = (int)(t / txy % nz);
    return Tile{(int)(t / txy / nz), zc * P, min(P, D - zc * P), (xy % ntx) * kTX, (xy / ntx) * kTY};
  };

  if (tid == 0) {
    for (int i = 0; i < kRingB; i++) {
      bar_init(&loaded[i]);
      bar_init(&done[i], P);
    }
    for (int b = 0; b < nbox; b++) {
      for (int i = 0; i < P + 2; i++) bar_init(&box_full[b][i]);
      bar_init(&box_free[b], P);
    }
    for (int i = 0; i < 2; i++) {
      bar_init(&acc_full[i], P);
      bar_init(&acc_free[i], 4);
    }
    bar_init(&fin, P);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tslot, ts.cols);
  fence_before();
  __syncthreads();
  fence_after();
  const unsigned tmem = tslot;

  const bool one = elect_one();
  if (warp == 4 && one) {  // copies: the planes' boxes pass by pass, the weight copies in order
    bool ok = true;
    int it = 0, boxes = 0;  // tiles done, boxes issued (all passes of all tiles in order)
    int64_t bt = blockIdx.x;  // tile and pass of the next box
    int bp = 0;
    auto issue_box = [&]() {
      const Tile t = tile_at(bt);
      const int b = boxes % nbox;
      if (boxes >= nbox && !bar_wait(&box_free[b], ((boxes / nbox) - 1) & 1)) return false;
      // planes past the grid read zero, and count towards the barriers of every box
      for (int k = 0; k < P + 2; k++) {
        const int i = BWD ? P + 1 - k : k;  // in the order the taps need them
        bar_expect(&box_full[b][i], plane_bytes);
        tma_box(sm + b * box_bytes + i * plane_bytes, &tm, t.x0, t.y0, t.z0 - 1 + i, bp * gp, &box_full[b][i]);
      }
      boxes++;
      if (++bp == npass) {
        bp = 0;
        bt += gridDim.x;
      }
      return true;
    };
    int s = 0, c = 0;
    unsigned turn = 1;  // a ring buffer's first use does not wait
    for (int64_t t = blockIdx.x; t < ts.tiles && ok; t += gridDim.x, it++) {
      const uint16_t *wt = wpack + (int64_t)tile_at(t).nt * nch * (b_bytes / 2);
      for (int q = 0; q < nch && ok; q++, c++) {
        if (q % per == 0)
          while (ok && bt < ts.tiles && boxes < it * npass + q / per + nbox) ok = issue_box();
        ok = ok && (c < ring || bar_wait(&done[s], turn));
        if (!ok) break;
        bar_expect(&loaded[s], b_bytes);
        bulk_copy(sb + s * b_bytes, wt + (int64_t)q * (b_bytes / 2), b_bytes, &loaded[s]);
        if (++s == ring) {
          s = 0;
          turn ^= 1u;
        }
      }
    }
    // every copy lands before the shared memory is released
    for (int q = max(0, c - ring); q < c; q++) bar_wait(&loaded[q % ring], (q / ring) & 1);
    for (int q = max(0, boxes - nbox); q < boxes; q++)
      for (int i = 0; i < P + 2; i++) bar_wait(&box_full[q % nbox][i], (q / nbox) & 1);
  } else if (warp < P && one) {  // MMAs of plane `warp`
    const uint32_t idesc = instr_desc(nt_n);
    const unsigned ahi = (unsigned)(smem_desc(0, kGroupBytes, kRowBytes) >> 32), bhi = (unsigned)(smem_desc(0, lbo_b, 128) >> 32);
    const unsigned blo = (unsigned)smem_desc(su32(sb), lbo_b, 128), bj = (2 * lbo_b) >> 4;
    bool ok = true;
    int s = 0, tc = 0, it = 0, box_n = 0;
    unsigned turn = 0;  // phase of the ring buffer
    for (int64_t t = blockIdx.x; t < ts.tiles && ok; t += gridDim.x, it++) {
      const bool live = warp < tile_at(t).np;  // a plane past the grid keeps the barriers only
      const int as = it % nacc;
      if (it >= nacc) ok = bar_wait(&acc_free[as], ((it / nacc) - 1) & 1);
      fence_after();
      const unsigned d = tmem + (unsigned)((as * P + warp) * nt_n);
      unsigned acc = 0;  // 0 for the accumulator's first MMA
      for (int ps = 0; ps < npass && ok; ps++, box_n++) {
        const int b = box_n % nbox;
        const unsigned ph = (box_n / nbox) & 1;
        const unsigned box = (unsigned)smem_desc(su32(sm + b * box_bytes + warp * plane_bytes), kGroupBytes, kRowBytes);
        // the taps of the pass with JN group pairs
        auto run = [&](auto pairs) {
          constexpr int JN = decltype(pairs)::value;
          for (int r = 0; r < 9; r++) {  // (kz, ky): three taps
            // the tap's shift, mirrored in the backward pass
            const int sz = BWD ? 2 - r / 3 : r / 3, sy = BWD ? 2 - r % 3 : r % 3;
            if (r % 3 == 0) ok = bar_wait(&box_full[b][warp + sz], ph);
            const unsigned al = box + (((unsigned)sz * plane_bytes + (unsigned)sy * kRowBytes) >> 4);
#pragma unroll
            for (int kx = 0; kx < 3; kx++) {
              if (tc == 0) ok = ok && bar_wait(&loaded[s], turn);
              if (!ok) return;
              fence_after();
              const unsigned bl = blo + ((unsigned)(s * b_bytes + tc * t_bytes) >> 4);
              if (live) {
#pragma unroll
                for (int j = 0; j < JN; j++) {
                  mma_ss(d, al + (BWD ? 2 - kx : kx) + j * ((2 * kGroupBytes) >> 4), ahi, bl + j * bj, bhi, idesc, acc);
                  acc = 1u;
                }
              }
              if (++tc == taps) {
                mma_commit(&done[s]);
                tc = 0;
                if (++s == ring) {
                  s = 0;
                  turn ^= 1u;
                }
              }
            }
          }
          mma_commit(&box_free[b]);
        };
        switch (min(gp, ts.G - ps * gp) / 2) {
          case 1: run(std::integral_constant<int, 1>{}); break;
          case 2: run(std::integral_constant<int, 2>{}); break;
          case 3: run(std::integral_constant<int, 3>{}); break;
          case 4: run(std::integral_constant<int, 4>{}); break;
          case 5: run(std::integral_constant<int, 5>{}); break;
          default: run(std::integral_constant<int, 6>{});
        }
      }
      if (ok) mma_commit(&acc_full[as]);
    }
    mma_commit(&fin);
    bar_wait(&fin, 0);
  } else if (warp > 4) {  // results: warp q reads TMEM lanes 32 q .. 32 q + 31 (tile rows 4 q .. 4 q + 3)
    const int quad = warp & 3, m = quad * 32 + lane;
    const int64_t nv = (int64_t)D * H * W;
    using Out = typename std::conditional<BWD, float, uint16_t>::type;
    bool ok = true;
    int it = 0, bias_nt = -1;
    for (int64_t t = blockIdx.x; t < ts.tiles; t += gridDim.x, it++) {
      const Tile tl = tile_at(t);
      const int as = it % nacc;
      if (tl.nt != bias_nt) {
        asm volatile("bar.sync 1, 128;" ::: "memory");
        for (int i = tid - 160; i < nt_n; i += 128)
          sbias[i] = bias && tl.nt * nt_n + i < n_out ? __ldg(bias + tl.nt * nt_n + i) : 0.f;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        bias_nt = tl.nt;
      }
      // once a wait gave up, this and the block's later tiles get NaN
      ok = ok && __all_sync(0xffffffffu, bar_wait(&acc_full[as], (it / nacc) & 1));
      fence_after();
      const int ox = tl.x0 + (m & 7), oy = tl.y0 + (m >> 3);
      const bool in = ox < W && oy < H;
      for (int p = 0; p < tl.np; p++) {
        Out *o = static_cast<Out *>(yout) + (int64_t)tl.nt * nt_n * nv + ((int64_t)(tl.z0 + p) * H + oy) * W + ox;
        for (int c0 = 0; c0 < nt_n; c0 += 16) {
          uint32_t r[16];
          tmem_ld16(r, tmem + ((unsigned)(quad * 32) << 16) + (unsigned)((as * P + p) * nt_n + c0));
          const int nc = min(16, n_out - tl.nt * nt_n - c0);
          Out v[16];
#pragma unroll
          for (int j = 0; j < 16; j++) {
            if constexpr (BWD) {
              v[j] = ok ? __uint_as_float(r[j]) : __uint_as_float(0x7FC00000u);
            } else {
              float f = __uint_as_float(r[j]) + sbias[c0 + j];
              if (relu) f = relu_nan(f);
              v[j] = ok ? __bfloat16_as_ushort(__float2bfloat16_rn(f)) : (uint16_t)0x7FC0;
            }
          }
          if (in) {
            if (nc == 16) {
#pragma unroll
              for (int j = 0; j < 16; j++) o[j * nv] = v[j];
            } else {
#pragma unroll
              for (int j = 0; j < 16; j++)
                if (j < nc) o[j * nv] = v[j];
            }
          }
          o += 16 * nv;
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(&acc_free[as]);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, ts.cols);
}

int pow2_cols(int n) {
  int c = 32;
  while (c < n) c *= 2;
  return c;
}

// shapes of the tile form for n_rows output channels and `groups` channel groups, on an SM whose
// registers hold reg_blocks blocks; false when no shape fits
bool tile_shape(int n_rows, int groups, int64_t tiles_xy, int D, int reg_blocks, TileShape *out) {
  const int n16 = (n_rows + 15) / 16 * 16;
  TileShape ts{};
  ts.nt_n = n16 < kMaxN ? n16 : kMaxN;
  ts.ntiles = (n_rows + ts.nt_n - 1) / ts.nt_n;
  ts.G = (groups + 1) / 2 * 2;
  // groups per pass: the largest of 12, 8, 4 that divides the groups rounded up to 4 and leaves
  // room for the N tile. It sets the order of the FP32 sums, and with it the rounding of the
  // stored BF16 activations (which a ReLU network amplifies) and of the gradients, so it depends
  // on the channels alone, not on the grid or on the planes per block.
  int gp = 0;
  const int g4 = (groups + 3) / 4 * 4;
  for (int cand : {12, 8, 4})
    if (!gp && g4 % cand == 0 && 3 * kGroupBytes * cand + 4 * ts.nt_n * cand * 16 <= 200 * 1024) gp = cand;
  if (!gp) return false;
  if (gp > ts.G) gp = ts.G;
  ts.gp = gp;
  const int npass = ts.npass = (ts.G + gp - 1) / gp;
  double best = 0;
  for (int planes : {4, 2, 1})
    for (int nacc : {2, 1})
      for (int nbox = 1; nbox <= kMaxBox; nbox++)
        for (int taps : {9, 3, 1})
          for (int ring = 2; ring <= kRingB; ring++) {
            if (nacc * planes * ts.nt_n > kTmemCols) continue;
            const int cols = pow2_cols(nacc * planes * ts.nt_n);
            const int box = kGroupBytes * gp * (planes + 2), copy = taps * ts.nt_n * gp * 16;
            int smem = nbox * box + ring * copy;
            if (smem > kSmBlock) continue;
            // the shared memory keeps the blocks an SM can hold within its TMEM columns, so an
            // allocation never waits
            const int floor_smem = kSmPerSM / (kTmemCols / cols + 1) - 1024 + 16;
            if (smem < floor_smem) smem = floor_smem;
            const int occ = std::min({kTmemCols / cols, kSmPerSM / (smem + 2560), reg_blocks});
            const int64_t tiles = tiles_xy * ((D + planes - 1) / planes) * ts.ntiles;
            // a model in SM clocks: an MMA of M = 128, K = 16 reads 4 KB of A and 32 nt_n bytes of B
            // at 128 B per clock or computes nt_n / 2 clocks, and its issue takes about 110 clocks of
            // its warp (all measured); a weight copy takes about 1500 clocks of latency and 24 B per
            // clock and SM; the epilogue, about 60 clocks per column, runs beside the next tile's MMAs
            // with two accumulator sets; a box's load runs beside the MMAs before it with two buffers;
            // else only the SM's other blocks hide them
            const double one = std::max(32.0 + ts.nt_n / 4.0, ts.nt_n / 2.0);
            const double mma = 27.0 * (ts.G / 2) * planes * one;                     // tensor pipe
            const double chain = 27.0 * (ts.G / 2) * std::max(planes * one, 110.0);  // issue of one warp
            const double trip = 27.0 * npass / taps * (1500.0 + copy / 24.0) / (ring - 1);
            const double body = std::max(chain, trip);
            const double load = 1500.0 + box / 30.0 * 0.5, epi = 500.0 + 60.0 * planes * ts.nt_n;
            const double l2 = 27.0 * ts.G * 16 * ts.nt_n / 24.0;
            const double turns = std::ceil(tiles / (kSms * (double)occ));               // tiles per block
            const double share = std::min((double)occ, std::ceil(tiles / (double)kSms));  // blocks on an SM
            // one block's time per tile, or the SM's pipes shared by its blocks
            const double each = std::max(body + (nbox == 1 ? npass * load : 0.0), share * std::max(mma, l2));
            const double cost = (nbox == 1 ? 0.0 : load) +
                                (nacc == 2 ? turns * std::max(each, epi) + epi : turns * (each + epi));
            if (best == 0 || cost < best) {
              best = cost;
              ts.planes = planes;
              ts.nacc = nacc;
              ts.nbox = nbox;
              ts.taps = taps;
              ts.ring = ring;
              ts.cols = cols;
              ts.smem = smem;
              ts.tiles = tiles;
              ts.grid = (int)std::min<int64_t>(tiles, (int64_t)kSms * occ);
              *out = ts;
            }
          }
  return best > 0;
}

unsigned blocks_x(int64_t n, int threads, int64_t most) {
  const int64_t b = (n + threads - 1) / threads;
  return (unsigned)(b < most ? b : most);
}

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

// the tile form of the forward (x) or backward-data (dy) convolution of `in`; n_rows GEMM output
// channels, n_red real source channels (forward: cin; backward: cout, with cop = the part stride)
template <bool BWD>
cudaError_t run_tile(const void *in, const uint16_t *w, const float *b, int n_rows, int n_red, int cop, int groups, int D,
                     int H, int W, int relu, void *y, cudaStream_t s) {
  const int64_t nv = (int64_t)D * H * W;
  const int64_t tiles_xy = (int64_t)((W + kTX - 1) / kTX) * ((H + kTY - 1) / kTY);
  TileShape ts;
  if (tiles_xy > 0x7fffffff || D > 65535 || !tile_shape(n_rows, groups, tiles_xy, D, kTileBlocks[BWD], &ts) || ts.ntiles > 65535)
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(tile_conv_kernel<BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmBlock);
  if (e != cudaSuccess) return e;
  const size_t pack_elems = (size_t)ts.ntiles * ts.npass * 27 * ts.nt_n * ts.gp * 8;
  const size_t src_bytes = align256((size_t)ts.G * nv * 16);
  unsigned char *buf = nullptr;
  e = cudaMallocAsync(reinterpret_cast<void **>(&buf), src_bytes + pack_elems * 2, s);
  if (e != cudaSuccess) return e;
  uint16_t *src = reinterpret_cast<uint16_t *>(buf), *wp = reinterpret_cast<uint16_t *>(buf + src_bytes);
  CUtensorMap tm;
  e = box_map(&tm, src, D, H, W, ts.G, ts.gp);
  if (e == cudaSuccess) {
    const unsigned nx = blocks_x(nv, 256, 65536), nsrc = nx * (unsigned)(BWD ? cop / 8 : ts.G);
    const unsigned npack = blocks_x((int64_t)pack_elems / 8, 256, 4096);
    tile_prep_kernel<BWD><<<nsrc + npack, 256, 0, s>>>(in, nv, n_red, cop, w, n_rows, ts, src, wp, (int)nx, (int)nsrc);
    tile_conv_kernel<BWD><<<ts.grid, kTileThreads, ts.smem, s>>>(tm, wp, b, n_rows, ts, D, H, W, relu, y);
    e = cudaGetLastError();
  }
  const cudaError_t f = cudaFreeAsync(buf, s);
  return e != cudaSuccess ? e : f;
}

// ---- weight gradient: D_t[r][ci] = sum_p A[r][p] x[ci][p + off(t)], r = (part, channel) of the
// split gradient. The three parts of up to 42 channels are the M = 128 rows of one operand
// that is kept in TMEM, so the taps of a block share one load of it and an MMA reads only the
// x view from shared memory (B, MN-major: a core matrix is 8 x-voxels along K of 8 channels).
// With both operands in shared memory an MMA of N = 32 reads 5 KB (40 clocks) for 16 clocks of
// math; from TMEM the read is 1 KB. A block owns a slice of voxel tiles, a group of T taps of
// one kz (9 up to 32 channels, else 3 of one ky) and up to 112 input channels, one
// accumulator of nt_n columns per tap. The three parts are added in the epilogue, so each
// accumulator's chain is a third as long as with one for all parts.
//
// Warp 4 copies the stages (a gradient tile, contiguous in the tile-ordered split copy, and the
// x box), warps 0-3 move the gradient rows from shared memory into one of two TMEM buffers,
// warp 5 + t issues the MMAs of tap t (one thread's issue, about 45 clocks, takes three times
// as long as an MMA of N = 32). Bound: the tensor pipe at small N and the hand-over of the
// gradient buffers. Measured at 65 x 129 x 129 voxels, 28 x 28 channels: 1362 -> 215 us (im2col
// rows gathered by the threads before); 56 x 56 channels at 33 x 65 x 65: 511 -> 126 us.
constexpr int kWgA = 384;          // first TMEM column of the two gradient buffers (64 columns each)
constexpr int kWgAccCols = 368;    // accumulator columns: 368 + 16 (bias) = 384
constexpr int kWgMaxRing = 8;      // most stages in flight
constexpr int kWgRows = 42;        // gradient channels per M tile (3 parts: 126 rows)
constexpr int kWgSlice = 48;       // most tiles per slice: 6144 voxels, 384 sums per accumulator
constexpr int kWgThin = 8;         // times as many on grids of one or two rows (one of a tile's 8 MMAs is not zero)
constexpr int kWorkSlice = 2048;    // voxels per slice the size of `work` is counted by

// dyt[mt][tile][y][r][8 x]: the split gradient of the rows r = part cm + c of M tile mt
// (channel mt cm + c), per voxel tile (the ncopy tiles from `first` on) and tile row; zero outside
// the grid and past cout. A block turns one tile of up to 32 channels through shared memory, so that both its reads
// (8 voxels of a row) and its writes (16 bytes of consecutive channels) are contiguous.
__device__ __forceinline__ void split_tile_block(const float *__restrict__ dy, int cout, int cm, int ntx, int nty, int first,
                                                 int ncopy, int D, int H, int W, uint16_t *__restrict__ dyt, int tile,
                                                 int mt, int c0) {
  __shared__ float st[32][kM + 1];
  const int x0 = tile % ntx * kTX, y0 = tile / ntx % nty * kTY, z = tile / ntx / nty;
  const int nc = min(32, cm - c0);
  for (int i = threadIdx.x; i < nc * kM; i += 256) {
    const int c = i / kM, v = i % kM, x = x0 + (v & 7), y = y0 + (v >> 3), co = mt * cm + c0 + c;
    st[c][v] = (co < cout && x < W && y < H) ? __ldg(dy + (((int64_t)co * D + z) * H + y) * W + x) : 0.f;
  }
  __syncthreads();
  const int64_t base = ((int64_t)mt * ncopy + (tile - first)) * kTY * (3 * cm);
  for (int i = threadIdx.x; i < 32 * kTY; i += 256) {
    const int c = i & 31, y = i >> 5;
    if (c >= nc) continue;
    uint16_t h[3][8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
      uint16_t t[3];
      split3(st[c][y * 8 + e], t);
#pragma unroll
      for (int s = 0; s < 3; s++) h[s][e] = t[s];
    }
#pragma unroll
    for (int s = 0; s < 3; s++)
      *reinterpret_cast<uint4 *>(dyt + (base + (int64_t)y * (3 * cm) + s * cm + c0 + c) * 8) = pack8(h[s]);
  }
}

struct WgShape {
  int T, nt_n, ntile;      // taps per block, input channels per block, N tiles
  int cm, mt;              // gradient channels per M tile, M tiles
  int G, ntx, nty, tiles;  // source groups, voxel tiles
  int slices, per;         // slices, tiles per slice
  int slice0;              // first slice of the launch
  int first, ncopy;        // first tile and tiles of its slices, those in the copy of the gradient
  int ring, smem;
};

// x alone, for grids where the two copies' own launches cost nothing: wgrad_prep_kernel's shared
// memory leaves its x blocks fewer on an SM
__global__ void __launch_bounds__(256) group_major_kernel(const uint16_t *__restrict__ x, int64_t nv, int cin,
                                                          uint16_t *__restrict__ src, int nx) {
  group_major_block(x, nv, cin, src, blockIdx.x, nx);
}
// Voxels up to which the two copies are one launch. One launch against two, 28 and 56 channels: 17 x 33 x
// 33 voxels 31.6 / 33.7 and 45.7 / 48.7 us a call, 49 x 97 x 97 (461 thousand) 157.0 / 160.9 and 475.0 /
// 477.0, 65 x 129 x 129 (1.08 million) 338.4 / 339.7 and 1023.4 / 1021.9.
constexpr int64_t kPrepVoxels = 1 << 20;

// the copies of a weight gradient: blocks below nsrc x, the others the gradient tiles
__global__ void __launch_bounds__(256) wgrad_prep_kernel(const float *__restrict__ dy, const uint16_t *__restrict__ x,
                                                         int64_t nv, int cin, int cout, WgShape g, int D, int H, int W,
                                                         uint16_t *__restrict__ src, uint16_t *__restrict__ dyt, int nx,
                                                         int nsrc) {
  const int b = blockIdx.x;
  if (b < nsrc) {
    group_major_block(x, nv, cin, src, b, nx);
    return;
  }
  const int chunks = (g.cm + 31) / 32;  // of 32 channels of an M tile
  for (int64_t i = b - nsrc; i < (int64_t)g.ncopy * chunks * g.mt; i += gridDim.x - nsrc) {
    const int r = (int)(i / g.ncopy);
    __syncthreads();  // the tile before has been read
    split_tile_block(dy, cout, g.cm, g.ntx, g.nty, g.first, g.ncopy, D, H, W, dyt, g.first + (int)(i % g.ncopy), r / chunks,
                     r % chunks * 32);
  }
}

// Tiles that reach over the grid's edge multiply their zero gradients there with the x values
// beside them: voxel W (H) with x at W - 1 (H - 1), which the taps of kx = 0 (ky = 0) must not use
// so. That adds nothing unless such an x is not finite.
__device__ __forceinline__ bool tap_reaches(int t, int H, int W) {
  return (t % 3 == 0 && W % kTX != 0) || (t / 3 % 3 == 0 && H % kTY != 0);
}
// such a tap's sum over the grid's voxels in tiles t0 .. t1 - 1, by a warp (dy, x: of the output and
// input channel); ends as soon as a NaN settles it
__device__ __forceinline__ float tap_over_grid(const float *dy, const uint16_t *x, int t, int t0, int t1, int ntx, int plane, int D,
                                            int H, int W) {
  double acc = 0.0;
  for (int i = t0; i < t1 && !__any_sync(0xffffffffu, acc != acc); i++) {
    const int z = i / plane, y0 = i % plane / ntx * kTY, x0 = i % ntx * kTX, zz = z + t / 9 - 1;
    for (int v = threadIdx.x & 31; v < kM; v += 32) {
      const int y = y0 + (v >> 3), xx = x0 + (v & 7), py = y + t / 3 % 3 - 1, px = xx + t % 3 - 1;
      if (y < H && xx < W && zz >= 0 && zz < D && py >= 0 && py < H && px >= 0 && px < W)
        acc += (double)__ldg(dy + ((int64_t)z * H + y) * W + xx) *
               (double)__uint_as_float((uint32_t)__ldg(x + ((int64_t)zz * H + py) * W + px) << 16);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return (float)acc;
}

template <int T>
__global__ void __launch_bounds__(32 * (5 + T), 1)
    wgrad_kernel(const __grid_constant__ CUtensorMap tm, const uint16_t *__restrict__ dyt, WgShape g, int D, int H, int W,
                 int cin, int cout, const float *__restrict__ dy, const uint16_t *__restrict__ x, float *__restrict__ part) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(128) uint4 ones[8];  // a core matrix of BF16 ones (the bias gradient)
  __shared__ uint64_t full[kWgMaxRing], free_[kWgMaxRing], a_full[2], a_free[2], fin;
  __shared__ unsigned tslot;
  __shared__ int okslot;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  // the blocks of one slice are neighbours in the grid: its voxels are read while L2 holds them
  constexpr int ngrp = 27 / T;
  const int grp = blockIdx.x % ngrp, nt = blockIdx.x / ngrp % g.ntile, mt = blockIdx.x / ngrp / g.ntile;
  const int slice = g.slice0 + blockIdx.y;
  const int tap0 = grp * T, kz = tap0 / 9, ky0 = tap0 / 3 % 3;
  const bool bias = tap0 / 9 == 1 && (T == 9 || ky0 == 1) && nt == 0;
  const int R = 3 * g.cm, plane = g.ntx * g.nty;
  const int box_bytes = g.nt_n / 8 * kGroupBytes, a_bytes = R * kTY * 16;
  const int stage = (box_bytes + a_bytes + 127) / 128 * 128;  // box, then gradient rows [y][r][8 x]
  // the slice's tiles whose plane z + kz - 1 is inside the grid (the others add nothing)
  const int t0 = max(slice * g.per, kz == 0 ? plane : 0);
  const int t1 = min(min((slice + 1) * g.per, g.tiles), kz == 2 ? plane * (D - 1) : g.tiles);
  const int n = max(0, t1 - t0);

  if (tid == 0) {
    for (int i = 0; i < g.ring; i++) {
      bar_init(&full[i]);
      bar_init(&free_[i], T);
    }
    for (int i = 0; i < 2; i++) {
      bar_init(&a_full[i], 4);
      bar_init(&a_free[i], T);
    }
    bar_init(&fin, T);
    okslot = 1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 8) ones[tid] = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) tmem_alloc(&tslot, kTmemCols);
  fence_before();
  __syncthreads();
  fence_after();
  const unsigned tmem = tslot;

  const bool one = elect_one();
  if (warp < 4) {  // gradient rows into TMEM: thread = row, 64 columns = 128 voxels
    const int r = warp * 32 + lane;
    bool ok = true;
    for (int i = 0; i < n; i++) {
      const int b = i & 1, st = i % g.ring;
      ok = __all_sync(0xffffffffu, bar_wait(&full[st], (i / g.ring) & 1) && (i < 2 || bar_wait(&a_free[b], ((i >> 1) - 1) & 1)));
      if (!ok) break;
      fence_after();
      const uint4 *q = reinterpret_cast<const uint4 *>(sm + st * stage + box_bytes) + r;
      const unsigned a = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(kWgA + b * 64);
#pragma unroll
      for (int c = 0; c < 4; c++) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; k++) v[k] = r < R ? q[(4 * c + k) * R] : make_uint4(0u, 0u, 0u, 0u);
        tmem_st16(a + 16 * c, v);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(&a_full[b]);
    }
    if (!ok) atomicExch(&okslot, 0);
  } else if (warp == 4 && one) {  // copies
    const uint16_t *src = dyt + ((int64_t)mt * g.ncopy + (t0 - g.first)) * (a_bytes / 2);
    bool ok = true;
    int i = 0;
    for (; i < n; i++) {
      const int s = i % g.ring, tile = t0 + i;
      if (i >= g.ring && !bar_wait(&free_[s], ((i / g.ring) - 1) & 1)) {
        ok = false;
        break;
      }
      bar_expect(&full[s], box_bytes + a_bytes);
      bulk_copy(sm + s * stage + box_bytes, src + (int64_t)i * (a_bytes / 2), a_bytes, &full[s]);
      tma_box(sm + s * stage, &tm, tile % g.ntx * kTX, tile / g.ntx % g.nty * kTY, tile / plane + kz - 1,
              nt * (g.nt_n / 8), &full[s]);
    }
    for (int q = max(0, i - g.ring); q < i; q++) ok = bar_wait(&full[q % g.ring], (q / g.ring) & 1) && ok;
    if (!ok) atomicExch(&okslot, 0);
  } else if (warp >= 5 && one) {  // MMAs of tap w of the group
    const int w = warp - 5;
    const uint32_t idesc = instr_desc(g.nt_n) | (1u << 16), idesc1 = instr_desc(16) | (1u << 16);  // B MN-major
    const unsigned dhi = (unsigned)(smem_desc(0, kRowBytes, kGroupBytes) >> 32);
    const unsigned dlo0 =
        (unsigned)smem_desc(su32(sm) + (unsigned)((ky0 + w / 3) * kRowBytes + w % 3 * 16), kRowBytes, kGroupBytes);
    const uint64_t d1 = smem_desc(su32(ones), 0, 0);
    const unsigned d1lo = (unsigned)d1, d1hi = (unsigned)(d1 >> 32);
    const unsigned dt = tmem + (unsigned)(w * g.nt_n), db = tmem + (unsigned)(T * g.nt_n);
    const bool ones_too = bias && w == 0;
    bool ok = true;
    for (int i = 0; i < n; i++) {
      const int b = i & 1, s = i % g.ring;
      if (!bar_wait(&a_full[b], (i >> 1) & 1) || !bar_wait(&full[s], (i / g.ring) & 1)) {
        ok = false;
        break;
      }
      fence_after();
      const unsigned dlo = dlo0 + ((unsigned)(s * stage) >> 4), a = tmem + (unsigned)(kWgA + b * 64);
#pragma unroll
      for (int ks = 0; ks < 8; ks++) {  // 16 voxels: tile rows 2 ks, 2 ks + 1
        const unsigned acc = (i > 0 || ks > 0) ? 1u : 0u;
        mma_ts(dt, a + ks * 8, dlo + ((2 * ks * kRowBytes) >> 4), dhi, idesc, acc);
        if (ones_too) mma_ts(db, a + ks * 8, d1lo, d1hi, idesc1, acc);
      }
      mma_commit(&a_free[b]);
      mma_commit(&free_[s]);
    }
    mma_commit(&fin);
    if (!bar_wait(&fin, 0)) ok = false;
    if (!ok) atomicExch(&okslot, 0);
  }
  __syncthreads();
  const bool ok = *(volatile int *)&okslot != 0;
  fence_after();
  // part[slice][co][t cin + ci], then the bias sum: the accumulators go to shared memory (the
  // stages' space), where every thread adds the three parts' rows of its channels
  float *se = reinterpret_cast<float *>(sm);
  const int ncol = T * g.nt_n + (bias ? 16 : 0), pitch = ncol + 1;
  if (warp < 4)
    for (int c0 = 0; c0 < ncol; c0 += 16) {
      uint32_t v[16];
      tmem_ld16(v, tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0);
#pragma unroll
      for (int j = 0; j < 16; j++) se[tid * pitch + c0 + j] = n > 0 ? __uint_as_float(v[j]) : 0.f;
    }
  __syncthreads();
  const int64_t row = 27 * (int64_t)cin + 1;
  for (int c = warp; c < g.cm; c += 5 + T) {
    const int co = mt * g.cm + c;
    if (co >= cout) break;
    const float *s0 = se + c * pitch, *s1 = s0 + g.cm * pitch, *s2 = s1 + g.cm * pitch;
    float *out = part + ((int64_t)slice * cout + co) * row;
    // NaN once a value is not finite; such values are looked at after the loop, which a test and
    // a vote inside it had made slower (28 x 28 channels: 340 against 350 us a call)
    float worst = 0.f;
    for (int t = 0; t < T; t++)
      for (int j = lane; j < g.nt_n; j += 32) {
        const int ci = nt * g.nt_n + j, q = t * g.nt_n + j;
        if (ci < cin) {
          const float v = ok ? s0[q] + (s1[q] + s2[q]) : __uint_as_float(0x7FC00000u);
          out[(int64_t)(tap0 + t) * cin + ci] = v;
          worst = fmaf(v, 0.f, worst);
        }
      }
    if (__any_sync(0xffffffffu, worst != 0.f) && ok)
      for (int o = 0; o < T * g.nt_n; o++) {
        const int t = o / g.nt_n, ci = nt * g.nt_n + o % g.nt_n;
        const int64_t nv = (int64_t)D * H * W;
        if (ci >= cin || !tap_reaches(tap0 + t, H, W) || isfinite(s0[o] + (s1[o] + s2[o]))) continue;
        const float v = tap_over_grid(dy + co * nv, x + ci * nv, tap0 + t, t0, t1, g.ntx, plane, D, H, W);
        __syncwarp();
        if (lane == 0) out[(int64_t)(tap0 + t) * cin + ci] = v;
      }
    if (bias && lane == 0) {
      const int q = T * g.nt_n;
      out[row - 1] = ok ? s0[q] + (s1[q] + s2[q]) : __uint_as_float(0x7FC00000u);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, kTmemCols);
}

// dw[co][ci][t] and db[co]: the slices' partial sums. A block owns 32 outputs; warp k adds
// the slices k, k + 8, ... in order, then the eight sums are added in order (one thread per
// output, all slices in one chain, took 64 us at 28 x 28 channels and 528 slices; 9 us now).
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float *__restrict__ part, int nslice, int cin, int cout,
                                                           float *__restrict__ dw, float *__restrict__ db) {
  __shared__ float sh[8][32];
  const int64_t row = 27 * (int64_t)cin + 1, total = cout * row;
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  for (int64_t i0 = (int64_t)blockIdx.x * 32; i0 < total; i0 += (int64_t)gridDim.x * 32) {
    const int64_t i = i0 + lane;
    float acc = 0.f;
    if (i < total)
#pragma unroll 4
      for (int sl = k; sl < nslice; sl += 8) acc += __ldg(part + sl * total + i);
    sh[k][lane] = acc;
    __syncthreads();
    if (k == 0 && i < total) {
#pragma unroll
      for (int q = 1; q < 8; q++) acc += sh[q][lane];
      const int co = (int)(i / row), j = (int)(i % row);
      if (j == row - 1) {
        if (db) db[co] = acc;
      } else {
        dw[((int64_t)co * cin + j % cin) * 27 + j / cin] = acc;
      }
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t conv3d_forward_tc(const uint16_t *x, const uint16_t *w, const float *b, int cin, int cout, int D, int H,
                              int W, int relu, uint16_t *y, cudaStream_t s) {
  return run_tile<false>(x, w, b, cout, cin, 8, (cin + 7) / 8, D, H, W, relu, y, s);
}

cudaError_t conv3d_backward_data_tc(const float *dy, const uint16_t *w, int cin, int cout, int D, int H, int W,
                                    float *dx, cudaStream_t s) {
  const int cop = (cout + 7) / 8 * 8;
  return run_tile<true>(dy, w, nullptr, cin, cout, cop, 3 * cop / 8, D, H, W, 0, dx, s);
}

// floats the caller's scratch holds: one 128-row-padded im2col row set per 2048 voxels and
// output channel (the partial sums below need less for all but small grids)
int64_t conv3d_backward_weight_tc_work(int cin, int cout, int D, int H, int W) {
  const int cp = (cin + 7) / 8 * 8;
  const int64_t nv = (int64_t)D * H * W;
  const int64_t nslice = (nv + kWorkSlice - 1) / kWorkSlice;
  const int64_t mpad = ((int64_t)27 * cp + 1 + 127) / 128 * 128;
  const int n16 = (cout + 15) / 16 * 16;
  const int nt_n = n16 < kMaxN ? n16 : kMaxN;
  const int64_t ncol = (int64_t)((cout + nt_n - 1) / nt_n) * nt_n;
  return nslice * ncol * mpad;
}

cudaError_t conv3d_backward_weight_tc(const float *dy, const uint16_t *x, int cin, int cout, int D, int H, int W,
                                      float *dw, float *db, float *work, cudaStream_t s) {
  const int64_t nv = (int64_t)D * H * W;
  WgShape g{};
  g.ntx = (W + kTX - 1) / kTX;
  g.nty = (H + kTY - 1) / kTY;
  const int64_t tiles = (int64_t)g.ntx * g.nty * D;
  if ((nv + kWorkSlice - 1) / kWorkSlice > 65535) return cudaErrorInvalidValue;  // the limit the size of `work` assumes
  g.tiles = (int)tiles;
  g.mt = (cout + kWgRows - 1) / kWgRows;
  g.cm = (cout + g.mt - 1) / g.mt;
  g.G = (cin + 7) / 8;
  const int n16 = (cin + 15) / 16 * 16;
  g.T = n16 <= 32 ? 9 : 3;
  const int most = kWgAccCols / g.T / 16 * 16;
  g.ntile = (n16 + most - 1) / most;
  g.nt_n = ((n16 + g.ntile - 1) / g.ntile + 15) / 16 * 16;
  const int combos = 27 / g.T * g.ntile * g.mt;
  // one block per SM (all its TMEM): as many slices as fill whole waves of the SMs, at most
  // kWgSlice tiles each, and on small grids at least two tiles
  const int cap = H <= 2 ? kWgThin * kWgSlice : kWgSlice;
  const int64_t waves = ((int64_t)combos * ((tiles + cap - 1) / cap) + kSms - 1) / kSms;
  int64_t slices = std::max<int64_t>(1, waves * kSms / combos);
  slices = std::max<int64_t>(std::min(slices, (tiles + 1) / 2), (tiles + cap - 1) / cap);
  g.per = (int)((tiles + slices - 1) / slices);
  g.slices = (int)((tiles + g.per - 1) / g.per);
  const int stage = (g.nt_n / 8 * kGroupBytes + 3 * g.cm * kTY * 16 + 127) / 128 * 128;
  g.ring = std::min(kWgMaxRing, kSmBlock / stage);
  g.smem = std::max({g.ring * stage, kM * (g.T * g.nt_n + 17) * 4, kSmPerSM / 2});  // one block per SM, as its TMEM is one block's
  const auto kernel = g.T == 9 ? wgrad_kernel<9> : wgrad_kernel<3>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmBlock);
  if (e != cudaSuccess) return e;
  const size_t src_bytes = align256((size_t)g.G * nv * 16);
  // The copy of the gradient holds whole tiles: on thin grids many times the gradient's size. It
  // is at most about twice that of a grid of full tiles, and the slices take turns with it.
  const int64_t tile_bytes = (int64_t)g.mt * kTY * 3 * g.cm * 16;
  const int64_t most_bytes = std::max<int64_t>(2 * tile_bytes * (nv / kM), 256 << 20);
  int64_t turn = std::min(g.slices, 65535);  // slices of a launch: its grid's y
  if (tile_bytes * tiles > most_bytes) turn = std::max<int64_t>(1, std::min(turn, most_bytes / (tile_bytes * g.per)));
  const size_t dyt_bytes = align256((size_t)(tile_bytes * std::min(tiles, turn * g.per)));
  const int64_t part_floats = (int64_t)g.slices * cout * (27 * (int64_t)cin + 1);
  const bool own = part_floats > conv3d_backward_weight_tc_work(cin, cout, D, H, W);
  unsigned char *buf = nullptr;
  e = cudaMallocAsync(reinterpret_cast<void **>(&buf), src_bytes + dyt_bytes + (own ? part_floats * 4 : 0), s);
  if (e != cudaSuccess) return e;
  uint16_t *src = reinterpret_cast<uint16_t *>(buf), *dyt = reinterpret_cast<uint16_t *>(buf + src_bytes);
  float *part = own ? reinterpret_cast<float *>(buf + src_bytes + dyt_bytes) : work;
  CUtensorMap tm;
  e = box_map(&tm, src, D, H, W, g.G, g.nt_n / 8);
  if (e == cudaSuccess) {
    const unsigned nx = blocks_x(nv, 256, 65536), nsrc = nx * (unsigned)g.G;
    const bool apart = nv > kPrepVoxels;
    if (apart) group_major_kernel<<<nsrc, 256, 0, s>>>(x, nv, cin, src, (int)nx);
    for (int64_t sl = 0; sl < g.slices; sl += turn) {
      const int ns = (int)std::min<int64_t>(turn, g.slices - sl);
      g.slice0 = (int)sl;
      g.first = (int)(sl * g.per);
      g.ncopy = (int)std::min<int64_t>((int64_t)ns * g.per, tiles - g.first);
      const unsigned ntl = blocks_x((int64_t)g.ncopy * ((g.cm + 31) / 32) * g.mt, 1, 1 << 30);
      const unsigned nx_here = apart || sl > 0 ? 0 : nsrc;
      wgrad_prep_kernel<<<nx_here + ntl, 256, 0, s>>>(dy, x, nv, cin, cout, g, D, H, W, src, dyt, (int)nx, (int)nx_here);
      kernel<<<dim3((unsigned)combos, (unsigned)ns), 32 * (5 + g.T), g.smem, s>>>(tm, dyt, g, D, H, W, cin, cout, dy, x, part);
    }
    wgrad_reduce_kernel<<<blocks_x((int64_t)cout * (27 * (int64_t)cin + 1), 32, 65536), 256, 0, s>>>(part, g.slices, cin,
                                                                                                  cout, dw, db);
    e = cudaGetLastError();
  }
  const cudaError_t f = cudaFreeAsync(buf, s);
  return e != cudaSuccess ? e : f;
}

}  // namespace fwi_tc
