// Learned warm start: a residual 3D convolutional network on the spherical grid
// (3x3x3 kernels, zero padding in r and theta, periodic in phi), bfloat16
// weights and activations, float32 accumulation, trained by its own kernels.
//
//   h1 = relu(conv(a; w1) + b1)                   1 -> 32   CUDA cores
//   h_k = h_{k-1} + relu(conv(h_{k-1}; wk) + bk)  32 -> 32  tensor cores (k = 2..5)
//   out = a + conv(h5; w6) + b6                   32 -> 1   tensor cores (forward; dgrad on CUDA cores)
//
// The 32 -> 32 layers are implicit GEMMs (voxels x 32 outputs, K = 27 taps x 32).
// Forward and dgrad run on the tcgen05 tensor cores with TMEM accumulators
// (conv32_tc_kernel): for each (r, theta) tap pair one 128-row window of a
// shared-memory slab of the neighbouring rows is the A operand and the three
// phi taps' weights side by side are B (N = 96), so one MMA computes all three
// phi taps of a window; the epilogue adds them with a one-row shift each.
// dgrad is the same kernel with the mirrored, transposed kernel. The weight
// gradient (wgrad32_tc_kernel) also runs on tcgen05: K = the voxels, M = three
// neighbouring shells' rows x 32 input channels, N = three azimuth taps x 32
// output channels, both operands MN-major, accumulated in TMEM over all of a
// CTA's rows. The one-channel layers run on the CUDA cores (thin_conv_kernel)
// but for their weight gradients (mma.sync, thin_wgrad_kernel).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <cmath>
#include <type_traits>
#include <vector>

#include "tsp_internal.h"

struct tsp_net_s;

// Device error word of this translation unit: a tensor-core wait that gives up
// sets it (no trap); tsp_device_status reads and clears it.
static __device__ int g_conv_error_word;

namespace tsp {

static cudaError_t take_conv_error(int* out, cudaStream_t st) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbolAsync(&v, g_conv_error_word, sizeof(int), 0, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  const int zero = 0;
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(g_conv_error_word, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  *out |= v << 8;
  return e;
}

namespace {
struct ConvErrorRegistrar {
  ConvErrorRegistrar() { register_error_reader(&take_conv_error); }
};
ConvErrorRegistrar conv_error_registrar;

constexpr int CH = 32;

struct Dims {
  int B, Nr, Ne, Na;
  int64_t V;  // voxels per sample
};

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::);
}
// 16-byte copy that reads `src_bytes` (16 or 0) bytes and zero-fills the rest
__device__ __forceinline__ void cp_async16_zfill(void* smem, const void* gmem, uint32_t src_bytes) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(src_bytes));
}

// ---------------------------------------------------------------------------
// 32 -> 32 implicit GEMM on the 5th-generation tensor cores (tcgen05, TMEM).
// MODE 0 forward (bias, ReLU, residual, mask, bf16 out), MODE 1 dgrad
// (accumulate into float32 G), MODE 2 the 32 -> 1 output layer (weights in
// output channel 0, the others zero; out = a + z_0 + b into float32 G, with
// the one-channel input a passed as Y).
//
// Output positions of one shell are flattened with the two periodic halo
// columns of every theta-row, o = e * (N_a + 2) + p, p = 1..N_a the azimuth
// bins (p = 0 and N_a + 1 are computed and discarded); a "chunk" is T tiles of
// 128 consecutive positions. A shell buffer holds the theta-rows a chunk
// needs from one shell (halo columns included, zeros outside the grid),
// a row of 64 bytes (32 channels) per position under the 64-byte swizzle, as
// TMA lands a theta-row (row 0 a zero pad). The A operand of an (r, theta) tap
// pair is one 128-row window of a shell buffer: the swizzle follows the
// address, so a window may start at any row (starting all of them on a
// multiple of eight rows changed nothing). The weights (B: rows of one tap and
// output channel, 64 bytes of input channels) sit in the same layout, loaded
// once per CTA; three azimuth taps' rows follow one another (N = 96).
//
// Persistent CTAs take work items (sample, chunk, run of consecutive shells).
// Walking along r, a ring of three to six shell buffers holds shells r-1, r,
// r+1 and those loaded ahead, so each step loads one new shell. One thread
// issues the step's 9 windows x T tiles x 2 K halves (M = 128, N = 96, K = 16,
// bf16 x bf16 -> f32) shell by shell, committing after the outgoing shell's
// taps so that its buffer is refilled while the other MMAs run; accumulators
// rotate through NB TMEM buffers so that the epilogue groups read one step's
// (tcgen05.ld 32x32b) while the tensor cores work on the next.
//
// Batch 8 of 64 x 48 x 96 on GB300: output layer 138 us, bound by the MMAs
// (about 100 cycles each over the 80 steps of the longest CTA, 67 with N = 32:
// most of it the window's read from shared memory, so fewer, wider MMAs win; the
// CTAs' mean is 67 steps); forward layer 168 and dgrad 267,
// bound by the epilogue (157 and 249 with half of the MMAs left out). With the
// operands read back one step ahead in registers (56 / 224 registers a thread
// by setmaxnreg) 169 and 262.
// ---------------------------------------------------------------------------
constexpr int WROWS = 27 * CH;  // weight rows, 64 bytes each
// Default bound of every mbarrier wait of the tensor-core kernels, in SM clock
// cycles (about one second): a kernel argument, so that a test can shorten it.
constexpr long long TC_WAIT_BUDGET = 2000000000LL;

// Tiles per chunk and shell-buffer geometry for an azimuth count (host and
// device agree). Slab columns per theta-row: the N_a bins plus the two halo
// columns, padded to a multiple of 8 so that every TMA box (N_a bins of one
// theta-row, stored from column 1) starts on a 512-byte boundary, a period of
// the swizzle; the data start at buffer row TC_BASE. A 128-row tile
// yields TC_TOUT outputs (its first and last rows only feed their neighbours'
// azimuth taps), T tiles per chunk; a chunk's inputs span nrows theta-rows.
constexpr int TC_BASE = 7;
constexpr int TC_TOUT = 126;
// Epilogue: a group of four warps (one per TMEM lane quarter) per tile of a
// step; the CTA is an MMA warp, three loader warps and two groups.
constexpr int TC_THREADS = 128 + 256;
// Most tiles per step (2: two TMEM buffers of 192 columns, measured faster
// than 1 tile per step with five buffers of 96).
#ifndef TC_TILES
#define TC_TILES 2
#endif
constexpr int TC_MAX_SLOTS = 6;
struct TcPlan {
  int T, NB, colsP, nrows, SBP;  // NB: accumulator buffers of T x 96 TMEM columns (of 512)
  int NS;                        // shell buffers of the ring
  size_t smem;
};
__host__ __device__ inline TcPlan tc_plan(int Na) {
  TcPlan pl{1, 5, (Na + 2 + 7) / 8 * 8, 0, 0, 3, 0};
  const size_t most = 232448 - 1024 - 5120;  // static shared memory: barriers, bias, the epilogue's row exchange
  for (int T = TC_TILES; T >= 1; --T) {
    pl.T = T;
    pl.NB = 512 / (96 * T);
    pl.nrows = TC_TOUT * T / pl.colsP + 4;
    pl.SBP = (TC_BASE + pl.nrows * pl.colsP + 2 + 7) / 8 * 8;  // + the largest shift; a multiple of the swizzle's period
    pl.smem = 3 * size_t(pl.SBP) * 64 + size_t(WROWS) * 64;
    if (pl.smem <= most) break;
  }
  while (pl.NS < TC_MAX_SLOTS && pl.smem + size_t(pl.SBP) * 64 <= most) {
    ++pl.NS;
    pl.smem += size_t(pl.SBP) * 64;
  }
  return pl;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// Shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
// offsets, descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return uint64_t((addr & 0x3FFFFu) >> 4) | (uint64_t((lbo >> 4) & 0x3FFFu) << 16) |
         (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (uint64_t(1) << 46);
}
// Instruction descriptor, kind::f16: f32 accumulator, bf16 A and B, both
// K-major, N = 96 (three azimuth taps x 32 output channels), M = 128.
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((96u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// N consecutive accumulator columns (N = 8 or 16) of this thread's TMEM lane, no wait.
template <int N>
__device__ __forceinline__ void tmem_ld_nowait(uint32_t taddr, uint32_t (&r)[N]) {
  static_assert(N == 8 || N == 16, "8 or 16 columns");
  if constexpr (N == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
  }
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// One 5-D tiled TMA box (coordinates innermost first) into shared memory,
// completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                           uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
      "[%7];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}

// 16-byte channel chunk c of position u in rows of 64 bytes (32 channels) under
// the 64-byte swizzle: address bits 4-5 exclusive-or bits 7-8 (the rows start
// 512-byte aligned).
__device__ __forceinline__ uint4* row_chunk(unsigned char* rows, int u, int c) {
  return reinterpret_cast<uint4*>(rows + u * 64 + ((c ^ ((u >> 1) & 3)) << 4));
}

// Load shell rr of sample b, for the chunk whose first output theta-row is
// e_lo + 1, into a shell buffer (one warp): buffer row TC_BASE + j * colsP + p
// holds theta-row e_lo + j, column p (p = 1..N_a: azimuth p - 1; p = 0 and
// N_a + 1: the periodic halo, azimuths N_a - 1 and 0). Lane 0 registers the
// bytes and issues one TMA box per theta-row for columns
// 1..N_a (zeros outside the grid); all lanes copy the halo columns with
// 16-byte cp.async (zero-filled outside the grid), then arrive on `bar`.
__device__ __forceinline__ void tc_load_shell(const CUtensorMap* map, const Dims& d, const bf16* __restrict__ X, int b,
                                              int rr, int e_lo, const TcPlan& pl, unsigned char* buf, uint64_t* bar,
                                              int lane) {
  const int Na = d.Na;
  if (lane == 0) {
    mbar_expect_tx(bar, uint32_t(pl.nrows * Na * 64));
    for (int j = 0; j < pl.nrows; ++j)
      tma_load_5d(buf + size_t(TC_BASE + j * pl.colsP + 1) * 64, map, 0, 0, e_lo + j, rr, b, bar);
  }
  const bool shell_ok = rr >= 0 && rr < d.Nr;
  for (int i = lane; i < pl.nrows * 8; i += 32) {
    const int c = i & 3, side = (i >> 2) & 1, j = i >> 3;
    const int ee = e_lo + j;
    const bool ok = shell_ok && ee >= 0 && ee < d.Ne;
    const int aa = side == 0 ? Na - 1 : 0;
    const bf16* src = ok ? X + (((size_t(b) * d.Nr + rr) * d.Ne + ee) * Na + aa) * CH + c * 8 : X;
    cp_async16_zfill(row_chunk(buf, TC_BASE + j * pl.colsP + (side == 0 ? 0 : Na + 1), c), src, ok ? 16u : 0u);
  }
  cp_async_wait_all();
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // halo copies -> tensor-core reads
  mbar_arrive(bar);
}

// Epilogue of one tile of a step (run by a group of four warps, warp w reading
// TMEM lane quarter w & 3). The tile's accumulators sit in TMEM columns col ..
// col + 95: row m holds, for position c_m = o0 + 126 t - 1 + m, the three
// azimuth-tap partial sums z_dai(c_m) (32 columns each). The output at c_m is
// z_0(c_m - 1) + z_1(c_m) + z_2(c_m + 1): rows m - 1 and m + 1 come from the
// neighbouring lanes by shuffle and, across a warp boundary, through `xch`.
// Rows m = 1..126 are outputs. Forward: y = x + relu(z + bias) with x the
// layer input (the residual), plus the ReLU mask; dgrad: G += z, and, if Y is
// given, Y = the updated G gated by the mask of the layer below, in bf16 (the
// next dgrad's input). The voxel of row m is vox, if valid. Operands read back from memory (the residual x, or
// the gradient being accumulated) are fetched by tc_epilogue_fetch before the
// step's accumulators are ready, so their latency overlaps the wait. Each
// group takes one tile with all its channels: with both groups on both tiles,
// half the channels each, every step waited for TMEM, the exchange and the
// shuffles twice (forward layer, batch 8 of 64 x 48 x 96 on GB300: 216 us,
// 204 without).
// 32-byte global accesses: a thread's row of channels is contiguous, so each
// covers whole sectors (16-byte ones cover half sectors, a row apart per lane).
struct __align__(32) b32x8 {
  uint32_t v[8];
};
__device__ __forceinline__ b32x8 ldg32(const void* p) {
  b32x8 r;
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
                 "=r"(r.v[7])
               : "l"(p));
  return r;
}
__device__ __forceinline__ void stg32(void* p, const b32x8& r) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r.v[0]), "r"(r.v[1]), "r"(r.v[2]),
               "r"(r.v[3]), "r"(r.v[4]), "r"(r.v[5]), "r"(r.v[6]), "r"(r.v[7])
               : "memory");
}

// g_z = bf16(g_h where the forward pre-activation was positive, else 0) of 16 channels.
__device__ __forceinline__ b32x8 gated16(const float (&g)[16], uint32_t mask) {
  b32x8 o;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const __nv_bfloat162 z = __floats2bfloat162_rn((mask >> (2 * u)) & 1u ? g[2 * u] : 0.0f,
                                                   (mask >> (2 * u + 1)) & 1u ? g[2 * u + 1] : 0.0f);
    o.v[u] = *reinterpret_cast<const uint32_t*>(&z);
  }
  return o;
}

template <int MODE>
struct EpiIn {
  b32x8 x[CH / 16];  // forward: residual of the tile's row (bf16)
  b32x8 g[CH / 8];   // dgrad: G of the tile's row (float32)
  uint32_t mask;     // dgrad: ReLU mask of the next layer's gradient
  float a;           // output layer: the network input a at the tile's row
};
template <int MODE>
__device__ __forceinline__ void tc_epilogue_fetch(size_t vox, bool valid, const bf16* __restrict__ Xres,
                                                  const float* __restrict__ G, const uint32_t* __restrict__ mask,
                                                  EpiIn<MODE>& in) {
  if (MODE == 0) {
#pragma unroll
    for (int h = 0; h < CH / 16; ++h)
      if (valid) in.x[h] = ldg32(Xres + vox * CH + 16 * h);
  } else if (MODE == 2) {  // Xres: the one-channel input a
    in.a = valid ? __bfloat162float(Xres[vox]) : 0.0f;
  } else {
#pragma unroll
    for (int h = 0; h < CH / 8; ++h)
      if (valid) in.g[h] = ldg32(G + vox * CH + 8 * h);
    in.mask = valid && mask ? mask[vox] : 0u;
  }
}
// Empty asm through which a value passes: the compiler may not compute with
// it earlier (it would wait for the load there).
__device__ __forceinline__ void pin(b32x8& r) {
  asm volatile(""
               : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]), "+r"(r.v[6]),
                 "+r"(r.v[7]));
}

// One accumulator column of this thread's TMEM lane, no wait.
__device__ __forceinline__ void tmem_ld1_nowait(uint32_t taddr, uint32_t& r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
}

// xb: this group's exchange buffer of the step ([quarter][0: z_0 of the last row, 1: z_2 of the first][channel]).
template <int MODE>
__device__ __forceinline__ void tc_epilogue(size_t vox, bool valid, uint32_t ta, EpiIn<MODE>& in,
                                            const float* __restrict__ s_bias, bf16* __restrict__ Y,
                                            uint32_t* __restrict__ mask, float* __restrict__ G, int qd, int group,
                                            int lane, float (*xb)[2][CH]) {
  if (MODE == 2) {  // output layer (32 -> 1, output channel 0): out = a + z_0 + b
    uint32_t r0, r1, r2;
    tmem_ld1_nowait(ta, r0);
    tmem_ld1_nowait(ta + 32, r1);
    tmem_ld1_nowait(ta + 64, r2);
    tmem_wait();
    if (lane == 31) xb[qd][0][0] = __uint_as_float(r0);
    if (lane == 0) xb[qd][1][0] = __uint_as_float(r2);
    asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory");
    float up = __shfl_up_sync(0xffffffffu, __uint_as_float(r0), 1);
    float dn = __shfl_down_sync(0xffffffffu, __uint_as_float(r2), 1);
    if (lane == 0) up = qd > 0 ? xb[qd - 1][0][0] : 0.0f;
    if (lane == 31) dn = qd < 3 ? xb[qd + 1][1][0] : 0.0f;
    asm volatile("" : "+f"(in.a));
    if (valid) G[vox] = in.a + ((up + __uint_as_float(r1) + dn) + s_bias[0]);
    return;
  }
  uint32_t r0[2][16], r1[2][16], r2[2][16];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    tmem_ld_nowait(ta + 16 * h, r0[h]);
    tmem_ld_nowait(ta + 64 + 16 * h, r2[h]);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) tmem_ld_nowait(ta + 32 + 16 * h, r1[h]);
  tmem_wait();
  if (lane == 31)
#pragma unroll
    for (int j = 0; j < CH; j += 4)
      *reinterpret_cast<uint4*>(&xb[qd][0][j]) =
          make_uint4(r0[j / 16][j % 16], r0[j / 16][j % 16 + 1], r0[j / 16][j % 16 + 2], r0[j / 16][j % 16 + 3]);
  if (lane == 0)
#pragma unroll
    for (int j = 0; j < CH; j += 4)
      *reinterpret_cast<uint4*>(&xb[qd][1][j]) =
          make_uint4(r2[j / 16][j % 16], r2[j / 16][j % 16 + 1], r2[j / 16][j % 16 + 2], r2[j / 16][j % 16 + 3]);
  asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory");
  uint32_t bits = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // 16 channels at a time
    // neighbours' taps: rows m-1 (z_0) and m+1 (z_2); all shuffles first so that their latencies overlap
    float up[16], dn[16], acc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) up[j] = __shfl_up_sync(0xffffffffu, __uint_as_float(r0[h][j]), 1);
#pragma unroll
    for (int j = 0; j < 16; ++j) dn[j] = __shfl_down_sync(0xffffffffu, __uint_as_float(r2[h][j]), 1);
    if (lane == 0)
#pragma unroll
      for (int j = 0; j < 16; ++j) up[j] = qd > 0 ? xb[qd - 1][0][16 * h + j] : 0.0f;
    if (lane == 31)
#pragma unroll
      for (int j = 0; j < 16; ++j) dn[j] = qd < 3 ? xb[qd + 1][1][16 * h + j] : 0.0f;
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j] = up[j] + __uint_as_float(r1[h][j]) + dn[j];
    if (!valid) continue;
    if (MODE == 0) {
      pin(in.x[h]);
      b32x8 ov;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = 2 * u, co = 16 * h + j;
        const float y0 = acc[j] + s_bias[co], y1 = acc[j + 1] + s_bias[co + 1];
        bits |= (y0 > 0.0f ? 1u : 0u) << co;
        bits |= (y1 > 0.0f ? 1u : 0u) << (co + 1);
        const float2 xf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&in.x[h].v[u]));
        const __nv_bfloat162 o = __floats2bfloat162_rn(xf.x + fmaxf(y0, 0.0f), xf.y + fmaxf(y1, 0.0f));
        ov.v[u] = *reinterpret_cast<const uint32_t*>(&o);
      }
      stg32(Y + vox * CH + 16 * h, ov);
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        b32x8 g = in.g[2 * h + i];
        pin(g);
#pragma unroll
        for (int u = 0; u < 8; ++u) g.v[u] = __float_as_uint(__uint_as_float(g.v[u]) + acc[8 * i + u]);
        stg32(G + vox * CH + 16 * h + 8 * i, g);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[8 * i + u] = __uint_as_float(g.v[u]);
      }
      if (Y) stg32(Y + vox * CH + 16 * h, gated16(acc, in.mask >> (16 * h)));
    }
  }
  if (MODE == 0 && valid) mask[vox] = bits;
}

// AND of `p` over the 128 threads of an epilogue group (its named barrier):
// their decision to go on or give up is taken together, so none waits at the
// epilogue's barrier for a warp that has left.
__device__ __forceinline__ bool epilogue_and(bool p, int group) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred pi, po;\n setp.ne.u32 pi, %1, 0;\n bar.red.and.pred po, %2, 128, pi;\n selp.u32 %0, 1, 0, po;\n}"
      : "=r"(r)
      : "r"(uint32_t(p)), "r"(1 + group)
      : "memory");
  return r != 0;
}

// Bounded wait on an mbarrier phase (at most `budget` SM cycles) that also
// gives up when another role of the CTA has already given up (s_abort); sets
// s_abort on its own timeout.
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, volatile int* s_abort, long long budget) {
  const long long t0 = clock64();
  while (!mbar_try(bar, parity)) {
    if (*s_abort) return false;
    if (clock64() - t0 > budget) {
      *s_abort = 1;
      return false;
    }
  }
  return true;
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(ok));
  return ok != 0;
}
// Issue of an MMA / a commit by the one calling thread.
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}


// Steps ahead of which the dgrad's epilogue asks for the gradient it adds to
// (it comes from DRAM, 128 bytes a thread; the threads hold one step's at a
// time: a layer of batch 8, 64 x 48 x 96 takes 281 us without, 267 with).
constexpr int TC_AHEAD = 2;

template <int MODE>
__global__ void __launch_bounds__(TC_THREADS, 1) conv32_tc_kernel(const __grid_constant__ CUtensorMap xmap, Dims d, int rseg,
                                                           const bf16* __restrict__ X, const bf16* __restrict__ W,
                                                           const float* __restrict__ bias, bf16* __restrict__ Y,
                                                           uint32_t* __restrict__ mask, float* __restrict__ G,
                                                           long long budget, int stall_loader) {
  extern __shared__ __align__(1024) unsigned char smem[];
  // full[s]: shell slot s loaded (32 loader arrivals + TMA bytes); empty[s]: its last MMA done (commit);
  // tfull[j]: TMEM buffer j holds a finished step (commit); tempty[j]: drained (one arrival per thread of the groups)
  __shared__ __align__(8) uint64_t full[TC_MAX_SLOTS], empty[TC_MAX_SLOTS], tfull[5], tempty[5];
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_abort;
  __shared__ __align__(16) float xch[2][2][4][2][CH];  // epilogue: rows that cross a warp boundary [group][step parity]
  __shared__ float s_bias[CH];
  const TcPlan pl = tc_plan(d.Na);
  const int cols = pl.colsP, P = d.Ne * cols;
  const int T = pl.T, SBP = pl.SBP;
  const int NB = pl.NB;
  const uint32_t ncols = 512u;  // NB accumulator buffers of T x 96 columns
  const int NS = pl.NS;
  unsigned char* s_w = smem + NS * size_t(SBP) * 64;           // WROWS rows of 64 B, swizzled like the shells
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nq = (P + TC_TOUT * T - 1) / (TC_TOUT * T), nseg = (d.Nr + rseg - 1) / rseg;
  const int items = d.B * nq * nseg;

  if (smem_u32(smem) & 511u) {  // the swizzle pattern repeats every 512 bytes: report, touch nothing
    if (tid == 0) atomicOr(&g_conv_error_word, 2);
    return;
  }
  // ---- set-up, all threads: zero the shell buffers (pad rows and padding columns stay zero), weights,
  // barriers, TMEM ----
  for (int i = tid; i < NS * SBP * 4; i += blockDim.x)
    reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 27 * CH * 4; i += blockDim.x) {  // row = tap * 32 + output channel, K = input channel
    const int row = i >> 2, c = i & 3;
    cp_async16(s_w + row * 64 + ((c ^ ((row >> 1) & 3)) << 4), W + size_t(row) * CH + c * 8);
  }
  cp_async_wait_all();
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor-core reads
  if (tid < CH) s_bias[tid] = MODE == 0 || (MODE == 2 && tid == 0) ? bias[tid] : 0.0f;
  if (tid == 0) {
    s_abort = 0;
    for (int s = 0; s < NS; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 32;" ::"r"(smem_u32(&full[s])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
    }
    for (int j = 0; j < NB; ++j) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&tfull[j])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&tempty[j])), "r"(128 * T)
                   : "memory");
    }
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;

  // Every role walks the same sequence: items, their steps r = r0..r1-1 (global
  // step K, TMEM buffer K mod NB) and their shell loads r0-1..r1 (global load G,
  // slot G % NS, the n-th use of a slot being phase n of its barriers).
  if (warp == 0) {  // ---- MMA issuer: one lane walks the schedule and issues ----
    if (elect_one()) {
      const uint64_t wd0 = umma_desc(smem_u32(s_w), 16, 512) | (uint64_t(4) << 61);
      int K = 0, G0 = 0, kb = 0;  // step, shell loads so far, TMEM buffer of step K
      uint32_t kph = 0;           // phase of buffer kb's barriers for step K
      bool go = true;
      for (int item = blockIdx.x; item < items && go; item += gridDim.x) {
        const int seg = item % nseg, q = (item / nseg) % nq;
        const int r0 = seg * rseg, n = min(rseg, d.Nr - r0);
        const int o0 = q * TC_TOUT * T, e_lo = (o0 - 1 + cols) / cols - 2;  // floor((o0 - 1) / cols) - 1
        for (int i = 0; i < n && go; ++i, ++K) {
          if (K >= NB && !tc_wait(&tempty[kb], kph ^ 1u, &s_abort, budget)) {
            go = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t acc0 = tmem + uint32_t(kb) * uint32_t(T) * 96;
          for (int dri = 0; dri < 3; ++dri) {
            const int Gl = G0 + i + dri, slot = Gl % NS;
            if (!tc_wait(&full[slot], uint32_t(Gl / NS) & 1u, &s_abort, budget)) {
              go = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t xd0 = umma_desc(smem_u32(smem + size_t(slot) * SBP * 64), 16, 512) | (uint64_t(4) << 61);
            for (int t = 0; t < T; ++t) {
              // tile rows m = 0..127 are the positions o0 + 126 t - 1 + m (input column p of each)
              const int orel = o0 + TC_TOUT * t - 1 - e_lo * cols;
#pragma unroll
              for (int dei = 0; dei < 3; ++dei) {
                const uint32_t srow = uint32_t(orel + (dei - 1) * cols + TC_BASE);
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                  // B: the three azimuth taps (dri, dei, 0..2) x 32 output channels, contiguous rows
                  const uint64_t ad = xd0 + ((srow * 64u + uint32_t(kk) * 32u) >> 4);
                  const uint64_t bd = wd0 + ((uint32_t(dri * 9 + dei * 3) * CH * 64u + uint32_t(kk) * 32u) >> 4);
                  tc_mma(acc0 + uint32_t(t) * 96, ad, bd, TC_IDESC, (dri | dei | kk) != 0);
                }
              }
            }
            if (dri == 0 || i == n - 1) tc_commit(&empty[slot]);  // this load's last use
          }
          if (go) tc_commit(&tfull[kb]);
          if (++kb == NB) kb = 0, kph ^= 1u;
        }
        G0 += n + 2;
      }
      if (!go) {  // let issued MMAs land before TMEM is released
        const long long t0 = clock64();
        while (clock64() - t0 < budget / 8) {
        }
      }
    }
    __syncwarp();
  } else if (warp < 4 && !stall_loader) {  // ---- shell loaders: warp w the loads w - 1 mod 3 (a test may stall them) ----
    int G0 = 0;
    bool go = true;
    for (int item = blockIdx.x; item < items && go; item += gridDim.x) {
      const int seg = item % nseg, rest = item / nseg, q = rest % nq, b = rest / nq;
      const int r0 = seg * rseg, n = min(rseg, d.Nr - r0);
      const int e_lo = (q * TC_TOUT * T - 1 + cols) / cols - 2;
      for (int j = 0; j < n + 2; ++j) {
        const int Gl = G0 + j, slot = Gl % NS;
        if (Gl % 3 != warp - 1) continue;
        if (Gl >= NS && !__all_sync(0xffffffffu, tc_wait(&empty[slot], uint32_t(Gl / NS - 1) & 1u, &s_abort, budget))) {
          go = false;
          break;
        }
        tc_load_shell(&xmap, d, X, b, r0 - 1 + j, e_lo, pl, smem + size_t(slot) * SBP * 64, &full[slot], lane);
      }
      G0 += n + 2;
    }
  } else if (warp >= 4 && (warp >> 2) - 1 < T) {  // ---- epilogue (one tile per step: the second group idle) ----
    const int qd = warp & 3;            // TMEM lane quarter this warp may read
    const int group = (warp >> 2) - 1;  // the tile of every step that this group takes
    const int m = 32 * qd + lane;       // tile row of this thread
    const size_t plane = size_t(d.Ne) * d.Na;
    int K = 0, kb = 0;
    uint32_t kph = 0;
    bool go = true;
    for (int item = blockIdx.x; item < items && go; item += gridDim.x) {
      const int seg = item % nseg, rest = item / nseg, q = rest % nq, b = rest / nq;
      const int r0 = seg * rseg, n = min(rseg, d.Nr - r0);
      // row m of the tile is position c = o0 + 126 t - 1 + m of the (theta, padded phi) plane
      const int c = q * TC_TOUT * T + TC_TOUT * group - 1 + m;
      const int e = c >= 0 ? c / cols : -1, p = c - e * cols;
      const bool valid = m >= 1 && m <= TC_TOUT && c < P && p >= 1 && p <= d.Na;
      size_t vox = valid ? (size_t(b) * d.Nr * d.Ne + e) * d.Na + (p - 1) + size_t(r0) * plane : 0;
      const size_t vstep = valid ? plane : 0;
      for (int i = 0; i < n; ++i, ++K, vox += vstep) {
        EpiIn<MODE> in;
        tc_epilogue_fetch<MODE>(vox, valid, MODE == 2 ? Y : X, G, mask, in);  // mode 2: Y carries the input a
        if (MODE == 1 && valid && i + TC_AHEAD < n)  // the gradient row of a later step, one 128-byte line
          asm volatile("prefetch.global.L2 [%0];" ::"l"(G + (vox + TC_AHEAD * vstep) * CH));
        if (!epilogue_and(tc_wait(&tfull[kb], kph, &s_abort, budget), group)) {
          go = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ta = tmem + (uint32_t(32 * qd) << 16) + uint32_t(kb * T + group) * 96;
        tc_epilogue<MODE>(vox, valid, ta, in, s_bias, Y, mask, G, qd, group, lane, xch[group][K & 1]);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(&tempty[kb]);
        if (++kb == NB) kb = 0, kph ^= 1u;
      }
    }
  }
  __syncthreads();
  if (tid == 0 && s_abort) atomicOr(&g_conv_error_word, 1);  // TSP_DEVERR_WAIT_TIMEOUT once shifted
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// ---------------------------------------------------------------------------
// 32 -> 32 weight gradient on the tcgen05 tensor cores:
//   dW[tap][co][ci] = sum_u H[u shell r + dr, row e + de][ci] Gz[u - da][co],
//   tap = (dr+1) 9 + (de+1) 3 + (da+1), u over the N_a periodic azimuths.
// K = the azimuths of one output theta-row (16 per MMA). A = H, M = 128: the
// rows (r-1, r, r+1; e + de) x 32 input channels (96; the last 32 rows repeat
// whatever follows and are not read back). B = Gz, N = 96: the output row's
// gradient three times, rotated by the azimuth tap. Both are MN-major with a
// 64-byte swizzle, the layout in which TMA lands a theta-row of 32 bf16
// channels ([azimuth][channel], 64 bytes per azimuth): 32-element blocks along
// M / N one theta-row apart (the descriptor's leading offset), 8 azimuths 512
// bytes apart along K (its stride offset). Three accumulator tiles (de) of 96
// columns collect every row the CTA processes; the epilogue writes the CTA's
// partial dW, which part_reduce_kernel sums in a fixed order.
//
// A CTA takes a contiguous run of output rows (b, r, e) and walks along e, so
// of the nine H rows an output row needs only the three of e + 1 are new: a
// ring of H slots (three rows each) and one of Gz slots (three copies), one
// elected lane issuing six boxes per row. The copies' wrapped azimuth (TMA
// fills it with zeros) is patched from the unrotated copy by a warp of its
// own.
//
// Measured at batch 8, 64 x 48 x 96 on GB300: 435 us a layer before (N = 32
// with one MMA per azimuth tap over 16-byte channel planes, all nine rows
// loaded again for every output row), 195 us now. It is bound by the tensor
// cores (about 130 cycles per MMA): fewer bytes loaded or longer rings change
// nothing, a third of the MMAs takes 139 us. Issued by one elected lane: with
// elect.sync around every MMA the same kernel took 243 us.
// ---------------------------------------------------------------------------
constexpr int WG_MAX_SLOTS = 5;
__host__ __device__ inline int wg_slot(int Na) { return 3 * Na * 64; }  // bytes of three theta-rows
// slots of the two rings: as many as fit
__host__ __device__ inline int wg_h_slots(int Na) { return 8 * wg_slot(Na) + 2048 <= 232448 ? 5 : 4; }
__host__ __device__ inline int wg_g_slots(int Na) { return 7 * wg_slot(Na) + 2048 <= 232448 ? 3 : 2; }
// Dynamic shared memory of a launch: the slots, at least 116 KB so that one
// CTA (which allocates all 512 TMEM columns) holds a multiprocessor.
inline int wg_smem(int Na) { return std::max((wg_h_slots(Na) + wg_g_slots(Na)) * wg_slot(Na), 116 * 1024); }
// kind::f16: f32 accumulator, bf16 A and B, both MN-major, N = 96, M = 128.
constexpr uint32_t WG_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((96u >> 3) << 17) |
                              ((128u >> 4) << 24);
// Descriptor of an MN-major operand with 64-byte swizzle (layout type 4):
// leading offset between 32-element blocks along M / N, stride offset between
// groups of eight along K.
__device__ __forceinline__ uint64_t wg_desc(uint32_t addr, uint32_t lbo) {
  return umma_desc(addr, lbo, 512) | (uint64_t(4) << 61);
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// AND of p over the 128 epilogue threads of wgrad32_tc_kernel (named barrier 2).
__device__ __forceinline__ bool wg_epilogue_and(bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred pi, po;\n setp.ne.u32 pi, %1, 0;\n bar.red.and.pred po, 2, 128, pi;\n selp.u32 %0, 1, 0, po;\n}"
      : "=r"(r)
      : "r"(uint32_t(p))
      : "memory");
  return r != 0;
}

// Warp 0 issues the MMAs, warp 1 the loads, warp 2 patches, warps 4-7 read the accumulators
// back at the end. hmap / gmap: boxes of one theta-row (32 channels x N_a).
// part: [gridDim.x][27][32][32], bpart: [gridDim.x][32].
__global__ void __launch_bounds__(256, 1) wgrad32_tc_kernel(const __grid_constant__ CUtensorMap hmap,
                                                            const __grid_constant__ CUtensorMap gmap, Dims d,
                                                            float* __restrict__ part, float* __restrict__ bpart,
                                                            long long budget) {
  extern __shared__ __align__(1024) unsigned char smem[];
  // hfull / gfull[s]: slot s loaded (TMA bytes); gready[s]: copies patched (one arrival per lane of warp 2);
  // hempty / gempty[s]: the slot's MMAs done (commit), and for Gz its column sums (four warps);
  // done: every MMA of the CTA done (commit)
  __shared__ __align__(8) uint64_t hfull[WG_MAX_SLOTS], hempty[WG_MAX_SLOTS], gfull[3], gready[3], gempty[3], done;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_abort;
  __shared__ float s_cs[4][CH];
  const int Na = d.Na, ROW = Na * 64, SLOT = wg_slot(Na), NH = wg_h_slots(Na), NG = wg_g_slots(Na);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t rows = int64_t(d.B) * d.Nr * d.Ne;
  const int64_t row0 = rows * blockIdx.x / gridDim.x, row1 = rows * (blockIdx.x + 1) / gridDim.x;
  if (smem_u32(smem) & 511u) {  // the swizzle pattern repeats every 512 bytes: report, touch nothing
    if (tid == 0) atomicOr(&g_conv_error_word, 2);
    return;
  }
  if (tid == 0) {
    s_abort = 0;
    for (int k = 0; k < WG_MAX_SLOTS; ++k) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&hfull[k])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&hempty[k])) : "memory");
    }
    for (int k = 0; k < 3; ++k) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&gfull[k])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 32;" ::"r"(smem_u32(&gready[k])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 5;" ::"r"(smem_u32(&gempty[k])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  unsigned char* const gbase = smem + size_t(NH) * SLOT;

  // Both roles walk the CTA's rows in runs of one column (b, r): a run of n
  // rows takes n + 2 H loads (theta-rows e - 1 .. e + n) and n Gz loads.
  if (warp == 0) {  // ---- MMA issuer: one lane ----
    if (elect_one()) {
      bool go = true;
      uint32_t started = 0;
      int h0 = 0, gi = 0;  // H loads before this run, Gz loads so far
      for (int64_t row = row0; row < row1 && go;) {
        const int n = int(min(row1 - row, int64_t(d.Ne) - row % d.Ne));
        for (int i = 0; i < n; ++i, ++gi) {
          const int gs = gi % NG;
          for (int k = i == 0 ? 0 : 2; k < 3 && go; ++k)
            go = tc_wait(&hfull[(h0 + i + k) % NH], uint32_t((h0 + i + k) / NH) & 1u, &s_abort, budget);
          if (!go || !tc_wait(&gready[gs], uint32_t(gi / NG) & 1u, &s_abort, budget)) {
            go = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t bd0 = wg_desc(smem_u32(gbase + size_t(gs) * SLOT), uint32_t(ROW));
          for (int k = 0; k < 3; ++k) {  // theta tap
            const uint64_t ad0 = wg_desc(smem_u32(smem + size_t((h0 + i + k) % NH) * SLOT), uint32_t(ROW));
#pragma unroll 2
            for (int u = 0; u < Na / 16; ++u)  // 16 azimuths: 1024 bytes
              tc_mma(tmem + uint32_t(k) * 96, ad0 + uint64_t(u) * 64, bd0 + uint64_t(u) * 64, WG_IDESC,
                     started | uint32_t(u));
          }
          started = 1;
          tc_commit(&gempty[gs]);
          tc_commit(&hempty[(h0 + i) % NH]);
          if (i == n - 1) {
            tc_commit(&hempty[(h0 + i + 1) % NH]);
            tc_commit(&hempty[(h0 + i + 2) % NH]);
          }
        }
        h0 += n + 2;
        row += n;
      }
      if (go) {
        tc_commit(&done);
      } else {  // let issued MMAs land before TMEM is released
        const long long t0 = clock64();
        while (clock64() - t0 < budget / 8) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 2) {  // ---- the rotated copies' wrapped azimuths, from the unrotated one ----
    for (int gi = 0; gi < int(row1 - row0); ++gi) {
      const int gs = gi % NG;
      if (!__all_sync(0xffffffffu, tc_wait(&gfull[gs], uint32_t(gi / NG) & 1u, &s_abort, budget))) break;
      unsigned char* const g = gbase + size_t(gs) * SLOT;
      if (lane < 4) *row_chunk(g, Na - 1, lane) = *row_chunk(g + ROW, 0, lane);
      else if (lane < 8) *row_chunk(g + 2 * ROW, 0, lane - 4) = *row_chunk(g + ROW, Na - 1, lane - 4);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // -> tensor-core reads
      mbar_arrive(&gready[gs]);
    }
  } else if (warp == 1) {  // ---- loader: one lane ----
    if (lane == 0) {
      bool go = true;
      int h = 0, gi = 0;
      for (int64_t row = row0; row < row1 && go;) {
        const int n = int(min(row1 - row, int64_t(d.Ne) - row % d.Ne));
        const int e0 = int(row % d.Ne), r = int((row / d.Ne) % d.Nr), b = int(row / (int64_t(d.Ne) * d.Nr));
        for (int j = 0; j < n + 2 && go; ++j, ++h) {  // H rows e0 - 1 + j, then (from the third on) Gz row e0 + j - 2
          const int hs = h % NH;
          if (h >= NH && !tc_wait(&hempty[hs], uint32_t(h / NH - 1) & 1u, &s_abort, budget)) {
            go = false;
            break;
          }
          mbar_arrive_expect_tx(&hfull[hs], uint32_t(SLOT));
          for (int k = 0; k < 3; ++k)  // out-of-grid theta-rows and shells read as zeros
            tma_load_5d(smem + size_t(hs) * SLOT + size_t(k) * ROW, &hmap, 0, 0, e0 - 1 + j, r + k - 1, b, &hfull[hs]);
          if (j < 2) continue;
          const int gs = gi % NG;
          if (gi >= NG && !tc_wait(&gempty[gs], uint32_t(gi / NG - 1) & 1u, &s_abort, budget)) {
            go = false;
            break;
          }
          mbar_arrive_expect_tx(&gfull[gs], uint32_t(SLOT));
          for (int k = 0; k < 3; ++k)  // copy k holds Gz at azimuth u - (k - 1)
            tma_load_5d(gbase + size_t(gs) * SLOT + size_t(k) * ROW, &gmap, 0, 1 - k, e0 + j - 2, r, b, &gfull[gs]);
          ++gi;
        }
        row += n;
      }
    }
    __syncwarp();
  } else if (warp >= 4) {  // ---- epilogue: the CTA's partial dW ----
    // meanwhile: the column sums of Gz (the bias gradient) from the unrotated
    // copy; a thread adds its eight channels of every 32nd azimuth, in order:
    // a row's (at most six) plainly, the rows with the remainder of each
    // addition kept (a plain chain over all of a CTA's rows, 485 values at
    // batch 8 of 64 x 48 x 96, is off by its length)
    const int c8 = tid & 3, u0 = (tid - 128) >> 2;
    float cs[8], rem[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) cs[i] = rem[i] = 0.0f;
    for (int gi = 0; gi < int(row1 - row0); ++gi) {
      const int gs = gi % NG;
      if (!__all_sync(0xffffffffu, tc_wait(&gfull[gs], uint32_t(gi / NG) & 1u, &s_abort, budget))) break;
      unsigned char* const g = gbase + size_t(gs) * SLOT + ROW;
      float rs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int u = u0; u < Na; u += 32) {
        const uint4 v = *row_chunk(g, u, c8);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
          rs[2 * i] += f.x;
          rs[2 * i + 1] += f.y;
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float t = cs[i] + rs[i], z = t - cs[i];
        rem[i] += (cs[i] - (t - z)) + (rs[i] - z);
        cs[i] = t;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&gempty[gs]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {  // the 8 threads of a channel group in a warp, then the 4 warps in order
      if (rem[i] == rem[i]) cs[i] += rem[i];  // (an infinite sum has no remainder)
      cs[i] += __shfl_xor_sync(0xffffffffu, cs[i], 4);
      cs[i] += __shfl_xor_sync(0xffffffffu, cs[i], 8);
      cs[i] += __shfl_xor_sync(0xffffffffu, cs[i], 16);
      if (lane < 4) s_cs[warp - 4][8 * lane + i] = cs[i];
    }
    const int q = warp & 3;  // shell tap; quarter 3 holds the rows beyond the three
    float* out = part + size_t(blockIdx.x) * 27 * CH * CH;
    const bool ok = wg_epilogue_and(tc_wait(&done, 0u, &s_abort, budget));
    if (ok && q == 3)
      bpart[size_t(blockIdx.x) * CH + lane] = ((s_cs[0][lane] + s_cs[1][lane]) + s_cs[2][lane]) + s_cs[3][lane];
    if (ok && q < 3) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int t = 0; t < 9; ++t) {  // theta tap, azimuth tap
        const int tap = 9 * q + t;
        uint32_t v[16];
        for (int h = 0; h < 2; ++h) {  // output channels 16 h .. 16 h + 15 of input channel ci = lane
          tmem_ld_nowait<16>(tmem + (uint32_t(32 * q) << 16) + uint32_t(t * 32 + 16 * h), v);
          tmem_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) out[(size_t(tap) * CH + 16 * h + j) * CH + lane] = __uint_as_float(v[j]);
        }
      }
    }
  }
  __syncthreads();
  if (tid == 0 && s_abort) atomicOr(&g_conv_error_word, 1);  // TSP_DEVERR_WAIT_TIMEOUT once shifted
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ---------------------------------------------------------------------------
// CUDA-core layers and element-wise pieces
// ---------------------------------------------------------------------------
__global__ void to_bf16_kernel(const float* __restrict__ x, bf16* __restrict__ y, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

// Weight preparation from the float32 masters: bf16 tensors for the tensor-core
// layers (forward [tap][co][ci], dgrad [tap'][ci][co] with tap' the mirrored tap)
// and bf16-rounded float copies for the CUDA-core layers.
__global__ void prep_weights_kernel(const float* __restrict__ w, bf16* __restrict__ wf, bf16* __restrict__ wd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 27 * CH * CH) return;
  const int tap = i / (CH * CH), co = (i / CH) % CH, ci = i % CH;
  const bf16 v = __float2bfloat16_rn(w[i]);
  wf[i] = v;
  wd[(size_t(26 - tap) * CH + ci) * CH + co] = v;
}

// Output layer weights w6 [27][32] in the 32 -> 32 layout [27][co][ci]:
// output channel 0 holds them, the other 31 are zero.
__global__ void pad_w6_kernel(const float* __restrict__ w6, bf16* __restrict__ wf6) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 27 * CH * CH) return;
  const int tap = i / (CH * CH), co = (i / CH) % CH, ci = i % CH;
  wf6[i] = __float2bfloat16_rn(co == 0 ? w6[tap * CH + ci] : 0.0f);
}

__global__ void round_bf16_kernel(const float* __restrict__ w, float* __restrict__ out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = __bfloat162float(__float2bfloat16_rn(w[i]));
}

// Packed pairs of float32 (two independent IEEE multiply-adds per instruction).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// Layers with one channel on the input side, 32 on the output side; the 27
// taps are summed in order, two channels per instruction:
//   MODE 0, input layer:  h1 = relu(conv(a; w1) + b1), and its mask;
//   MODE 1, output layer backward: g_h[v][ci] = sum_tap w6[tap][ci] g_out[v - d_tap],
//           and gz = g_h gated by the mask of the layer below, in bf16.
// A thread takes eight neighbouring azimuths and eight channels: every weight
// read from shared memory (two 16-byte reads a tap) then serves eight voxels,
// and four lanes write a voxel's row. With one voxel and all channels per
// thread the weight reads, which return 512 bytes a warp however many lanes
// share them, bound it. Batch 8 of 64 x 48 x 96 on GB300: input layer 221 us
// before (scalar reads), 156 with two voxels a thread, 130 now; output layer
// backward with its gate 352, 183 and 132 us.
constexpr int THIN_V = 8, THIN_C = 8;  // voxels and channels per thread
template <int MODE>
__global__ void __launch_bounds__(128) thin_conv_kernel(Dims d, const bf16* __restrict__ a, const float* __restrict__ gout,
                                                        const float* __restrict__ w, const float* __restrict__ b1,
                                                        bf16* __restrict__ h, uint32_t* __restrict__ mask,
                                                        float* __restrict__ gh) {
  __shared__ __align__(16) float sw[27 * CH];
  for (int i = threadIdx.x; i < 27 * CH; i += blockDim.x) sw[i] = w[i];
  __syncthreads();
  const int64_t gi = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int c0 = int(gi & 3) * THIN_C;
  const int64_t g0 = (gi >> 2) * THIN_V;  // the first voxel (N_a is a multiple of 32)
  if (g0 >= int64_t(d.B) * d.V) return;
  const int Na = d.Na;
  const int64_t row = g0 / Na;
  const int a0 = int(g0 - row * Na), e = int(row % d.Ne), r = int((row / d.Ne) % d.Nr);
  const int64_t v0 = row * Na;  // first voxel of this theta-row
  f32x2 acc[THIN_V][THIN_C / 2];
#pragma unroll
  for (int c = 0; c < THIN_C / 2; ++c) {
    const f32x2 z = MODE == 0 ? pack2(b1[c0 + 2 * c], b1[c0 + 2 * c + 1]) : pack2(0.0f, 0.0f);
#pragma unroll
    for (int v = 0; v < THIN_V; ++v) acc[v][c] = z;
  }
#pragma unroll 1
  for (int t9 = 0; t9 < 9; ++t9) {
    const int dr = MODE == 0 ? t9 / 3 - 1 : 1 - t9 / 3, de = MODE == 0 ? t9 % 3 - 1 : 1 - t9 % 3;
    if (r + dr < 0 || r + dr >= d.Nr || e + de < 0 || e + de >= d.Ne) continue;
    const int64_t q = v0 + (int64_t(dr) * d.Ne + de) * Na;
    const int al = a0 == 0 ? Na - 1 : a0 - 1, ar = a0 + THIN_V == Na ? 0 : a0 + THIN_V;
    float s[THIN_V + 2];  // the scalar field at azimuths a0 - 1 .. a0 + 8
    if (MODE == 0) {
      const uint4 m = *reinterpret_cast<const uint4*>(a + q + a0);
      const uint32_t mw[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&mw[i]));
        s[1 + 2 * i] = f.x;
        s[2 + 2 * i] = f.y;
      }
      s[0] = __bfloat162float(a[q + al]);
      s[THIN_V + 1] = __bfloat162float(a[q + ar]);
    } else {
#pragma unroll
      for (int i = 0; i < THIN_V / 4; ++i) {
        const float4 m = *reinterpret_cast<const float4*>(gout + q + a0 + 4 * i);
        s[1 + 4 * i] = m.x;
        s[2 + 4 * i] = m.y;
        s[3 + 4 * i] = m.z;
        s[4 + 4 * i] = m.w;
      }
      s[0] = gout[q + al];
      s[THIN_V + 1] = gout[q + ar];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int o = MODE == 0 ? k : 2 - k;
      const ulonglong2* wr = reinterpret_cast<const ulonglong2*>(sw + (t9 * 3 + k) * CH + c0);
      const ulonglong2 w0 = wr[0], w1 = wr[1];
#pragma unroll
      for (int v = 0; v < THIN_V; ++v) {
        const f32x2 sv = pack2(s[v + o], s[v + o]);
        acc[v][0] = fma2(w0.x, sv, acc[v][0]);
        acc[v][1] = fma2(w0.y, sv, acc[v][1]);
        acc[v][2] = fma2(w1.x, sv, acc[v][2]);
        acc[v][3] = fma2(w1.y, sv, acc[v][3]);
      }
    }
  }
#pragma unroll
  for (int v = 0; v < THIN_V; ++v) {
    const size_t vox = size_t(g0 + v);
    uint8_t* const mb = reinterpret_cast<uint8_t*>(mask + vox) + (c0 >> 3);  // this thread's byte of the mask word
    float z[THIN_C];
#pragma unroll
    for (int c = 0; c < THIN_C / 2; ++c) unpack2(acc[v][c], z[2 * c], z[2 * c + 1]);
    uint32_t bits = MODE == 1 ? *mb : 0u;
    if (MODE == 0) {
#pragma unroll
      for (int c = 0; c < THIN_C; ++c) bits |= (z[c] > 0.0f ? 1u : 0u) << c;
      *mb = uint8_t(bits);
    } else {
      b32x8 o;
#pragma unroll
      for (int c = 0; c < THIN_C; ++c) o.v[c] = __float_as_uint(z[c]);
      stg32(gh + vox * CH + c0, o);
    }
    uint4 y;  // relu(z) and the gated gradient: z where the bit is set
    uint32_t* yw = reinterpret_cast<uint32_t*>(&y);
#pragma unroll
    for (int c = 0; c < THIN_C / 2; ++c) {
      const __nv_bfloat162 p = __floats2bfloat162_rn((bits >> (2 * c)) & 1u ? z[2 * c] : 0.0f,
                                                     (bits >> (2 * c + 1)) & 1u ? z[2 * c + 1] : 0.0f);
      yw[c] = *reinterpret_cast<const uint32_t*>(&p);
    }
    *reinterpret_cast<uint4*>(h + vox * CH + c0) = y;
  }
}

// g_out = 2 (out - target) / n; shares[block] = the block's share of
// sum (out - target)^2 / n (double), summed by ordered_sum_kernel.
constexpr int MSE_BLOCKS = 152 * 8;
__global__ void mse_kernel(const float* __restrict__ out, const float* __restrict__ tgt, int64_t n,
                           float* __restrict__ g, double* __restrict__ shares) {
  double acc = 0.0;
  const double inv = 1.0 / double(n);
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float diff = out[i] - tgt[i];
    g[i] = float(2.0 * inv * double(diff));
    acc += double(diff) * double(diff) * inv;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) shares[blockIdx.x] = v;
  }
}

// *out = sum of part[0 .. n) in a fixed order (one warp: strided lane sums,
// then a shuffle tree), so the loss repeats bit for bit.
__global__ void ordered_sum_kernel(const double* __restrict__ part, int n, double* __restrict__ out) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) v += part[i];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) *out = v;
}

// ---------------------------------------------------------------------------
// Weight gradients of the one-sided layers (one channel on one side, 32 on the
// other), in one pass over the voxels:
//   mode 0 (output layer 32 -> 1): dw[tap][c] = sum_v g1[v] X[v + d_tap][c]
//                                            = sum_u X[u][c] g1[u - d_tap],  db = sum g1
//   mode 1 (input layer 1 -> 32):  dw[tap][c] = sum_v gz[v][c] a1[v + d_tap],
//                                  gz = g_h where the pre-activation was positive, db[c] = sum gz
// Both read dw[tap][c] = sum_u P[u][c] s(u + sigma d_tap): P the 32-channel
// operand (X, or the gated g_h), s the scalar field (g1, or a1), sigma = -1 / +1.
// A contraction over the voxels (M = 27 taps, N = 32 channels): mma.sync
// m16n8k16, whose fragments come straight from the staged rows; the pass is
// bound by reading P, so tcgen05's rate and its accumulators' read-back would
// buy nothing. Of the two operands one is bf16 and the other float32 (X and
// g1; a1 and g_h): the float32 one is cut into three bf16 parts whose sum it
// is exactly (8 + 8 + 8 bits), so every product is exact, and every 16 voxels'
// sums (the highest parts' by themselves: nearly exact) start from zero and are
// added, rounded to nearest, to float32 sums outside the tensor core, whose own
// running sums are cut off.
// A CTA takes tiles of ET theta-rows and stages the 3 x (ET + 2) rows of s
// around one, each three times, rotated by the azimuth tap, so that a tap's two
// neighbouring azimuths are one aligned word; its 8 warps take 16 azimuths of a
// row at a time. P goes from memory to the fragments of B: column n of tile j
// is channel 4 n + j, so a lane's four columns of a voxel are one vector load,
// and the next 16 voxels' loads are issued before this one's matrix steps.
// (Staged in shared memory, split there: mode 1 at 242 us, 150 in mode 0.) Row
// 27 of A is ones in mode 1: db. Each CTA writes its sums to its row of `part`
// (THIN_OUT floats: 27 x 32 weights, then 32 biases); part_reduce_kernel adds
// the rows in a fixed order (deterministic). Batch 8 of 64 x 48 x 96 on GB300,
// mode 0 / 1: 226 / 230 us with float32 FMAs of channel pairs, 117 / 132 now.
// ---------------------------------------------------------------------------
constexpr int THIN_OUT = 27 * CH + CH;

// theta-rows per tile: the largest power of two <= 16 with ET N_a <= 384
inline int thin_et(int Na) {
  int et = 1;
  while (et < 16 && 2 * et * Na <= 384) et *= 2;
  return et;
}
// bytes of a staged row of s (an odd number of 16-byte chunks: N_a is a multiple of 32)
__host__ __device__ inline int thin_row(int Na) { return Na * 2 + 16; }
inline size_t thin_smem(int Na, int mode) {
  return std::max(size_t(mode == 1 ? 1 : 3) * 9 * (thin_et(Na) + 2) * thin_row(Na), sizeof(float) * 8 * THIN_OUT);
}

// f = hi + mid + lo, each a bf16 (the bits of its upper half), exactly: the
// three bytes of its significand. An infinity or a NaN is all three: beside an
// infinite hi, zeros would make NaN of its products with infinities.
struct Split3 {
  uint32_t p[3];  // lo, mid, hi
};
__device__ __forceinline__ Split3 split3(float f) {
  const uint32_t b = __float_as_uint(f);
  const bool finite = (b & 0x7f800000u) != 0x7f800000u;
  uint32_t hi = b & 0xffff0000u;
  if (f != f) hi |= 0x00400000u;
  const float r = f - __uint_as_float(hi);
  const uint32_t mid = finite ? __float_as_uint(r) & 0xffff0000u : hi;
  Split3 o;
  o.p[0] = (finite ? __float_as_uint(r - __uint_as_float(mid)) : hi) >> 16;
  o.p[1] = mid >> 16;
  o.p[2] = hi >> 16;
  return o;
}
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// P of a lane's four voxels (2 t, 2 t + 1, 2 t + 8, 2 t + 9) of 16, channels 4 g .. 4 g + 3.
template <int MODE>
struct ThinP {
  float4 f[MODE == 1 ? 4 : 1];
  uint32_t m[MODE == 1 ? 4 : 1];
  uint2 x[MODE == 1 ? 1 : 4];
  __device__ __forceinline__ void load(const float* __restrict__ gh, const uint32_t* __restrict__ mask,
                                       const bf16* __restrict__ X32, int64_t v, int g, int t) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t vi = v + 2 * t + (i & 1) + 8 * (i >> 1);
      if (MODE == 1) {
        f[i] = __ldg(reinterpret_cast<const float4*>(gh + vi * CH + 4 * g));
        m[i] = __ldg(mask + vi);
      } else {
        x[i] = __ldg(reinterpret_cast<const uint2*>(X32 + vi * CH + 4 * g));
      }
    }
  }
};

template <int MODE>
__global__ void __launch_bounds__(256, 2) thin_wgrad_kernel(Dims d, int ET, const float* __restrict__ g1,
                                                            const bf16* __restrict__ X32, const float* __restrict__ gh,
                                                            const uint32_t* __restrict__ mask,
                                                            const bf16* __restrict__ a1, float* __restrict__ part) {
  constexpr int NP = MODE == 1 ? 3 : 1, NS = MODE == 1 ? 1 : 3;  // parts of P and of s
  extern __shared__ __align__(16) unsigned char thin_sm[];
  const int Na = d.Na, ETS = ET + 2, SR = thin_row(Na), planeS = 9 * ETS * SR;
  unsigned char* sS = thin_sm;  // [NS][azimuth tap][3][ET + 2] rows of bf16
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  // the rows of A of this lane: window element m = o 9 + oe 3 + k, s at (r + o - 1, e + oe - 1, a + k - 1)
  int aoff[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int m = 8 * j + g;
    aoff[j] = (((m % 3) * 3 + m / 9) * ETS + (m / 3) % 3) * SR + 4 * t;
  }
  const uint32_t row3 = MODE == 1 && g == 3 ? 0x3f803f80u : 0u;  // rows 27 (ones) and 28-31 (zeros)
  float sum[2][4][4], gsum = 0.0f;
#pragma unroll
  for (int i = 0; i < 32; ++i) sum[i / 16][i / 4 % 4][i % 4] = 0.0f;
  const int nET = (d.Ne + ET - 1) / ET, per_row = Na / 16;
  const int64_t tiles = int64_t(d.B) * d.Nr * nET;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int e0 = int(tile % nET) * ET, r = int((tile / nET) % d.Nr), b = int(tile / (int64_t(nET) * d.Nr));
    const int ETe = min(ET, d.Ne - e0);
    const int64_t v0 = ((int64_t(b) * d.Nr + r) * d.Ne + e0) * Na;  // first voxel of the tile (rows are contiguous)
    ThinP<MODE> next;
    if (warp < ETe * per_row) next.load(gh, mask, X32, v0 + warp * 16, g, t);
    __syncthreads();  // the previous tile is no longer read
    for (int row = warp; row < 3 * ETS; row += 8) {  // a warp per row, its loads first
      const int rr = row / ETS, ee = row - rr * ETS, rg = r - 1 + rr, eg = e0 - 1 + ee;
      const bool in = rg >= 0 && rg < d.Nr && eg >= 0 && eg < d.Ne;
      const int64_t q0 = int64_t(b) * d.V + (int64_t(rg) * d.Ne + eg) * Na + lane;
      float v[6];  // N_a <= 192
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        v[i] = 0.0f;
        if (in && 32 * i < Na) v[i] = MODE == 1 ? __bfloat162float(a1[q0 + 32 * i]) : g1[q0 + 32 * i];
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        if (32 * i >= Na) break;
        if (MODE == 0 && rr == 1 && ee >= 1 && ee <= ETe) gsum += v[i];
        Split3 f;
        if (MODE == 1) f.p[0] = __float_as_uint(v[i]) >> 16;
        else f = split3(v[i]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {  // position a of copy k holds azimuth a + k - 1
          int pos = lane + 32 * i + 1 - k;
          pos = pos < 0 ? pos + Na : (pos >= Na ? pos - Na : pos);
          unsigned char* q = sS + (k * 3 * ETS + row) * SR + 2 * pos;
#pragma unroll
          for (int n = 0; n < NS; ++n) *reinterpret_cast<unsigned short*>(q + n * planeS) = (unsigned short)(f.p[n]);
        }
      }
    }
    __syncthreads();
    for (int grp = warp; grp < ETe * per_row; grp += 8) {
      const ThinP<MODE> p = next;
      if (grp + 8 < ETe * per_row) next.load(gh, mask, X32, v0 + (grp + 8) * 16, g, t);
      const int el = grp / per_row, a0 = (grp - el * per_row) * 16;
      const unsigned char* arow = sS + el * SR + 2 * a0;
      uint32_t bf[NP][4][2];  // [part][tile j: channel 4 g + j][azimuths 2 t, 2 t + 1; 8 on]
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (MODE == 1) {
            Split3 q[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float4 f4 = p.f[2 * h + i];
              const float v = j == 0 ? f4.x : j == 1 ? f4.y : j == 2 ? f4.z : f4.w;
              q[i] = split3((p.m[2 * h + i] >> (4 * g + j)) & 1u ? v : 0.0f);
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) bf[k][j][h] = q[0].p[k] | (q[1].p[k] << 16);
          } else {
            const uint32_t u0 = j < 2 ? p.x[2 * h].x : p.x[2 * h].y, u1 = j < 2 ? p.x[2 * h + 1].x : p.x[2 * h + 1].y;
            bf[0][j][h] = __byte_perm(u0, u1, j & 1 ? 0x7632 : 0x5410);
          }
        }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        float hi[4][4], lo[4][4];  // sums of the highest parts' products, of the other two's
#pragma unroll
        for (int i = 0; i < 16; ++i) hi[i / 4][i % 4] = lo[i / 4][i % 4] = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          uint32_t af[4];
#pragma unroll
          for (int j = 0; j < 2; ++j) {  // rows 16 mt + 8 j + g: azimuths 2 t, 2 t + 1, then 8 on
            const unsigned char* q = arow + (NS == 3 ? k : 0) * planeS + aoff[2 * mt + j];
            const bool on = mt + j < 2 || g < 3;
            af[j] = on ? *reinterpret_cast<const uint32_t*>(q) : row3;
            af[2 + j] = on ? *reinterpret_cast<const uint32_t*>(q + 16) : row3;
          }
#pragma unroll
          for (int n = 0; n < 4; ++n)
            mma_16816(k == 2 ? hi[n] : lo[n], af, bf[NP == 3 ? k : 0][n][0], bf[NP == 3 ? k : 0][n][1]);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) sum[mt][i / 4][i % 4] += hi[i / 4][i % 4] + lo[i / 4][i % 4];
      }
    }
  }
  // the 8 warps' sums, added in order
  __syncthreads();
  float* red = reinterpret_cast<float*>(thin_sm) + warp * THIN_OUT;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int m = 16 * mt + g + 8 * (i >> 1), c = 4 * (2 * t + (i & 1)) + n;
        // mode 1: the window offset is d_tap; mode 0: it is -d_tap
        if (m < 27) red[(MODE == 1 ? m : 26 - m) * CH + c] = sum[mt][n][i];
        else if (MODE == 1 && m == 27) red[27 * CH + c] = sum[mt][n][i];
      }
  if (MODE == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gsum += __shfl_xor_sync(0xffffffffu, gsum, o);
    red[27 * CH + lane] = lane == 0 ? gsum : 0.0f;
  }
  __syncthreads();
  for (int i = tid; i < THIN_OUT; i += 256) {
    float v = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += reinterpret_cast<float*>(thin_sm)[k * THIN_OUT + i];
    part[size_t(blockIdx.x) * THIN_OUT + i] = v;
  }
}

// out[i] += sum_k part[k][i] for i < n (rows of `stride` floats), k in order:
// 32 outputs per CTA, warp w takes rows w, w + 32, ...
__global__ void __launch_bounds__(1024) part_reduce_kernel(const float* __restrict__ part, int rows, int stride, int n,
                                                           float* __restrict__ out) {
  __shared__ float s[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  float v = 0.0f;
  if (i < n)
    for (int k = warp; k < rows; k += 32) v += part[size_t(k) * stride + i];
  s[warp][lane] = v;
  __syncthreads();
  if (warp == 0 && i < n) {
    // compensated: this chain's rounding was most of a gradient's error (in
    // double it takes half as long again as the whole kernel)
    float t = 0.0f, c = 0.0f;
    for (int w = 0; w < 32; ++w) {
      const float x = s[w][lane], y = t + x, z = y - t;
      c += (t - (y - z)) + (x - z);
      t = y;
    }
    out[i] += c == c ? t + c : t;  // (an infinite sum has no remainder)
  }
}

int blocks_for(int64_t n, int threads) { return int(std::min<int64_t>((n + threads - 1) / threads, 1 << 30)); }

}  // namespace
}  // namespace tsp

using namespace tsp;

// Parameter layout (float32, flat): w1 [27][32][1], b1 [32], w2..w5 [27][32][32],
// b2..b5 [32], w6 [27][1][32], b6 [1].
struct tsp_net_s {
  Dims d{};
  int max_batch = 0;
  int device = 0;
  size_t n_params = 0;
  size_t off_w[6], off_b[6];
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  bf16 *wf[4] = {nullptr, nullptr, nullptr, nullptr}, *wd[4] = {nullptr, nullptr, nullptr, nullptr};
  float *w1r = nullptr, *w6r = nullptr;
  bf16* wf6 = nullptr;  // output layer weights in the 32 -> 32 layout (tensor-core forward)
  bf16* a16 = nullptr;
  bf16* h[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  uint32_t* mask[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  float *out = nullptr, *gout = nullptr, *gh = nullptr;
  bf16* gz[2] = {nullptr, nullptr};  // gated gradients: a dgrad reads one and writes the other
  double* loss = nullptr;
  double* loss_part = nullptr;  // per-block shares of the loss
  float* part = nullptr;  // per-CTA partial sums of the weight / bias gradient reductions
  int part_rows = 0;
  float* wpart = nullptr;  // per-CTA partial 32 -> 32 weight gradients [SMs][27][32][32]
  std::vector<void*> allocs;
  int adam_step = 0;
  bool prepared = false;  // wf / wd / w1r / w6r / wf6 hold the current parameters
  CUtensorMap map_h[5];  // TMA descriptors of the activations h1..h5 (inputs of the 32 -> 32 layers)
  CUtensorMap map_gz[2];  // and of the gated gradients (inputs of dgrad)
};

namespace {


// TMA descriptor of a bf16 activation tensor [B][N_r][N_e][N_a][32]: a 5-D
// tiled map (channels innermost) whose box is a theta-row, 32 channels x N_a
// azimuths, 64-byte swizzle; out-of-range theta-rows and shells read as zeros.
tsp_status encode_act_map(CUtensorMap* m, const bf16* base, const Dims& d) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    TSP_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !fn) return fail(TSP_ECUDA, "cuTensorMapEncodeTiled is not available");
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  const cuuint64_t dims[5] = {cuuint64_t(CH), cuuint64_t(d.Na), cuuint64_t(d.Ne), cuuint64_t(d.Nr), cuuint64_t(d.B)};
  const cuuint64_t strides[4] = {cuuint64_t(CH) * 2, cuuint64_t(CH) * 2 * d.Na, cuuint64_t(CH) * 2 * d.Na * d.Ne,
                                 cuuint64_t(CH) * 2 * d.Na * d.Ne * d.Nr};
  const cuuint32_t box[5] = {cuuint32_t(CH), cuuint32_t(d.Na), 1u, 1u, 1u};
  const cuuint32_t es[5] = {1u, 1u, 1u, 1u, 1u};
  const CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16*>(base), dims, strides, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(TSP_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string(int(r)) + ")");
  return TSP_OK;
}

template <class T>
tsp_status net_alloc(tsp_net n, T** p, size_t count) {
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * count);
  if (e != cudaSuccess) return cuda_fail(e, "tsp_net_create: allocation");
  n->allocs.push_back(*p);
  return TSP_OK;
}

int g_sm_count = 152;  // multiprocessors of the device the network lives on (set at creation)

// Allow f the most dynamic shared memory a block may have on this device
// (the opt-in limit less f's static shared memory). The attribute belongs to
// the function, not to a net, so it is set to the largest value once instead
// of to one net's need (nets of several azimuth counts may coexist).
template <class F>
tsp_status allow_max_smem(F* f, int dev) {
  int optin = 0;
  TSP_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  cudaFuncAttributes fa{};
  TSP_CUDA(cudaFuncGetAttributes(&fa, f));
  TSP_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - int(fa.sharedSizeBytes)));
  return TSP_OK;
}

tsp_status set_attrs(int Na) {
  int dev = 0;
  TSP_CUDA(cudaGetDevice(&dev));
  TSP_CUDA(cudaDeviceGetAttribute(&g_sm_count, cudaDevAttrMultiProcessorCount, dev));
  int optin = 0;
  TSP_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  if (int(tc_plan(Na).smem) + 4096 > optin || wg_smem(Na) + 4096 > optin || int(thin_smem(Na, 1)) + 4096 > optin || int(thin_smem(Na, 0)) + 4096 > optin)
    return fail(TSP_ENOTSUP, "tsp_net_create: the azimuth count needs more shared memory than a block may have");
  tsp_status st = allow_max_smem(conv32_tc_kernel<0>, dev);
  if (st == TSP_OK) st = allow_max_smem(conv32_tc_kernel<1>, dev);
  if (st == TSP_OK) st = allow_max_smem(conv32_tc_kernel<2>, dev);
  if (st == TSP_OK) st = allow_max_smem(wgrad32_tc_kernel, dev);
  if (st == TSP_OK) st = allow_max_smem(thin_wgrad_kernel<0>, dev);
  if (st == TSP_OK) st = allow_max_smem(thin_wgrad_kernel<1>, dev);
  return st;
}

// Armed by tsp_debug_tc_stall: the wait budget (cycles) of the next
// tensor-core convolution launch, whose loader then stalls; 0 = not armed.
std::atomic<long long> g_tc_stall{0};

// Persistent launch: work items (sample, chunk, run of rseg shells), about
// four per multiprocessor, one CTA per multiprocessor (its shared memory).
void conv32(int mode, const Dims& d, int B, const CUtensorMap& xmap, const bf16* X, const bf16* W, const float* bias,
            bf16* Y, uint32_t* mask, float* G, cudaStream_t st) {
  Dims db = d;
  db.B = B;
  const TcPlan pl = tc_plan(d.Na);
  const int P = d.Ne * (d.Na + 2);
  const int nq = (P + TC_TOUT * pl.T - 1) / (TC_TOUT * pl.T);
  const int64_t steps = int64_t(B) * nq * d.Nr;
  const int rseg = int(std::max<int64_t>(2, std::min<int64_t>(d.Nr, steps / (4 * int64_t(g_sm_count)))));
  const int64_t items = int64_t(B) * nq * ((d.Nr + rseg - 1) / rseg);
  const unsigned grid = unsigned(std::min<int64_t>(items, g_sm_count));
  // the one-shot test hook of tsp_debug_tc_stall: this launch's loader issues
  // nothing and its waits give up after the armed number of cycles
  const long long armed = g_tc_stall.exchange(0);
  const long long budget = armed > 0 ? armed : TC_WAIT_BUDGET;
  const int stall = armed > 0 ? 1 : 0;
  if (mode == 0)
    conv32_tc_kernel<0><<<grid, TC_THREADS, pl.smem, st>>>(xmap, db, rseg, X, W, bias, Y, mask, G, budget, stall);
  else if (mode == 1)
    conv32_tc_kernel<1><<<grid, TC_THREADS, pl.smem, st>>>(xmap, db, rseg, X, W, bias, Y, mask, G, budget, stall);
  else conv32_tc_kernel<2><<<grid, TC_THREADS, pl.smem, st>>>(xmap, db, rseg, X, W, bias, Y, mask, G, budget, stall);
}

tsp_status prepare_weights(tsp_net n, cudaStream_t st) {
  for (int k = 0; k < 4; ++k)
    prep_weights_kernel<<<(27 * CH * CH + 255) / 256, 256, 0, st>>>(n->params + n->off_w[k + 1], n->wf[k], n->wd[k]);
  round_bf16_kernel<<<(27 * CH + 255) / 256, 256, 0, st>>>(n->params + n->off_w[0], n->w1r, 27 * CH);
  round_bf16_kernel<<<(27 * CH + 255) / 256, 256, 0, st>>>(n->params + n->off_w[5], n->w6r, 27 * CH);
  pad_w6_kernel<<<(27 * CH * CH + 255) / 256, 256, 0, st>>>(n->params + n->off_w[5], n->wf6);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

tsp_status net_forward(tsp_net n, const float* a, int B, cudaStream_t st) {
  const Dims& d = n->d;
  Dims db = d;
  db.B = B;
  const int64_t nv = int64_t(B) * d.V;
  if (!n->prepared) {  // the bf16 / rounded copies, refreshed only after the parameters change
    tsp_status s = prepare_weights(n, st);
    if (s != TSP_OK) return s;
    n->prepared = true;
  }
  to_bf16_kernel<<<blocks_for(nv, 256), 256, 0, st>>>(a, n->a16, nv);
  thin_conv_kernel<0><<<blocks_for(nv / THIN_V * 4, 128), 128, 0, st>>>(db, n->a16, nullptr, n->w1r, n->params + n->off_b[0],
                                                               n->h[0], n->mask[0], nullptr);
  for (int k = 0; k < 4; ++k)
    conv32(0, d, B, n->map_h[k], n->h[k], n->wf[k], n->params + n->off_b[k + 1], n->h[k + 1], n->mask[k + 1], nullptr,
           st);
  conv32(2, d, B, n->map_h[4], n->h[4], n->wf6, n->params + n->off_b[5], n->a16, nullptr, n->out, st);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

}  // namespace

extern "C" tsp_status tsp_net_create(int n_r, int n_e, int n_a, int max_batch, tsp_net* out) {
  if (!out) return fail(TSP_EINVAL, "tsp_net_create: out is NULL");
  *out = nullptr;
  if (n_r <= 0 || n_e <= 0 || max_batch <= 0) return fail(TSP_EINVAL, "tsp_net_create: bad size");
  if (n_a % 32 != 0 || n_a < 32 || n_a > 192)
    return fail(TSP_ENOTSUP, "tsp_net_create: the azimuth count must be a multiple of 32 in [32, 192]");
  tsp_net n = new (std::nothrow) tsp_net_s();
  if (!n) return fail(TSP_ENOMEM, "tsp_net_create: host allocation");
  n->d = Dims{max_batch, n_r, n_e, n_a, int64_t(n_r) * n_e * n_a};
  n->max_batch = max_batch;
  cudaGetDevice(&n->device);
  size_t off = 0;
  const size_t wsz[6] = {27 * CH, 27 * CH * CH, 27 * CH * CH, 27 * CH * CH, 27 * CH * CH, 27 * CH};
  const size_t bsz[6] = {CH, CH, CH, CH, CH, 1};
  for (int k = 0; k < 6; ++k) {
    n->off_w[k] = off;
    off += wsz[k];
    n->off_b[k] = off;
    off += bsz[k];
  }
  n->n_params = off;
  const int64_t nv = int64_t(max_batch) * n->d.V;
  tsp_status st = TSP_OK;
  if (st == TSP_OK) st = net_alloc(n, &n->params, off);
  if (st == TSP_OK) st = net_alloc(n, &n->grads, off);
  if (st == TSP_OK) st = net_alloc(n, &n->m, off);
  if (st == TSP_OK) st = net_alloc(n, &n->v, off);
  for (int k = 0; k < 4 && st == TSP_OK; ++k) {
    st = net_alloc(n, &n->wf[k], 27 * CH * CH);
    if (st == TSP_OK) st = net_alloc(n, &n->wd[k], 27 * CH * CH);
  }
  if (st == TSP_OK) st = net_alloc(n, &n->w1r, 27 * CH);
  if (st == TSP_OK) st = net_alloc(n, &n->w6r, 27 * CH);
  if (st == TSP_OK) st = net_alloc(n, &n->wf6, 27 * CH * CH);
  if (st == TSP_OK) st = net_alloc(n, &n->a16, nv);
  for (int k = 0; k < 5 && st == TSP_OK; ++k) {
    st = net_alloc(n, &n->h[k], nv * CH);
    if (st == TSP_OK) st = net_alloc(n, &n->mask[k], nv);
  }
  if (st == TSP_OK) st = net_alloc(n, &n->out, nv);
  if (st == TSP_OK) st = net_alloc(n, &n->gout, nv);
  if (st == TSP_OK) st = net_alloc(n, &n->gh, nv * CH);
  for (int k = 0; k < 2 && st == TSP_OK; ++k) st = net_alloc(n, &n->gz[k], nv * CH);
  if (st == TSP_OK) st = net_alloc(n, &n->loss, 1);
  if (st == TSP_OK) st = net_alloc(n, &n->loss_part, MSE_BLOCKS);
  if (st == TSP_OK) st = set_attrs(n_a);
  if (st == TSP_OK) {  // one row per CTA of the reductions (2 per multiprocessor, THIN_OUT floats)
    n->part_rows = 2 * g_sm_count;
    st = net_alloc(n, &n->part, size_t(n->part_rows) * THIN_OUT);
    if (st == TSP_OK) st = net_alloc(n, &n->wpart, size_t(g_sm_count) * 27 * CH * CH);
  }
  for (int k = 0; k < 5 && st == TSP_OK; ++k) st = encode_act_map(&n->map_h[k], n->h[k], n->d);
  for (int k = 0; k < 2 && st == TSP_OK; ++k) st = encode_act_map(&n->map_gz[k], n->gz[k], n->d);
  if (st == TSP_OK) {
    cudaError_t e = cudaMemset(n->params, 0, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, sizeof(float) * off);
    if (e != cudaSuccess) st = cuda_fail(e, "tsp_net_create: clear");
  }
  if (st != TSP_OK) {
    tsp_net_destroy(n);
    return st;
  }
  *out = n;
  return TSP_OK;
}

extern "C" void tsp_net_destroy(tsp_net n) {
  if (!n) return;
  for (void* p : n->allocs) cudaFree(p);
  delete n;
}

extern "C" tsp_status tsp_debug_tc_stall(int64_t wait_cycles) {
  if (wait_cycles <= 0 || wait_cycles > TC_WAIT_BUDGET)
    return fail(TSP_EINVAL, "tsp_debug_tc_stall: wait_cycles must be in 1 .. " + std::to_string(TC_WAIT_BUDGET));
  g_tc_stall.store((long long)wait_cycles);
  return TSP_OK;
}

extern "C" tsp_status tsp_net_num_params(tsp_net n, size_t* count) {
  if (!n || !count) return fail(TSP_EINVAL, "tsp_net_num_params: NULL argument");
  *count = n->n_params;
  return TSP_OK;
}

extern "C" tsp_status tsp_net_set_params(tsp_net n, const float* host, size_t count) {
  if (!n || !host || count != n->n_params) return fail(TSP_EINVAL, "tsp_net_set_params: bad argument");
  TSP_CUDA(cudaMemcpy(n->params, host, sizeof(float) * count, cudaMemcpyHostToDevice));
  TSP_CUDA(cudaMemset(n->m, 0, sizeof(float) * count));
  TSP_CUDA(cudaMemset(n->v, 0, sizeof(float) * count));
  n->adam_step = 0;
  n->prepared = false;
  return TSP_OK;
}

extern "C" tsp_status tsp_net_get_params(tsp_net n, float* host, size_t count) {
  if (!n || !host || count != n->n_params) return fail(TSP_EINVAL, "tsp_net_get_params: bad argument");
  TSP_CUDA(cudaMemcpy(host, n->params, sizeof(float) * count, cudaMemcpyDeviceToHost));
  return TSP_OK;
}

extern "C" tsp_status tsp_net_get_state(tsp_net n, float* params, float* m, float* v, size_t count,
                                        int* adam_step) {
  if (!n || !params || !m || !v || !adam_step || count != n->n_params)
    return fail(TSP_EINVAL, "tsp_net_get_state: bad argument");
  tsp_status st = check_device(n->device);
  if (st != TSP_OK) return st;
  TSP_CUDA(cudaDeviceSynchronize());  // Adam steps enqueued on any stream have landed
  TSP_CUDA(cudaMemcpy(params, n->params, sizeof(float) * count, cudaMemcpyDeviceToHost));
  TSP_CUDA(cudaMemcpy(m, n->m, sizeof(float) * count, cudaMemcpyDeviceToHost));
  TSP_CUDA(cudaMemcpy(v, n->v, sizeof(float) * count, cudaMemcpyDeviceToHost));
  *adam_step = n->adam_step;
  return TSP_OK;
}

extern "C" tsp_status tsp_net_set_state(tsp_net n, const float* params, const float* m, const float* v,
                                        size_t count, int adam_step) {
  if (!n || !params || !m || !v || count != n->n_params || adam_step < 0)
    return fail(TSP_EINVAL, "tsp_net_set_state: bad argument");
  tsp_status st = check_device(n->device);
  if (st != TSP_OK) return st;
  TSP_CUDA(cudaDeviceSynchronize());  // no kernel of an earlier call still reads the old state
  TSP_CUDA(cudaMemcpy(n->params, params, sizeof(float) * count, cudaMemcpyHostToDevice));
  TSP_CUDA(cudaMemcpy(n->m, m, sizeof(float) * count, cudaMemcpyHostToDevice));
  TSP_CUDA(cudaMemcpy(n->v, v, sizeof(float) * count, cudaMemcpyHostToDevice));
  n->adam_step = adam_step;
  n->prepared = false;
  return TSP_OK;
}

extern "C" tsp_status tsp_net_get_grads(tsp_net n, float* host, size_t count) {
  if (!n || !host || count != n->n_params) return fail(TSP_EINVAL, "tsp_net_get_grads: bad argument");
  TSP_CUDA(cudaMemcpy(host, n->grads, sizeof(float) * count, cudaMemcpyDeviceToHost));
  return TSP_OK;
}

extern "C" tsp_status tsp_net_forward(tsp_net n, const float* a, int batch, float* out, void* stream) {
  TSP_RANGE("tsp_net_forward");
  if (!n || !a || !out || batch <= 0 || batch > n->max_batch) return fail(TSP_EINVAL, "tsp_net_forward: bad argument");
  tsp_status st = check_device(n->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  st = net_forward(n, a, batch, cs);
  if (st != TSP_OK) return st;
  TSP_CUDA(cudaMemcpyAsync(out, n->out, sizeof(float) * size_t(batch) * n->d.V, cudaMemcpyDeviceToDevice, cs));
  return TSP_OK;
}

namespace {
// dW (27 x 32 x 32, added) and db (32, added) of 32 -> 32 layer k + 1 from its
// input h[k] and the gated gradient gz[z]: the tcgen05 kernel's per-CTA
// partials, then their fixed-order sums.
void wgrad32_tc(tsp_net n, int k, int z, int batch, float* dW, float* dbias, cudaStream_t cs) {
  Dims db = n->d;
  db.B = batch;
  const int64_t rows = int64_t(batch) * db.Nr * db.Ne;
  const int grid = int(std::min<int64_t>(rows, g_sm_count));
  wgrad32_tc_kernel<<<grid, 256, wg_smem(db.Na), cs>>>(n->map_h[k], n->map_gz[z], db, n->wpart, n->part, TC_WAIT_BUDGET);
  part_reduce_kernel<<<27 * CH * CH / 32, 1024, 0, cs>>>(n->wpart, grid, 27 * CH * CH, 27 * CH * CH, dW);
  part_reduce_kernel<<<1, 1024, 0, cs>>>(n->part, grid, CH, CH, dbias);
}

// Weight and bias gradient of a one-sided layer (mode 0: output layer from
// g_out and h5; mode 1: input layer from the gated g_h and a): per-CTA
// partial sums, then a fixed-order reduction added to dw (27 x 32) and db (nb).
void thin_wgrad(tsp_net n, int mode, const Dims& db, float* dw, float* dbias, int nb, cudaStream_t cs) {
  const int et = thin_et(db.Na);
  const int64_t tiles = int64_t(db.B) * db.Nr * ((db.Ne + et - 1) / et);
  const int grid = int(std::min<int64_t>(tiles, n->part_rows));
  const size_t sm = thin_smem(db.Na, mode);
  if (mode == 0)
    thin_wgrad_kernel<0><<<grid, 256, sm, cs>>>(db, et, n->gout, n->h[4], nullptr, nullptr, nullptr, n->part);
  else
    thin_wgrad_kernel<1><<<grid, 256, sm, cs>>>(db, et, nullptr, nullptr, n->gh, n->mask[0], n->a16, n->part);
  part_reduce_kernel<<<(27 * CH + 31) / 32, 1024, 0, cs>>>(n->part, grid, THIN_OUT, 27 * CH, dw);
  part_reduce_kernel<<<1, 1024, 0, cs>>>(n->part + 27 * CH, grid, THIN_OUT, nb, dbias);
}
}  // namespace

extern "C" tsp_status tsp_net_loss_grad(tsp_net n, const float* a, const float* target, int batch, double* loss_host,
                                        void* stream) {
  TSP_RANGE("tsp_net_loss_grad");
  if (!n || !a || !target || batch <= 0 || batch > n->max_batch)
    return fail(TSP_EINVAL, "tsp_net_loss_grad: bad argument");
  tsp_status st = check_device(n->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  st = net_forward(n, a, batch, cs);
  if (st != TSP_OK) return st;
  const Dims& d = n->d;
  Dims db = d;
  db.B = batch;
  const int64_t nv = int64_t(batch) * d.V;
  TSP_CUDA(cudaMemsetAsync(n->grads, 0, sizeof(float) * n->n_params, cs));
  const int mse_blocks = int(std::min<int64_t>(blocks_for(nv, 256), MSE_BLOCKS));
  mse_kernel<<<mse_blocks, 256, 0, cs>>>(n->out, target, nv, n->gout, n->loss_part);
  ordered_sum_kernel<<<1, 32, 0, cs>>>(n->loss_part, mse_blocks, n->loss);
  // output layer
  thin_wgrad(n, 0, db, n->grads + n->off_w[5], n->grads + n->off_b[5], 1, cs);
  thin_conv_kernel<1><<<blocks_for(nv / THIN_V * 4, 128), 128, 0, cs>>>(db, nullptr, n->gout, n->w6r, nullptr, n->gz[0],
                                                               n->mask[4], n->gh);
  // residual 32 -> 32 layers, last to first: each dgrad also gates the
  // gradient it leaves for the layer below, into the other buffer
  for (int k = 3; k >= 0; --k) {
    const int z = (3 - k) & 1;
    wgrad32_tc(n, k, z, batch, n->grads + n->off_w[k + 1], n->grads + n->off_b[k + 1], cs);
    conv32(1, d, batch, n->map_gz[z], n->gz[z], n->wd[k], nullptr, k > 0 ? n->gz[1 - z] : nullptr,
           k > 0 ? n->mask[k] : nullptr, n->gh, cs);
  }
  // input layer (ReLU gate applied inside)
  thin_wgrad(n, 1, db, n->grads + n->off_w[0], n->grads + n->off_b[0], CH, cs);
  TSP_CUDA(cudaGetLastError());
  if (loss_host) {
    TSP_CUDA(cudaMemcpyAsync(loss_host, n->loss, sizeof(double), cudaMemcpyDeviceToHost, cs));
    TSP_CUDA(cudaStreamSynchronize(cs));
  }
  return TSP_OK;
}

extern "C" tsp_status tsp_net_adam(tsp_net n, float lr, float beta1, float beta2, float eps, float weight_decay,
                                   void* stream) {
  TSP_RANGE("tsp_net_adam");
  if (!n) return fail(TSP_EINVAL, "tsp_net_adam: NULL net");
  n->adam_step += 1;
  n->prepared = false;
  return tsp_adam(n->params, n->grads, n->m, n->v, int64_t(n->n_params), lr, beta1, beta2, eps, weight_decay,
                  n->adam_step, stream);
}

extern "C" tsp_status tsp_net_activation(tsp_net n, int layer, int batch, void* host) {
  if (!n || !host || layer < 0 || layer > 5 || batch <= 0 || batch > n->max_batch)
    return fail(TSP_EINVAL, "tsp_net_activation: bad argument");
  const size_t nv = size_t(batch) * n->d.V;
  if (layer < 5) TSP_CUDA(cudaMemcpy(host, n->h[layer], sizeof(bf16) * nv * CH, cudaMemcpyDeviceToHost));
  else TSP_CUDA(cudaMemcpy(host, n->out, sizeof(float) * nv, cudaMemcpyDeviceToHost));
  return TSP_OK;
}
