// Precomputed segment lists (the paper's steps 1-3 stored once, Sec. 3 and
// Sec. 4.4's stored region indices and lengths; step 4 repeated): per ray the
// (voxel, length) pairs of its valid segments in order along the ray,
// compressed (no padding slots: Eq. 8's padded arrays are not needed), and
// optionally their transpose per voxel (ray, length). Forward and adjoint on
// these lists stream 8 bytes per segment: the lists are read once, coalesced,
// and multiply an input gathered from L2 (the volume, or the detector values),
// summed per output row in registers.
#include <atomic>
#include <cstring>
#include <limits>

#include "tsp_kernels.cuh"

// One direction of the lists: rows (rays or voxels) with their entries
// (column index, length). The voxel-major entries lie row after row. The
// ray-major ones are interleaved within slices of 32 rows, 8 x 4 pixels of a
// detector (RowOrder): the slice's first entries, row by row, then the second
// ones of the rows that have two, and so on, so that a warp with a row per
// lane reads consecutive words and its lanes, neighbouring rays, gather from
// few voxels. A slice takes the words off[32 s] .. off[32 s + 32] either way:
// no padding.
// The order of the ray-major rows: views in turn, each in bands of four
// detector rows, a band column by column. Free-form rays (W = 0) keep theirs.
struct RowOrder {
  int H = 1, W = 0;
  __host__ __device__ int64_t ray(int64_t p) const {
    if (W == 0) return p;
    const int64_t view = p / (int64_t(H) * W);
    const int64_t in_view = p - view * (int64_t(H) * W), band = in_view / (4 * int64_t(W));
    const int64_t in_band = in_view - band * (4 * int64_t(W));
    const int h = H - 4 * int(band) < 4 ? H - 4 * int(band) : 4;
    const int64_t col = in_band / h, row = 4 * band + (in_band - col * h);
    return (view * H + row) * W + col;
  }
  __host__ __device__ int64_t row(int64_t r) const {  // ray's inverse
    if (W == 0) return r;
    const int64_t view = r / (int64_t(H) * W);
    const int in_view = int(r - view * (int64_t(H) * W)), i = in_view / W, col = in_view - i * W, band = i / 4;
    const int h = H - 4 * band < 4 ? H - 4 * band : 4;
    return view * (int64_t(H) * W) + 4 * int64_t(band) * W + int64_t(col) * h + (i - 4 * band);
  }
};

struct SegList {
  int64_t n_rows = 0, n_cols = 0, S = 0;
  int64_t* off = nullptr;   // [n_rows + 1] row offsets
  uint32_t* idx = nullptr;  // [S] column
  float* len = nullptr;     // [S]
};

struct tsp_segments_s {
  int64_t n_rays = 0, n_segs = 0, V = 0;
  SegList fwd;  // ray-major: rows = rays in `order`, columns = voxels
  RowOrder order;
  SegList adj;  // voxel-major (transposed): rows = voxels, columns = rays
  bool has_adj = false;
  std::vector<void*> held;  // the allocations that hold them
  size_t bytes = 0;
  int device = 0;
};

namespace tsp {
namespace {

struct CountOnlyOp {
  int* __restrict__ counts;
  int n;
  __device__ __forceinline__ bool begin(int64_t) {
    n = 0;
    return true;
  }
  __device__ __forceinline__ void operator()(int, float) { ++n; }
  __device__ __forceinline__ void end(int64_t ray) { counts[ray] = n; }
};

// The fill walk repeats the count walk bit for bit (same code, no FMA
// contraction), so each ray fills exactly its slots; the bound check only
// guards memory should that ever fail, and flags the error word.
// Four entries leave at a time (16 bytes of columns, 16 of lengths), the first
// and last of a row singly: an entry by itself is two 4-byte writes to lines of
// its own (11 M segments of 0.3 M rays, 206 -> 143 us). The entries go ray after
// ray (off: the rays' offsets), or (ROWS) those of the rows p0 .. p1 - 1 row
// after row from word 0 on (off: the rows' offsets); rays of other rows leave
// at once.
template <bool ROWS>
struct FillOp {
  const int64_t* __restrict__ off;
  RowOrder order;
  int64_t p0, p1;
  uint32_t* __restrict__ vox;
  float* __restrict__ len;
  int64_t pos, lim, out;  // entries seen, row end, entries written
  uint32_t v0, v1, v2;    // entries out .. pos - 1
  float l0, l1, l2;
  bool bad;
  __device__ __forceinline__ bool begin(int64_t ray) {
    bad = false;
    const int64_t i = ROWS ? order.row(ray) : ray, base = ROWS ? off[p0] : 0;
    if (ROWS && (i < p0 || i >= p1)) return false;
    pos = out = off[i] - base;
    lim = off[i + 1] - base;
    v0 = v1 = v2 = 0u;
    l0 = l1 = l2 = 0.0f;
    return true;
  }
  __device__ __forceinline__ void drain() {  // the pending entries one by one
    if (out < pos) vox[out] = v0, len[out] = l0;
    if (out + 1 < pos) vox[out + 1] = v1, len[out + 1] = l1;
    if (out + 2 < pos) vox[out + 2] = v2, len[out + 2] = l2;
    out = pos;
  }
  __device__ __forceinline__ void operator()(int v, float dl) {
    if (pos >= lim) {  // one too many: flagged, not written
      bad = true;
      return;
    }
    const int at = int(pos & 3);
    if (at == 3) {
      if (pos - out == 3) {
        *reinterpret_cast<uint4*>(vox + out) = make_uint4(v0, v1, v2, uint32_t(v));
        *reinterpret_cast<float4*>(len + out) = make_float4(l0, l1, l2, dl);
      } else {
        drain();
        vox[pos] = uint32_t(v);
        len[pos] = dl;
      }
      out = ++pos;
      return;
    }
    if (pos == out) v0 = uint32_t(v), l0 = dl;
    else if (pos == out + 1) v1 = uint32_t(v), l1 = dl;
    else v2 = uint32_t(v), l2 = dl;
    ++pos;
  }
  __device__ __forceinline__ void end(int64_t) {
    drain();
    if (pos != lim || bad) atomicOr(&g_tsp_error_word, 2);
  }
};

// ---- exclusive scan of int32 counts into int64 offsets (out[n] = total) ----
constexpr int SCAN_T = 1024, SCAN_E = 2;  // threads, elements per thread

__device__ __forceinline__ int64_t block_incl_scan(int64_t v, int64_t* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  if (lane == 31) sh[warp] = v;
  __syncthreads();
  if (warp == 0) {
    int64_t w = lane < int(blockDim.x >> 5) ? sh[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    sh[lane] = w;
  }
  __syncthreads();
  if (warp > 0) v += sh[warp - 1];
  __syncthreads();
  return v;
}

__global__ void scan_blocks_kernel(const int* __restrict__ in, int64_t n, int64_t* __restrict__ block_sums) {
  __shared__ int64_t sh[32];
  const int64_t base = int64_t(blockIdx.x) * SCAN_T * SCAN_E + int64_t(threadIdx.x) * SCAN_E;
  int64_t s = 0;
  for (int k = 0; k < SCAN_E; ++k)
    if (base + k < n) s += in[base + k];
  const int64_t incl = block_incl_scan(s, sh);
  if (threadIdx.x == blockDim.x - 1) block_sums[blockIdx.x] = incl;
}

// one block: exclusive scan of the block sums in place, total at [nb]
__global__ void scan_sums_kernel(int64_t* __restrict__ sums, int64_t nb) {
  __shared__ int64_t sh[32];
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t c0 = 0; c0 < nb; c0 += blockDim.x) {
    const int64_t i = c0 + threadIdx.x;
    const int64_t v = i < nb ? sums[i] : 0;
    const int64_t incl = block_incl_scan(v, sh);
    const int64_t base = carry;
    if (i < nb) sums[i] = base + incl - v;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = base + incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void scan_final_kernel(const int* __restrict__ in, int64_t n, const int64_t* __restrict__ sums,
                                  int64_t* __restrict__ out) {
  __shared__ int64_t sh[32];
  const int64_t base = int64_t(blockIdx.x) * SCAN_T * SCAN_E + int64_t(threadIdx.x) * SCAN_E;
  int64_t v[SCAN_E];
  int64_t s = 0;
  for (int k = 0; k < SCAN_E; ++k) {
    v[k] = base + k < n ? in[base + k] : 0;
    s += v[k];
  }
  int64_t run = block_incl_scan(s, sh) - s + sums[blockIdx.x];
  for (int k = 0; k < SCAN_E; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
    int64_t nb = gridDim.x;
    out[n] = sums[nb];
  }
}

constexpr int64_t scan_words(int64_t n) { return (n + SCAN_T * SCAN_E - 1) / (SCAN_T * SCAN_E) + 1; }

// sums: scan_words(n) words of scratch.
tsp_status exclusive_scan(const int* in, int64_t n, int64_t* out, int64_t* sums, cudaStream_t st) {
  if (n == 0) {
    TSP_CUDA(cudaMemsetAsync(out, 0, sizeof(int64_t), st));
    return TSP_OK;
  }
  const int64_t nb = scan_words(n) - 1;
  scan_blocks_kernel<<<unsigned(nb), SCAN_T, 0, st>>>(in, n, sums);
  scan_sums_kernel<<<1, 1024, 0, st>>>(sums, nb);
  scan_final_kernel<<<unsigned(nb), SCAN_T, 0, st>>>(in, n, sums, out);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

// Entries per key of the sorted keys (cnt zeroed before): a key's first entry
// subtracts its index, its last adds one more than its own.
__global__ void key_counts_kernel(const uint32_t* __restrict__ keys, int64_t S, uint32_t key_max,
                                  unsigned* __restrict__ cnt) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < S; i += int64_t(gridDim.x) * blockDim.x) {
    const uint32_t k = keys[i];
    const uint32_t at = min(k, key_max);  // the clamp only guards memory
    if (i == 0 || keys[i - 1] != k) atomicAdd(cnt + at, 0u - unsigned(i));
    if (i == S - 1 || keys[i + 1] != k) atomicAdd(cnt + at, unsigned(i) + 1u);
  }
}

// Offsets of the keys below 2^RB after one pass: where each digit begins.
__global__ void digit_offsets_kernel(const int64_t* __restrict__ base, int64_t n_tiles, int64_t n_rows,
                                     int64_t* __restrict__ off) {
  const int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (v <= n_rows) off[v] = base[v * n_tiles];
}

// ---- voxel-major transpose: stable LSD radix sort of the entries by voxel ----
// Keys are the voxel ids of the ray-major entries, carried with their ray id
// and length, RB bits of the key per pass. A pass counts each tile's digits,
// scans the counts digit-major (digit 0 of every tile, then digit 1, ...) and
// scatters: an entry goes to its digit's base in its tile plus the number of
// same-digit entries before it in the tile. Every pass keeps the order of
// equal digits, so after the last one each voxel's entries are in ray-major
// order (by ray, then along the ray): the same rows on every build.
constexpr int RB = 8, RD = 1 << RB;  // key bits per pass, digits
constexpr int RW = 8, RK = 8;        // warps per block, entries per lane
constexpr int RT = RW * 32 * RK;     // entries per tile

__global__ void __launch_bounds__(RW * 32) radix_hist_kernel(const uint32_t* __restrict__ keys, int64_t S, int shift, int64_t n_tiles,
                                                             int* __restrict__ hist) {
  __shared__ int h[RD];
  for (int d = threadIdx.x; d < RD; d += blockDim.x) h[d] = 0;
  __syncthreads();
  const int64_t t = blockIdx.x, e0 = t * RT;
  for (int j = threadIdx.x; j < RT; j += blockDim.x) {
    const int64_t i = e0 + j;
    if (i < S) atomicAdd(&h[(keys[i] >> shift) & (RD - 1)], 1);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < RD; d += blockDim.x) hist[int64_t(d) * n_tiles + t] = h[d];
}

// One pass over a tile of RT entries (RD == threads per block). Ranking: a
// warp takes its 32 * RK consecutive entries in RK rounds of 32; lanes with
// equal digits find each other (match), take the warp's running count for the
// digit plus the number of such lanes below them, and the lowest of them
// advances the count. The warps' counts become offsets in warp order and the
// digits' totals offsets in digit order, which sorts the tile by digit in
// shared memory; the tile then leaves as one contiguous run per digit.
__global__ void __launch_bounds__(RW * 32) radix_scatter_kernel(
    const uint32_t* __restrict__ keys, const uint32_t* __restrict__ rays, const float* __restrict__ lens, int64_t S,
    int shift, int64_t n_tiles, const int64_t* __restrict__ base, uint32_t* __restrict__ keys_out,
    uint32_t* __restrict__ rays_out, float* __restrict__ lens_out) {
  __shared__ int cnt[RW][RD];
  __shared__ int start[RD];
  __shared__ int64_t scan_sh[32];
  __shared__ uint32_t sk[RT], sr[RT];
  __shared__ float sl[RT];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int d = lane; d < RD; d += 32) cnt[warp][d] = 0;
  __syncwarp();
  const int64_t t = blockIdx.x, w0 = t * RT + int64_t(warp) * (32 * RK);
  const unsigned below = (1u << lane) - 1u;
  uint32_t key[RK], ray[RK];
  float len[RK];
  int rank[RK];
#pragma unroll
  for (int k = 0; k < RK; ++k) {
    const int64_t i = w0 + k * 32 + lane;
    const bool ok = i < S;
    key[k] = ok ? keys[i] : 0u;
    ray[k] = ok ? rays[i] : 0u;
    len[k] = ok ? lens[i] : 0.0f;
    const uint32_t d = ok ? (key[k] >> shift) & (RD - 1) : uint32_t(RD);  // past the end: a class of its own
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    rank[k] = ok ? cnt[warp][d] + __popc(peers & below) : 0;
    __syncwarp();
    if (ok && (peers & below) == 0) cnt[warp][d] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {
    const int d = threadIdx.x;
    int run = 0;
    for (int w = 0; w < RW; ++w) {
      const int c = cnt[w][d];
      cnt[w][d] = run;
      run += c;
    }
    const int64_t incl = block_incl_scan(run, scan_sh);
    start[d] = int(incl - run);
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < RK; ++k) {
    if (w0 + k * 32 + lane >= S) continue;
    const uint32_t d = (key[k] >> shift) & (RD - 1);
    const int lp = start[d] + cnt[warp][d] + rank[k];
    sk[lp] = key[k];
    sr[lp] = ray[k];
    sl[lp] = len[k];
  }
  __syncthreads();
  const int n = int(S - t * RT < RT ? S - t * RT : RT);
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const uint32_t kk = sk[j];
    const uint32_t d = (kk >> shift) & (RD - 1);
    const int64_t g = base[int64_t(d) * n_tiles + t] + (j - start[d]);
    if (keys_out) keys_out[g] = kk;
    rays_out[g] = sr[j];
    lens_out[g] = sl[j];
  }
}

// ray id of every ray-major entry (warp per ray)
__global__ void ray_ids_kernel(const int64_t* __restrict__ off, int64_t n_rays, uint32_t* __restrict__ rid) {
  const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n_rays) return;
  for (int64_t s = off[w] + lane; s < off[w + 1]; s += 32) rid[s] = uint32_t(w);
}


// Counts per ray into the order of the rows.
__global__ void order_counts_kernel(const int* __restrict__ counts, int64_t n_rows, RowOrder order,
                                    int* __restrict__ out) {
  const int64_t row = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (row < n_rows) out[row] = counts[order.ray(row)];
}

// Entries into the interleaved order, a warp per slice, a row per lane: from
// ray after ray (their offsets off_in), or, with off_in NULL, the rows p0 ..
// n_rows - 1 row after row from word 0 on (p0 a multiple of 32).
__global__ void __launch_bounds__(256) interleave_kernel(const int64_t* __restrict__ off, int64_t p0, int64_t n_rows,
                                                         RowOrder order, const int64_t* __restrict__ off_in,
                                                         const uint32_t* __restrict__ idx_in,
                                                         const float* __restrict__ len_in,
                                                         uint32_t* __restrict__ idx, float* __restrict__ len) {
  const int64_t row = p0 + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
  const int64_t o0 = off[min(row, n_rows)], o1 = off[min(row + 1, n_rows)];
  const int n = int(o1 - o0), most = __reduce_max_sync(0xffffffffu, n);
  const int64_t from = off_in == nullptr ? o0 - off[p0] : (row < n_rows ? off_in[order.ray(row)] : 0);
  int64_t q = __shfl_sync(0xffffffffu, o0, 0);
#pragma unroll 4
  for (int k = 0; k < most; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, k < n);
    if (k < n) {
      const int64_t to = q + __popc(m & below);
      idx[to] = idx_in[from + k];
      len[to] = len_in[from + k];
    }
    q += __popc(m);
  }
}

// The entries of the rays a .. z - 1 ray after ray (to: their offsets, from ray
// a's) out of the interleaved rows from p0 (a multiple of 32) on.
__global__ void __launch_bounds__(256) export_kernel(const int64_t* __restrict__ off, int64_t p0, int64_t n_rows,
                                                     RowOrder order, const uint32_t* __restrict__ idx,
                                                     const float* __restrict__ len, int64_t a, int64_t z,
                                                     const int64_t* __restrict__ to, uint32_t* __restrict__ idx_out,
                                                     float* __restrict__ len_out) {
  const int64_t row = p0 + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
  const int64_t o0 = off[min(row, n_rows)], o1 = off[min(row + 1, n_rows)];
  const int n = int(o1 - o0), most = __reduce_max_sync(0xffffffffu, n);
  const int64_t ray = row < n_rows ? order.ray(row) : -1;
  const bool mine = ray >= a && ray < z;
  const int64_t out = mine ? to[ray - a] - to[0] : 0;
  int64_t q = __shfl_sync(0xffffffffu, o0, 0);
  for (int k = 0; k < most; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, k < n);
    if (mine && k < n) {
      const int64_t at = q + __popc(m & below);
      idx_out[out + k] = idx[at];
      len_out[out + k] = len[at];
    }
    q += __popc(m);
  }
}

// ---- forward: W warps per slice of 32 rows, a row per lane ----
// Each warp takes an equal run of the slice's steps. Every step reads
// consecutive words; while all rows last (k < the slice's shortest), SLICE_U
// steps at a time, their loads issued before their gathers. A lane adds its
// row's terms in order, and the W sums are added in order: no atomics, the
// same bits on every call. With EPI the rows end in SIRT's residual
// R (y - sum). NB volumes per pass over the lists.
//
// Bound by the gathers' L1 wavefronts (a warp's 32 rays of a detector tile
// are at some ten voxels a step) and, for long rows, by HBM. On GB300, F of
// one volume (us; the flat stream with a segmented reduction that stood here,
// whose lanes at successive segments of one ray gathered from 32 lines; this
// with rows in detector order; in 8 x 4 tiles; split over 2 / 4 / 8 warps):
// 3.1 M rays of 49 segments 363, 297, 277, 272 / 286 / 336; 2.1 M rays of 142
// segments 679, 490, 464, 445 / 436 / 455; 0.6 M rays of 68 segments 118, 145,
// 140, 118 / 113 / 112; 16 k rays of 49 segments 39, 66, 72, 41 / 31 / 30; four
// volumes, 0.8 M rays of 49 segments 375, 212, 180, 174 / 168 / 189.
constexpr int SLICE_U = 8, SLICE_T = 4;

template <int W, int NB, bool EPI>
__global__ void __launch_bounds__(256) slice_forward_kernel(const int64_t* __restrict__ off,
                                                            const uint32_t* __restrict__ idx,
                                                            const float* __restrict__ len, int64_t n_rows,
                                                            RowOrder order, uint32_t col_max,
                                                            const float* __restrict__ src, int64_t src_stride,
                                                            float* __restrict__ dst, int64_t dst_stride, int nb,
                                                            const float* __restrict__ R,
                                                            const float* __restrict__ y) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = warp % W;
  const int64_t row = (int64_t(blockIdx.x) * (8 / W) + warp / W) * 32 + lane;
  const int64_t o0 = off[min(row, n_rows)], o1 = off[min(row + 1, n_rows)];
  const int n = int(o1 - o0);
  const int least = __reduce_min_sync(0xffffffffu, n), most = __reduce_max_sync(0xffffffffu, n);
  int k = most * part / W;
  const int last = most * (part + 1) / W;
  int64_t q = __shfl_sync(0xffffffffu, o0, 0);  // the slice's entries of step k
  q += __reduce_add_sync(0xffffffffu, min(n, k));
  float acc[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) acc[b] = 0.0f;
  for (; k + SLICE_U <= min(least, last); k += SLICE_U, q += 32 * SLICE_U) {
    uint32_t i[SLICE_U];
    float l[SLICE_U];
#pragma unroll
    for (int u = 0; u < SLICE_U; ++u) {
      i[u] = min(__ldg(idx + q + 32 * u + lane), col_max);  // the clamp only guards memory: columns are valid
      l[u] = __ldg(len + q + 32 * u + lane);
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (NB > 1 && b >= nb) break;
      float x[SLICE_U];
#pragma unroll
      for (int u = 0; u < SLICE_U; ++u) x[u] = __ldg(src + b * src_stride + i[u]);
#pragma unroll
      for (int u = 0; u < SLICE_U; ++u) acc[b] = fmaf(x[u], l[u], acc[b]);
    }
  }
  const unsigned below = (1u << lane) - 1u;
  for (; k < last; k += SLICE_T) {  // rows that have ended leave no gap
    uint32_t i[SLICE_T];
    float l[SLICE_T];
    bool in[SLICE_T];
#pragma unroll
    for (int u = 0; u < SLICE_T; ++u) {
      in[u] = k + u < last && k + u < n;
      const unsigned m = __ballot_sync(0xffffffffu, in[u]);
      const int64_t at = q + __popc(m & below);
      q += __popc(m);
      i[u] = in[u] ? min(__ldg(idx + at), col_max) : 0u;
      l[u] = in[u] ? __ldg(len + at) : 0.0f;
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (NB > 1 && b >= nb) break;
      float x[SLICE_T];
#pragma unroll
      for (int u = 0; u < SLICE_T; ++u) x[u] = in[u] ? __ldg(src + b * src_stride + i[u]) : 0.0f;
#pragma unroll
      for (int u = 0; u < SLICE_T; ++u) acc[b] = fmaf(x[u], l[u], acc[b]);
    }
  }
  __shared__ float sums[8][NB][32];  // the parts' sums, added in order
#pragma unroll
  for (int b = 0; b < NB; ++b) sums[warp][b][lane] = acc[b];
  __syncthreads();
  if (part > 0) return;
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int w = 1; w < W; ++w) acc[b] = __fadd_rn(acc[b], sums[warp + w][b][lane]);
  if (row >= n_rows) return;
  const int64_t ray = order.ray(row);
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (NB > 1 && b >= nb) break;
    dst[b * dst_stride + ray] = EPI ? __fmul_rn(R[ray], __fsub_rn(y[ray], acc[b])) : acc[b];
  }
}

// ---- adjoint: G lanes per row of the voxel-major lists ----
// A row's entries are the rays of neighbouring pixels, so consecutive lanes
// gather from few sectors. A lane reads four consecutive entries (16 bytes of
// columns, 16 of lengths; the row's ends masked) U times before their gathers;
// a shuffle tree sums the lanes: fixed order, no atomics. With EPI the rows
// end in SIRT's update x += C sum (clamped at 0 if asked) instead of a store.
template <int G, int U, int NB, bool EPI>
__global__ void __launch_bounds__(256) row_group_kernel(const int64_t* __restrict__ off,
                                                        const uint32_t* __restrict__ idx,
                                                        const float* __restrict__ len, int64_t n_rows,
                                                        uint32_t col_max, const float* __restrict__ src,
                                                        int64_t src_stride, float* __restrict__ dst,
                                                        int64_t dst_stride, int nb, int flag,
                                                        const float* __restrict__ C) {
  const int64_t row = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) / G;
  const int sub = threadIdx.x % G;
  float acc[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) acc[b] = 0.0f;
  if (row < n_rows) {
    const int64_t s0 = off[row], s1 = off[row + 1];
    for (int64_t s = (s0 & ~int64_t(3)) + 4 * sub; s < s1; s += 4 * G * U) {
      uint32_t i[4 * U];
      float l[4 * U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int64_t sk = s + 4 * G * k;
        uint4 iv = make_uint4(0u, 0u, 0u, 0u);
        float4 lv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (sk < s1) {  // (the arrays are allocated to a multiple of four entries)
          iv = __ldcs(reinterpret_cast<const uint4*>(idx + sk));
          lv = __ldcs(reinterpret_cast<const float4*>(len + sk));
        }
        const uint32_t ia[4] = {iv.x, iv.y, iv.z, iv.w};
        const float la[4] = {lv.x, lv.y, lv.z, lv.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool in = sk + j >= s0 && sk + j < s1;
          i[4 * k + j] = in ? min(ia[j], col_max) : 0xffffffffu;  // the clamp only guards memory: columns are valid
          l[4 * k + j] = la[j];
        }
      }
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        if (NB > 1 && b >= nb) break;
        float x[4 * U];
#pragma unroll
        for (int j = 0; j < 4 * U; ++j) x[j] = i[j] != 0xffffffffu ? __ldg(src + b * src_stride + i[j]) : 0.0f;
#pragma unroll
        for (int j = 0; j < 4 * U; ++j)
          if (i[j] != 0xffffffffu) acc[b] = fmaf(x[j], l[j], acc[b]);
      }
    }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (NB > 1 && b >= nb) break;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) acc[b] += __shfl_down_sync(0xffffffffu, acc[b], o, G);
    if (sub == 0 && row < n_rows) {
      float* p = dst + b * dst_stride + row;
      if (EPI) {
        float v = fmaf(C[row], acc[b], *p);
        *p = flag ? fmaxf(v, 0.0f) : v;
      } else {
        *p = flag ? *p + acc[b] : acc[b];
      }
    }
  }
}

// adjoint without the transposed lists: one atomic per run of neighbouring
// rays on the same voxel (a warp per slice, a row per lane)
__global__ void __launch_bounds__(256) seg_scatter_kernel(const int64_t* __restrict__ off,
                                                          const uint32_t* __restrict__ vox,
                                                          const float* __restrict__ len, RowOrder order,
                                                          const float* __restrict__ y, float* __restrict__ g,
                                                          int64_t n_rays) {
  const int64_t row = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
  const int64_t o0 = off[min(row, n_rays)], o1 = off[min(row + 1, n_rays)];
  const int n = int(o1 - o0), most = __reduce_max_sync(0xffffffffu, n);
  int64_t q = __shfl_sync(0xffffffffu, o0, 0);
  const float yv = n > 0 ? y[order.ray(row)] : 0.0f;
  for (int k = 0; k < most; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, k < n);
    const int64_t at = q + __popc(m & below);
    q += __popc(m);
    if (k < n && yv != 0.0f) {
      const int v = int(vox[at]);
      RunSum run;
      run.set(v);
      const float c = run.sum(__fmul_rn(yv, len[at]));
      if (run.head) atomicAdd(g + v, c);
    }
    __syncwarp();
  }
}

template <int W>
void slices(const SegList& l, RowOrder order, const float* rho, float* y, int k, const float* R, const float* y_meas,
            cudaStream_t st) {
  const unsigned blocks = unsigned((l.n_rows + 256 / W - 1) / (256 / W));
  const uint32_t cm = uint32_t(l.n_cols - 1);
  if (R)
    slice_forward_kernel<W, 1, true><<<blocks, 256, 0, st>>>(l.off, l.idx, l.len, l.n_rows, order, cm, rho, l.n_cols, y,
                                                             l.n_rows, 1, R, y_meas);
  else if (k == 1)
    slice_forward_kernel<W, 1, false><<<blocks, 256, 0, st>>>(l.off, l.idx, l.len, l.n_rows, order, cm, rho, l.n_cols,
                                                              y, l.n_rows, 1, nullptr, nullptr);
  else
    slice_forward_kernel<W, 4, false><<<blocks, 256, 0, st>>>(l.off, l.idx, l.len, l.n_rows, order, cm, rho, l.n_cols,
                                                              y, l.n_rows, k, nullptr, nullptr);
}

// y = F rho, or with R the residual R (y_meas - F rho) of one volume.
tsp_status list_forward(const SegList& l, RowOrder order, const float* rho, float* y, int nb, const float* R,
                        const float* y_meas, cudaStream_t st) {
  for (int b0 = 0; b0 < nb; b0 += 4) {
    const int k = std::min(4, nb - b0);
    const float* sp = rho + b0 * l.n_cols;
    float* dp = y + b0 * l.n_rows;
    if (l.S < 24 * l.n_rows || (l.S < 96 * l.n_rows && l.n_rows >= (1 << 20)))
      slices<2>(l, order, sp, dp, k, R, y_meas, st);
    else
      slices<4>(l, order, sp, dp, k, R, y_meas, st);
  }
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

template <int G, int U>
void row_groups(const SegList& l, const float* src, float* dst, int k, int flag, const float* C, cudaStream_t st) {
  const unsigned blocks = unsigned((l.n_rows * G + 255) / 256);
  const uint32_t cm = uint32_t(l.n_cols - 1);
  if (C)
    row_group_kernel<G, U, 1, true><<<blocks, 256, 0, st>>>(l.off, l.idx, l.len, l.n_rows, cm, src, l.n_cols, dst,
                                                            l.n_rows, 1, flag, C);
  else if (k == 1)
    row_group_kernel<G, U, 1, false><<<blocks, 256, 0, st>>>(l.off, l.idx, l.len, l.n_rows, cm, src, l.n_cols,
                                                             dst, l.n_rows, 1, flag, nullptr);
  else
    row_group_kernel<G, U, 4, false><<<blocks, 256, 0, st>>>(l.off, l.idx, l.len, l.n_rows, cm, src, l.n_cols,
                                                             dst, l.n_rows, k, flag, nullptr);
}

// rho (+)= F^T y from the voxel-major lists (flag: accumulate), or with C the
// update rho += C F^T y of one volume (flag: clamp at 0). Lanes per row by the
// mean row: measured on GB300 (us with 4 / 8 / 16 / 32 lanes; the flat stream
// and the warp per row that stood here in the last column): 3 entries 18 / 21 /
// 34 / 57, 26; 58 entries 116 / 112 / 125 / 181, 110; 132 entries, four volumes
// 229 / 193 / 195 / 255, 363; 224 entries 266 / 258 / 225 / 227, 236; 414
// entries 628 / 588 / 500 / 510, 570; 526 entries 431 / 380 / 297 / 275, 311.
// Few rows leave the chip idle: two reads in flight then (674 entries, 9000
// rows: 46 / 39 with one / two, 62 before).
tsp_status list_adjoint(const SegList& l, const float* y, float* rho, int nb, int flag, const float* C,
                        cudaStream_t st) {
  for (int b0 = 0; b0 < nb; b0 += 4) {
    const int k = std::min(4, nb - b0);
    const float* sp = y + b0 * l.n_cols;
    float* dp = rho + b0 * l.n_rows;
    if (l.S < 24 * l.n_rows) row_groups<4, 1>(l, sp, dp, k, flag, C, st);
    else if (l.S < 160 * l.n_rows) row_groups<8, 1>(l, sp, dp, k, flag, C, st);
    else if (l.S < 448 * l.n_rows) row_groups<16, 1>(l, sp, dp, k, flag, C, st);
    else if (l.n_rows > 152 * 64) row_groups<32, 1>(l, sp, dp, k, flag, C, st);
    else row_groups<32, 2>(l, sp, dp, k, flag, C, st);
  }
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

// ---- SIRT on the stored lists (same update as tsp_sirt) ----
__global__ void fill_kernel(float* __restrict__ a, int64_t n, float v) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    a[i] = v;
}

// a[i] = 1 / a[i], 0 where a[i] <= 0 (rays missing the grid, voxels no ray meets)
__global__ void recip_kernel(float* __restrict__ a, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float v = a[i];
    a[i] = v > 0.0f ? __frcp_rn(v) : 0.0f;
  }
}

// x += C * g, clamped at 0 if asked
__global__ void xupdate_kernel(float* __restrict__ x, const float* __restrict__ g, const float* __restrict__ C,
                               int64_t n, int nonneg) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    float v = fmaf(C[i], g[i], x[i]);
    if (nonneg) v = fmaxf(v, 0.0f);
    x[i] = v;
  }
}

unsigned ew_blocks(int64_t n) { return unsigned(std::min<int64_t>((n + 255) / 256, 152 * 16)); }
size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Device allocations held together. The spares are those that a chunked driver
// keeps from one build's scratch to the next.
struct Blocks {
  std::vector<void*> held;
  void* spare[2] = {nullptr, nullptr};
  size_t spare_bytes[2] = {0, 0};
  void release() {
    for (void* p : held) cudaFree(p);
    held.clear();
  }
  void release_spare(int i) {
    cudaFree(spare[i]);
    spare[i] = nullptr;
    spare_bytes[i] = 0;
  }
  void release_spares() {
    release_spare(0);
    release_spare(1);
  }
};

// Limits that tsp_debug_segments_memory changes: the largest block of several
// arrays, and the most scratch per segment that a build may take.
constexpr int64_t BLOCK_MOST = int64_t(512) << 20;
std::atomic<int64_t> g_block_most{BLOCK_MOST}, g_scratch_most{std::numeric_limits<int64_t>::max()};

// Several arrays in one device allocation, 256-byte aligned each (in the spare
// one if it is large enough), as long as they are small: an allocation and its
// release take some 60 us however few bytes they are of. Together above
// BLOCK_MOST bytes each gets its own: the driver clears a large block that was
// freed behind the kernels that follow (a first pass over 2.5 GB of lists took
// 530 us instead of 320 after a build with its scratch in one block). Every
// array passes the allocation hook: in a block all before its one allocation,
// else each before its own.
struct Carve {
  std::vector<std::pair<void**, size_t>> parts;
  template <class T>
  void add(T** p, int64_t count) {
    parts.emplace_back(reinterpret_cast<void**>(p), align256(sizeof(T) * size_t(count > 0 ? count : 1)));
  }
  size_t bytes() const {
    size_t b = 0;
    for (const auto& p : parts) b += p.second;
    return b;
  }
  // spare: the block to use or to become. On failure nothing is held that was not before; *injected: by the test hook.
  cudaError_t allocate(Blocks& blocks, int spare = -1, bool* injected = nullptr) const {
    auto hook = [&]() {
      const cudaError_t e = dev_malloc_hook();
      if (e != cudaSuccess && injected) *injected = true;
      return e;
    };
    if (int64_t(bytes()) > g_block_most.load()) {
      if (spare >= 0) blocks.release_spare(spare);
      const size_t before = blocks.held.size();
      for (const auto& p : parts) {
        cudaError_t e = hook();
        if (e == cudaSuccess) e = cudaMalloc(p.first, p.second);
        if (e != cudaSuccess) {
          for (; blocks.held.size() > before; blocks.held.pop_back()) cudaFree(blocks.held.back());
          return e;
        }
        blocks.held.push_back(*p.first);
      }
      return cudaSuccess;
    }
    for (size_t i = 0; i < parts.size(); ++i) {  // one allocation that stands for all of them
      const cudaError_t e = hook();
      if (e != cudaSuccess) return e;
    }
    void* block = nullptr;
    if (spare >= 0 && blocks.spare_bytes[spare] >= bytes()) {
      block = blocks.spare[spare];
    } else {
      if (spare >= 0) blocks.release_spare(spare);
      const cudaError_t e = cudaMalloc(&block, bytes());
      if (e != cudaSuccess) return e;
      if (spare >= 0) {
        blocks.spare[spare] = block;
        blocks.spare_bytes[spare] = bytes();
      } else {
        blocks.held.push_back(block);
      }
    }
    char* at = static_cast<char*>(block);
    for (const auto& p : parts) {
      *p.first = at;
      at += p.second;
    }
    return cudaSuccess;
  }
};

}  // namespace
}  // namespace tsp

using namespace tsp;

static tsp_status build_lists(tsp_grid grid, tsp_geom geom, int transpose, Blocks& scratch, tsp_segments* out,
                              void* stream);

extern "C" void tsp_segments_destroy(tsp_segments s) {
  if (!s) return;
  for (void* p : s->held) cudaFree(p);
  delete s;
}

// The rows' entries into the interleaved order, from the walk in pieces of whole
// slices through a staging buffer, so that lists of any size take a bounded
// scratch: each piece is one more walk in which the rays of other pieces leave
// at once (200 M segments of 3 M rays in 256 MB: 7 pieces).
constexpr int64_t STAGE_MOST = int64_t(512) << 20;
static tsp_status fill_rows(tsp_grid grid, tsp_geom geom, const tsp_launch& l, SegList& f, RowOrder order,
                            cudaStream_t cs) {
  if (f.S == 0) return TSP_OK;
  const int64_t n_slices = (f.n_rows + 31) / 32;
  std::vector<int64_t> first;  // offsets of the slices, once one piece is not enough
  int64_t widest = f.S;
  auto slices = [&]() -> tsp_status {
    first.assign(size_t(n_slices + 1), f.S);
    TSP_CUDA(cudaMemcpy2DAsync(first.data(), sizeof(int64_t), f.off, 32 * sizeof(int64_t), sizeof(int64_t),
                               size_t(n_slices), cudaMemcpyDeviceToHost, cs));
    TSP_CUDA(cudaStreamSynchronize(cs));
    widest = 0;
    for (int64_t k = 0; k < n_slices; ++k) widest = std::max(widest, first[size_t(k + 1)] - first[size_t(k)]);
    return TSP_OK;
  };
  int64_t most = std::min(f.S, std::min(g_scratch_most.load(), STAGE_MOST) / 8);  // entries
  if (most < f.S) {
    const tsp_status st = slices();
    if (st != TSP_OK) return st;
    most = std::max(most, widest);
  }
  uint32_t* xi = nullptr;
  if (dev_malloc_hook() != cudaSuccess) return fail(TSP_ENOMEM, "tsp_segments_build: out of device memory (staging)");
  for (;;) {  // (the lengths after the columns, on a multiple of four entries)
    const cudaError_t e = cudaMalloc(&xi, size_t(8 * ((most + 3) & ~int64_t(3))));
    if (e == cudaSuccess) break;
    cudaGetLastError();  // not sticky: clear it
    if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "tsp_segments_build: staging");
    if (first.empty()) {
      const tsp_status st = slices();
      if (st != TSP_OK) return st;
    }
    if (most / 2 < std::max(widest, int64_t(1) << 17))
      return fail(TSP_ENOMEM, "tsp_segments_build: out of device memory (staging)");
    most /= 2;
  }
  float* xl = reinterpret_cast<float*>(xi + ((most + 3) & ~int64_t(3)));
  for (int64_t s0 = 0, s1; s0 < n_slices; s0 = s1) {
    s1 = n_slices;
    if (!first.empty())
      for (s1 = s0 + 1; s1 < n_slices && first[size_t(s1 + 1)] - first[size_t(s0)] <= most;) ++s1;
    FillOp<true> op;
    op.off = f.off;
    op.order = order;
    op.p0 = 32 * s0;
    op.p1 = std::min(32 * s1, f.n_rows);
    op.vox = xi;
    op.len = xl;
    launch_trace(grid, geom, l, op, cs);
    interleave_kernel<<<unsigned((op.p1 - op.p0 + 255) / 256), 256, 0, cs>>>(f.off, op.p0, op.p1, order, nullptr, xi,
                                                                            xl, f.idx, f.len);
  }
  cudaError_t e = cudaGetLastError();
  const cudaError_t done = cudaStreamSynchronize(cs);
  cudaFree(xi);
  if (e == cudaSuccess) e = done;
  return e == cudaSuccess ? TSP_OK : cuda_fail(e, "tsp_segments_build: filling the lists");
}

// One allocation for the lists and two for the build's scratch: with one per
// array and the scans' own, allocating and freeing took longer than the kernels
// of a build of 11 M segments (2.2 ms a build with its release, 1.3 now).
extern "C" tsp_status tsp_segments_build(tsp_grid grid, tsp_geom geom, int transpose, tsp_segments* out,
                                         void* stream) {
  Blocks scratch;
  const tsp_status st = build_lists(grid, geom, transpose, scratch, out, stream);
  scratch.release_spares();
  return st;
}

static tsp_status build_lists(tsp_grid grid, tsp_geom geom, int transpose, Blocks& scratch, tsp_segments* out,
                              void* stream) {
  TSP_RANGE("tsp_segments_build");
  if (!out) return fail(TSP_EINVAL, "tsp_segments_build: out is NULL");
  *out = nullptr;
  tsp_status st = check_trace_args(grid, geom, grid, geom, 1, nullptr, "tsp_segments_build");
  if (st != TSP_OK) return st;
  if (geom->n_rays >= (int64_t(1) << 31) || grid->voxels() >= (int64_t(1) << 31))
    return fail(TSP_ENOTSUP, "tsp_segments_build: 2^31 or more rays or voxels");
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  tsp_segments s = new (std::nothrow) tsp_segments_s();
  if (!s) return fail(TSP_ENOMEM, "tsp_segments_build: host allocation");
  const int64_t n_rays = geom->n_rays, V = grid->voxels();
  s->n_rays = n_rays;
  s->V = V;
  s->device = grid->device;
  if (int64_t(geom->n_views) * geom->H * geom->W == n_rays) s->order = RowOrder{geom->H, geom->W};
  Blocks lists;
  auto bail = [&](tsp_status r) {
    cudaStreamSynchronize(cs);
    scratch.release();
    lists.release();
    tsp_segments_destroy(s);
    return r;
  };
#define SEG_TRY(call)                                                                        \
  do {                                                                                       \
    cudaError_t e__ = (call);                                                                \
    if (e__ == cudaErrorMemoryAllocation) {                                                  \
      cudaGetLastError(); /* not sticky: clear it */                                         \
      return bail(fail(TSP_ENOMEM, std::string("tsp_segments_build: out of device memory at ") + #call)); \
    }                                                                                        \
    if (e__ != cudaSuccess) return bail(cuda_fail(e__, #call));                              \
  } while (0)
  SegList &f = s->fwd, &t = s->adj;
  f.n_rows = t.n_cols = n_rays;
  f.n_cols = t.n_rows = V;
  Carve entries, first;
  int *counts = nullptr, *ordered = nullptr;
  int64_t *ray_off = nullptr, *row_off = nullptr, *sums = nullptr;
  first.add(&counts, n_rays);
  first.add(&ordered, n_rays);
  first.add(&row_off, n_rays + 1);
  first.add(&sums, scan_words(n_rays));
  if (transpose) first.add(&ray_off, n_rays + 1);
  SEG_TRY(first.allocate(scratch, 0));
  const tsp_launch l = preferred_launch(grid, geom, false);
  CountOnlyOp cop;
  cop.counts = counts;
  launch_trace(grid, geom, l, cop, cs);
  const unsigned row_blocks = unsigned((n_rays + 255) / 256);
  order_counts_kernel<<<row_blocks, 256, 0, cs>>>(counts, n_rays, s->order, ordered);
  st = exclusive_scan(ordered, n_rays, row_off, sums, cs);
  if (st == TSP_OK && transpose) st = exclusive_scan(counts, n_rays, ray_off, sums, cs);
  if (st != TSP_OK) return bail(st);
  SEG_TRY(cudaMemcpyAsync(&s->n_segs, row_off + n_rays, sizeof(int64_t), cudaMemcpyDeviceToHost, cs));
  SEG_TRY(cudaStreamSynchronize(cs));
  const int64_t S = s->n_segs;
  if (S >= (int64_t(1) << 32)) return bail(fail(TSP_ENOTSUP, "tsp_segments_build: 2^32 or more segments"));
  f.S = t.S = S;
  entries.add(&f.off, n_rays + 1);
  entries.add(&f.idx, S);
  entries.add(&f.len, S);
  if (transpose) {
    entries.add(&t.off, V + 1);
    entries.add(&t.idx, S);
    entries.add(&t.len, S);
  }
  SEG_TRY(entries.allocate(lists));
  SEG_TRY(cudaMemcpyAsync(f.off, row_off, sizeof(int64_t) * size_t(n_rays + 1), cudaMemcpyDeviceToDevice, cs));
  if (!transpose) {
    st = fill_rows(grid, geom, l, f, s->order, cs);
    if (st != TSP_OK) return bail(st);
  } else {
    // Radix sort by voxel of the entries ray after ray, X: `passes` stable passes
    // between the buffers A = (ka, t.idx, t.len) and B = (kb, rb, lb) of (key,
    // ray, length), so that the last one reads B and writes A; its keys give
    // the row offsets. The first reads X and its ray ids, which start in the ray
    // array that it does not write. f holds nothing of its own until the end:
    // with X in scratch it is B's keys and lengths, and X is interleaved into
    // it last (16 bytes a segment of scratch, 12 for one pass). Where that does
    // not fit, X is filled into f and gives up its place to the sort after the
    // first pass (4, 12, 8, 12 bytes for one to four passes), and f is filled by
    // one more walk.
    int bits = 1;
    while (bits < 32 && (uint64_t(V - 1) >> bits) != 0) ++bits;
    const int passes = (bits + RB - 1) / RB;
    const bool first_to_a = (passes - 1) % 2 == 0;
    const int64_t n_rt = (S + RT - 1) / RT;
    uint32_t *xi = nullptr, *ka = nullptr, *kb = nullptr, *rb = nullptr;
    float *xl = nullptr, *lb = nullptr;
    int *rhist = nullptr, *vcount = nullptr;
    int64_t *rbase = nullptr, *rsums = nullptr;
    bool in_place = false;
    for (;; in_place = true) {
      Carve second;
      second.add(&rb, S);
      if (!in_place) {
        second.add(&xi, S);
        second.add(&xl, S);
        if (passes > 1) second.add(&ka, S);
      } else if (passes > 1 && first_to_a) {
        second.add(&ka, S);
      } else if (passes > 1) {
        second.add(&kb, S);
        second.add(&lb, S);
      }
      second.add(&rhist, RD * n_rt);
      second.add(&rbase, RD * n_rt + 1);
      second.add(&vcount, V);
      second.add(&rsums, scan_words(std::max(RD * n_rt, V)));
      bool injected = false;
      const cudaError_t e = int64_t(second.bytes()) > g_scratch_most.load() ? cudaErrorMemoryAllocation
                                                                           : second.allocate(scratch, 1, &injected);
      if (e == cudaSuccess) break;
      if (e != cudaErrorMemoryAllocation || in_place || injected) SEG_TRY(e);
      cudaGetLastError();  // not sticky: clear it
    }
    if (in_place) {
      xi = f.idx;
      xl = f.len;
    }
    if (!in_place || first_to_a) {
      kb = f.idx;
      lb = f.len;
    } else {
      ka = f.idx;
    }
    FillOp<false> fop;
    fop.off = ray_off;
    fop.vox = xi;
    fop.len = xl;
    launch_trace(grid, geom, l, fop, cs);
    if (S > 0) {
      uint32_t* rid = first_to_a ? rb : t.idx;
      ray_ids_kernel<<<unsigned((n_rays * 32 + 255) / 256), 256, 0, cs>>>(ray_off, n_rays, rid);
      const uint32_t *ik = xi, *ir = rid;
      const float* il = xl;
      for (int p = 0; p < passes; ++p) {
        const int shift = p * RB;
        radix_hist_kernel<<<unsigned(n_rt), RW * 32, 0, cs>>>(ik, S, shift, n_rt, rhist);
        st = exclusive_scan(rhist, RD * n_rt, rbase, rsums, cs);
        if (st != TSP_OK) return bail(st);
        const bool to_a = (passes - 1 - p) % 2 == 0;
        uint32_t* ok_ = to_a ? ka : kb;
        uint32_t* orr = to_a ? t.idx : rb;
        float* ol = to_a ? t.len : lb;
        const unsigned g = unsigned(n_rt);
        radix_scatter_kernel<<<g, RW * 32, 0, cs>>>(ik, ir, il, S, shift, n_rt, rbase, ok_, orr, ol);
        SEG_TRY(cudaGetLastError());
        ik = ok_;
        ir = orr;
        il = ol;
      }
    }
    if (S > 0 && passes == 1) {
      digit_offsets_kernel<<<unsigned(V / 256 + 1), 256, 0, cs>>>(rbase, n_rt, V, t.off);
    } else {
      SEG_TRY(cudaMemsetAsync(vcount, 0, sizeof(int) * size_t(V), cs));
      if (S > 0)
        key_counts_kernel<<<152 * 16, 256, 0, cs>>>(ka, S, uint32_t(V - 1), reinterpret_cast<unsigned*>(vcount));
      st = exclusive_scan(vcount, V, t.off, rsums, cs);
      if (st != TSP_OK) return bail(st);
    }
    SEG_TRY(cudaGetLastError());
    if (!in_place) {
      interleave_kernel<<<row_blocks, 256, 0, cs>>>(f.off, 0, n_rays, s->order, ray_off, xi, xl, f.idx, f.len);
      SEG_TRY(cudaGetLastError());
    } else {
      SEG_TRY(cudaStreamSynchronize(cs));
      scratch.release();
      scratch.release_spares();
      st = fill_rows(grid, geom, l, f, s->order, cs);
      if (st != TSP_OK) return bail(st);
    }
    s->has_adj = true;
  }
  SEG_TRY(cudaStreamSynchronize(cs));
#undef SEG_TRY
  scratch.release();
  s->held = lists.held;
  s->bytes = entries.bytes();
  *out = s;
  return TSP_OK;
}

extern "C" tsp_status tsp_debug_segments_memory(int64_t block_most, int64_t scratch_most) {
  g_block_most.store(block_most < 0 ? BLOCK_MOST : block_most);
  g_scratch_most.store(scratch_most < 0 ? std::numeric_limits<int64_t>::max() : scratch_most);
  return TSP_OK;
}

extern "C" tsp_status tsp_segments_info(tsp_segments s, int64_t* n_rays, int64_t* n_segments, size_t* bytes) {
  if (!s) return fail(TSP_EINVAL, "tsp_segments_info: NULL handle");
  if (n_rays) *n_rays = s->n_rays;
  if (n_segments) *n_segments = s->n_segs;
  if (bytes) *bytes = s->bytes;
  return TSP_OK;
}

// The lists to the host ray after ray, in pieces of whole rays through device
// buffers of 40 MB (less where there is less); a host loop over the entries takes
// ten times as long. The host's pages are touched first: several copies into
// pages that are not mapped yet took as long as that loop (106 M segments: 640 ms;
// 49 now, 56 in one copy per array when the lists lay ray after ray).
extern "C" tsp_status tsp_segments_export(tsp_segments s, int64_t* ray_off, uint32_t* vox, float* len) {
  if (!s) return fail(TSP_EINVAL, "tsp_segments_export: NULL handle");
  tsp_status st = check_device(s->device);
  if (st != TSP_OK) return st;
  if (!ray_off && !vox && !len) return TSP_OK;
  const int64_t n = s->n_rays;
  std::vector<int64_t> off(size_t(n + 1)), to(size_t(n + 1), 0);  // of the rows, of the rays
  TSP_CUDA(cudaMemcpy(off.data(), s->fwd.off, sizeof(int64_t) * off.size(), cudaMemcpyDeviceToHost));
  const RowOrder order = s->order;
  if (order.W == 0) {
    to = off;
  } else {
    int64_t p = 0;
    for (int64_t r0 = 0; r0 < n; r0 += int64_t(order.H) * order.W)  // views, bands, columns, rows of a band
      for (int i0 = 0; i0 < order.H; i0 += 4)
        for (int64_t col = 0; col < order.W; ++col)
          for (int i = i0; i < std::min(i0 + 4, order.H); ++i, ++p)
            to[size_t(r0 + int64_t(i) * order.W + col + 1)] = off[size_t(p + 1)] - off[size_t(p)];
    for (int64_t r = 0; r < n; ++r) to[size_t(r + 1)] += to[size_t(r)];
  }
  if (ray_off) std::copy(to.begin(), to.end(), ray_off);
  if (s->n_segs == 0 || (!vox && !len)) return TSP_OK;
  if (vox) std::memset(vox, 0, sizeof(uint32_t) * size_t(s->n_segs));
  if (len) std::memset(len, 0, sizeof(float) * size_t(s->n_segs));
  int64_t widest = 0;
  for (int64_t r = 0; r < n; ++r) widest = std::max(widest, to[size_t(r + 1)] - to[size_t(r)]);
  int64_t most = std::max(widest, std::min(s->n_segs, int64_t(1) << 22)), rays = std::min(n, int64_t(1) << 20);
  char* stage = nullptr;
  for (;;) {  // [rays + 1] offsets, [most] columns, [most] lengths
    const cudaError_t e = cudaMalloc(&stage, size_t(8 * (rays + 1) + 8 * most));
    if (e == cudaSuccess) break;
    if (most / 2 < std::max(widest, int64_t(1) << 16)) return cuda_fail(e, "tsp_segments_export: staging");
    cudaGetLastError();  // not sticky: clear it
    most /= 2;
    rays = std::max<int64_t>(1, rays / 2);
  }
  int64_t* const d_to = reinterpret_cast<int64_t*>(stage);
  uint32_t* const d_vox = reinterpret_cast<uint32_t*>(stage + 8 * (rays + 1));
  float* const d_len = reinterpret_cast<float*>(d_vox + most);
  cudaError_t e = cudaSuccess;
  for (int64_t a = 0, z; a < n && e == cudaSuccess; a = z) {
    for (z = a + 1; z < n && z - a < rays && to[size_t(z + 1)] - to[size_t(a)] <= most;) ++z;
    const size_t m = size_t(to[size_t(z)] - to[size_t(a)]);
    if (m == 0) continue;
    // the rows of these rays lie in their bands (their ranges of rows and of rays are the same)
    int64_t p0 = a, p1 = z;
    if (order.W > 0) {
      const int64_t plane = int64_t(order.H) * order.W, band = 4 * int64_t(order.W);
      p0 = a / plane * plane + a % plane / band * band;
      const int64_t v = (z - 1) / plane * plane;
      p1 = v + std::min(plane, ((z - 1 - v) / band + 1) * band);
    }
    p0 = p0 / 32 * 32;
    e = cudaMemcpy(d_to, to.data() + a, sizeof(int64_t) * size_t(z - a + 1), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) break;
    export_kernel<<<unsigned((p1 - p0 + 255) / 256), 256>>>(s->fwd.off, p0, n, order, s->fwd.idx, s->fwd.len, a, z,
                                                           d_to, d_vox, d_len);
    e = cudaGetLastError();
    if (e == cudaSuccess && vox)
      e = cudaMemcpy(vox + to[size_t(a)], d_vox, sizeof(uint32_t) * m, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && len)
      e = cudaMemcpy(len + to[size_t(a)], d_len, sizeof(float) * m, cudaMemcpyDeviceToHost);
  }
  cudaFree(stage);
  return e == cudaSuccess ? TSP_OK : cuda_fail(e, "tsp_segments_export");
}

extern "C" tsp_status tsp_segments_export_transposed(tsp_segments s, int64_t* vox_off, uint32_t* ray, float* len) {
  if (!s) return fail(TSP_EINVAL, "tsp_segments_export_transposed: NULL handle");
  if (!s->has_adj) return fail(TSP_EINVAL, "tsp_segments_export_transposed: lists built without the transpose");
  tsp_status st = check_device(s->device);
  if (st != TSP_OK) return st;
  if (vox_off)
    TSP_CUDA(cudaMemcpy(vox_off, s->adj.off, sizeof(int64_t) * size_t(s->V + 1), cudaMemcpyDeviceToHost));
  if (ray && s->n_segs) {
    TSP_CUDA(cudaMemcpy(ray, s->adj.idx, sizeof(uint32_t) * size_t(s->n_segs), cudaMemcpyDeviceToHost));
  }
  if (len && s->n_segs) TSP_CUDA(cudaMemcpy(len, s->adj.len, sizeof(float) * size_t(s->n_segs), cudaMemcpyDeviceToHost));
  return TSP_OK;
}

extern "C" tsp_status tsp_segments_forward(tsp_segments s, const float* rho, float* y, int batch, void* stream) {
  TSP_RANGE("tsp_segments_forward");
  if (!s || !rho || !y || batch <= 0) return fail(TSP_EINVAL, "tsp_segments_forward: bad argument");
  tsp_status st = check_device(s->device);
  if (st != TSP_OK) return st;
  return list_forward(s->fwd, s->order, rho, y, batch, nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

extern "C" tsp_status tsp_segments_adjoint(tsp_segments s, const float* y, float* rho, int batch, int accumulate,
                                           void* stream) {
  TSP_RANGE("tsp_segments_adjoint");
  if (!s || !y || !rho || batch <= 0) return fail(TSP_EINVAL, "tsp_segments_adjoint: bad argument");
  tsp_status st = check_device(s->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  if (s->has_adj) return list_adjoint(s->adj, y, rho, batch, accumulate, nullptr, cs);
  if (!accumulate) TSP_CUDA(cudaMemsetAsync(rho, 0, sizeof(float) * size_t(s->V) * batch, cs));
  for (int b = 0; b < batch; ++b)
    seg_scatter_kernel<<<unsigned((s->n_rays + 255) / 256), 256, 0, cs>>>(s->fwd.off, s->fwd.idx, s->fwd.len, s->order,
                                                                          y + b * s->n_rays, rho + b * s->V, s->n_rays);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_segments_sirt_workspace_bytes(tsp_segments s, size_t* bytes) {
  if (!s || !bytes) return fail(TSP_EINVAL, "tsp_segments_sirt_workspace_bytes: NULL argument");
  *bytes = 2 * align256(sizeof(float) * size_t(s->n_rays)) + 2 * align256(sizeof(float) * size_t(s->V));
  return TSP_OK;
}

// R = 1 / (F 1), C = 1 / (F^T 1) from the lists (0 where a sum is 0); ones_v
// [V] and ones_r [n_rays] are scratch.
static tsp_status list_weights(tsp_segments s, float* R, float* C, float* ones_v, float* ones_r, cudaStream_t cs) {
  const int64_t nr = s->n_rays, V = s->V;
  fill_kernel<<<ew_blocks(V), 256, 0, cs>>>(ones_v, V, 1.0f);
  tsp_status st = list_forward(s->fwd, s->order, ones_v, R, 1, nullptr, nullptr, cs);
  if (st != TSP_OK) return st;
  recip_kernel<<<ew_blocks(nr), 256, 0, cs>>>(R, nr);
  fill_kernel<<<ew_blocks(nr), 256, 0, cs>>>(ones_r, nr, 1.0f);
  st = tsp_segments_adjoint(s, ones_r, C, 1, 0, cs);
  if (st != TSP_OK) return st;
  recip_kernel<<<ew_blocks(V), 256, 0, cs>>>(C, V);
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

extern "C" tsp_status tsp_segments_sirt_weights(tsp_segments s, float* R, float* C, void* stream) {
  if (!s || !R || !C) return fail(TSP_EINVAL, "tsp_segments_sirt_weights: NULL argument");
  tsp_status st = check_device(s->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  float* ones = nullptr;
  const int64_t n = std::max<int64_t>(std::max(s->n_rays, s->V), 1);
  TSP_CUDA(cudaMallocAsync(&ones, sizeof(float) * size_t(n) * 2, cs));
  st = list_weights(s, R, C, ones, ones + n, cs);
  cudaFreeAsync(ones, cs);
  return st;
}

extern "C" tsp_status tsp_segments_sirt(tsp_segments s, const float* y, float* x, int n_iter, int flags,
                                        void* workspace, size_t workspace_bytes, void* stream) {
  TSP_RANGE("tsp_segments_sirt");
  if (!s || !y || !x || !workspace) return fail(TSP_EINVAL, "tsp_segments_sirt: NULL argument");
  if (n_iter < 0) return fail(TSP_EINVAL, "tsp_segments_sirt: n_iter < 0");
  if (flags & ~(TSP_SIRT_NONNEG | TSP_SIRT_REUSE_WEIGHTS)) return fail(TSP_EINVAL, "tsp_segments_sirt: unknown flags");
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return fail(TSP_EINVAL, "tsp_segments_sirt: workspace not 256-byte aligned");
  size_t need = 0;
  tsp_segments_sirt_workspace_bytes(s, &need);
  if (workspace_bytes < need)
    return fail(TSP_EINVAL, "tsp_segments_sirt: workspace of " + std::to_string(workspace_bytes) + " bytes, " +
                                std::to_string(need) + " needed");
  tsp_status st = check_device(s->device);
  if (st != TSP_OK) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  const int64_t nr = s->n_rays, V = s->V;
  char* p = static_cast<char*>(workspace);
  float* R = reinterpret_cast<float*>(p);
  float* r = reinterpret_cast<float*>(p + align256(4 * size_t(nr)));
  float* C = reinterpret_cast<float*>(p + 2 * align256(4 * size_t(nr)));
  float* g = reinterpret_cast<float*>(p + 2 * align256(4 * size_t(nr)) + align256(4 * size_t(V)));
  if (!(flags & TSP_SIRT_REUSE_WEIGHTS)) {
    st = list_weights(s, R, C, g, r, cs);
    if (st != TSP_OK) return st;
  }
  for (int it = 0; it < n_iter; ++it) {
    st = list_forward(s->fwd, s->order, x, r, 1, R, y, cs);  // r = R (y - F x)
    if (st != TSP_OK) return st;
    if (s->has_adj) {  // x += C F^T r
      st = list_adjoint(s->adj, r, x, 1, flags & TSP_SIRT_NONNEG, C, cs);
      if (st != TSP_OK) return st;
    } else {
      st = tsp_segments_adjoint(s, r, g, 1, 0, stream);  // g = F^T r
      if (st != TSP_OK) return st;
      xupdate_kernel<<<ew_blocks(V), 256, 0, cs>>>(x, g, C, V, flags & TSP_SIRT_NONNEG);
    }
  }
  TSP_CUDA(cudaGetLastError());
  return TSP_OK;
}

// ---------------------------------------------------------------------------
// Chunked segment lists: SIRT over many independent reconstructions whose
// stored lists together exceed device memory. Lists are built for one chunk
// of instances at a time (as many, in order, as fit the byte budget), every
// iteration of those instances runs from the lists, and the chunk's lists
// are freed before the next chunk is built. Each instance gets the same
// iterates as tsp_segments_sirt on its own lists.
// ---------------------------------------------------------------------------
extern "C" tsp_status tsp_sirt_chunked(const tsp_batch_item* items, int n_items, int n_iter, int flags,
                                       size_t budget_bytes, int* n_chunks, size_t* peak_bytes, void* stream) {
  TSP_RANGE("tsp_sirt_chunked");
  if (!items || n_items <= 0) return fail(TSP_EINVAL, "tsp_sirt_chunked: no items");
  if (n_iter < 0) return fail(TSP_EINVAL, "tsp_sirt_chunked: n_iter < 0");
  if (flags & ~TSP_SIRT_NONNEG) return fail(TSP_EINVAL, "tsp_sirt_chunked: unknown flags");
  for (int i = 0; i < n_items; ++i)
    if (!items[i].grid || !items[i].geom || !items[i].y || !items[i].x)
      return fail(TSP_EINVAL, "tsp_sirt_chunked: item " + std::to_string(i) + " has a NULL member");
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  if (budget_bytes == 0) {  // default: 80% of what is free now
    size_t free_b = 0, total_b = 0;
    TSP_CUDA(cudaMemGetInfo(&free_b, &total_b));
    budget_bytes = free_b / 10 * 8;
  }
  std::vector<tsp_segments> chunk;
  Blocks scratch;
  size_t used = 0, peak = 0, ws_bytes = 0;
  void* ws = nullptr;
  int chunks = 0;
  auto release = [&]() {
    for (tsp_segments s : chunk) tsp_segments_destroy(s);
    chunk.clear();
    used = 0;
  };
  auto run_chunk = [&](int first) -> tsp_status {  // items first .. first + chunk.size() - 1
    for (size_t k = 0; k < chunk.size(); ++k) {
      size_t need = 0;
      tsp_segments_sirt_workspace_bytes(chunk[k], &need);
      if (need > ws_bytes) {
        if (ws) cudaFree(ws);
        ws = nullptr;
        ws_bytes = 0;
        cudaError_t e = dev_malloc(&ws, need);
        if (e == cudaErrorMemoryAllocation) {  // the builds' spare scratch first
          cudaGetLastError();  // not sticky: clear it
          scratch.release_spares();
          e = dev_malloc(&ws, need);
        }
        if (e != cudaSuccess) return cuda_fail(e, "tsp_sirt_chunked: workspace");
        ws_bytes = need;
      }
      const tsp_batch_item& it = items[first + int(k)];
      tsp_status st = tsp_segments_sirt(chunk[k], it.y, it.x, n_iter, flags, ws, ws_bytes, stream);
      if (st != TSP_OK) return st;
    }
    ++chunks;
    return TSP_OK;
  };
  tsp_status st = TSP_OK;
  int first = 0;
  for (int i = 0; i < n_items && st == TSP_OK; ++i) {
    tsp_segments s = nullptr;
    st = build_lists(items[i].grid, items[i].geom, 1, scratch, &s, stream);
    if (st == TSP_ENOMEM && !chunk.empty()) {  // no room next to the chunk: finish it, then retry alone
      scratch.release_spares();  // (the workspace may have to be allocated now)
      st = run_chunk(first);
      if (st == TSP_OK) {
        cudaError_t e = cudaStreamSynchronize(cs);
        if (e != cudaSuccess) st = cuda_fail(e, "tsp_sirt_chunked: sync");
      }
      release();
      first = i;
      if (st == TSP_OK) st = build_lists(items[i].grid, items[i].geom, 1, scratch, &s, stream);
    }
    if (st != TSP_OK) break;
    size_t b = 0;
    tsp_segments_info(s, nullptr, nullptr, &b);
    if (!chunk.empty() && used + b > budget_bytes) {  // over budget: run the chunk built so far first
      st = run_chunk(first);
      if (st == TSP_OK) {
        cudaError_t e = cudaStreamSynchronize(cs);
        if (e != cudaSuccess) st = cuda_fail(e, "tsp_sirt_chunked: sync");
      }
      release();
      first = i;
    }
    chunk.push_back(s);
    used += b;
    peak = std::max(peak, used);
  }
  if (st == TSP_OK && !chunk.empty()) {
    st = run_chunk(first);
    if (st == TSP_OK) {
      cudaError_t e = cudaStreamSynchronize(cs);
      if (e != cudaSuccess) st = cuda_fail(e, "tsp_sirt_chunked: sync");
    }
  }
  release();
  scratch.release_spares();
  if (ws) cudaFree(ws);
  if (n_chunks) *n_chunks = chunks;
  if (peak_bytes) *peak_bytes = peak;
  return st;
}
