// rf_stream.cu -- the bandwidth kernels of the step core:
//   rf_schedule_compact  active-frame mask -> index lists (warp ballot / popc scan)
//   rf_project           Eq. 3 latent trajectory projection (128-bit streaming)
//   rf_project_kv        rolling key/value cache of Appendix B.2 (bf16, 128-bit streaming)
//   rf_step              Euler update of the active frames (128-bit streaming)
//   rf_step_core         a whole step: the four above in one launch, then the attention
#include <cuda_runtime.h>

#include "rf_host.h"

namespace rf {
namespace {

constexpr int kMaxFrames = 4096;
constexpr int kCompactThreads = 256;

// ---------------------------------------------------------------------------------------
// Compaction.  Every block rebuilds the (tiny) active list in shared memory with a
// ballot/popc scan, block 0 publishes the lists and counts, and all blocks write the
// token index list with a grid-stride loop (int4 stores).
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kCompactThreads)
    compact_kernel(const uint8_t* __restrict__ mask, int F, int N, int32_t* __restrict__ active,
                   int32_t* __restrict__ skipped, int32_t* __restrict__ token_idx,
                   int32_t* __restrict__ counts) {
  __shared__ int s_active[kMaxFrames];
  __shared__ int s_chunk_base[kMaxFrames / 32 + 1];
  __shared__ int s_A;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nchunks = (F + 31) >> 5;
  // per-32-frame chunk population counts
  for (int c = warp; c < nchunks; c += kCompactThreads / 32) {
    const int f = c * 32 + lane;
    const bool on = f < F && mask[f] != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    if (lane == 0) s_chunk_base[c] = __popc(bal);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int c = 0; c < nchunks; ++c) {
      const int n = s_chunk_base[c];
      s_chunk_base[c] = run;
      run += n;
    }
    s_A = run;
  }
  __syncthreads();
  const int A = s_A;
  for (int c = warp; c < nchunks; c += kCompactThreads / 32) {
    const int f = c * 32 + lane;
    const bool on = f < F && mask[f] != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    const int below = __popc(bal & ((1u << lane) - 1u));
    const int pos_on = s_chunk_base[c] + below;
    if (on) s_active[pos_on] = f;
    if (blockIdx.x == 0 && f < F) {
      if (on)
        active[pos_on] = f;
      else
        skipped[(c * 32 + lane) - pos_on] = f;  // frames before f that are skipped
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    counts[0] = A;
    counts[1] = A * N;
  }
  if (token_idx == nullptr) return;
  __syncthreads();
  const int total = A * N;
  const int nvec = total >> 2;
  int4* out4 = reinterpret_cast<int4*>(token_idx);
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += gridDim.x * blockDim.x) {
    int t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = 4 * v + k;
      const int a = i / N;
      t[k] = s_active[a] * N + (i - a * N);
    }
    out4[v] = make_int4(t[0], t[1], t[2], t[3]);
  }
  for (int i = 4 * nvec + blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += gridDim.x * blockDim.x) {
    const int a = i / N;
    token_idx[i] = s_active[a] * N + (i - a * N);
  }
}

// ---------------------------------------------------------------------------------------
// Streaming kernels.  grid = (blocks per frame, F); a block walks its frame's float4s with
// a stride of (blocks per frame * threads), four independent 16-byte loads in flight.
// ---------------------------------------------------------------------------------------
constexpr int kStreamThreads = 256;
constexpr int kUnroll = 4;

__device__ __forceinline__ float4 ld_stream(const float4* p) { return __ldcs(p); }
__device__ __forceinline__ void st_stream(float4* p, float4 v) { __stcs(p, v); }

__global__ void __launch_bounds__(kStreamThreads)
    project_kernel(float4* __restrict__ ctx, const float4* __restrict__ z2,
                   const uint8_t* __restrict__ cur_slot, const float* __restrict__ alpha,
                   const float* __restrict__ beta, int F, int64_t E4) {
  const int f = blockIdx.y;
  const int c = cur_slot[f] & 1;
  const float a = alpha[f], b = beta[f];
  const float4* cur = z2 + (static_cast<int64_t>(c) * F + f) * E4;
  const float4* prev = z2 + (static_cast<int64_t>(c ^ 1) * F + f) * E4;
  float4* out = ctx + static_cast<int64_t>(f) * E4;
  const int64_t step = static_cast<int64_t>(gridDim.x) * kStreamThreads;
  int64_t i = static_cast<int64_t>(blockIdx.x) * kStreamThreads + threadIdx.x;
  if (b == 0.0f) {  // active frame (or alpha == 1): ctx = cur, prev never read
    for (; i + (kUnroll - 1) * step < E4; i += kUnroll * step) {
      float4 v[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) v[u] = ld_stream(cur + i + u * step);
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) st_stream(out + i + u * step, v[u]);
    }
    for (; i < E4; i += step) st_stream(out + i, ld_stream(cur + i));
    return;
  }
  for (; i + (kUnroll - 1) * step < E4; i += kUnroll * step) {
    float4 x[kUnroll], y[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      x[u] = ld_stream(cur + i + u * step);
      y[u] = ld_stream(prev + i + u * step);
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      float4 r;
      r.x = fmaf(a, x[u].x, b * y[u].x);
      r.y = fmaf(a, x[u].y, b * y[u].y);
      r.z = fmaf(a, x[u].z, b * y[u].z);
      r.w = fmaf(a, x[u].w, b * y[u].w);
      st_stream(out + i + u * step, r);
    }
  }
  for (; i < E4; i += step) {
    const float4 x = ld_stream(cur + i), y = ld_stream(prev + i);
    float4 r;
    r.x = fmaf(a, x.x, b * y.x);
    r.y = fmaf(a, x.y, b * y.y);
    r.z = fmaf(a, x.z, b * y.z);
    r.w = fmaf(a, x.w, b * y.w);
    st_stream(out + i, r);
  }
}

// Euler step over the active frames only.  The active count lives on the device, so the grid
// is fixed (a few waves) and walks (active frame, chunk of kStreamThreads*kUnroll float4s)
// pairs with a stride of gridDim.x chunks: the work spreads over every SM whatever A is.
__global__ void __launch_bounds__(kStreamThreads)
    step_kernel(float4* __restrict__ z2, const uint8_t* __restrict__ cur_slot,
                const float4* __restrict__ vel, const float* __restrict__ dt,
                const int32_t* __restrict__ active, const int32_t* __restrict__ counts, int F,
                int64_t E4) {
  constexpr int64_t kChunk = static_cast<int64_t>(kStreamThreads) * kUnroll;
  int A = counts[0];
  A = A < 0 ? 0 : (A > F ? F : A);
  const int64_t per_frame = (E4 + kChunk - 1) / kChunk;
  const int64_t total = per_frame * A;
  for (int64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const int a = static_cast<int>(c / per_frame);
    const int64_t base = (c - a * per_frame) * kChunk + threadIdx.x;
    const int f = active[a];
    if (f < 0 || f >= F) continue;
    const int sl = cur_slot[f] & 1;
    const float h = dt[f];
    const float4* z = z2 + (static_cast<int64_t>(sl) * F + f) * E4;
    float4* out = z2 + (static_cast<int64_t>(sl ^ 1) * F + f) * E4;
    const float4* v = vel + static_cast<int64_t>(f) * E4;
    float4 x[kUnroll], y[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t i = base + u * kStreamThreads;
      if (i < E4) {
        x[u] = ld_stream(z + i);
        y[u] = ld_stream(v + i);
      }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t i = base + u * kStreamThreads;
      if (i < E4) {
        float4 r;
        r.x = fmaf(h, y[u].x, x[u].x);
        r.y = fmaf(h, y[u].y, x[u].y);
        r.z = fmaf(h, y[u].z, x[u].z);
        r.w = fmaf(h, y[u].w, x[u].w);
        st_stream(out + i, r);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Rolling key/value cache (Appendix B.2).  blockIdx.y selects keys or values.  The grid walks
// (frame-list index, chunk) pairs over all F frames: list index a < A is the active frame
// active[a], whose fresh rows are stored into its cache's other slot (shift-and-store); the
// rest are skipped[a - A], whose rows are rewritten with Eq. 3 from the two cached states.
// Eight bf16 per 16-byte access; fp32 arithmetic, rounded to nearest even.
//
// Bound by HBM.  Every frame has work, so the grid has one CTA per chunk of 128 threads x 4 vectors
// (8 KB of each stream) and the scheduler deals them out; walking the chunks with a fixed grid of
// four CTAs of 256 threads per SM left the SMs' last chunks uneven.  Keyframe-only step of
// 33 x 3600 x 3072: 595 -> 570 us (7.2 TB/s; 7.1 TB/s is what torch.add's two reads and a
// write reach), all frames active 435 -> 405 us, 13 x 1560 x 1536: 52.1 -> 50.0 us.  256 threads
// 567 / 422 / 50.9, two or eight vectors per thread at 256 threads 568 / 414 / 50.2 and
// 676 / 522 / 59.8.
// ---------------------------------------------------------------------------------------
constexpr int kKvThreads = 128;
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t proj_pair(uint32_t cur, uint32_t prev, float a, float b) {
  const float lo = fmaf(a, bf16_lo(cur), b * bf16_lo(prev));
  const float hi = fmaf(a, bf16_hi(cur), b * bf16_hi(prev));
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// One chunk (kKvThreads x kUnroll vectors from `base`, this thread's first) of frame f's keys or
// values X and their cache Xc.
__device__ __forceinline__ void kv_chunk(uint16_t* X, int64_t row_stride, uint16_t* Xc,
                                         const uint8_t* cur_slot, const float* alpha,
                                         const float* beta, int F, int N, int D, int f,
                                         bool is_active, int64_t base) {
  const int D8 = D >> 3;  // 16-byte vectors per row
  const int64_t frame_vecs = static_cast<int64_t>(N) * D8;
  const int64_t slot_stride = static_cast<int64_t>(F) * N * D;  // elements between slots
  const bool contiguous = row_stride == D;  // K/V rows back to back: no row arithmetic
  const int sl = cur_slot[f] & 1;
  const uint4* cur = reinterpret_cast<const uint4*>(Xc + sl * slot_stride +
                                                    static_cast<int64_t>(f) * N * D);
  uint4* prev = reinterpret_cast<uint4*>(Xc + (sl ^ 1) * slot_stride +
                                         static_cast<int64_t>(f) * N * D);
  uint16_t* rows = X + static_cast<int64_t>(f) * N * row_stride;
  // vector index of the k-th vector of this thread inside the frame's K/V rows: (row, col)
  // advanced incrementally (one division per chunk, none per vector)
  int64_t off[kUnroll];
  {
    int64_t p = 0, q = base;
    if (!contiguous) {
      p = static_cast<uint32_t>(base) / static_cast<uint32_t>(D8);  // < 2^31 (host check)
      q = base - p * D8;
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      off[u] = contiguous ? base + u * kKvThreads : p * (row_stride >> 3) + q;
      if (!contiguous) {
        q += kKvThreads;
        while (q >= D8) {
          q -= D8;
          ++p;
        }
      }
    }
  }
  uint4* rv = reinterpret_cast<uint4*>(rows);
  if (is_active) {
    uint4 x[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (base + u * kKvThreads < frame_vecs) x[u] = __ldcs(rv + off[u]);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t v = base + u * kKvThreads;
      if (v < frame_vecs) __stcs(prev + v, x[u]);  // the other slot
    }
  } else {
    const float al = alpha[f], be = beta[f];
    uint4 x[kUnroll], y[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t v = base + u * kKvThreads;
      if (v < frame_vecs) {
        x[u] = __ldcs(cur + v);
        y[u] = __ldcs(prev + v);
      }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      if (base + u * kKvThreads < frame_vecs) {
        uint4 r;
        r.x = proj_pair(x[u].x, y[u].x, al, be);
        r.y = proj_pair(x[u].y, y[u].y, al, be);
        r.z = proj_pair(x[u].z, y[u].z, al, be);
        r.w = proj_pair(x[u].w, y[u].w, al, be);
        __stcs(rv + off[u], r);
      }
    }
  }
}

__global__ void __launch_bounds__(kKvThreads)
    project_kv_kernel(uint16_t* __restrict__ K, uint16_t* __restrict__ V, int64_t row_stride,
                      uint16_t* __restrict__ Kc, uint16_t* __restrict__ Vc,
                      const uint8_t* __restrict__ cur_slot, const float* __restrict__ alpha,
                      const float* __restrict__ beta, const int32_t* __restrict__ active,
                      const int32_t* __restrict__ skipped, const int32_t* __restrict__ counts,
                      int F, int N, int D) {
  uint16_t* X = blockIdx.y ? V : K;
  uint16_t* Xc = blockIdx.y ? Vc : Kc;
  int A = counts[0];
  A = A < 0 ? 0 : (A > F ? F : A);
  const int64_t frame_vecs = static_cast<int64_t>(N) * (D >> 3);  // 16-byte vectors
  constexpr int64_t kChunk = static_cast<int64_t>(kKvThreads) * kUnroll;
  const int64_t per_frame = (frame_vecs + kChunk - 1) / kChunk;
  const int64_t total = per_frame * F;
  for (int64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const int a = static_cast<int>(c / per_frame);
    const int64_t base = (c - a * per_frame) * kChunk + threadIdx.x;
    const bool is_active = a < A;
    const int f = is_active ? active[a] : skipped[a - A];
    if (f < 0 || f >= F) continue;
    kv_chunk(X, row_stride, Xc, cur_slot, alpha, beta, F, N, D, f, is_active, base);
  }
}

// ---------------------------------------------------------------------------------------
// A step's work beside its attention in one launch: compaction, Eq. 3 of the latents and of the
// cached keys and values, and the Euler update.  What each CTA does follows from its index:
//   0           the frame lists and counts
//   n_tok       one chunk of kTokChunk entries of one frame's part of the token list
//   n_lat       one chunk of one frame's latents: the context, and the next state if it is active
//   2 n_kv      one chunk of one frame's keys, then of its values
//
// The four parts depend only on the step's mask row, which every CTA reads for its own frame (the
// token list also needs the frame's rank, a block-wide count over the mask), so nothing waits
// for the lists.  A frame's context and next state are made by the same thread: the state is read
// once for both, and a context that reads the other slot has read it before it is overwritten.
//
// Bound by launches at small sizes and by HBM through the keys and values at large ones.  As four
// launches of their own (compaction, latents, keys and values before the attention, the Euler
// update after it) they cost the launch, ramp and drain of each: keyframe-only step of
// 13 x 1560 x 1536, 2.9 + 5.4 + 47 + 4.5 us in kernels, 44 us as one; four steps of 4 x 64 tokens
// replayed as a graph, 106.9 -> 86.4 us with the copies around it; a step of them from the host
// 57.4 -> 23.8 us.
// ---------------------------------------------------------------------------------------
constexpr int kTokChunk = 16 * kKvThreads;
constexpr int kFrontTiles = kMaxFrames / kKvThreads;  // mask tiles of one thread's register
static_assert(kFrontTiles <= 32, "one bit per tile of the mask");

struct FrontParams {
  const uint8_t *mask, *cur_slot;
  const float *alpha, *beta, *dt;
  int32_t *active, *skipped, *token_idx, *counts;
  float4 *ctx, *z2;
  const float4* v;
  uint16_t *K, *V, *Kc, *Vc;
  int64_t E4, kv_row_stride;
  int F, N, D;
  uint32_t n_tok, n_lat, n_kv;                            // CTAs of each part (n_kv: keys)
  uint32_t tok_per_frame, lat_per_frame, kv_per_frame;    // chunks per frame
};

// The active and skipped lists and the counts, by one CTA.
__device__ __forceinline__ void front_lists(const FrontParams& p) {
  __shared__ int s_count[2][kKvThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tiles = (p.F + kKvThreads - 1) / kKvThreads;
  uint32_t on = 0;  // bit t: frame t * kKvThreads + tid is active
#pragma unroll 4
  for (int t = 0; t < tiles; ++t) {
    const int f = t * kKvThreads + tid;
    if (f < p.F && p.mask[f] != 0) on |= 1u << t;
  }
  int run = 0;  // active frames before tile t
  for (int t = 0; t < tiles; ++t) {
    const bool mine = (on >> t) & 1u;
    const unsigned bal = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_count[t & 1][wid] = __popc(bal);
    __syncthreads();  // two rows of counts: tile t + 2 is written after everyone has read tile t
    int pos = run + __popc(bal & ((1u << lane) - 1u));
#pragma unroll
    for (int w = 0; w < kKvThreads / 32; ++w) {
      const int n = s_count[t & 1][w];
      if (w < wid) pos += n;
      run += n;
    }
    const int f = t * kKvThreads + tid;
    if (f < p.F) {
      if (mine)
        p.active[pos] = f;
      else
        p.skipped[f - pos] = f;  // frames before f that are skipped
    }
  }
  if (tid == 0) {
    p.counts[0] = run;
    p.counts[1] = run * p.N;
  }
}

__device__ __forceinline__ void front_tokens(const FrontParams& p, uint32_t c) {
  const int f = static_cast<int>(c / p.tok_per_frame);
  const uint32_t first = (c - f * p.tok_per_frame) * kTokChunk;
  if (p.mask[f] == 0) return;
  int rank = 0;  // active frames before f
  for (int g0 = 0; g0 < f; g0 += kKvThreads) {
    const int g = g0 + static_cast<int>(threadIdx.x);
    rank += __syncthreads_count(g < f && p.mask[g] != 0);
  }
  int32_t* out = p.token_idx + static_cast<int64_t>(rank) * p.N;
#pragma unroll 4
  for (int u = 0; u < kTokChunk / kKvThreads; ++u) {
    const uint32_t i = first + u * kKvThreads + threadIdx.x;  // past N by less than a chunk
    if (i < static_cast<uint32_t>(p.N)) out[i] = f * p.N + static_cast<int>(i);
  }
}

__device__ __forceinline__ float4 axpby(float a, float4 x, float b, float4 y) {
  return make_float4(fmaf(a, x.x, b * y.x), fmaf(a, x.y, b * y.y), fmaf(a, x.z, b * y.z),
                     fmaf(a, x.w, b * y.w));
}
__device__ __forceinline__ float4 axpy(float h, float4 v, float4 z) {
  return make_float4(fmaf(h, v.x, z.x), fmaf(h, v.y, z.y), fmaf(h, v.z, z.z), fmaf(h, v.w, z.w));
}

__device__ __forceinline__ void front_latent(const FrontParams& p, uint32_t c) {
  const int f = static_cast<int>(c / p.lat_per_frame);
  const int64_t base =
      static_cast<int64_t>(c - f * p.lat_per_frame) * (kKvThreads * kUnroll) + threadIdx.x;
  const bool is_active = p.mask[f] != 0;
  const int sl = p.cur_slot[f] & 1;
  const float a = p.alpha[f], b = p.beta[f], h = p.dt[f];
  const float4* cur = p.z2 + (static_cast<int64_t>(sl) * p.F + f) * p.E4;
  float4* other = p.z2 + (static_cast<int64_t>(sl ^ 1) * p.F + f) * p.E4;
  float4* out = p.ctx + f * p.E4;
  const float4* second = is_active ? p.v + f * p.E4 : other;
  if (is_active && b != 0.0f) {  // reads all three; no plan of rf_plan_build has such a frame
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t i = base + u * kKvThreads;
      if (i < p.E4) {
        const float4 x = ld_stream(cur + i), y = ld_stream(other + i), v = ld_stream(second + i);
        st_stream(out + i, axpby(a, x, b, y));
        st_stream(other + i, axpy(h, v, x));
      }
    }
    return;
  }
  const bool two = is_active || b != 0.0f;
  float4 x[kUnroll], y[kUnroll];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const int64_t i = base + u * kKvThreads;
    if (i < p.E4) {
      x[u] = ld_stream(cur + i);
      if (two) y[u] = ld_stream(second + i);
    }
  }
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const int64_t i = base + u * kKvThreads;
    if (i < p.E4) {
      if (is_active) st_stream(other + i, axpy(h, y[u], x[u]));
      st_stream(out + i, b == 0.0f ? x[u] : axpby(a, x[u], b, y[u]));
    }
  }
}

__global__ void __launch_bounds__(kKvThreads) front_kernel(const __grid_constant__ FrontParams p) {
  uint32_t c = blockIdx.x;
  if (c == 0) return front_lists(p);
  c -= 1;
  if (c < p.n_tok) return front_tokens(p, c);
  c -= p.n_tok;
  if (c < p.n_lat) return front_latent(p, c);
  c -= p.n_lat;
  const bool values = c >= p.n_kv;
  if (values) c -= p.n_kv;
  const int f = static_cast<int>(c / p.kv_per_frame);
  const int64_t base =
      static_cast<int64_t>(c - f * p.kv_per_frame) * (kKvThreads * kUnroll) + threadIdx.x;
  kv_chunk(values ? p.V : p.K, p.kv_row_stride, values ? p.Vc : p.Kc, p.cur_slot, p.alpha, p.beta,
           p.F, p.N, p.D, f, p.mask[f] != 0, base);
}

rf_status launch_front(const void* arg, cudaStream_t stream) {
  // an error that an earlier call left behind is reported while nothing has been enqueued
  if (rf_status st = launch_status("before rf_step_core")) return st;
  const FrontParams& p = *static_cast<const FrontParams*>(arg);
  front_kernel<<<1 + p.n_tok + p.n_lat + 2 * p.n_kv, kKvThreads, 0, stream>>>(p);
  return launch_status("front_kernel launch");
}

// Address ranges of a step's buffers, to see whether its parts may share a launch.
enum : uint32_t {
  kReads = 1,        // read by front_kernel
  kWrites = 2,       // written by front_kernel
  kEuler = 4,        // of the Euler update, which as a launch of its own follows the attention
  kAttn = 8,         // of the attention only
  kRows = 16,        // keys and values: may be slices of one buffer, rows interleaved
};
struct Range {
  uintptr_t lo, hi;
  uint32_t what;
};
bool overlap_matters(const Range& a, const Range& b) {
  if (a.lo >= b.hi || b.lo >= a.hi) return false;
  if ((a.what & b.what & kRows) != 0) return false;
  if ((a.what & b.what & kAttn) != 0) return false;
  if (((a.what | b.what) & kAttn) != 0) return ((a.what | b.what) & kEuler) != 0;
  return ((a.what | b.what) & kWrites) != 0;
}

// Blocks per frame so that the whole grid covers a few waves of the device even when only
// one frame is active, without launching blocks that would have nothing to do.
int blocks_per_frame(int64_t E4, int sm_count) {
  const int64_t per_block = static_cast<int64_t>(kStreamThreads) * kUnroll;
  int64_t bx = (E4 + per_block - 1) / per_block;
  const int64_t cap = 4LL * sm_count;
  if (bx > cap) bx = cap;
  if (bx < 1) bx = 1;
  return static_cast<int>(bx);
}

// Argument errors of the entry points, before anything is enqueued.
rf_status check_compact(const uint8_t* d_mask, int F, int N, const int32_t* d_active,
                        const int32_t* d_skipped, const int32_t* d_token_idx,
                        const int32_t* d_counts) {
  if (!d_mask || !d_active || !d_skipped || !d_counts) return RF_ERR_INVALID_ARG;
  if (F < 1 || F > kMaxFrames || N < 1) return RF_ERR_INVALID_ARG;
  if (static_cast<int64_t>(F) * N > 0x7FFFFFFF) return RF_ERR_INVALID_ARG;
  if (d_token_idx && !aligned16(d_token_idx)) return RF_ERR_MISALIGNED;
  return RF_OK;
}

rf_status check_project(const float* d_ctx, const float* d_z2, const uint8_t* d_cur_slot,
                        const float* d_alpha, const float* d_beta, int F, int64_t E) {
  if (!d_ctx || !d_z2 || !d_cur_slot || !d_alpha || !d_beta) return RF_ERR_INVALID_ARG;
  if (F < 1 || F > 65535 || E < 0) return RF_ERR_INVALID_ARG;
  if (E % 4 != 0) return RF_ERR_MISALIGNED;
  if (!aligned16(d_ctx) || !aligned16(d_z2)) return RF_ERR_MISALIGNED;
  return RF_OK;
}

rf_status check_step(const float* d_z2, const uint8_t* d_cur_slot, const float* d_v,
                     const float* d_dt, const int32_t* d_active, const int32_t* d_counts, int F,
                     int64_t E) {
  if (!d_z2 || !d_cur_slot || !d_v || !d_dt || !d_active || !d_counts) return RF_ERR_INVALID_ARG;
  if (F < 1 || F > 65535 || E < 0) return RF_ERR_INVALID_ARG;
  if (E % 4 != 0) return RF_ERR_MISALIGNED;
  if (!aligned16(d_z2) || !aligned16(d_v)) return RF_ERR_MISALIGNED;
  return RF_OK;
}

rf_status check_project_kv(const void* d_K, const void* d_V, int64_t kv_row_stride,
                           const void* d_Kc, const void* d_Vc, const uint8_t* d_cur_slot,
                           const float* d_alpha, const float* d_beta, const int32_t* d_active,
                           const int32_t* d_skipped, const int32_t* d_counts, int F, int N,
                           int D) {
  if (!d_K || !d_V || !d_Kc || !d_Vc || !d_cur_slot || !d_alpha || !d_beta || !d_active ||
      !d_skipped || !d_counts)
    return RF_ERR_INVALID_ARG;
  if (F < 1 || F > kMaxFrames || N < 1 || D < 8) return RF_ERR_INVALID_ARG;
  if (kv_row_stride < D) return RF_ERR_INVALID_ARG;
  if (static_cast<int64_t>(N) * (D / 8) > 0x7FFFFFFF) return RF_ERR_INVALID_ARG;
  if (D % 8 != 0 || kv_row_stride % 8 != 0) return RF_ERR_MISALIGNED;
  if (!aligned16(d_K) || !aligned16(d_V) || !aligned16(d_Kc) || !aligned16(d_Vc))
    return RF_ERR_MISALIGNED;
  return RF_OK;
}

}  // namespace
}  // namespace rf

using namespace rf;

extern "C" rf_status rf_schedule_compact(const uint8_t* d_mask, int F, int N, int32_t* d_active,
                                         int32_t* d_skipped, int32_t* d_token_idx,
                                         int32_t* d_counts, rf_stream_t stream) {
  if (rf_status st = check_compact(d_mask, F, N, d_active, d_skipped, d_token_idx, d_counts))
    return st;
  DeviceInfo di;
  if (rf_status st = current_device_info(&di)) return st;
  int blocks = 1;
  if (d_token_idx) {
    const int64_t nvec = (static_cast<int64_t>(F) * N + 3) / 4;
    int64_t b = (nvec + kCompactThreads - 1) / kCompactThreads;
    if (b > di.sm_count) b = di.sm_count;
    blocks = static_cast<int>(b < 1 ? 1 : b);
  }
  compact_kernel<<<blocks, kCompactThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      d_mask, F, N, d_active, d_skipped, d_token_idx, d_counts);
  return launch_status("compact_kernel launch");
}

extern "C" rf_status rf_project(float* d_ctx, const float* d_z2, const uint8_t* d_cur_slot,
                                const float* d_alpha, const float* d_beta, int F, int64_t E,
                                rf_stream_t stream) {
  if (rf_status st = check_project(d_ctx, d_z2, d_cur_slot, d_alpha, d_beta, F, E)) return st;
  if (E == 0) return RF_OK;
  DeviceInfo di;
  if (rf_status st = current_device_info(&di)) return st;
  const int64_t E4 = E / 4;
  dim3 grid(blocks_per_frame(E4, di.sm_count), F);
  project_kernel<<<grid, kStreamThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<float4*>(d_ctx), reinterpret_cast<const float4*>(d_z2), d_cur_slot,
      d_alpha, d_beta, F, E4);
  return launch_status("project_kernel launch");
}

extern "C" rf_status rf_step(float* d_z2, const uint8_t* d_cur_slot, const float* d_v,
                             const float* d_dt, const int32_t* d_active, const int32_t* d_counts,
                             int F, int64_t E, rf_stream_t stream) {
  if (rf_status st = check_step(d_z2, d_cur_slot, d_v, d_dt, d_active, d_counts, F, E)) return st;
  if (E == 0) return RF_OK;
  DeviceInfo di;
  if (rf_status st = current_device_info(&di)) return st;
  const int64_t E4 = E / 4;
  // enough chunks in flight to cover every SM a few times, never more than the largest A needs
  const int64_t chunk = static_cast<int64_t>(kStreamThreads) * kUnroll;
  int64_t blocks = ((E4 + chunk - 1) / chunk) * F;
  if (blocks > 8LL * di.sm_count) blocks = 8LL * di.sm_count;
  step_kernel<<<static_cast<int>(blocks), kStreamThreads, 0,
                reinterpret_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<float4*>(d_z2), d_cur_slot, reinterpret_cast<const float4*>(d_v), d_dt,
      d_active, d_counts, F, E4);
  return launch_status("step_kernel launch");
}

extern "C" rf_status rf_project_kv(void* d_K, void* d_V, int64_t kv_row_stride, void* d_Kc,
                                   void* d_Vc, const uint8_t* d_cur_slot, const float* d_alpha,
                                   const float* d_beta, const int32_t* d_active,
                                   const int32_t* d_skipped, const int32_t* d_counts, int F,
                                   int N, int D, rf_stream_t stream) {
  if (rf_status st = check_project_kv(d_K, d_V, kv_row_stride, d_Kc, d_Vc, d_cur_slot, d_alpha,
                                      d_beta, d_active, d_skipped, d_counts, F, N, D))
    return st;
  DeviceInfo di;
  if (rf_status st = current_device_info(&di)) return st;
  const int64_t frame_vecs = static_cast<int64_t>(N) * (D / 8);
  const int64_t chunk = static_cast<int64_t>(kKvThreads) * kUnroll;
  int64_t blocks = ((frame_vecs + chunk - 1) / chunk) * F;
  if (blocks > 0x7FFFFFFFLL) blocks = 0x7FFFFFFFLL;  // the kernel walks on from there
  dim3 grid(static_cast<unsigned>(blocks), 2);
  project_kv_kernel<<<grid, kKvThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      static_cast<uint16_t*>(d_K), static_cast<uint16_t*>(d_V), kv_row_stride,
      static_cast<uint16_t*>(d_Kc), static_cast<uint16_t*>(d_Vc), d_cur_slot, d_alpha, d_beta,
      d_active, d_skipped, d_counts, F, N, D);
  return launch_status("project_kv_kernel launch");
}

extern "C" rf_status rf_step_core(
    const uint8_t* d_mask, const uint8_t* d_cur_slot, const float* d_alpha, const float* d_beta,
    const float* d_dt, int F, int N, int64_t E, int H, int d, int32_t* d_active,
    int32_t* d_skipped, int32_t* d_token_idx, int32_t* d_counts, float* d_ctx, float* d_z2,
    const float* d_v, void* d_Kc, void* d_Vc, void* d_O, float* d_lse, const void* d_Q, void* d_K,
    void* d_V, int64_t qkv_row_stride, int64_t kv_row_stride, int64_t o_row_stride,
    float softmax_scale, void* d_workspace, int64_t workspace_bytes, int32_t* d_status,
    rf_stream_t stream) {
  const bool cache = d_Kc != nullptr || d_Vc != nullptr;
  if (rf_status st = check_compact(d_mask, F, N, d_active, d_skipped, d_token_idx, d_counts))
    return st;
  if (rf_status st = check_project(d_ctx, d_z2, d_cur_slot, d_alpha, d_beta, F, E)) return st;
  if (H < 1 || H > 65535 || (d != 64 && d != 128))
    return H < 1 || H > 65535 ? RF_ERR_INVALID_ARG : RF_ERR_UNSUPPORTED;
  const int D = H * d;
  if (cache)
    if (rf_status st = check_project_kv(d_K, d_V, kv_row_stride, d_Kc, d_Vc, d_cur_slot, d_alpha,
                                        d_beta, d_active, d_skipped, d_counts, F, N, D))
      return st;
  if (rf_status st = attn_check(d_O, d_Q, d_K, d_V, qkv_row_stride, o_row_stride, F, N, H, d,
                                d_active, d_counts, softmax_scale, d_workspace, workspace_bytes))
    return st;
  if (rf_status st = check_step(d_z2, d_cur_slot, d_v, d_dt, d_active, d_counts, F, E)) return st;

  FrontParams p;
  p.mask = d_mask;
  p.cur_slot = d_cur_slot;
  p.alpha = d_alpha;
  p.beta = d_beta;
  p.dt = d_dt;
  p.active = d_active;
  p.skipped = d_skipped;
  p.token_idx = d_token_idx;
  p.counts = d_counts;
  p.ctx = reinterpret_cast<float4*>(d_ctx);
  p.z2 = reinterpret_cast<float4*>(d_z2);
  p.v = reinterpret_cast<const float4*>(d_v);
  p.K = static_cast<uint16_t*>(d_K);
  p.V = static_cast<uint16_t*>(d_V);
  p.Kc = static_cast<uint16_t*>(d_Kc);
  p.Vc = static_cast<uint16_t*>(d_Vc);
  p.E4 = E / 4;
  p.kv_row_stride = kv_row_stride;
  p.F = F;
  p.N = N;
  p.D = D;
  constexpr int64_t kChunk = static_cast<int64_t>(kKvThreads) * kUnroll;
  const int64_t tok = d_token_idx ? (static_cast<int64_t>(N) + kTokChunk - 1) / kTokChunk : 0;
  const int64_t lat = (p.E4 + kChunk - 1) / kChunk;
  const int64_t kv = cache ? (static_cast<int64_t>(N) * (D / 8) + kChunk - 1) / kChunk : 0;

  // The parts share a launch unless their buffers overlap (a velocity that is a view of the
  // context or of the attention's output, say) or the grid could not hold them: then each is a
  // launch of its own, in order.
  const int64_t S_tok = static_cast<int64_t>(F) * N, f4 = 4 * static_cast<int64_t>(F);
  const int64_t kv_span = 2 * ((S_tok - 1) * kv_row_stride + D);
  const int64_t q_span = 2 * ((S_tok - 1) * qkv_row_stride + D);
  const int64_t o_span = 2 * ((S_tok - 1) * o_row_stride + D);
  const int64_t c_span = cache ? 4 * S_tok * D : 0;
  Range r[24];
  int n = 0;
  auto add = [&](const void* base, int64_t bytes, uint32_t what) {
    const uintptr_t lo = reinterpret_cast<uintptr_t>(base);
    if (base != nullptr && bytes > 0) r[n++] = Range{lo, lo + static_cast<uintptr_t>(bytes), what};
  };
  add(d_mask, F, kReads);
  add(d_cur_slot, F, kReads | kEuler);
  add(d_alpha, f4, kReads);
  add(d_beta, f4, kReads);
  add(d_dt, f4, kReads | kEuler);
  add(d_active, f4, kWrites);
  add(d_skipped, f4, kWrites);
  add(d_token_idx, 4 * S_tok, kWrites);
  add(d_counts, 8, kWrites);
  add(d_ctx, f4 * E, kWrites);
  add(d_z2, 2 * f4 * E, kWrites | kEuler);
  add(d_v, f4 * E, kReads | kEuler);
  if (cache) {
    add(d_K, kv_span, kWrites | kRows);
    add(d_V, kv_span, kWrites | kRows);
  }
  add(d_Kc, c_span, kWrites);
  add(d_Vc, c_span, kWrites);
  add(d_Q, q_span, kAttn);
  add(d_K, q_span, kAttn);
  add(d_V, q_span, kAttn);
  add(d_O, o_span, kAttn);
  add(d_lse, 4 * S_tok * H, kAttn);
  add(d_workspace, workspace_bytes, kAttn);
  add(d_status, 4, kAttn);
  bool together = lat * F + tok * F + 2 * kv * F < 0x7FFFFFFF;
  for (int i = 0; i < n && together; ++i)
    for (int j = 0; j < i && together; ++j) together = !overlap_matters(r[i], r[j]);

  if (together) {
    p.tok_per_frame = static_cast<uint32_t>(tok);
    p.lat_per_frame = static_cast<uint32_t>(lat);
    p.kv_per_frame = static_cast<uint32_t>(kv);
    p.n_tok = static_cast<uint32_t>(tok * F);
    p.n_lat = static_cast<uint32_t>(lat * F);
    p.n_kv = static_cast<uint32_t>(kv * F);
    // the Euler update goes in front of the attention, so that must be able to follow
    return attn_behind(Front{launch_front, &p}, d_O, d_lse, d_Q, d_K, d_V, qkv_row_stride,
                       o_row_stride, F, N, H, d, d_active, d_counts, softmax_scale, d_workspace,
                       workspace_bytes, d_status, stream);
  }
  if (rf_status st = rf_schedule_compact(d_mask, F, N, d_active, d_skipped, d_token_idx, d_counts,
                                         stream))
    return st;
  if (rf_status st = rf_project(d_ctx, d_z2, d_cur_slot, d_alpha, d_beta, F, E, stream)) return st;
  if (cache)
    if (rf_status st = rf_project_kv(d_K, d_V, kv_row_stride, d_Kc, d_Vc, d_cur_slot, d_alpha,
                                     d_beta, d_active, d_skipped, d_counts, F, N, D, stream))
      return st;
  if (rf_status st = rf_attn(d_O, d_lse, d_Q, d_K, d_V, qkv_row_stride, o_row_stride, F, N, H, d,
                             d_active, d_counts, softmax_scale, d_workspace, workspace_bytes,
                             d_status, stream))
    return st;
  return rf_step(d_z2, d_cur_slot, d_v, d_dt, d_active, d_counts, F, E, stream);
}
