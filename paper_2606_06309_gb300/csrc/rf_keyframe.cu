// rf_keyframe.cu -- inner products of the clean-latent proxies for keyframe selection.
//
// Sequential keyframe selection (Sec. 3.1, Eq. 1, Algorithm 1) compares each candidate frame
// with the latest keyframe by cosine similarity.  Which pairs are compared depends on earlier
// decisions, so the device computes every inner product <P_i, P_j> of the F frame proxies at
// once (the Gram matrix; its diagonal gives the norms) and the host runs the sequential rule
// over it (rf_keyframe_select in rf_plan.cpp).
//
// gram_kernel (gram_short_kernel where that is faster, see short_is_faster): split-K
// over the proxy length E.  Each CTA takes every n-th slice of up to 128
// elements of every frame, streams them through shared memory (cp.async, two or three stages,
// rows as they are in memory) and accumulates 8 x 8 frame pairs per thread in fp32, four
// elements at a time.  Only tiles on and above the diagonal have threads: with G = ceil(F/8)
// groups, tile (i <= j) pairs the frames i + aG with j + bG (a, b < 8), so that neighbouring
// threads read neighbouring rows, and KG = 2^n k-groups of tiles fill up to 256 threads, each
// group taking every KG-th quad of elements.  At the end the k-groups are summed in shared
// memory, then the two CTAs of a cluster through distributed shared memory, both as
// unevaluated pairs of floats (the fp64 units are few; a sum past their range is made again in
// 64 bits), and one fp64 atomic per entry and cluster reaches the result.  So only a thread's own
// chain of multiply-adds has the range of fp32: at most 96 of the 384 elements of a short
// CTA (four k-groups, above 56 frames), or a quarter of a long one's.
//
// What bounds it: at latent width (33 x 57600) launches, the final sums and the atomics; at
// hidden width instruction issue and shared-memory reads.  A tile of T x T costs 2T 16-byte
// shared-memory loads (four wavefronts each) for 4 T^2 multiply-adds per thread: at T = 4 the loads
// take twice the time of the arithmetic, at 8 the two are even.
// Measured (us, with the zero-fill; before: 4 x 4 tiles with rows transposed on the way to shared
// memory, an fp64 atomic per entry from each of up to 608 CTAs):
//   33 x 57600 24.6 -> 14.5, 13 x 24960 13.0 -> 10.3, 64 x 57600 48.3 -> 27.5,
//   21 x 18.4 M 736 -> 569 (2.7 TB/s), 33 x 11.1 M 1163 -> 712, 64 x 4 M 849 -> 652
// The error against 64 bits is 0.1 to 0.8 of what it was.  Clusters of eight left SMs without work
// for half of the time (they do not fill the chip's processing clusters evenly, and the rest ran
// as a second wave): 1040 us on 21 x 18.4 M.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "rf_host.h"
#include "rf_ptx.cuh"

namespace cg = cooperative_groups;

namespace rf {
namespace {

constexpr int kGramMaxF = 64;   // frames per call
constexpr int kGramK = 128;     // elements per stage
// floats per staged row: rows of neighbouring threads, and their neighbouring quads, in other banks
constexpr int kGramRow = kGramK + 12;
// two stages above 40 frames, where three would leave one CTA per SM
__host__ __device__ constexpr int gram_stages(int groups) { return groups > 5 ? 2 : 3; }
constexpr int kGramThreads = 256;     // at most
constexpr int kGramCluster = 2;
constexpr int kGramT = 8;             // frames per side of a thread's tile
// elements per CTA, at least (but for the last ones): fewer CTAs bring fewer sums to add up
// (33 x 57600: 192, 384, 768 elements take 18.6, 14.5, 17.1 us)
constexpr int kGramMinWork = 384;
constexpr int kGramMaxSmem = 112 * 1024;  // two CTAs per SM

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// a + b as an unevaluated sum (Knuth's two-sum): hi + lo is exact.
__device__ __forceinline__ void two_sum(float a, float b, float& hi, float& lo) {
  hi = a + b;
  const float t = hi - a;
  lo = (a - (hi - t)) + (b - t);
}

// Tile (i, j) of index t among those on and above the diagonal, row by row.
__device__ __forceinline__ void tile_of(int t, int groups, int& i, int& j) {
  i = 0;
  while (t >= groups - i) t -= groups - i++;
  j = t + i;
}

// VEC: rows start on 16-byte boundaries (base and row stride), so 16-byte copies can be used.
template <bool VEC, int STAGES>
__global__ void __launch_bounds__(kGramThreads, 2)
    gram_kernel(const float* __restrict__ P, int F, int64_t E, int64_t ld, int width, int groups,
                int tiles, int kgroups, int red_offset, double* __restrict__ out) {
  constexpr int T = kGramT;
  extern __shared__ __align__(16) float smem[];
  const int rows = T * groups;
  float* stage0 = smem;  // [STAGES][rows][kGramRow]
  const int stage_floats = rows * kGramRow;
  const int entries = tiles * T * T;
  float* part = smem;  // [kgroups][entries], reuses the stages
  float2* red = reinterpret_cast<float2*>(smem) + red_offset;  // [entries] sums, past both
  const int tid = threadIdx.x;
  // stage st of this CTA: elements [k0, k0 + width) with k0 = (blockIdx.x + st * gridDim.x) * width
  const int64_t slices = (E + width - 1) / width;
  const int nstages = static_cast<int>((slices - blockIdx.x + gridDim.x - 1) / gridDim.x);
  auto first = [&](int st) {
    return (blockIdx.x + static_cast<int64_t>(st) * gridDim.x) * width;
  };

  // this thread's tile and k-group; the last threads may have none
  const int g = tid / tiles;
  int i, j;
  tile_of(tid - g * tiles, groups, i, j);
  const bool works = g < kgroups;

  // rows past F stay zero
  for (int s = 0; s < STAGES; ++s)
    for (int v = F * kGramRow + tid; v < stage_floats; v += blockDim.x)
      stage0[s * stage_floats + v] = 0.f;

  auto load = [&](int st) {
    if (st < nstages) {
      const int64_t k0 = first(st);
      const int left = static_cast<int>(min(static_cast<int64_t>(width), E - k0));
      const uint32_t dst = smem_u32(stage0 + (st % STAGES) * stage_floats);
      if constexpr (VEC) {
        for (int v = tid; v < F * (kGramK / 4); v += blockDim.x) {
          const int r = v / (kGramK / 4), c = (v % (kGramK / 4)) * 4;
          const int bytes = max(0, min(4, left - c)) * 4;  // the rest is zero-filled
          cp_async16(dst + (r * kGramRow + c) * 4, P + r * ld + k0 + (bytes ? c : 0), bytes);
        }
      } else {
        for (int v = tid; v < F * kGramK; v += blockDim.x) {
          const int r = v / kGramK, c = v % kGramK;
          cp_async4(dst + (r * kGramRow + c) * 4, P + r * ld + k0 + (c < left ? c : 0),
                    c < left ? 4 : 0);
        }
      }
    }
    cp_async_commit();  // a group per stage, empty past the end
  };

  float acc[T][T] = {};
  for (int st = 0; st < STAGES - 1; ++st) load(st);
  for (int st = 0; st < nstages; ++st) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();  // stage st has landed; stage st - 1 has been consumed
    load(st + STAGES - 1);
    if (works) {
      const float* ta = stage0 + (st % STAGES) * stage_floats + i * kGramRow;
      const float* tb = ta + (j - i) * kGramRow;
      const int left = static_cast<int>(min(static_cast<int64_t>(width), E - first(st)));
      const int quads = (left + 3) / 4;
      for (int q = g; q < quads; q += kgroups) {
        float4 av[T];
#pragma unroll
        for (int a = 0; a < T; ++a)
          av[a] = *reinterpret_cast<const float4*>(ta + a * groups * kGramRow + 4 * q);
#pragma unroll
        for (int b = 0; b < T; ++b) {
          const float4 bv = *reinterpret_cast<const float4*>(tb + b * groups * kGramRow + 4 * q);
#pragma unroll
          for (int a = 0; a < T; ++a) {
            acc[a][b] = fmaf(av[a].x, bv.x, acc[a][b]);
            acc[a][b] = fmaf(av[a].y, bv.y, acc[a][b]);
            acc[a][b] = fmaf(av[a].z, bv.z, acc[a][b]);
            acc[a][b] = fmaf(av[a].w, bv.w, acc[a][b]);
          }
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();  // the stages are free
  if (works) {
    float4* dst = reinterpret_cast<float4*>(part + g * entries + (tid - g * tiles) * T * T);
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
      for (int b = 0; b < T; b += 4)
        dst[(a * T + b) / 4] = make_float4(acc[a][b], acc[a][b + 1], acc[a][b + 2], acc[a][b + 3]);
  }
  __syncthreads();
  for (int e = tid; e < entries; e += blockDim.x) {
    float hi = part[e], lo = 0.f;
    for (int q = 1; q < kgroups; ++q) {
      float err;
      two_sum(hi, part[q * entries + e], hi, err);
      lo += err;
    }
    red[e] = make_float2(hi, lo);
  }
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();  // every CTA's sums are in its shared memory
  const int rank = static_cast<int>(cluster.block_rank());
  for (int e = rank + kGramCluster * tid; e < entries; e += kGramCluster * blockDim.x) {
    float2 v[kGramCluster];
#pragma unroll
    for (int c = 0; c < kGramCluster; ++c) v[c] = *cluster.map_shared_rank(red + e, c);
    float hi = v[0].x, lo = v[0].y;
#pragma unroll
    for (int c = 1; c < kGramCluster; ++c) {
      float err;
      two_sum(hi, v[c].x, hi, err);
      lo += err + v[c].y;
    }
    int ti, tj;
    tile_of(e / (T * T), groups, ti, tj);
    const int a = (e / T) % T, b = e % T;
    const int fi = ti + a * groups, fj = tj + b * groups;
    if (fi < F && fj < F && (ti != tj || a <= b)) {
      double t = static_cast<double>(hi) + static_cast<double>(lo);
      if (!isfinite(t)) {
        // a pair of floats has the range of one: add the k-groups' sums again in 64 bits, which
        // leaves infinite and undefined only what is infinite or undefined in one k-group
        t = 0.0;
        for (int c = 0; c < kGramCluster; ++c) {
          const float* sums = cluster.map_shared_rank(part + e, c);
          for (int q = 0; q < kgroups; ++q) t += static_cast<double>(sums[q * entries]);
        }
      }
      atomicAdd(out + static_cast<int64_t>(fi) * F + fj, t);
      if (fi != fj) atomicAdd(out + static_cast<int64_t>(fj) * F + fi, t);
    }
  }
  cluster.sync();  // no CTA leaves while another reads its shared memory
}

// A grid of plain CTAs, each 128 elements of every frame (or a few such slices), TILE
// frames (>= F, padded with zeros).  Thread tiles are 4 x 4; (TILE/4)^2 threads form a
// k-group, and the 256/((TILE/4)^2) k-groups of a CTA take interleaved elements of each stage,
// so small F does not pay for a 64 x 64 product.  The Gram matrix is symmetric: thread tiles
// below the diagonal are skipped and the upper ones written to both halves.  The next stage's
// global loads are issued before the current stage is multiplied (register double buffer).
template <int TILE>
__global__ void __launch_bounds__(kGramThreads)
    gram_short_kernel(const float* __restrict__ P, int F, int64_t E, int64_t ld, double* __restrict__ G) {
  constexpr int TG = (TILE / 4) * (TILE / 4);  // threads per k-group
  static_assert(TILE % 8 == 0 && TG <= kGramThreads && kGramK % 16 == 0, "tile");
  constexpr int KG = kGramThreads / TG;          // k-groups per CTA (leftover threads only load)
  constexpr int kStageV = TILE * kGramK / 4;     // float4 per stage
  constexpr int NV = (kStageV + kGramThreads - 1) / kGramThreads;  // per thread
  __shared__ __align__(16) float tile[kGramK][TILE + 4];
  __shared__ float red[KG > 1 ? KG : 1][TG][16];
  const int g = threadIdx.x / TG, r = threadIdx.x % TG;
  const int ty = r / (TILE / 4), tx = r % (TILE / 4);
  const bool upper = g < KG && ty <= tx;
  float acc[4][4] = {};
  const bool vec_ok = (ld % 4 == 0) && ((reinterpret_cast<uintptr_t>(P) & 15) == 0);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kGramK;
  float4 pre[NV];
  // float4 v of a stage -> (frame lf, element lk): a warp's 32 consecutive v cover 8 frames x 16
  // elements (64 contiguous bytes per frame), so the transposed stores below spread over 16
  // banks (2-way) where 32 rows of one frame column would fall into 2 banks (16-way)
  auto frame_of = [](int v) { return ((v >> 5) % (TILE / 8)) * 8 + ((v & 31) >> 2); };
  auto elem_of = [](int v) { return ((v >> 5) / (TILE / 8)) * 16 + (v & 3) * 4; };
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const int v = threadIdx.x + q * kGramThreads;
      const int idx = v * 4;
      const int lf = frame_of(v), lk = elem_of(v);
      const float* prow = P + static_cast<int64_t>(lf) * ld + k0 + lk;
      if (idx >= kStageV * 4) {
        pre[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else if (lf < F && vec_ok && k0 + lk + 4 <= E) {
        pre[q] = __ldcs(reinterpret_cast<const float4*>(prow));
      } else {
        float t[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) t[e] = (lf < F && k0 + lk + e < E) ? prow[e] : 0.f;
        pre[q] = make_float4(t[0], t[1], t[2], t[3]);
      }
    }
  };
  int64_t k0 = static_cast<int64_t>(blockIdx.x) * kGramK;
  if (k0 < E) load(k0);
  for (; k0 < E; k0 += stride) {
    __syncthreads();  // the previous stage has been consumed
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const int v = threadIdx.x + q * kGramThreads;
      if (v * 4 >= kStageV * 4) break;
      const int lf = frame_of(v), lk = elem_of(v);
      tile[lk][lf] = pre[q].x;
      tile[lk + 1][lf] = pre[q].y;
      tile[lk + 2][lf] = pre[q].z;
      tile[lk + 3][lf] = pre[q].w;
    }
    __syncthreads();
    if (k0 + stride < E) load(k0 + stride);  // in flight while this stage is multiplied
    if (upper) {
#pragma unroll 4
      for (int k = g; k < kGramK; k += KG) {
        const float4 a = *reinterpret_cast<const float4*>(&tile[k][ty * 4]);
        const float4 b = *reinterpret_cast<const float4*>(&tile[k][tx * 4]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) acc[i][jj] = fmaf(av[i], bv[jj], acc[i][jj]);
      }
    }
  }
  if (KG > 1) {  // sum the k-groups' partial tiles
    if (g < KG) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) red[g][r][i * 4 + jj] = acc[i][jj];
    }
    __syncthreads();
    if (g != 0) return;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        float t = 0.f;
        for (int q = 0; q < KG; ++q) t += red[q][r][i * 4 + jj];
        acc[i][jj] = t;
      }
  }
  if (!upper) return;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int fi = ty * 4 + i, fj = tx * 4 + jj;
      if (fi < F && fj < F && acc[i][jj] != 0.f && (ty < tx || fi <= fj)) {
        atomicAdd(G + static_cast<int64_t>(fi) * F + fj, static_cast<double>(acc[i][jj]));
        if (fi != fj)
          atomicAdd(G + static_cast<int64_t>(fj) * F + fi, static_cast<double>(acc[i][jj]));
      }
    }
}

// Whether gram_short_kernel is the faster of the two.  On short proxies gram_kernel's clusters, its
// wider tiles' fewer threads and its sums cost more than one atomic per entry and CTA.
// gram_short_kernel's time grows with its CTAs, one per 128 elements (33 frames: about 5.6 us and
// 0.36 us per 1000 elements); gram_kernel's hardly does until its CTAs have more than their 384
// elements, and its level rises with the frames.  The lines lie where the two meet.  Short / long,
// in us: 1 x 24000 7.3 / 8.4, 46000 8.4 / 8.3; 13 x 10001 8.4 / 10.4, 24960 14.4 / 10.4; 33 x 12000
// 9.9 / 12.5, 24000 14.2 / 13.0, 27001 14.7 / 14.4, 57600 26.0 / 15.2; 56 x 20000 16.3 / 16.7, 30000
// 18.2 / 17.1; 64 x 2475 10.0 / 27.5, 30000 18.9 / 23.5, 42000 28.4 / 24.3.
// Long proxies whose rows are not 16-byte aligned go through 4-byte copies in gram_kernel, which
// bound it where there is little arithmetic per element (9 to 24 frames) or few threads to issue
// them (above 56): 16 x 1000001 49 / 44, 4000001 115 / 134; 21 x 2097153 110 / 113, 20 x 8000001 358 / 374;
// 57 x 67483 37.8 / 39.0, 64 x 400001 118 / 105, 1000001 235 / 244.
bool short_is_faster(int F, int64_t E, bool vec) {
  int64_t long_from = F > 48 ? 24576 : 20480;
  if (!vec && F > 16) long_from = F > 48 ? 32768 : 30720;
  if (F > 56) long_from = vec ? 36864 : 73728;  // 36 tiles: 144 threads, two stages
  if (F <= 2) long_from = 40960;
  if (E < long_from) return true;
  if (vec || F <= 8) return false;
  if (F <= 16) return E >= 1572864;
  if (F <= 24) return E >= 2097152;
  return F > 56 && E >= 786432;
}

}  // namespace
}  // namespace rf

using namespace rf;

extern "C" rf_status rf_frame_gram(const float* d_P, int F, int64_t E, int64_t ld, double* d_G,
                                   rf_stream_t stream) {
  if (!d_P || !d_G) return RF_ERR_INVALID_ARG;
  if (F < 1 || F > kGramMaxF || E < 1 || ld < E) return RF_ERR_INVALID_ARG;
  DeviceInfo di;
  if (rf_status st = current_device_info(&di)) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaError_t e = cudaMemsetAsync(d_G, 0, sizeof(double) * F * F, s))
    return fail(RF_ERR_CUDA, "cudaMemsetAsync(gram)", e);
  const bool vec = ld % 4 == 0 && aligned16(d_P);
  if (short_is_faster(F, E, vec)) {
    int64_t blocks = (E + kGramK - 1) / kGramK;
    if (blocks > 4LL * di.sm_count) blocks = 4LL * di.sm_count;
    const int b = static_cast<int>(blocks);
    if (F <= 16)
      gram_short_kernel<16><<<b, kGramThreads, 0, s>>>(d_P, F, E, ld, d_G);
    else if (F <= 24)
      gram_short_kernel<24><<<b, kGramThreads, 0, s>>>(d_P, F, E, ld, d_G);
    else if (F <= 40)
      gram_short_kernel<40><<<b, kGramThreads, 0, s>>>(d_P, F, E, ld, d_G);
    else if (F <= 48)
      gram_short_kernel<48><<<b, kGramThreads, 0, s>>>(d_P, F, E, ld, d_G);
    else
      gram_short_kernel<64><<<b, kGramThreads, 0, s>>>(d_P, F, E, ld, d_G);
    return launch_status("gram_short_kernel launch");
  }
  const int groups = (F + kGramT - 1) / kGramT, tiles = groups * (groups + 1) / 2;
  int kgroups = 1;
  while (kgroups < kGramK / 4 && 2 * kgroups * tiles <= kGramThreads) kgroups *= 2;
  const int threads = std::max(128, (kgroups * tiles + 31) / 32 * 32);
  const int64_t entries = static_cast<int64_t>(tiles) * kGramT * kGramT;
  const int64_t stage_bytes = static_cast<int64_t>(gram_stages(groups)) * kGramT * groups * kGramRow * 4;
  const int64_t red_offset = std::max(stage_bytes, kgroups * entries * 4) / 8;
  const int smem = static_cast<int>(8 * red_offset + entries * 8);
  if (smem > kGramMaxSmem || kGramMaxSmem > di.max_smem_optin)
    return fail(RF_ERR_UNSUPPORTED, "rf_frame_gram: shared memory");
  // two to four CTAs per SM, in whole clusters; fewer when their slices would get short.  All CTAs
  // walk the proxies together (slice by slice of 128 elements), so that at any time they read the
  // same few pages of each frame; up to one slice per CTA, the slices are cut to equal widths.
  const int per_sm = F <= 16 ? 4 : 2;
  int64_t ctas = std::min<int64_t>((E + kGramMinWork - 1) / kGramMinWork,
                                   static_cast<int64_t>(per_sm) * di.sm_count);
  ctas = (ctas + kGramCluster - 1) / kGramCluster * kGramCluster;
  const int width = static_cast<int>(
      std::min<int64_t>(kGramK, ((E + ctas - 1) / ctas + 3) / 4 * 4));  // starts stay 16-byte aligned
  const bool three = gram_stages(groups) == 3;
  auto kernel = vec ? (three ? gram_kernel<true, 3> : gram_kernel<true, 2>)
                    : (three ? gram_kernel<false, 3> : gram_kernel<false, 2>);
  static bool attr_set[2][2][64] = {};  // per device: the largest size a call can need
  if (di.device < 0 || di.device >= 64 || !attr_set[vec][three][di.device]) {
    if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kGramMaxSmem))
      return fail(RF_ERR_CUDA, "cudaFuncSetAttribute(gram_kernel)", e);
    if (di.device >= 0 && di.device < 64) attr_set[vec][three][di.device] = true;
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kGramCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = static_cast<size_t>(smem);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, d_P, F, E, ld, width, groups, tiles, kgroups,
                                         static_cast<int>(red_offset), d_G))
    return fail(RF_ERR_CUDA, "gram_kernel launch", e);
  return RF_OK;
}
