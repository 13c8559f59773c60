// The per-frame work queue and the setup kernels.
#include <cuda_runtime.h>

#include "anim_internal.h"
#include "dev_math.cuh"
#include "scan_core.cuh"
#include "smem_limit.h"

#define ANIM_MAX_KEYS_DEV 1024  // keys per clip (ANIM_MAX_KEYS in the ABI)

namespace anim {

// ------------------------------------------------------------ work queue
constexpr int kBucketThreads = 256;
constexpr int kBucketPer = kRangeCharsMax / kBucketThreads;  // characters per thread
static_assert(kBucketPer * kBucketThreads == kRangeCharsMax, "range size");

__device__ __forceinline__ int key_index(float tm, float rate, int nk, int *status) {
  if (!isfinite(tm)) {
    atomicOr(status, 1);
    return 0;
  }
  const float u = __fmul_rn(tm, rate);
  const int k = (int)floorf(u);
  int m = k % nk;
  return m < 0 ? m + nk : m;
}

// Block-wide exclusive scan of one int per thread; returns the prefix and
// writes the total to *total.
__device__ int block_excl_scan(int v, int *warp_sums, int *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int w = lane < nw ? warp_sums[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) warp_sums[lane] = w;
  }
  __syncthreads();
  const int before = (wid ? warp_sums[wid - 1] : 0) + x - v;
  if (threadIdx.x == blockDim.x - 1) *total = before + v;
  __syncthreads();
  return before;
}

// One CTA per range of <= kRangeCharsMax characters of one type: counting sort
// by key index k0 in shared memory, items of <= cap characters per (k0) bin
// written to the range's slot region, and empty items (count 0) in the
// region's remaining slots.  Regions are laid out in range order (types most
// costly first); the persistent kernel's producer warp skips empty slots.
__global__ void __launch_bounds__(kBucketThreads) k_bucket(const BucketArgs a) {
  __shared__ int s_hist[ANIM_MAX_KEYS_DEV];
  __shared__ int s_start[ANIM_MAX_KEYS_DEV];
  __shared__ int s_istart[ANIM_MAX_KEYS_DEV];
  __shared__ int s_warp[32];
  __shared__ int s_total, s_itotal;
  const int tid = threadIdx.x, nth = blockDim.x;
  // a frame kernel launched after this one with programmatic stream
  // serialization may start now; it waits for this grid's completion (and
  // its memory) in griddepcontrol.wait before reading the queue
  asm volatile("griddepcontrol.launch_dependents;");
  // launched the same way after the previous frame's kernel: the plan's
  // tables are read before waiting for it, the times (which the preceding
  // kernel may have written) and every write of this grid after
  const RangeDev R = a.ranges[blockIdx.x];
  const int nk = a.types[R.type].n_keys;
  const float rate = a.types[R.type].rate;
  const int cap = a.cap[R.type];
  const int region_end = (blockIdx.x + 1 < a.n_ranges) ? a.ranges[blockIdx.x + 1].region : a.n_slots;
  for (int b = tid; b < nk; b += nth) s_hist[b] = 0;
  int cid[kBucketPer], k[kBucketPer], pos[kBucketPer];
#pragma unroll
  for (int m = 0; m < kBucketPer; ++m) {
    const int i = tid + m * nth;
    cid[m] = i < R.count ? __ldg(a.type_chars + R.start + i) : -1;
    k[m] = 0;
    pos[m] = 0;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (blockIdx.x == 0 && tid == 0) *a.queue_head = 0;  // consumed by the next launch in stream order
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kBucketPer; ++m)
    if (cid[m] >= 0) {
      k[m] = key_index(a.time[cid[m]], rate, nk, a.status);
      pos[m] = atomicAdd(&s_hist[k[m]], 1);  // rank inside the bin
    }
  __syncthreads();
  // exclusive scans over the bins: character starts and item starts (one
  // warp's shuffles when the bins fit in a warp, else block-wide)
  const int per = (nk + nth - 1) / nth;
  const int b0 = min(nk, tid * per), b1 = min(nk, b0 + per);
  if (nk <= 32) {
    if (tid < 32) {
      const int h = tid < nk ? s_hist[tid] : 0, ih = (h + cap - 1) / cap;
      int x = h, ix = ih;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o), iy = __shfl_up_sync(0xffffffffu, ix, o);
        if (tid >= o) {
          x += y;
          ix += iy;
        }
      }
      if (tid < nk) {
        s_start[tid] = x - h;
        s_istart[tid] = ix - ih;
      }
      if (tid == 31) s_itotal = ix;
    }
  } else {
    int run = 0, irun = 0;
    for (int b = b0; b < b1; ++b) {
      run += s_hist[b];
      irun += (s_hist[b] + cap - 1) / cap;
    }
    int pre = block_excl_scan(run, s_warp, &s_total);
    int ipre = block_excl_scan(irun, s_warp, &s_itotal);
    for (int b = b0; b < b1; ++b) {
      s_start[b] = pre;
      s_istart[b] = ipre;
      pre += s_hist[b];
      ipre += (s_hist[b] + cap - 1) / cap;
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kBucketPer; ++m)
    if (cid[m] >= 0) a.sorted[R.start + s_start[k[m]] + pos[m]] = cid[m];
  for (int b = b0; b < b1; ++b) {
    const int cnt = s_hist[b];
    for (int m = 0; m * cap < cnt; ++m) {
      WorkItem w;
      w.start = R.start + s_start[b] + m * cap;
      w.count = min(cap, cnt - m * cap);
      w.type = R.type;
      w.k0 = b;
      a.items[R.region + s_istart[b] + m] = w;
    }
  }
  const WorkItem empty = {0, 0, R.type, 0};
  for (int sl = R.region + s_itotal + tid; sl < region_end; sl += nth) a.items[sl] = empty;
}

cudaError_t launch_bucket(const BucketArgs &a, cudaStream_t st) {
  if (a.n_ranges == 0) return cudaSuccess;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)a.n_ranges);
  lc.blockDim = dim3((unsigned)kBucketThreads);
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, k_bucket, a);
}

// ------------------------------------------------------------ setup kernels
// Arc angle between consecutive keys (shorter arc), stored in the pad slot
// of the first key of each pair: theta = 2 atan2(|a - b'|, |a + b'|) with
// b' = +-b on a's hemisphere, carrying the sign of that choice (slerp_pre).
// Keys loop, so key n_keys-1 pairs with key 0.
__global__ void k_prepare_keys(float4 *keys, int n_clips, int n_keys, int n) {
  const long long total = (long long)n_clips * n_keys * n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(i % n);
    const long long ck = i / n;
    const int k = (int)(ck % n_keys), c = (int)(ck / n_keys);
    const int k1 = (k + 1 == n_keys) ? 0 : k + 1;
    const float4 a = keys[2 * i];
    const float4 b = keys[2 * (((long long)c * n_keys + k1) * n + j)];
    const float sg = dot4(a, b) < 0.f ? -1.f : 1.f;
    float dm = 0.f, dp = 0.f, d;
    d = a.x - sg * b.x; dm += d * d; d = a.x + sg * b.x; dp += d * d;
    d = a.y - sg * b.y; dm += d * d; d = a.y + sg * b.y; dp += d * d;
    d = a.z - sg * b.z; dm += d * d; d = a.z + sg * b.z; dp += d * d;
    d = a.w - sg * b.w; dm += d * d; d = a.w + sg * b.w; dp += d * d;
    keys[2 * i + 1].w = copysignf(2.f * atan2f(sqrtf(dm), sqrtf(dp)), sg);  // the sign: b's hemisphere
  }
}

cudaError_t launch_prepare_keys(float4 *keys, int n_clips, int n_keys, int n, cudaStream_t st) {
  const long long total = (long long)n_clips * n_keys * n;
  const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  k_prepare_keys<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(keys, n_clips, n_keys, n);
  return cudaGetLastError();
}

// Inverse bind poses from a rest pose: thread 0 composes the rest pose down
// the joint list (parent before child) into inv_bind, then every thread
// replaces its model pose [R | t] by the rigid inverse [R^T | -R^T t].
__global__ void k_bind_from_rest(const int32_t *parent, const float *rest_q, const float *rest_t, int n,
                                 float4 *out) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < n; ++i) {
      const float4 q = normalize4(make_float4(rest_q[4 * i], rest_q[4 * i + 1], rest_q[4 * i + 2], rest_q[4 * i + 3]));
      Aff L = aff_from_qt(q, rest_t[3 * i], rest_t[3 * i + 1], rest_t[3 * i + 2]);
      const int p = parent[i];
      if (p >= 0) {
        Aff M;
        M.r0 = out[3 * p];
        M.r1 = out[3 * p + 1];
        M.r2 = out[3 * p + 2];
        L = aff_mul(M, L);
      }
      out[3 * i] = L.r0;
      out[3 * i + 1] = L.r1;
      out[3 * i + 2] = L.r2;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float4 a = out[3 * i], b = out[3 * i + 1], c = out[3 * i + 2];
    // R^T rows are the columns of R
    const float tx = -(a.x * a.w + b.x * b.w + c.x * c.w);
    const float ty = -(a.y * a.w + b.y * b.w + c.y * c.w);
    const float tz = -(a.z * a.w + b.z * b.w + c.z * c.w);
    out[3 * i] = make_float4(a.x, b.x, c.x, tx);
    out[3 * i + 1] = make_float4(a.y, b.y, c.y, ty);
    out[3 * i + 2] = make_float4(a.z, b.z, c.z, tz);
  }
}

cudaError_t launch_bind_from_rest(const int32_t *parent, const float *rest_q, const float *rest_t, int n,
                                  float4 *inv_bind, cudaStream_t st) {
  k_bind_from_rest<<<1, 256, 0, st>>>(parent, rest_q, rest_t, n, inv_bind);
  return cudaGetLastError();
}

}  // namespace anim
