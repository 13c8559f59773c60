// The segmented Hierarchy-Scan (Eq. 1) with rigid transforms kept as
// (quaternion, translation) pairs -- 32 bytes per joint instead of a 48-byte
// 3x4 matrix -- while it runs in shared memory (scan_core.cuh):
//   MODE 0  the plain fused frame (Simulation -> Hierarchy-Scan -> Bind
//           MeshPose, Sec. 1 steps 1-3): local poses sampled from the clips;
//   MODE 1  the forward from given local poses q [total][4] (normalized
//           here), t [total][3], skin and / or model matrices out;
//   MODE 2  the frame with layered blending (up to 4 clips by per-character
//           weights and an additive layer, sample_layers);
//   MODE 3  the plain frame followed by linear blend skinning: the bind pass
//           leaves the skin matrices' rows in shared memory (a third plane
//           beside q and t) for the skinning pass, and writes them to global
//           memory only if the caller wants them.
// The smaller item footprint lets more characters be in flight per SM, which
// is what bounds the latency-limited scan passes.  The segment tables are
// staged by cp.async during pass 1a; one character of a pure chain longer
// than 1,024 joints takes a two-level chain scan (chain_scan_qt) instead of
// the segment walks and pointer jumping.  The bind pass normalizes
// the composed quaternion once (removing the norm drift of long products),
// forms M = [R(q) | t] and writes M and / or S = M B straight to global
// memory.  Item pipeline of scan_core.cuh: producer warp, 8 compute warps,
// work queue.
#include <cuda_runtime.h>

#include "anim_internal.h"
#include "dev_math.cuh"
#include "scan_core.cuh"
#include "smem_limit.h"

namespace anim {

namespace {

__device__ __forceinline__ QT shfl_up_qt(const QT &a, int o) {
  QT r;
  r.q.x = __shfl_up_sync(0xffffffffu, a.q.x, o);
  r.q.y = __shfl_up_sync(0xffffffffu, a.q.y, o);
  r.q.z = __shfl_up_sync(0xffffffffu, a.q.z, o);
  r.q.w = __shfl_up_sync(0xffffffffu, a.q.w, o);
  r.t.x = __shfl_up_sync(0xffffffffu, a.t.x, o);
  r.t.y = __shfl_up_sync(0xffffffffu, a.t.y, o);
  r.t.z = __shfl_up_sync(0xffffffffu, a.t.z, o);
  r.t.w = 0.f;
  return r;
}

// A pure chain, one character per item: joint j's model pose is the product
// L_0 ... L_j (Eq. 1 along the one path).  Each compute thread composes its
// run of J consecutive joints in place (J = ceil(n / 256) rounded up to
// odd); a warp-shuffle scan over the runs' products and a scan of the 8 warp
// totals give each run the product of everything before it, which the run
// then applies in place.  Two barriers instead of the segment walks and
// pointer-jumping rounds, so a 2,048-deep chain is never walked more than J
// levels by one thread.
__device__ __forceinline__ void chain_scan_qt(int n, float4 *P, QT *wtot, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  // an odd run length: the lanes' slots (J float4 apart) fall in distinct banks
  const int J = ((n + kComputeThreads - 1) / kComputeThreads) | 1;
  const int j0 = min(n, tid * J), j1 = min(n, j0 + J);
  QT acc = qt_identity();
  for (int j = j0; j < j1; ++j) {
    const QT L = lds_qt(P, j, n);
    acc = j == j0 ? L : qt_mul(acc, L);
    if (j > j0) sts_qt(P, j, n, acc);
  }
  QT x = acc;  // inclusive scan of the run products over the warp's lanes
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const QT y = shfl_up_qt(x, o);
    if (lane >= o) x = qt_mul(y, x);
  }
  QT ex = shfl_up_qt(x, 1);
  if (lane == 0) ex = qt_identity();
  if (lane == 31) wtot[warp] = x;
  compute_sync();
  QT wp = qt_identity();
  for (int w = 0; w < warp; ++w) wp = w == 0 ? wtot[0] : qt_mul(wp, wtot[w]);
  if (tid > 0) {
    const QT E = warp == 0 ? ex : lane == 0 ? wp : qt_mul(wp, ex);
    for (int j = j0; j < j1; ++j) sts_qt(P, j, n, qt_mul(E, lds_qt(P, j, n)));
  }
  compute_sync();
}

// Linear blend skinning of the item's characters: vertex v of character c
// goes to sum_k w_k S_{b_k} [p; 1] with normal normalize(sum_k w_k R_{b_k} n)
// (rigid skin matrices), written as 6 floats at the character's vertex
// offset.  S is kept in three planes of n rows, character c's from P + c * cs.
// A thread loads a vertex's record once for the item's characters.  ZEROS:
// only the vertices whose first weight is zero, testing their slots; the
// records of all others have no zero weight (pack_influences).
// Bound by shared-memory bandwidth: a warp reads 4 bones x 3 rows, 48 wave
// fronts per 32 vertices, 29 of the about 48 us this pass takes of the 104 us
// frame (4,097 characters, 1,500 vertices each, 147 MB out; 125 us with the
// scan on 3x4 matrices, 55 without this pass).  Storing through a staging
// buffer as consecutive words took 3 us more than these 24-byte rows, the
// streaming hint 1.5 us less.
template <bool ZEROS>
__device__ __forceinline__ void skin_mesh(const ItemBuf &b, const float4 *P, int cs, float *verts, int tid) {
  const int nv = b.T.n_verts, n = b.T.n, C = b.C;
  const float4 *mesh = b.T.mesh;
  for (int v = tid; v < nv; v += kComputeThreads) {
    const float4 r0 = __ldg(mesh + v), r1 = __ldg(mesh + nv + v), r2 = __ldg(mesh + 2 * nv + v);
    const float w[4] = {r1.z, r1.w, r2.x, r2.y};
    const uint32_t b01 = __float_as_uint(r2.z), b23 = __float_as_uint(r2.w);
    if (ZEROS && w[0] != 0.f) continue;
    for (int c = 0; c < C; ++c) {
      const float4 *Sc = P + c * cs;
      float px = 0.f, py = 0.f, pz = 0.f, nx = 0.f, ny = 0.f, nz = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (ZEROS && w[k] == 0.f) continue;
        const uint32_t bb = k < 2 ? b01 : b23;
        const float4 *S = Sc + (k & 1 ? bb >> 16 : bb & 0xFFFFu);
        const float4 s0 = S[0], s1 = S[n], s2 = S[2 * n];
        px = fmaf(w[k], fmaf(s0.x, r0.x, fmaf(s0.y, r0.y, fmaf(s0.z, r0.z, s0.w))), px);
        py = fmaf(w[k], fmaf(s1.x, r0.x, fmaf(s1.y, r0.y, fmaf(s1.z, r0.z, s1.w))), py);
        pz = fmaf(w[k], fmaf(s2.x, r0.x, fmaf(s2.y, r0.y, fmaf(s2.z, r0.z, s2.w))), pz);
        nx = fmaf(w[k], fmaf(s0.x, r0.w, fmaf(s0.y, r1.x, s0.z * r1.y)), nx);
        ny = fmaf(w[k], fmaf(s1.x, r0.w, fmaf(s1.y, r1.x, s1.z * r1.y)), ny);
        nz = fmaf(w[k], fmaf(s2.x, r0.w, fmaf(s2.y, r1.x, s2.z * r1.y)), nz);
      }
      const float l2 = nx * nx + ny * ny + nz * nz;
      const float inv = l2 > 0.f ? rsqrtf(l2) : 0.f;
      float2 *out = reinterpret_cast<float2 *>(verts + b.voff[c] * 6) + 3 * (size_t)v;
      __stcs(out + 0, make_float2(px, py));
      __stcs(out + 1, make_float2(pz, nx * inv));
      __stcs(out + 2, make_float2(ny * inv, nz * inv));
    }
  }
}

template <int MODE, int MINB>
__global__ void __launch_bounds__(kCtaThreads, MINB) k_scan_qt(const ScanArgs a) {
  extern __shared__ __align__(128) float4 sm[];
  __shared__ ItemBuf bufs[2];
  __shared__ QT wtot[kComputeWarps];  // chain scan: the warps' run products
  constexpr int kPlanes = MODE == 3 ? 3 : 2;
  const int tid = threadIdx.x;
  // launched with programmatic stream serialization (after the work-queue
  // kernel, for the frame): wait for the preceding grid to complete before
  // reading anything it may have written.  The next launch may start now
  // (the next frame's work-queue kernel reads only plan tables before its
  // own wait) -- in the plain frame only once this grid's wait is over, as
  // the chain-walk kernel launched after it may then read the work queue
  // without a wait of its own (WalkArgs::pred_waited).
  // The forward from local poses (fixed work items) prefetches its first
  // wave's rows of q and t into L2 before the wait, and each next item's
  // while the current one runs.
  if (MODE != 0) asm volatile("griddepcontrol.launch_dependents;");
  const RowPrefetch pf = MODE == 1 ? RowPrefetch{{a.q, a.t, nullptr, nullptr}, {4, 3, 0, 0}, 0} : RowPrefetch{};
  if (MODE == 1 && tid >= kComputeThreads)
    prefetch_first_wave(bufs[1], a.n_items, a.items, a.types, a.item_chars, a.row_off, pf);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (MODE == 0) asm volatile("griddepcontrol.launch_dependents;");
  const int n_items = a.n_items;

  if (tid >= kComputeThreads) {
    producer_loop<MODE == 1 ? 1 : 0>(bufs, a.queue_head, n_items, a.items, a.types, a.item_chars, a.row_off,
                                     a.time, a.blend_w, a.status, MODE == 3 ? a.vert_off : nullptr,
                                     MODE == 2 ? LayerIn{a.layer_w, a.add_w} : LayerIn{nullptr, nullptr}, pf);
    return;
  }

  int cur = 0;
  handoff_sync();
  for (;;) {
    const ItemBuf &b = bufs[cur];
    if (b.item < 0) break;
    const int C = b.C, n = b.T.n, nseg = b.T.nseg;
    const int cs2 = 2 * n + 1;  // float4 stride between characters (16 B skew) of pairs
    const int cs = MODE == 3 ? cs2 + n : cs2;  // with the third plane
    const ItemLayout Lt = item_layout_qt(sm, C, n, nseg, kPlanes);
    float4 *P = Lt.P;

    // ---- pass 1a: local poses (q, t) from the clips or the caller's rows;
    // tables staged alongside
    if (MINB == 2) pass2_touch(b, tid);
    stage_tables(b, Lt, tid);
    if (MODE == 1) {
      // character-major: consecutive lanes read consecutive rows
      const float4 *q4 = reinterpret_cast<const float4 *>(a.q);
      const int32_t *gat = b.T.gather;
      const int CN = C * n;
#pragma unroll 2
      for (int idx = tid; idx < CN; idx += kComputeThreads) {
        const int c = (int)b.divN.div(idx), j = idx - c * n;
        const long long row = b.off[c] + (gat ? __ldg(gat + j) : j);
        const float4 q = normalize4(__ldg(q4 + row));
        const float *tp = a.t + 3 * row;
        sts_qt(P + c * cs, j, n, QT{q, make_float4(__ldg(tp), __ldg(tp + 1), __ldg(tp + 2), 0.f)});
      }
    } else if (MODE == 2) {
      const int W = n * b.cgroups, cpt = b.cpt;
      for (int idx = tid; idx < W; idx += kComputeThreads) {
        const int grp = (int)b.divN.div(idx), j = idx - grp * n;
        sample_layers<MINB == 2>(b, j, grp * cpt, min(C, (grp + 1) * cpt), P, cs);
      }
    } else {
      const int nk = b.T.n_keys, k0 = b.k0, k1 = (k0 + 1 == nk) ? 0 : k0 + 1;
      const float4 *KA0 = b.T.keys + (size_t)k0 * n * 2;
      const float4 *KA1 = b.T.keys + (size_t)k1 * n * 2;
      const float4 *KB0 = b.T.keys + (size_t)(nk + k0) * n * 2;
      const float4 *KB1 = b.T.keys + (size_t)(nk + k1) * n * 2;
      const bool two = b.T.n_clips >= 2;
      // joint-major: a thread loads joint j's key records once and samples
      // them for its group of characters (the pass-3 grouping)
      const int W = n * b.cgroups, cpt = b.cpt;
      for (int idx = tid; idx < W; idx += kComputeThreads) {
        const int grp = (int)b.divN.div(idx), j = idx - grp * n;
        const Key a0 = ldg_key(KA0 + 2 * j), a1 = ldg_key(KA1 + 2 * j);
        Key b0 = a0, b1 = a1;
        if (two) {
          b0 = ldg_key(KB0 + 2 * j);
          b1 = ldg_key(KB1 + 2 * j);
        }
        const int c1 = min(C, (grp + 1) * cpt);
        for (int c = grp * cpt; c < c1; ++c) {
          const float al = b.alpha[c];
          float4 q = slerp_pre(a0.q, a1.q, a0.t.w, al);
          float tx = fmaf(al, a1.t.x - a0.t.x, a0.t.x), ty = fmaf(al, a1.t.y - a0.t.y, a0.t.y),
                tz = fmaf(al, a1.t.z - a0.t.z, a0.t.z);
          if (two) {
            const float4 qb = slerp_pre(b0.q, b1.q, b0.t.w, al);
            const float w = b.blend[c];
            q = slerp_unit(q, qb, w);
            tx = fmaf(w, fmaf(al, b1.t.x - b0.t.x, b0.t.x) - tx, tx);
            ty = fmaf(w, fmaf(al, b1.t.y - b0.t.y, b0.t.y) - ty, ty);
            tz = fmaf(w, fmaf(al, b1.t.z - b0.t.z, b0.t.z) - tz, tz);
          }
          sts_qt(P + c * cs, j, n, QT{q, make_float4(tx, ty, tz, 0.f)});
        }
      }
    }
    cp_async_wait_all();  // this thread's table copies (stage_tables)
    compute_sync();

    // ---- pass 1b: running products along segments; pass 2: pointer jumping
    // over segments -- or, for one character of a pure chain of more than
    // 1,024 joints, the chain scan (same-box A/B: config 3's 2,048-joint
    // chains 54.2 -> 43.8 us per frame; the forward on config 2, whose
    // 1,024-joint dragon it would also take, 50.6 -> 51.3 us)
    const bool chain = b.T.chain && C == 1 && n > 1024;
    if (chain) {
      chain_scan_qt(n, P, wtot, tid);
    } else {
      const Entry<uint2> first = pass2_first(b, tid);
      pass1b_qt(b, Lt, P, cs, tid);
      compute_sync();
      pass2_qt(b, Lt, P, cs, tid, first);
    }

    // ---- pass 3: model pose, normalize, matrix, (bind,) store
    {
      const int W = n * b.cgroups, cpt = b.cpt;
      float4 *skin4 = reinterpret_cast<float4 *>(a.skin);
      float4 *model4 = reinterpret_cast<float4 *>(a.model);
      const bool skin = MODE != 1 || skin4 != nullptr, model = MODE == 1 && model4 != nullptr;
      for (int idx = tid; idx < W; idx += kComputeThreads) {
        const int grp = (int)b.divN.div(idx), j = idx - grp * n;
        const uint32_t info = Lt.jinfo[j];
        const int g = (int)(info & kJ16Seg);
        Aff B;
        if (skin) B = ldg_aff(b.T.inv_bind + 3 * j);
        const int c1 = min(C, (grp + 1) * cpt);
        for (int c = grp * cpt; c < c1; ++c) {
          QT m = lds_qt(P + c * cs, j, n);
          if (!chain && (info & kJ16Link))
            m = qt_mul(lds_qt(info & kJ16Odd ? Lt.Y1 : Lt.Y0, c * nseg + g, C * nseg), m);
          const Aff M = aff_from_qt(normalize4(m.q), m.t.x, m.t.y, m.t.z);
          if (model) stg_aff(model4 + (b.off[c] + j) * 3, M);
          if (MODE == 3) {  // the joint's own slots: nobody else reads them in this pass
            const Aff S = aff_mul(M, B);
            float4 *Pj = P + c * cs + j;
            Pj[0] = S.r0;
            Pj[n] = S.r1;
            Pj[2 * n] = S.r2;
            if (skin4) stg_aff(skin4 + (b.off[c] + j) * 3, S);
          } else if (skin) {
            stg_aff(skin4 + (b.off[c] + j) * 3, aff_mul(M, B));
          }
        }
      }
    }
    if (MODE == 3) {
      compute_sync();
      skin_mesh<false>(b, P, cs, a.verts, tid);
      // the few meshes with such vertices: their threads write them again
      if (b.T.mesh_zeros) skin_mesh<true>(b, P, cs, a.verts, tid);
    }
    cur ^= 1;
    handoff_sync();
  }
  if (tid == 0 && a.done) last_cta_reset(a.queue_head, a.done);
}

template <int MODE, int MINB>
static cudaError_t launch_qt(const ScanArgs &a, const LaunchCfg &cfg, cudaStream_t st) {
  static SmemLimit lim;
  cudaError_t e = ensure_smem_limit((const void *)k_scan_qt<MODE, MINB>, lim, cfg.smem);
  if (e != cudaSuccess) return e;
  // programmatic stream serialization: the CTAs become resident while the
  // preceding kernel runs and wait in griddepcontrol.wait
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)cfg.ctas);
  lc.blockDim = dim3((unsigned)cfg.threads);
  lc.dynamicSmemBytes = cfg.smem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, k_scan_qt<MODE, MINB>, a);
}

}  // namespace

size_t scan_smem_bytes(int n, int nseg, int C) { return scan_item_bytes(n, nseg, C); }
size_t scan_qt_smem_bytes(int n, int nseg, int C) { return qt_item_bytes(n, nseg, C); }
size_t scan_skin_smem_bytes(int n, int nseg, int C) { return qt_item_bytes(n, nseg, C, 3); }

cudaError_t launch_scan_qt(int mode, const ScanArgs &a, const LaunchCfg &cfg, cudaStream_t st) {
  const bool m3 = cfg.min_blocks >= 3;
  if (mode == 0) return m3 ? launch_qt<0, 3>(a, cfg, st) : launch_qt<0, 2>(a, cfg, st);
  if (mode == 1) return m3 ? launch_qt<1, 3>(a, cfg, st) : launch_qt<1, 2>(a, cfg, st);
  if (mode == 2) return m3 ? launch_qt<2, 3>(a, cfg, st) : launch_qt<2, 2>(a, cfg, st);
  return m3 ? launch_qt<3, 3>(a, cfg, st) : launch_qt<3, 2>(a, cfg, st);
}

}  // namespace anim
