// Headless rasterization of the skinned crowd (the picture the paper draws
// through a graphics API, Sec. 4 and Fig. 6), as plain CUDA: no graphics
// stack, a visibility buffer of 64-bit keys in device memory.
//
// Rules (fixed so that results are reproducible): character c stands at
// world offset (col * spacing, -row * spacing, 0), col = c % cols,
// row = c / cols; an orthographic camera looking down -Z maps a world point
// to screen (ox + scale X, oy - scale Y) with depth d = (2 - Z) / 4 (smaller
// is nearer).  Screen positions are snapped to 1/256 pixel (round to
// nearest, halves away from zero); pixel (x, y) is covered when its centre
// (x + 0.5, y + 0.5) is inside the triangle by 64-bit integer edge
// functions of the snapped positions, the triangle oriented to positive
// area, with the tie rule that a centre on an edge a->b belongs to it when
// b - a points down (dy > 0) or horizontally left (dy == 0, dx < 0); zero-
// area triangles cover nothing.  Visibility: the smallest key
// (depth bits << 32 | id), id = c * 4096 + face, by atomicMin.
#include <cuda_runtime.h>

#include <algorithm>

#include "anim_internal.h"
#include "dev_math.cuh"
#include "smem_limit.h"

namespace anim {

namespace {

constexpr int kRasterThreads = 256;
constexpr int kRasterMaxFaces = 4096;  // per type (the ids' 12 bits)

// Launched with programmatic stream serialization: the triangle kernel may
// start once every CTA here has seen the preceding grid complete, so it can
// read the vertices at once and waits only before it touches vis.
__global__ void k_raster_clear(unsigned long long *vis, long long n) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    vis[i] = ~0ull;
}

// A vertex (x, y) of character c on the screen in 1/256 pixel units, before
// rounding.  The products are fused as written: ids and colours depend on
// every bit of the snapped positions.
__device__ __forceinline__ float2 to_screen(const RasterArgs &a, int c, float x, float y) {
  const float wx = fmaf((float)(c % a.cols), a.spacing, x), wy = fmaf(-(float)(c / a.cols), a.spacing, y);
  return make_float2(fmaf(a.scale, wx, a.ox) * 256.f, fmaf(-a.scale, wy, a.oy) * 256.f);
}

__device__ __forceinline__ void put_pixel(unsigned long long *at, float e0, float e1, float e2, float D0, float D1,
                                          float D2, float inv_area, unsigned int id) {
  float d = fmaf(e2, D2, fmaf(e0, D0, e1 * D1)) * inv_area;
  d = fmaxf(d, 0.f);
  atomicMin(at, ((unsigned long long)__float_as_uint(d) << 32) | id);
}

// Depth of a vertex.
__device__ __forceinline__ float depth_of(float z) { return (2.f - z) * 0.25f; }

// One triangle in 64-bit arithmetic straight from the vertices: whatever
// the 32-bit path below does not take (far off-screen or non-finite
// positions, triangles of 64 pixels and more).  The warp takes it together,
// a pixel per lane along the longer side of its box: such triangles have up
// to tens of thousands of pixels, and a lane walking one alone is what the
// launch then waits for (1920x1080, 142 pixels per unit, 30 characters of 308
// faces: 2,311 us with every triangle on a lane of its own, 2,785 with the
// small ones taken by the warp first, 969 as it is).
__device__ __noinline__ void raster_tri_wide(const RasterArgs &a, const float *vb, const int32_t *face, int c,
                                             unsigned int id, int lane) {
  long long X[3], Y[3];
  float D[3];
  for (int k = 0; k < 3; ++k) {
    const float *v = vb + 6 * (long long)__ldg(face + k);
    const float2 p = to_screen(a, c, __ldcg(v), __ldcg(v + 1));
    X[k] = llroundf(p.x);
    Y[k] = llroundf(p.y);
    D[k] = depth_of(__ldcg(v + 2));
  }
  long long area = (X[1] - X[0]) * (Y[2] - Y[0]) - (Y[1] - Y[0]) * (X[2] - X[0]);
  if (area == 0) return;
  if (area < 0) {
    long long t = X[1];
    X[1] = X[2];
    X[2] = t;
    t = Y[1];
    Y[1] = Y[2];
    Y[2] = t;
    const float td = D[1];
    D[1] = D[2];
    D[2] = td;
    area = -area;
  }
  const long long xmin = min(X[0], min(X[1], X[2])), xmax = max(X[0], max(X[1], X[2]));
  const long long ymin = min(Y[0], min(Y[1], Y[2])), ymax = max(Y[0], max(Y[1], Y[2]));
  const long long px0 = max(0ll, (xmin - 128 + 255) >> 8), px1 = min((long long)a.width - 1, (xmax - 128) >> 8);
  const long long py0 = max(0ll, (ymin - 128 + 255) >> 8), py1 = min((long long)a.height - 1, (ymax - 128) >> 8);
  if (px1 < px0 || py1 < py0) return;
  const float inv_area = 1.f / (float)area;
  const bool cols = px1 - px0 < py1 - py0;
  const int len = (int)(cols ? py1 - py0 : px1 - px0), lines = (int)(cols ? px1 - px0 : py1 - py0);
  for (int line = 0; line <= lines; ++line) {
    for (int at = lane; at <= len; at += 32) {
      const long long px = px0 + (cols ? line : at), py = py0 + (cols ? at : line);
      const long long cx = px * 256 + 128, cy = py * 256 + 128;
      long long e[3];
      bool inside = true;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int ia = (k + 1) % 3, ib = (k + 2) % 3;
        const long long dx = X[ib] - X[ia], dy = Y[ib] - Y[ia];
        e[k] = dx * (cy - Y[ia]) - dy * (cx - X[ia]);
        inside = inside && (e[k] > 0 || (e[k] == 0 && (dy > 0 || (dy == 0 && dx < 0))));
      }
      if (inside)
        put_pixel(a.vis + py * a.width + px, (float)e[0], (float)e[1], (float)e[2], D[0], D[1], D[2], inv_area, id);
    }
  }
}

// A snapped coordinate the 32-bit path cannot hold (or NaN): its triangles
// take the wide path.
constexpr int kFar = (int)0x80000000;
__device__ __forceinline__ int snap_32(float v) {
  const float s = roundf(v);  // halves away from zero, as llroundf
  return fabsf(s) < 1073741824.f ? (int)s : kFar;
}

__device__ __forceinline__ int2 snapped_corner(const RasterArgs &a, int c, const float *v) {
  const float2 s = to_screen(a, c, __ldcg(v), __ldcg(v + 1));
  return make_int2(snap_32(s.x), snap_32(s.y));
}

// The sides of the image a snapped position lies past, so that no pixel
// centre is at or beyond it: 1 left, 2 right, 4 above, 8 below.
__device__ __forceinline__ unsigned outside(const RasterArgs &a, int X, int Y) {
  if (X == kFar || Y == kFar) return 0;
  return (X < 128 ? 1u : 0u) | (((X + 127) >> 8) >= a.width ? 2u : 0u) | (Y < 128 ? 4u : 0u) |
         (((Y + 127) >> 8) >= a.height ? 8u : 0u);
}

// The bracket an edge puts on the positions p of a line where its value
// r - 256 b p can be >= 0: p <= r q + up and p >= r q + down, a hundredth
// generous on the side it bounds and without effect on the other.  An edge
// along the line (b == 0) empties it when r < 0, and bounds neither side
// otherwise.
struct Bracket {
  float q, up, down;
};
__device__ __forceinline__ Bracket bracket_of(int b) {
  Bracket k;
  k.q = b == 0 ? 1e12f : __fdividef(1.f, (float)(b * 256));
  k.up = b > 0 ? 0.01f : 1e9f;
  k.down = b < 0 ? -0.01f : -3e38f;
  return k;
}
__device__ __forceinline__ void narrow(const Bracket &k, int r, float &lo, float &hi) {
  const float x = (float)r;
  hi = fminf(hi, fmaf(x, k.q, k.up));
  lo = fmaxf(lo, fmaf(x, k.q, k.down));
}

// What a warp keeps of its 32 triangles for the pixel pass, a column each.
// A triangle is cut into lines along the longer side of its box: rows, or
// columns.  Edge k is opposite corner k; r is its value at the first line's
// first pixel centre less the tie rule's bias, a line adds 256 a, a pixel
// along it takes off 256 b.
struct WarpTris {
  int4 r[32], a[32], b[32];  // of the three edges; w: index of the first line's first pixel; face (bits 0-11),
                             // biases (12-14), lines are columns (15); 1 / area
  float4 D[32];
  unsigned px[64];           // pixels to test: triangle (5 bits), line (7), position along it (7)
};

// The warp's pixel W.px[i] of character c's triangles: the exact test, the
// depth, the visibility buffer.
__device__ __forceinline__ void test_pixel(const RasterArgs &a, const WarpTris &W, int i, unsigned cid) {
  const unsigned px = W.px[i];
  const int t = px & 31u, l = px >> 5 & 127u, p = px >> 12 & 127u;
  const int4 r = W.r[t], u = W.a[t], b = W.b[t];
  const int e0 = r.x + (l * u.x - p * b.x) * 256, e1 = r.y + (l * u.y - p * b.y) * 256,
            e2 = r.z + (l * u.z - p * b.z) * 256;
  if ((e0 | e1 | e2) < 0) return;
  const float4 D = W.D[t];
  const unsigned idb = (unsigned)u.w;
  put_pixel(a.vis + (r.w + (idb >> 15 ? p * a.width + l : l * a.width + p)), (float)(e0 + (int)(idb >> 12 & 1u)),
            (float)(e1 + (int)(idb >> 13 & 1u)), (float)(e2 + (int)(idb >> 14 & 1u)), D.x, D.y, D.z,
            __int_as_float(b.w), cid + (idb & 4095u));
}

// One CTA per character.  What bounds the kernel is the instructions per
// triangle, row and pixel, not the vertices' bytes, so
//   - a character's vertices are snapped once into shared memory (each is a
//     corner of up to three and more faces); a character wholly past one side
//     of the image ends there;
//   - edge functions are 32-bit: with both extents of a triangle below 2^14
//     (64 pixels) every |dx|, |dy| and distance to a pixel centre inside its
//     bounding box is below 2^14, so each value fits in 30 bits;
//   - a warp sets 32 triangles up, a lane walks its triangle's lines and lists
//     their covered pixels, and the warp takes the list a pixel per lane: most
//     lines of the mesh's slivers cover no pixel or one, and testing each
//     where it is found would leave most lanes idle;
//   - lines run along the longer side of the triangle's box, which halves
//     their number for slivers in every direction;
//   - a line's covered run is bracketed from the three edges by float
//     division (a hundredth of a pixel wider than exact, far above the float
//     error over at most 64 pixels) and only the pixels in the bracket are
//     tested exactly: a sliver covers about one pixel of the sixteen of its
//     box.
// The tie rule enters as a bias: a centre on an edge that does not own it
// counts as just outside.
// Measured (4,097 characters of 1,498 faces, 1920x1080, 40 % of them below
// the image, all three launches): 422 us with a triangle per lane in 64-bit
// arithmetic from global vertices, 226 with staged vertices and 32-bit
// edges, 176 with a row per lane, 109 as it is (82.3 M warp instructions at
// 76 % issue; the vertices' 147 MB take 22 us).  A 5-CTA build spills: 116
// against 112; three CTAs per SM: 122.
// ALL_STAGED: every mesh fits the stage.  Otherwise the characters of the
// larger ones snap each triangle's corners as they come to it: 1,500 of 4,500
// vertices and 4,096 faces, 64 columns, take 177 us (686 with a triangle per
// lane in 64 bits, 2,582 with these meshes left to raster_tri_wide).
template <bool ALL_STAGED>
__global__ void __launch_bounds__(kRasterThreads, 4) k_raster_tris(const __grid_constant__ RasterArgs a) {
  extern __shared__ int2 sxy[];
  __shared__ WarpTris tris[kRasterThreads / 32];
  __shared__ unsigned codes[kRasterThreads / 32];
  __shared__ unsigned wide_faces[kRasterMaxFaces / 32];  // a bit per face
  const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;");
  const TypeDev &T = a.types[a.char_type[c]];
  const int nf = T.n_faces, nv = nf > 0 ? T.n_verts : 0;
  const float *vb = a.verts + a.vert_off[c] * 6;
  float *sd = reinterpret_cast<float *>(sxy + a.stage_verts);
  const bool staged = ALL_STAGED || nv <= a.stage_verts;
  unsigned code = staged ? 15u : 0u;  // no vertices: past every side
  if (staged) {
    if ((reinterpret_cast<uintptr_t>(vb) & 7u) == 0) {
      const float2 *v2 = reinterpret_cast<const float2 *>(vb);
#pragma unroll 2
      for (int v = tid; v < nv; v += kRasterThreads) {
        const float2 p = __ldcg(v2 + 3 * v);
        const float z = __ldcg(vb + 6 * v + 2);
        const float2 s = to_screen(a, c, p.x, p.y);
        const int2 xy = make_int2(snap_32(s.x), snap_32(s.y));
        sxy[v] = xy;
        sd[v] = depth_of(z);
        code &= outside(a, xy.x, xy.y);
      }
    } else {
      for (int v = tid; v < nv; v += kRasterThreads) {
        const float2 s = to_screen(a, c, __ldcg(vb + 6 * v), __ldcg(vb + 6 * v + 1));
        const int2 xy = make_int2(snap_32(s.x), snap_32(s.y));
        sxy[v] = xy;
        sd[v] = depth_of(__ldcg(vb + 6 * v + 2));
        code &= outside(a, xy.x, xy.y);
      }
    }
  }
  code = __reduce_and_sync(0xffffffffu, code);
  if (lane == 0) codes[warp] = code;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kRasterThreads / 32; ++i) code &= codes[i];
  // the visibility buffer is cleared; waited for on every path, so that the
  // resolve, which follows this grid alone, follows the clear too
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (code) return;
  WarpTris &W = tris[warp];
  const int32_t *faces = T.faces;
  const unsigned cid = (unsigned)c * 4096u;
  unsigned any_wide = 0;
  int f = tid;
  int n0 = 0, n1 = 0, n2 = 0;  // the next face's corners, a pass ahead
  if (f < nf) {
    n0 = __ldg(faces + 3 * f);
    n1 = __ldg(faces + 3 * f + 1);
    n2 = __ldg(faces + 3 * f + 2);
  }
  for (; f - lane < nf; f += kRasterThreads) {
    int i0 = n0, i1 = n1, i2 = n2;
    if (f + kRasterThreads < nf) {
      n0 = __ldg(faces + 3 * (f + kRasterThreads));
      n1 = __ldg(faces + 3 * (f + kRasterThreads) + 1);
      n2 = __ldg(faces + 3 * (f + kRasterThreads) + 2);
    }
    bool wide = false;
    int lines = 0, X0 = 0, Y0 = 0, X1 = 0, Y1 = 0, X2 = 0, Y2 = 0, px0 = 0, pw = 0, py0 = 0, ph = 0, area = 0;
    if (f < nf) {
      const int2 p0 = staged ? sxy[i0] : snapped_corner(a, c, vb + 6 * (long long)i0),
                 p1 = staged ? sxy[i1] : snapped_corner(a, c, vb + 6 * (long long)i1),
                 p2 = staged ? sxy[i2] : snapped_corner(a, c, vb + 6 * (long long)i2);
      X0 = p0.x, Y0 = p0.y, X1 = p1.x, Y1 = p1.y, X2 = p2.x, Y2 = p2.y;
      const int xmin = min(X0, min(X1, X2)), xmax = max(X0, max(X1, X2));
      const int ymin = min(Y0, min(Y1, Y2)), ymax = max(Y0, max(Y1, Y2));
      wide = xmin == kFar || ymin == kFar;  // the smallest integer
      if (!wide) {
        px0 = max(0, (xmin + 127) >> 8);
        py0 = max(0, (ymin + 127) >> 8);
        pw = min(a.width - 1, (xmax - 128) >> 8) - px0;
        ph = min(a.height - 1, (ymax - 128) >> 8) - py0;
        if (pw >= 0 && ph >= 0) {
          wide = xmax - xmin >= 16384 || ymax - ymin >= 16384;
          if (!wide) {
            area = (X1 - X0) * (Y2 - Y0) - (Y1 - Y0) * (X2 - X0);
            lines = area != 0 ? min(pw, ph) + 1 : 0;
          }
        }
      }
    }
    const unsigned wides = __ballot_sync(0xffffffffu, wide);
    if (lane == 0) wide_faces[f >> 5] = wides;
    any_wide |= wides;
    const int most = __reduce_max_sync(0xffffffffu, lines);
    if (most == 0) continue;
    if (area < 0) {
      int t = X1;
      X1 = X2;
      X2 = t;
      t = Y1;
      Y1 = Y2;
      Y2 = t;
      t = i1;
      i1 = i2;
      i2 = t;
      area = -area;
    }
    const int dx0 = X2 - X1, dy0 = Y2 - Y1, dx1 = X0 - X2, dy1 = Y0 - Y2, dx2 = X1 - X0, dy2 = Y1 - Y0;
    const int cx = px0 * 256 + 128, cy = py0 * 256 + 128;
    const int b0 = (dy0 > 0 || (dy0 == 0 && dx0 < 0)) ? 0 : 1;
    const int b1 = (dy1 > 0 || (dy1 == 0 && dx1 < 0)) ? 0 : 1;
    const int b2 = (dy2 > 0 || (dy2 == 0 && dx2 < 0)) ? 0 : 1;
    const bool cols = pw < ph;
    int r0 = dx0 * (cy - Y1) - dy0 * (cx - X1) - b0;
    int r1 = dx1 * (cy - Y2) - dy1 * (cx - X2) - b1;
    int r2 = dx2 * (cy - Y0) - dy2 * (cx - X0) - b2;
    const int u0 = cols ? -dy0 : dx0, u1 = cols ? -dy1 : dx1, u2 = cols ? -dy2 : dx2;
    const int s0 = cols ? -dx0 : dy0, s1 = cols ? -dx1 : dy1, s2 = cols ? -dx2 : dy2;
    if (lines > 0) {
      W.r[lane] = make_int4(r0, r1, r2, py0 * a.width + px0);  // below 2^28
      W.a[lane] = make_int4(u0, u1, u2, f | (b0 | b1 << 1 | b2 << 2 | (cols ? 8 : 0)) << 12);
      W.b[lane] = make_int4(s0, s1, s2, __float_as_int(1.f / (float)area));
      W.D[lane] = staged ? make_float4(sd[i0], sd[i1], sd[i2], 0.f)
                         : make_float4(depth_of(__ldcg(vb + 6 * (long long)i0 + 2)),
                                       depth_of(__ldcg(vb + 6 * (long long)i1 + 2)),
                                       depth_of(__ldcg(vb + 6 * (long long)i2 + 2)), 0.f);
    }
    const Bracket k0 = bracket_of(s0), k1 = bracket_of(s1), k2 = bracket_of(s2);
    const float len = (float)max(pw, ph);
    int listed = 0;
    for (int line = 0; line < most; ++line) {
      float lo = 0.f, hi = len;
      narrow(k0, r0, lo, hi);
      narrow(k1, r1, lo, hi);
      narrow(k2, r2, lo, hi);
      int p = __float2int_ru(lo);
      int n = line < lines ? __float2int_rd(fmaxf(hi, -1.f)) - p + 1 : 0;
      r0 += u0 * 256;
      r1 += u1 * 256;
      r2 += u2 * 256;
      unsigned more;
      while ((more = __ballot_sync(0xffffffffu, n > 0)) != 0) {
        if (n > 0) W.px[listed + __popc(more & ((1u << lane) - 1u))] = (unsigned)(lane | line << 5 | p << 12);
        listed += __popc(more);
        ++p;
        --n;
        if (listed >= 32) {
          __syncwarp();
          listed -= 32;
          test_pixel(a, W, listed + lane, cid);
          __syncwarp();  // read before the next lines' pixels overwrite it
        }
      }
    }
    __syncwarp();
    if (lane < listed) test_pixel(a, W, lane, cid);
    __syncwarp();  // the triangles are read before the next 32
  }
  if (any_wide == 0) return;
  __syncwarp();
  for (f = tid - lane; f < nf; f += kRasterThreads)  // the warp's own faces again
    for (unsigned w = wide_faces[f >> 5]; w; w &= w - 1u) {
      const int g = f + __ffs(w) - 1;
      raster_tri_wide(a, vb, faces + 3 * g, c, cid + (unsigned)g, lane);
    }
}

__global__ void k_raster_resolve(const RasterArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long long n = (long long)a.width * a.height;
  const float lx = 0.3f, ly = 0.5f, lz = 0.8f, ln = rsqrtf(lx * lx + ly * ly + lz * lz);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const unsigned long long key = a.vis[i];
    const unsigned int id = key == ~0ull ? 0xFFFFFFFFu : (unsigned int)(key & 0xFFFFFFFFull);
    if (a.ids) a.ids[i] = id;
    if (!a.rgba) continue;
    if (id == 0xFFFFFFFFu) {
      a.rgba[i] = 0xFF201810u;  // background (A B G R bytes)
      continue;
    }
    const int c = (int)(id >> 12), f = (int)(id & 4095u);
    const TypeDev &T = a.types[a.char_type[c]];
    const float *vb = a.verts + a.vert_off[c] * 6;
    float nx = 0.f, ny = 0.f, nz = 0.f;
    for (int k = 0; k < 3; ++k) {
      const float *v = vb + 6 * (long long)__ldg(T.faces + 3 * f + k);
      nx += __ldg(v + 3);
      ny += __ldg(v + 4);
      nz += __ldg(v + 5);
    }
    const float nn = nx * nx + ny * ny + nz * nz;
    const float lam = nn > 0.f ? fabsf(nx * lx + ny * ly + nz * lz) * ln * rsqrtf(nn) : 0.f;
    const float g = 0.25f + 0.75f * lam;
    const unsigned int h = (unsigned int)c * 2654435761u;  // per-character tint
    const float r = g * (0.6f + 0.4f * ((h >> 8) & 255u) / 255.f), gg = g * (0.6f + 0.4f * ((h >> 16) & 255u) / 255.f),
                b = g * (0.6f + 0.4f * ((h >> 24) & 255u) / 255.f);
    a.rgba[i] = 0xFF000000u | ((unsigned int)(b * 255.f) << 16) | ((unsigned int)(gg * 255.f) << 8) |
                (unsigned int)(r * 255.f);
  }
}

}  // namespace

template <class... Args>
static cudaError_t launch_chained(void (*k)(Args...), unsigned grid, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3((unsigned)kRasterThreads);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, k, args...);
}

cudaError_t launch_raster(const RasterArgs &a, int n_chars, bool all_staged, cudaStream_t st) {
  const long long n = (long long)a.width * a.height;
  const unsigned blocks = (unsigned)std::max(1ll, std::min((n + 255) / 256, 4096ll));
  cudaError_t e = launch_chained(k_raster_clear, blocks, 0, st, a.vis, n);
  if (e != cudaSuccess) return e;
  if (n_chars > 0) {
    static SmemLimit lims[2];
    const auto kernel = all_staged ? k_raster_tris<true> : k_raster_tris<false>;
    const size_t smem = 12 * (size_t)a.stage_verts;
    e = ensure_smem_limit((const void *)kernel, lims[all_staged], smem);
    if (e != cudaSuccess) return e;
    e = launch_chained(kernel, (unsigned)n_chars, smem, st, a);
    if (e != cudaSuccess) return e;
  }
  return launch_chained(k_raster_resolve, blocks, 0, st, a);
}

}  // namespace anim
