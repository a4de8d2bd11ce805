// Monte Carlo ray tracing of the hand (Section 3.1, "Rendering") and its derivative
// with edge sampling for the visibility discontinuities (the renderer of Li et al.
// 2018 that the paper builds on; Section 1 and Section 3.1).
//
// Primary rays of a pinhole camera are coherent, so the forward and the interior
// backward work on 8x4-pixel sub-tiles, one warp per sub-tile at a time.
//
// Candidate lists (forward).  A triangle can only be hit in its screen box (padded by
// half a pixel), so a sub-tile needs the triangle records whose boxes meet it; of its
// pixels, those that the triangle can cover (tri_pixel_mask) are kept with the record:
//   k_bin (count)  each (view, record) pair counts itself into the sub-tiles its box
//                  meets;
//   k_bin_alloc    each sub-tile gets a pool range for its K records and 1-16 work
//                  items of consecutive samples (more for longer lists, so no single
//                  warp holds up the launch);
//   k_background   sub-tiles that no record meets get the background (second stream);
//   k_bin (fill)   the pairs write their records, boxes, depths and pixel masks into
//                  the ranges;
//   k_bin_sort     each list is sorted by nearest camera depth.
// k_gather (a frustum walk of the LBVH per sub-tile) makes the backward's own lists
// when the forward's cannot be reused.
//
// Shading:
//   k_shade_fwd    warps take work items; the warp stages the item's candidates in
//                  shared memory (what their intersection needs, the camera's part
//                  already worked out), each lane (pixel) makes its samples (Philox
//                  jitter) and walks the candidates that can cover its pixel (a bit
//                  transpose of the lists' pixel masks), in depth order, with the same
//                  float32 Moller-Trumbore test and closest-hit rule as a per-ray
//                  traversal, stopping at the first candidate nearer than none of its
//                  hits; shades, and writes per-item sums.  The warp finishing a
//                  sub-tile's last item sums the items in item order (deterministic)
//                  and writes the pixels.
//   k_shade_bwd    the same samples re-traced (no hit records are kept between
//                  the passes); every hit is differentiated at the fixed ray, a lane's
//                  hits triangle by triangle in windows of 16 samples, and a triangle's
//                  sums of a window are added to memory (single instance: one partial
//                  per SM).
//   k_reduce_partials  fixed-order sum of the partials.
//
// Per-ray LBVH traversal (trace) serves the hr_trace entry point and the sub-tiles
// with more candidates than a list holds (k_overflow, and edge rays landing there).
//   k_silhouettes  per view, edges whose faces face opposite ways from the camera
//                  (plus boundary edges), compacted in edge order.
//   k_edge_samples the boundary term: samples on silhouette edges, f+ and f- by
//                  two rays over the candidate list of the sample's sub-tile, mapped
//                  to vertices by the projection Jacobian.
//   k_normal_gather  adjoint of the area-weighted vertex normals.
//
// Batches (hr_batch_create): every kernel runs over all instances of the batch in
// one launch.  Sub-tiles are numbered over all views of all instances (a view table
// maps a sub-tile to its view, instance, resolution and samples per pixel); each
// instance has its own BVH, vertices, normals and region of the work-item table.
// Warps take items of one instance, then of others with items left; a batch's backward
// adds its sums straight into its instance's gradient.  A single-instance call is a batch of one
// with a uniform view layout (no table).
#include <type_traits>

#include "hr_internal.h"

namespace hr {

namespace {

constexpr int kRenderThreads = 128;   // 4 warps per block
constexpr int kWarps = kRenderThreads / 32;
constexpr int kFwdMinBlocks = 7;      // launch bound of the forward shader (72 registers)
constexpr int kBwdMinBlocks = 4;      // launch bound of the backward shader (128 registers)
constexpr int kBlocksPerSm = 8;       // largest persistent grid
constexpr int kSubW = 8, kSubH = 4;   // sub-tile; lane = pixel
constexpr int kLeafCap = 512;         // candidates per sub-tile
constexpr int kFrontCap = 256;        // breadth-first frontier per level (dense meshes need the width)

// Self-check of an index read from device memory (BVH children, candidate records,
// pool offsets, work items): out of range sets a status bit and the caller skips
// the access.
__device__ __forceinline__ bool in_range(int* status, long long i, long long lo, long long hi) {
  if (i >= lo && i < hi) return true;
  set_status(status, kStatusIndex);
  return false;
}

struct Hit {
  int tri;
  float t, u, v;
};

__device__ __forceinline__ bool slab(float lx, float ly, float lz, float hx, float hy, float hz, float3 o,
                                     float3 inv, float tmax_in, float& tentry) {
  float t0x = (lx - o.x) * inv.x, t1x = (hx - o.x) * inv.x;
  float t0y = (ly - o.y) * inv.y, t1y = (hy - o.y) * inv.y;
  float t0z = (lz - o.z) * inv.z, t1z = (hz - o.z) * inv.z;
  float tmin = fmaxf(fmaxf(fminf(t0x, t1x), fminf(t0y, t1y)), fmaxf(fminf(t0z, t1z), 0.0f));
  float tmax = fminf(fminf(fmaxf(t0x, t1x), fmaxf(t0y, t1y)), fminf(fmaxf(t0z, t1z), tmax_in));
  tentry = tmin;
  return tmin <= tmax;
}

// reciprocal for the slab tests only (never for a hit decision): the approximate
// reciprocal is off by a couple of ulp, far inside the padding of the leaf boxes
__device__ __forceinline__ float safe_inv(float d) {
  return __fdividef(1.0f, fabsf(d) > 1e-20f ? d : copysignf(1e-20f, d));
}

// work counters of the statistics build (HR_STATS): estimator samples resolved,
// rays made individually, BVH nodes visited, Moller-Trumbore tests, hits, candidates read
// by a sub-tile's warp or tested against an edge ray
struct Counts {
  unsigned samples = 0, rays = 0, nodes = 0, tris = 0, hits = 0, cands = 0;
};

template <bool STATS>
__device__ __forceinline__ void isect(const float4* __restrict__ tris, int k, float3 o, float3 d, Hit& h,
                                      Counts& cnt) {
  if (STATS) ++cnt.tris;
  float4 a = __ldg(&tris[3 * k]), b = __ldg(&tris[3 * k + 1]), c = __ldg(&tris[3 * k + 2]);
  float3 v0 = make_float3(a.x, a.y, a.z), e1 = make_float3(a.w, b.x, b.y), e2 = make_float3(b.z, b.w, c.x);
  int id = __float_as_int(c.y);
  float t, u, v;
  if (mt_hit(o, d, v0, e1, e2, t, u, v)) {
    if (t < h.t || (t == h.t && id < h.tri)) {
      h.tri = id;
      h.t = t;
      h.u = u;
      h.v = v;
    }
  }
}

// One node of a closest-hit traversal; false when there is no next one.
template <bool STATS>
__device__ __forceinline__ bool visit_node(const Node* __restrict__ nodes, const float4* __restrict__ tris, float3 o,
                                           float3 d, float3 inv, Hit& h, int (&stack)[kStack], int& sp, int& node,
                                           int* status, Counts& cnt) {
  const float4* np = reinterpret_cast<const float4*>(nodes + node);
  if (STATS) ++cnt.nodes;
  float4 a = __ldg(np), b = __ldg(np + 1), c = __ldg(np + 2);
  int4 dd = __ldg(reinterpret_cast<const int4*>(np + 3));
  float tl, tr;
  bool hl = slab(a.x, a.y, a.z, a.w, b.x, b.y, o, inv, h.t, tl);
  bool hrr = slab(b.z, b.w, c.x, c.y, c.z, c.w, o, inv, h.t, tr);
  if (hl && dd.x < 0) {
    isect<STATS>(tris, ~dd.x, o, d, h, cnt);
    hl = false;
  }
  if (hrr && dd.y < 0) {
    isect<STATS>(tris, ~dd.y, o, d, h, cnt);
    hrr = false;
  }
  if (hl && hrr) {
    int nearc = dd.x, farc = dd.y;
    if (tr < tl) {
      nearc = dd.y;
      farc = dd.x;
    }
    if (sp < kStack) {
      stack[sp++] = farc;
    } else {
      set_status(status, kStatusLimit);
    }
    node = nearc;
  } else if (hl) {
    node = dd.x;
  } else if (hrr) {
    node = dd.y;
  } else {
    if (sp == 0) return false;
    node = stack[--sp];
  }
  return true;
}
__device__ __forceinline__ float3 slab_inv(float3 d) { return make_float3(safe_inv(d.x), safe_inv(d.y), safe_inv(d.z)); }

// Closest hit against the LBVH (root = internal node 0); ties in t go to the lower
// triangle id.  At most `max_visits` internal nodes are visited (a well-formed tree
// never needs more than F - 1); past it the status records a limit error.
template <bool STATS>
__device__ Hit trace(const Node* __restrict__ nodes, const float4* __restrict__ tris, float3 o, float3 d,
                     int* status, Counts& cnt, int max_visits) {
  Hit h{-1, INFINITY, 0.0f, 0.0f};
  const float3 inv = slab_inv(d);
  int stack[kStack];
  int sp = 0;
  int node = 0;
  for (int visits = 0;; ++visits) {
    if (visits >= max_visits) {
      set_status(status, kStatusLimit);
      break;
    }
    if (!visit_node<STATS>(nodes, tris, o, d, inv, h, stack, sp, node, status, cnt)) break;
  }
  return h;
}

template <bool STATS>
__device__ __forceinline__ void flush_counts(const Counts& c, unsigned long long* out) {
  if (!STATS) return;
  unsigned v[kStatsPer] = {c.samples, c.rays, c.nodes, c.tris, c.hits, c.cands};
  for (int k = 0; k < kStatsPer; ++k) {
    unsigned long long x = v[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(out + k, x);
  }
}

struct Shading {
  float3 l, lrgb;
  float ka, kd;
};

// candidate pool and work items shared by the gather / shade / combine kernels
struct Work {
  float4* bb;      // [pool] screen box (x0, y0, x1, y1) of the candidate
  float* z;        // [pool] nearest camera depth (sorted within a sub-tile)
  int* rec;        // [pool] triangle record
  unsigned* pm;    // [pool] pixels of the sub-tile (bit = lane) that the triangle can cover
  int pool_cap;
  int2* st;        // [sub-tiles] (pool offset, K): K = 0 no ray can hit, K < 0 per-ray
                   // traversal (-1: too many candidates; -(n + 1): n found no pool room)
  int4* items;     // [items] (sub-tile, chunk, chunks, first item of the sub-tile)
  int item_cap;
  float4* part;    // [items][32] forward per-item sums (r, g, b, misses)
  double* extra64; // [n_inst][6V] backward sums of meshes beyond shared memory (float64
                   // atomics: long runs of cancelling contributions)
  float* extra;    // [n_inst][8V] backward sums: shading blocks of a batch, and work
                   // done outside the shading blocks
  unsigned* ctr;   // [ctr_words(n_inst)] sub-tile counter, pool fill, per instance
                   // front items and taken items, the overflow count, per instance back
                   // items, then per instance a 64-bit allocation word
  int* ovf;        // [sub-tiles] sub-tiles whose items did not fit their instance's
                   // region (k_overflow does them whole)
  int* trace;      // [items] region slots (+ instance base) of the items of sub-tiles
                   // without a candidate list (k_overflow traces them ray by ray)
  unsigned* st_done;   // [sub-tiles] forward items finished (the last one combines)
  int4* cand_st;       // [sub-tiles] forward lists k_bin_sort orders: (sub-tile, pool offset, K, 0)
                       // (count: ctr_sort)
  unsigned* bin;       // [sub-tiles] records binned per sub-tile, then the fill's slot counter
  int* bvh_need;       // [n_inst] set when a sub-tile is listed for per-ray traversal
  unsigned long long* fx;   // [n_inst][6V] fixed-point backward sums (HR_DETERMINISTIC)
  bool det;                 // HR_DETERMINISTIC: every vertex-gradient sum goes to fx
};

struct RenderArgs {
  const Node* nodes;       // instance 0; instance i at + i node_stride
  const float4* tris;      // instance i at + 3 i node_stride
  const float* verts;      // instance i at + 3 i V
  const int* faces;
  const float* normals;    // instance i at + 3 i V
  const float* albedo;
  float4* frec;            // shading records by face id; instance i at + kFaceRec i node_stride
  const Cam* cams;         // [views]
  const float* bg;
  int N, H, W, spp, V;     // uniform layout (single instance)
  const ViewRec* vt;       // batch view table, nullptr = uniform layout
  const InstRec* it;       // batch instance table
  const int* active;       // batch: instances with 0 are skipped (retired), or null
  const int* act_off;      // with `active`: [2][n_inst + 1] active sub-tile / view prefix sums
  int n_inst, nviews, total_st;
  int num_sms;
  int node_stride;
  int cand_per_chunk, max_chunks;   // work-item split (tuning)
  const float* uv;        // [V][2] texture coordinates (shared by all instances)
  const float* tex;       // [tex_h][tex_w][3] albedo texture, or null: per-vertex albedo
  int tex_w, tex_h;
  float* d_tex;           // dL/dtexture (accumulated), or null
  uint2 key;
  uint32_t ctr1_hi;  // instance << 16
  uint32_t iter4;    // iter << 4 (kernels refresh it from iter_dev when given)
  const uint32_t* iter_dev;
  Shading sh;
  int* status;
  int max_visits;    // F + 1
  Work wk;
};

// bilinear texture lookup at the interpolated uv of a hit: texel coordinates
// x = uv_x W - 0.5, y = uv_y H - 0.5 and their floors are float32 decisions; the
// four texels (clamped to the edge) and their weights
struct TexSample {
  int i0, i1, j0, j1;
  int cell;   // the unclamped corner (x + 1 in the low half, y + 1 above): -1 .. size each
  float fx, fy;
};
__device__ __forceinline__ void tex_corners(const RenderArgs& a, TexSample& ts) {
  const int xi = (ts.cell & 0xffff) - 1, yi = (ts.cell >> 16) - 1;
  ts.i0 = min(max(xi, 0), a.tex_w - 1);
  ts.i1 = min(max(xi + 1, 0), a.tex_w - 1);
  ts.j0 = min(max(yi, 0), a.tex_h - 1);
  ts.j1 = min(max(yi + 1, 0), a.tex_h - 1);
}
__device__ __forceinline__ TexSample tex_coords(const RenderArgs& a, float4 t01, float4 t2, float u, float v) {
  const float w = __fsub_rn(__fsub_rn(1.0f, u), v);
  const float2 t0 = make_float2(t01.x, t01.y), t1 = make_float2(t01.z, t01.w);
  const float ux = __fmaf_rn(v, t2.x, __fmaf_rn(u, t1.x, __fmul_rn(w, t0.x)));
  const float uy = __fmaf_rn(v, t2.y, __fmaf_rn(u, t1.y, __fmul_rn(w, t0.y)));
  const float x = __fmaf_rn(ux, (float)a.tex_w, -0.5f), y = __fmaf_rn(uy, (float)a.tex_h, -0.5f);
  const float xf = floorf(x), yf = floorf(y);
  TexSample ts;
  ts.fx = __fsub_rn(x, xf);
  ts.fy = __fsub_rn(y, yf);
  const int xi = (int)fminf(fmaxf(xf, -1.0f), (float)a.tex_w), yi = (int)fminf(fmaxf(yf, -1.0f), (float)a.tex_h);
  ts.cell = (xi + 1) | ((yi + 1) << 16);
  tex_corners(a, ts);
  return ts;
}

__device__ __forceinline__ float3 tex_texel(const RenderArgs& a, int i, int j) {
  return ld3(a.tex + 3 * ((size_t)j * a.tex_w + i));
}

// Value arithmetic of the shading, every rounding spelled out: a pixel has the same bits
// whichever kernel shades it and however the code around is compiled.  The loss's
// adjoint is the sign of image - observation, so a last bit that moves can turn a pixel's
// gradient round (left to the compiler's contraction, one channel of 50 million turned
// and moved a texture gradient by 2e-4 of its norm).
// a b + c d, the first product exact
__device__ __forceinline__ float mul_add2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
// the orders are those that images have always had: of the upper pair of texels the product
// with fx is exact in red and green, that with 1 - fx in blue
__device__ __forceinline__ float3 tex_albedo(const RenderArgs& a, const TexSample& ts) {
  const float3 t00 = tex_texel(a, ts.i0, ts.j0), t10 = tex_texel(a, ts.i1, ts.j0);
  const float3 t01 = tex_texel(a, ts.i0, ts.j1), t11 = tex_texel(a, ts.i1, ts.j1);
  const float fx = ts.fx, fy = ts.fy, gx = __fsub_rn(1.0f, fx), gy = __fsub_rn(1.0f, fy);
  return make_float3(mul_add2(gy, mul_add2(fx, t10.x, gx, t00.x), fy, mul_add2(gx, t01.x, fx, t11.x)),
                     mul_add2(gy, mul_add2(fx, t10.y, gx, t00.y), fy, mul_add2(gx, t01.y, fx, t11.y)),
                     mul_add2(gy, mul_add2(gx, t00.z, fx, t10.z), fy, mul_add2(gx, t01.z, fx, t11.z)));
}

// Shading record of a face, kFaceRec float4 words:
//   0-2  (n_k, vertex index k)   unit normals of the corners
//   3-5  (albedo_k, e1 component k)
//   6    (e2, v_0.x)
//   7    (uv_0, uv_1)            (texture coordinates: with a texture)
//   8    (uv_2, v_0.y, v_0.z)
// A hit reads its face in a few 16-byte loads that depend on nothing but the face id,
// instead of the indices and then 18 to 27 scalar loads behind them.  Rewritten by
// every render call (from the current normals, albedo and vertices); an index outside
// the model is taken as vertex 0 (the build has reported it).
__device__ __forceinline__ void write_face_record(const RenderArgs& a, int f) {
  int i[3];
  float3 n[3], c[3], v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    i[k] = __ldg(&a.faces[3 * f + k]);
    if (i[k] < 0 || i[k] >= a.V) i[k] = 0;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    n[k] = ld3(a.normals + 3 * i[k]);
    c[k] = ld3(a.albedo + 3 * i[k]);
    v[k] = ld3(a.verts + 3 * i[k]);
  }
  const float3 e1 = dsub(v[1], v[0]), e2 = dsub(v[2], v[0]);
  float4* r = a.frec + (size_t)kFaceRec * f;
#pragma unroll
  for (int k = 0; k < 3; ++k) r[k] = make_float4(n[k].x, n[k].y, n[k].z, __int_as_float(i[k]));
  r[3] = make_float4(c[0].x, c[0].y, c[0].z, e1.x);
  r[4] = make_float4(c[1].x, c[1].y, c[1].z, e1.y);
  r[5] = make_float4(c[2].x, c[2].y, c[2].z, e1.z);
  r[6] = make_float4(e2.x, e2.y, e2.z, v[0].x);
  float2 t2 = make_float2(0.0f, 0.0f);
  if (a.tex) {
    const float2* uv = reinterpret_cast<const float2*>(a.uv);
    const float2 t0 = __ldg(uv + i[0]), t1 = __ldg(uv + i[1]);
    t2 = __ldg(uv + i[2]);
    r[7] = make_float4(t0.x, t0.y, t1.x, t1.y);
  }
  r[8] = make_float4(t2.x, t2.y, v[0].y, v[0].z);
}

// the records of every active instance, by all threads of the grid
__device__ __forceinline__ void write_face_records(const RenderArgs& a);

__device__ __forceinline__ float3 xyz(float4 q) { return make_float3(q.x, q.y, q.z); }

// radiance of a hit: the albedo times the light's colour, and the factor k = ka + kd sigma
// of all three channels, whose product a sum takes unrounded
__device__ __forceinline__ float3 shade(const RenderArgs& a, const Hit& h, float& k) {
  const float4* r = a.frec + (size_t)kFaceRec * h.tri;
  const float3 n0 = xyz(__ldg(r)), n1 = xyz(__ldg(r + 1)), n2 = xyz(__ldg(r + 2));
  const float3 nm = interp_normal(h.u, h.v, n0, n1, n2);
  const float ndl = ddot(nm, a.sh.l);
  float sigma = 0.0f;
  if (ndl > 0.0f) sigma = __fmul_rn(ndl, rsqrtf(__fmaf_rn(nm.z, nm.z, mul_add2(nm.x, nm.x, nm.y, nm.y))));
  k = __fmaf_rn(a.sh.kd, sigma, a.sh.ka);
  float3 alb;
  if (a.tex) {
    alb = tex_albedo(a, tex_coords(a, __ldg(r + 7), __ldg(r + 8), h.u, h.v));
  } else {
    const float3 a0 = xyz(__ldg(r + 3)), a1 = xyz(__ldg(r + 4)), a2 = xyz(__ldg(r + 5));
    const float w = __fsub_rn(__fsub_rn(1.0f, h.u), h.v);
    alb = make_float3(__fmaf_rn(h.v, a2.x, mul_add2(w, a0.x, h.u, a1.x)), __fmaf_rn(h.v, a2.y, mul_add2(w, a0.y, h.u, a1.y)),
                      __fmaf_rn(h.v, a2.z, mul_add2(w, a0.z, h.u, a1.z)));
  }
  return make_float3(__fmul_rn(alb.x, a.sh.lrgb.x), __fmul_rn(alb.y, a.sh.lrgb.y), __fmul_rn(alb.z, a.sh.lrgb.z));
}
__device__ __forceinline__ float3 radiance(const RenderArgs& a, const Hit& h) {
  float k;
  const float3 f = shade(a, h, k);
  return make_float3(__fmul_rn(f.x, k), __fmul_rn(f.y, k), __fmul_rn(f.z, k));
}

__device__ __forceinline__ Cam load_cam(const Cam* cams, int view) {
  Cam c;
  const float* src = reinterpret_cast<const float*>(cams + view);
  float* dst = reinterpret_cast<float*>(&c);
#pragma unroll
  for (int i = 0; i < 20; ++i) dst[i] = __ldg(src + i);
  return c;
}

// a work item's camera, copied into the warp's shared-memory slot (lane i < 20 copies
// word i) so that the shaders read it from there instead of holding 20 registers
__device__ __forceinline__ const Cam& warp_cam(Cam* slot, const Cam* cams, int view) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  if (lane < 20) reinterpret_cast<float*>(slot)[lane] = __ldg(reinterpret_cast<const float*>(cams + view) + lane);
  __syncwarp();
  return *slot;
}

// sample-stream iteration: the device counter when the caller gave one
__device__ __forceinline__ RenderArgs with_iter(RenderArgs a) {
  if (a.iter_dev) a.iter4 = (*a.iter_dev) << 4;
  return a;
}

// the same arguments with the scene pointers of instance `inst`
__device__ __forceinline__ RenderArgs for_inst(RenderArgs a, int inst) {
  a.nodes += (size_t)inst * a.node_stride;
  a.tris += (size_t)inst * 3 * a.node_stride;
  a.verts += (size_t)inst * 3 * a.V;
  a.normals += (size_t)inst * 3 * a.V;
  a.frec += (size_t)inst * kFaceRec * a.node_stride;
  return a;
}

// a batch instance still being refined (hr_batch_set_active)
__device__ __forceinline__ bool inst_active(const RenderArgs& a, int inst) {
  return !a.active || __ldg(&a.active[inst]) != 0;
}

__device__ __forceinline__ void write_face_records(const RenderArgs& a) {
  const int F = a.max_visits - 1;
  const long long n = (long long)a.n_inst * F;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int inst = (int)(i / F);
    if (inst_active(a, inst)) write_face_record(for_inst(a, inst), (int)(i - (long long)inst * F));
  }
}
__global__ void k_face_records(RenderArgs a) { write_face_records(a); }

// work-item region of an instance
__device__ __forceinline__ int inst_ibase(const RenderArgs& a, int inst) { return a.vt ? a.it[inst].ibase : 0; }
__device__ __forceinline__ int inst_icap(const RenderArgs& a, int inst) {
  return a.vt ? a.it[inst].icap : a.wk.item_cap;
}

// sample s of pixel (px, py) of a view of width W whose counter word is ctr1
__device__ __forceinline__ void jitter(const RenderArgs& a, uint32_t ctr1, int W, int px, int py, int s, float& u1,
                                       float& u2) {
  uint4 r = philox4x32_10(make_uint4((uint32_t)(py * W + px), ctr1, (uint32_t)s, a.iter4), a.key);
  u1 = u24(r.x);
  u2 = u24(r.y);
}


__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
  return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

template <class T>
__device__ __forceinline__ void add3(T* dst, int i, float x, float y, float z) {
  atomicAdd(&dst[3 * i], x);
  atomicAdd(&dst[3 * i + 1], y);
  atomicAdd(&dst[3 * i + 2], z);
}

// Fixed-point sums (HR_DETERMINISTIC): a contribution x is added as the 64-bit integer
// round(x 2^40) (two's complement in an unsigned word); integer addition is exact and
// associative, so the sums do not depend on the order of the atomics.
constexpr double kFixScale = 1099511627776.0;   // 2^40
__device__ __forceinline__ unsigned long long to_fixed(float x) {
  return (unsigned long long)__double2ll_rn((double)x * kFixScale);
}
__device__ __forceinline__ void add_fixed(unsigned long long* p, float x) { atomicAdd(p, to_fixed(x)); }
template <>
__device__ __forceinline__ void add3<unsigned long long>(unsigned long long* dst, int i, float x, float y, float z) {
  add_fixed(&dst[3 * i], x);
  add_fixed(&dst[3 * i + 1], y);
  add_fixed(&dst[3 * i + 2], z);
}
__device__ __forceinline__ float from_fixed(unsigned long long v) {
  return (float)((double)(long long)v * (1.0 / kFixScale));
}

// ---------------------------------------------------------------------------------
// sub-tiles, frustum gathering
// ---------------------------------------------------------------------------------
struct SubTile {
  int view;          // global view (camera index)
  int inst;          // instance
  int x0, y0;
  int H, W, spp;
  uint32_t ctr1;     // Philox counter word of the view
  long long pix0;    // first pixel of the view
};

__device__ __forceinline__ int subtile_count(const RenderArgs& a) { return a.total_st; }

// global view holding sub-tile st: binary search of the view table (views are in
// sub-tile order)
__device__ __forceinline__ int view_of_subtile(const RenderArgs& a, int st) {
  int lo = 0, hi = a.nviews - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(&a.vt[mid].st0) <= st) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// the view of global view index g (uniform layout: computed)
__device__ __forceinline__ void view_info(const RenderArgs& a, int g, SubTile& t, int& st0, int& nsx) {
  t.view = g;
  if (a.vt) {
    const ViewRec* v = a.vt + g;
    t.inst = __ldg(&v->inst);
    t.ctr1 = __ldg(&v->ctr1);
    t.H = __ldg(&v->H);
    t.W = __ldg(&v->W);
    t.spp = __ldg(&v->spp);
    t.pix0 = __ldg(&v->pix0);
    st0 = __ldg(&v->st0);
    nsx = __ldg(&v->nsx);
  } else {
    t.inst = 0;
    t.ctr1 = (uint32_t)g | a.ctr1_hi;
    t.H = a.H;
    t.W = a.W;
    t.spp = a.spp;
    t.pix0 = (long long)g * a.H * a.W;
    nsx = (a.W + kSubW - 1) / kSubW;
    st0 = g * nsx * ((a.H + kSubH - 1) / kSubH);
  }
}

__device__ __forceinline__ SubTile subtile(const RenderArgs& a, int st) {
  SubTile t;
  int g;
  if (a.vt) {
    g = view_of_subtile(a, st);
  } else {
    const int nsx = (a.W + kSubW - 1) / kSubW, nsy = (a.H + kSubH - 1) / kSubH;
    g = st / (nsx * nsy);
  }
  int st0, nsx;
  view_info(a, g, t, st0, nsx);
  const int rem = st - st0;
  t.x0 = (rem % nsx) * kSubW;
  t.y0 = (rem / nsx) * kSubH;
  return t;
}

// The sub-tiles a kernel visits: all of them, or in a batch with retired instances
// those of the active instances, numbered 0 .. visit_count - 1 in instance order
// (prefix sums act_off, made by k_active_layout before the render kernels), so that a
// mostly retired batch costs no pass over the retired instances' sub-tiles.
__device__ __forceinline__ int visit_count(const RenderArgs& a) {
  return a.act_off ? __ldg(&a.act_off[a.n_inst]) : a.total_st;
}
// the instance k with off[k] <= i < off[k + 1] (off: n_inst + 1 prefix sums)
__device__ __forceinline__ int active_inst(const int* off, int n, int i) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(&off[mid]) <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ int visit_subtile(const RenderArgs& a, int i) {
  if (!a.act_off) return i;
  const int k = active_inst(a.act_off, a.n_inst, i);
  return __ldg(&a.it[k].st0) + (i - __ldg(&a.act_off[k]));
}
// views likewise (the edge-sampling kernel)
__device__ __forceinline__ int visit_views(const RenderArgs& a) {
  return a.act_off ? __ldg(&a.act_off[a.n_inst + 1 + a.n_inst]) : a.nviews;
}
__device__ __forceinline__ int visit_view(const RenderArgs& a, int j) {
  if (!a.act_off) return j;
  const int* off = a.act_off + a.n_inst + 1;
  const int k = active_inst(off, a.n_inst, j);
  return __ldg(&a.it[k].view0) + (j - __ldg(&off[k]));
}

// act_off = prefix sums over the instances of (active ? sub-tiles : 0) and
// (active ? views : 0); one block, each thread a contiguous run of instances
constexpr int kLayoutThreads = 1024;
__global__ void __launch_bounds__(kLayoutThreads) k_active_layout(const InstRec* __restrict__ it,
                                                                  const int* __restrict__ active, int n,
                                                                  int* __restrict__ act_off) {
  __shared__ int sst[kLayoutThreads], svw[kLayoutThreads];
  const int per = (n + kLayoutThreads - 1) / kLayoutThreads;
  const int i0 = min(n, threadIdx.x * per), i1 = min(n, i0 + per);
  int st = 0, vw = 0;
  for (int i = i0; i < i1; ++i)
    if (active[i]) {
      st += it[i].nst;
      vw += it[i].nviews;
    }
  sst[threadIdx.x] = st;
  svw[threadIdx.x] = vw;
  __syncthreads();
  for (int d = 1; d < kLayoutThreads; d <<= 1) {   // inclusive scan
    const int a = threadIdx.x >= d ? sst[threadIdx.x - d] : 0, b = threadIdx.x >= d ? svw[threadIdx.x - d] : 0;
    __syncthreads();
    sst[threadIdx.x] += a;
    svw[threadIdx.x] += b;
    __syncthreads();
  }
  st = sst[threadIdx.x] - st;
  vw = svw[threadIdx.x] - vw;
  for (int i = i0; i < i1; ++i) {
    act_off[i] = st;
    act_off[n + 1 + i] = vw;
    if (active[i]) {
      st += it[i].nst;
      vw += it[i].nviews;
    }
  }
  if (threadIdx.x == kLayoutThreads - 1) {
    act_off[n] = sst[threadIdx.x];
    act_off[n + 1 + n] = svw[threadIdx.x];
  }
}

__device__ __forceinline__ unsigned lanemask_lt() { return (1u << (threadIdx.x & 31)) - 1u; }

__device__ __forceinline__ int warp_append(bool want, int value, int* arr, int count, int cap, bool& ovf) {
  unsigned b = __ballot_sync(0xffffffffu, want);
  int idx = count + __popc(b & lanemask_lt());
  if (want && idx < cap) arr[idx] = value;
  int n = count + __popc(b);
  if (n > cap) ovf = true;
  return n;
}

__device__ __forceinline__ bool box_in_frustum(const float4* pl, float lx, float ly, float lz, float hx, float hy,
                                               float hz) {
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    float4 p = pl[i];
    float x = p.x >= 0.0f ? hx : lx, y = p.y >= 0.0f ? hy : ly, z = p.z >= 0.0f ? hz : lz;
    if (p.x * x + p.y * y + p.z * z < p.w) return false;
  }
  return true;
}

struct GatherSmem {        // per warp
  int leaf[kLeafCap];
  float key[kLeafCap];
  int idx[kLeafCap];
  int front[2][kFrontCap];
  float4 pl[5];
};

// screen positions of a triangle's corners and how far (in pixels, x and y) its edges
// are moved outward by a pixel test that must keep every pixel a sample can hit it in;
// not positive: no such test (the box alone)
struct ScreenTri {
  float x[3], y[3];
  float margin;
};

// screen box (padded by half a pixel; unbounded if a vertex is not in front of the
// camera) and nearest camera depth of triangle record k
//
// The margin: a sample the float32 intersection accepts lies within the rounding of
// that test and of this projection from the triangle.  Both are a few float32 steps
// (2^-24) of the camera distance in pixels; the test's part grows by the edges'
// foreshortening, at most |edge| in pixels over the triangle's height on the screen.
// 32 steps of a generous distance plus 1/16 pixel covers them many times over; where
// that exceeds half a pixel (slivers, extreme cameras), or is not a number, the box,
// which is padded by half a pixel, decides alone.
template <bool TRI = false>
__device__ __forceinline__ void project_record(const RenderArgs& a, const Cam& cam, int k, float4& bb, float& zmin,
                                               ScreenTri* st = nullptr) {
  float4 t0 = __ldg(&a.tris[3 * k]), t1 = __ldg(&a.tris[3 * k + 1]), t2 = __ldg(&a.tris[3 * k + 2]);
  float3 v[3] = {make_float3(t0.x, t0.y, t0.z), make_float3(t0.x + t0.w, t0.y + t1.x, t0.z + t1.y),
                 make_float3(t0.x + t1.z, t0.y + t1.w, t0.z + t2.x)};
  float bx0 = INFINITY, by0 = INFINITY, bx1 = -INFINITY, by1 = -INFINITY;
  zmin = INFINITY;
  bool front = true;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    float X = cam.R[0] * v[m].x + cam.R[1] * v[m].y + cam.R[2] * v[m].z + cam.t[0];
    float Y = cam.R[3] * v[m].x + cam.R[4] * v[m].y + cam.R[5] * v[m].z + cam.t[1];
    float Z = cam.R[6] * v[m].x + cam.R[7] * v[m].y + cam.R[8] * v[m].z + cam.t[2];
    zmin = fminf(zmin, Z);
    front = front && Z > 1e-4f;
    float iz = 1.0f / Z;
    float sx = cam.fx * X * iz + cam.cx, sy = cam.fy * Y * iz + cam.cy;
    bx0 = fminf(bx0, sx);
    bx1 = fmaxf(bx1, sx);
    by0 = fminf(by0, sy);
    by1 = fmaxf(by1, sy);
    if (TRI) {
      st->x[m] = sx;
      st->y[m] = sy;
    }
  }
  if (TRI) {
    const float dx1 = st->x[1] - st->x[0], dy1 = st->y[1] - st->y[0];
    const float dx2 = st->x[2] - st->x[0], dy2 = st->y[2] - st->y[0];
    const float area = fabsf(dx1 * dy2 - dx2 * dy1);
    const float longest = fmaxf(fmaxf(fabsf(dx1) + fabsf(dy1), fabsf(dx2) + fabsf(dy2)),
                                fabsf(dx2 - dx1) + fabsf(dy2 - dy1));
    const float focal = fabsf(cam.fx) + fabsf(cam.fy);
    const float edge = fabsf(t0.w) + fabsf(t1.x) + fabsf(t1.y) + fabsf(t1.z) + fabsf(t1.w) + fabsf(t2.x);
    const float dist = fabsf(v[0].x) + fabsf(v[0].y) + fabsf(v[0].z) + edge + fabsf(cam.t[0]) + fabsf(cam.t[1]) +
                       fabsf(cam.t[2]) + fabsf(cam.c[0]) + fabsf(cam.c[1]) + fabsf(cam.c[2]);
    const float screen = fabsf(bx0) + fabsf(bx1) + fabsf(by0) + fabsf(by1) + fabsf(cam.cx) + fabsf(cam.cy);
    const float px = focal / zmin;
    const float grow = 1.0f + edge * px * longest / area;
    const float m = 0.0625f + 1.9073486e-6f * (px * dist * grow + screen);
    // the height test keeps the orientation's sign, and so the edges' sides, certain
    st->margin = front && m <= 0.5f && area > m * longest ? m : 0.0f;
  }
  if (front) {
    bb = make_float4(bx0 - 0.5f, by0 - 0.5f, bx1 + 0.5f, by1 + 0.5f);
  } else {
    bb = make_float4(-INFINITY, -INFINITY, INFINITY, INFINITY);
    zmin = -INFINITY;
  }
}

// Frustum traversal for the sub-tile with pixels [x0, x0+8) x [y0, y0+4): the four
// planes through the camera centre and the rectangle padded by half a pixel, and
// the camera's forward plane.  Leaves into gs.leaf; returns their count, or -1 when
// the sub-tile needs more than kLeafCap candidates or kFrontCap frontier nodes.
// plane q (0-4) of the sub-tile's frustum: the four planes through the camera centre
// and the rectangle padded by half a pixel, and the camera's forward plane (n, n . c)
__device__ __forceinline__ float4 frustum_plane(const Cam& cam, int x0, int y0, int q) {
  float ax = __fdividef((float)x0 - 0.5f - cam.cx, cam.fx);
  float bx = __fdividef((float)(x0 + kSubW) + 0.5f - cam.cx, cam.fx);
  float ay = __fdividef((float)y0 - 0.5f - cam.cy, cam.fy);
  float by = __fdividef((float)(y0 + kSubH) + 0.5f - cam.cy, cam.fy);
  float3 nc = q == 0   ? make_float3(1.0f, 0.0f, -ax)
              : q == 1 ? make_float3(-1.0f, 0.0f, bx)
              : q == 2 ? make_float3(0.0f, 1.0f, -ay)
              : q == 3 ? make_float3(0.0f, -1.0f, by)
                       : make_float3(0.0f, 0.0f, 1.0f);
  float3 nw = make_float3(cam.R[0] * nc.x + cam.R[3] * nc.y + cam.R[6] * nc.z,
                          cam.R[1] * nc.x + cam.R[4] * nc.y + cam.R[7] * nc.z,
                          cam.R[2] * nc.x + cam.R[5] * nc.y + cam.R[8] * nc.z);
  return make_float4(nw.x, nw.y, nw.z, nw.x * cam.c[0] + nw.y * cam.c[1] + nw.z * cam.c[2]);
}

template <bool STATS>
__device__ int frustum_leaves(const RenderArgs& a, const Cam& cam, int x0, int y0, GatherSmem& gs, Counts& cnt) {
  const int lane = threadIdx.x & 31;
  if (lane < 5) gs.pl[lane] = frustum_plane(cam, x0, y0, lane);
  if (lane == 0) gs.front[0][0] = 0;
  __syncwarp();
  int n = 1, cur = 0, K = 0, levels = 0;
  bool ovf = false;
  while (n > 0 && !ovf) {
    int nn = 0;
    for (int base = 0; base < n; base += 32) {
      const int i = base + lane;
      bool kl = false, kr = false;
      int cl = 0, cr = 0;
      if (i < n) {
        int node = gs.front[cur][i];
        if (!in_range(a.status, node, 0, a.max_visits)) node = 0;
        const float4* np = reinterpret_cast<const float4*>(a.nodes + node);
        float4 p = __ldg(np), q = __ldg(np + 1), r = __ldg(np + 2);
        int4 dd = __ldg(reinterpret_cast<const int4*>(np + 3));
        if (STATS) ++cnt.nodes;
        kl = box_in_frustum(gs.pl, p.x, p.y, p.z, p.w, q.x, q.y);
        kr = box_in_frustum(gs.pl, q.z, q.w, r.x, r.y, r.z, r.w);
        cl = dd.x;
        cr = dd.y;
        if (cl == cr) kr = false;   // a one-triangle tree stores its leaf twice
      }
      nn = warp_append(kl && cl >= 0, cl, gs.front[cur ^ 1], nn, kFrontCap, ovf);
      nn = warp_append(kr && cr >= 0, cr, gs.front[cur ^ 1], nn, kFrontCap, ovf);
      K = warp_append(kl && cl < 0, ~cl, gs.leaf, K, kLeafCap, ovf);
      K = warp_append(kr && cr < 0, ~cr, gs.leaf, K, kLeafCap, ovf);
    }
    __syncwarp();
    cur ^= 1;
    n = nn;
    if (++levels > a.max_visits) {   // deeper than any well-formed tree: report and stop
      if (lane == 0) set_status(a.status, kStatusLimit);
      ovf = true;
    }
  }
  return ovf ? -1 : K;
}

// work items of a sub-tile with K candidates (K < 0: per-ray traversal): one per
// `cand_per_chunk` candidates, at most max_chunks and spp
// (K = -1: more candidates than the gather's list holds; K < -1: -(K + 1) candidates
// that found no room in the pool.)  The split depends on the geometry only, never on
// which sub-tiles the pool served first, so sums over a sub-tile's items are
// reproducible.
__device__ __forceinline__ int chunks_for(const RenderArgs& a, int K, int spp) {
  int c = K == -1 ? a.max_chunks : (K < 0 ? -K - 1 : K) / a.cand_per_chunk;
  return max(1, min(min(c, a.max_chunks), spp));
}

// Work-item order.  A warp's item costs about (samples per lane) x (kSampleCost + K)
// candidate tests: a sample's own work (jitter, direction, shading or
// differentiation) weighs about kSampleCost tests (measured on the paper-shaped
// workload).  Items are taken from one counter, so the launch ends when the last
// item taken finishes; heavy items taken last leave most warps idle for the length
// of one heavy item.  Items whose cost exceeds twice the split's target
// (cand_per_chunk x spp) are therefore allocated from the front of the instance's
// item region and the others from its back, and the shaders take the front first.
// Per instance the counters are: front items (ctr[2 + 2i]), taken items
// (ctr[3 + 2i]), back items (ctr[3 + 2n + i]), and a 64-bit allocation word
// (front | back << 32) that decides, in one atomic, whether a group still fits.
constexpr int kSampleCost = 16;
__device__ __forceinline__ bool heavy_item(const RenderArgs& a, int K, int C, int spp) {
  const int k = K == -1 ? kLeafCap : (K < 0 ? -K - 1 : K);
  const int ns = (spp + C - 1) / C;
  return (long long)ns * (k + kSampleCost) > 2LL * a.cand_per_chunk * spp;
}
__device__ __forceinline__ unsigned* back_count(const RenderArgs& a, int inst) {
  return a.wk.ctr + 3 + 2 * a.n_inst + inst;
}
__device__ __forceinline__ unsigned long long* alloc_word(const RenderArgs& a, int inst) {
  return reinterpret_cast<unsigned long long*>(a.wk.ctr + ctr_alloc_base(a.n_inst)) + inst;
}
// reserve C consecutive slots of instance inst's region (lane 0 calls); -1 when the
// region has no room for them
__device__ __forceinline__ int alloc_items(const RenderArgs& a, int inst, int C, bool heavy, int icap) {
  const unsigned long long v =
      atomicAdd(alloc_word(a, inst), heavy ? (unsigned long long)C : ((unsigned long long)C << 32));
  const long long front = (long long)(v & 0xffffffffull), back = (long long)(v >> 32);
  if (front + back + C > icap) return -1;
  if (heavy) {
    atomicAdd(&a.wk.ctr[2 + 2 * inst], (unsigned)C);
    return (int)front;
  }
  atomicAdd(back_count(a, inst), (unsigned)C);
  return (int)(icap - back - C);
}

// the C items at table index `gi` belong to a sub-tile without a candidate list: list
// them for k_overflow (all lanes call)
__device__ __forceinline__ void note_trace_items(const RenderArgs& a, int gi, int C) {
  int base = 0;
  if ((threadIdx.x & 31) == 0) base = (int)atomicAdd(&a.wk.ctr[ctr_trace(a.n_inst)], (unsigned)C);
  base = __shfl_sync(0xffffffffu, base, 0);
  for (int c = threadIdx.x & 31; c < C; c += 32)
    if (base + c < a.wk.item_cap) a.wk.trace[base + c] = gi + c;
}


// bit p of the result: candidate box `b` (screen pixels, closed) meets pixel p of the
// 8x4 sub-tile at (x0, y0), i.e. b.x <= px + 1, b.z >= px, b.y <= py + 1, b.w >= py
// with pixel p at (x0 + p % 8, y0 + p / 8).  The float subtractions round
// monotonically and integers are exact, so the column and row bounds never exclude a
// pixel that meets the box; a NaN bound keeps the whole range.
__device__ __forceinline__ unsigned box_pixel_mask(float4 b, int x0, int y0) {
  const int cx0 = (int)fminf(fmaxf(ceilf(__fsub_rn(b.x, (float)(x0 + 1))), 0.0f), 8.0f);
  const int cx1 = (int)fmaxf(fminf(floorf(__fsub_rn(b.z, (float)x0)), 7.0f), -1.0f);
  const int ry0 = (int)fminf(fmaxf(ceilf(__fsub_rn(b.y, (float)(y0 + 1))), 0.0f), 4.0f);
  const int ry1 = (int)fmaxf(fminf(floorf(__fsub_rn(b.w, (float)y0)), 3.0f), -1.0f);
  if (cx0 > cx1 || ry0 > ry1) return 0u;
  const unsigned cols = (0xffu >> (7 - cx1)) & (0xffu << cx0);
  const unsigned rows = (0xffffffffu >> (8 * (3 - ry1))) & (0xffffffffu << (8 * ry0));
  return rows & (cols * 0x01010101u);
}

// 32 x 32 bit matrix held one row per lane (bit p of lane l's word) -> its transpose
// (bit l of lane p's word), by five butterfly stages that swap off-diagonal blocks
__device__ __forceinline__ unsigned warp_transpose32(unsigned x) {
  const int lane = threadIdx.x & 31;
  const unsigned m[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int j = 16 >> s;
    const unsigned t = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? ((x & ~m[s]) | ((t & ~m[s]) >> j)) : ((x & m[s]) | ((t & m[s]) << j));
  }
  return x;
}

// bits of box_pixel_mask's pixels that also meet the triangle moved outward by its
// margin: for each edge the pixel's corner farthest inside decides, so with E = A x +
// B y + C >= 0 inside, pixel (c, r) stays when A c + B r + C' >= 0, C' the edge's value
// at the sub-tile's first pixel plus that corner's and the margin's share; every row's
// columns are then an interval
__device__ __forceinline__ unsigned tri_pixel_mask(float4 b, const ScreenTri& t, int x0, int y0) {
  unsigned mask = box_pixel_mask(b, x0, y0);
  if (!(t.margin > 0.0f) || !mask) return mask;
  float px[3], py[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    px[k] = t.x[k] - (float)x0;
    py[k] = t.y[k] - (float)y0;
  }
  const float area = (px[1] - px[0]) * (py[2] - py[0]) - (px[2] - px[0]) * (py[1] - py[0]);
  const float sg = area < 0.0f ? -1.0f : 1.0f;
  float lo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, hi[4] = {7.0f, 7.0f, 7.0f, 7.0f};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int q = (k + 1) % 3;
    const float A = sg * (py[k] - py[q]), B = sg * (px[q] - px[k]);
    const float C = -(A * px[k] + B * py[k]) + t.margin * (fabsf(A) + fabsf(B)) + fmaxf(A, 0.0f) + fmaxf(B, 0.0f);
    const float inv = 1.0f / fmaxf(fabsf(A), 1e-20f);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float c = (B * (float)r + C) * inv;   // columns c' >= -c (A >= 0) or c' <= c
      if (A >= 0.0f) lo[r] = fmaxf(lo[r], -c);
      else hi[r] = fminf(hi[r], c);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int c0 = (int)fminf(ceilf(lo[r]), 8.0f), c1 = (int)fmaxf(floorf(hi[r]), -1.0f);
    const unsigned cols = c0 <= c1 ? (0xffu >> (7 - c1)) & (0xffu << c0) : 0u;
    mask &= (cols << (8 * r)) | ~(0xffu << (8 * r));
  }
  return mask;
}

// A warp's candidates in shared memory: what the intersection of a primary ray with
// each needs.  Primary rays start at the camera centre o, so of Moller-Trumbore's
// s = o - v0, q = s x e1 and e2 . q only depend on the candidate; they are computed
// once (the same operations, so the same float32 values) instead of once per ray.
// Arrays of float4: lanes reading neighbouring candidates meet no bank conflict.
// 32 of them, one per lane; longer lists pass through the tile in windows (a tile of 48, with
// two masks per lane, took 9 % more of a batch of 64 hands: 10.3 -> 9.4 ms).
constexpr int kCandCap = 32;
struct CandTile {
  float4 e1[kCandCap];   // e1, depth below which no ray's hit lets the candidate matter
  float4 e2[kCandCap];   // e2, triangle id
  float4 s[kCandCap];    // s, e2 . q
  float4 q[kCandCap];    // q
};

// candidates [c0, c0 + n), n <= kCandCap, of the list at `off` into the tile (one per lane);
// returns the lane's pixel's candidates, bit i = slot i
template <bool STATS>
__device__ __forceinline__ unsigned stage_candidates(const RenderArgs& a, CandTile& ct, int off, int c0, int n,
                                                     float3 o, Counts& cnt) {
  const int lane = threadIdx.x & 31;
  unsigned pm = 0u;
  if (lane < n) {
    const int i = off + c0 + lane;
    const float z = __ldg(&a.wk.z[i]);
    const int k = __ldg(&a.wk.rec[i]);
    pm = __ldg(&a.wk.pm[i]);
    if (STATS) ++cnt.cands;
    if (pm && in_range(a.status, k, 0, a.max_visits - 1)) {
      const float4 ta = __ldg(&a.tris[3 * k]), tb = __ldg(&a.tris[3 * k + 1]), tc = __ldg(&a.tris[3 * k + 2]);
      const float3 e1 = make_float3(ta.w, tb.x, tb.y), e2 = make_float3(tb.z, tb.w, tc.x);
      const float3 s = dsub(o, xyz(ta)), q = dcross(s, e1);
      if (!in_range(a.status, __float_as_int(tc.y), 0, a.max_visits - 1)) pm = 0u;
      ct.e1[lane] = make_float4(e1.x, e1.y, e1.z, z - (1e-4f * fabsf(z) + 1e-6f));
      ct.e2[lane] = make_float4(e2.x, e2.y, e2.z, tc.y);
      ct.s[lane] = make_float4(s.x, s.y, s.z, ddot(e2, q));
      ct.q[lane] = make_float4(q.x, q.y, q.z, 0.0f);
    } else {
      pm = 0u;
    }
  }
  __syncwarp();
  return warp_transpose32(pm);
}

// Walk of the candidates in m (bit i = slot i, in depth order) by a lane's S
// rays: the float32 Moller-Trumbore test and closest-hit rule of mt_hit / trace, with
// the candidate's part taken from the tile.  u, v >= 0 and u + v <= 1 imply u <= 1, and
// det = 0 makes u infinite or not a number, which fails the test, so both of mt_hit's
// checks are kept; 1 / det is the correctly rounded reciprocal in both.  A lane stops at
// the first candidate nearer than none of its hits (the list is depth-sorted).  Rays
// that take no part start with t = -1, nearer than any hit.
template <bool STATS, int S>
__device__ __forceinline__ void walk_candidates(const CandTile& ct, unsigned m, const float3 (&d)[S],
                                                Hit (&h)[S], bool& done, Counts& cnt) {
  while (m) {
    const int i = __ffs(m) - 1;
    m &= m - 1u;
    const float4 c1 = ct.e1[i];
    float tmax = h[0].t;
#pragma unroll
    for (int j = 1; j < S; ++j) tmax = fmaxf(tmax, h[j].t);
    if (tmax < c1.w) {
      done = true;
      break;
    }
    const float4 c2 = ct.e2[i], c3 = ct.s[i], c4 = ct.q[i];
    const float3 e1 = xyz(c1), e2 = xyz(c2), s = xyz(c3), q = xyz(c4);
    const int id = __float_as_int(c2.w);
#pragma unroll
    for (int j = 0; j < S; ++j) {
      if (STATS && h[j].t >= 0.0f) ++cnt.tris;
      const float3 p = dcross(d[j], e2);
      const float inv = __frcp_rn(ddot(e1, p));
      const float u = __fmul_rn(ddot(s, p), inv);
      const float v = __fmul_rn(ddot(d[j], q), inv);
      const float t = __fmul_rn(c3.w, inv);
      if (fminf(u, v) >= 0.0f && __fadd_rn(u, v) <= 1.0f && t > 0.0f &&
          (t < h[j].t || (t == h[j].t && id < h[j].tri)))
        h[j] = Hit{id, t, u, v};
    }
  }
}

// what a warp keeps of the sub-tile it works on
struct WarpTile {
  CandTile cand;
  SubTile t;
  Cam cam;
};

// sub-tile t into the warp's tile, with its candidates where they fit (all lanes call);
// m0: the lane's pixel's candidates, bit i = slot i
template <bool STATS>
__device__ __forceinline__ void stage_tile(const RenderArgs& a, WarpTile& wt, const SubTile& t, int off, int K, unsigned& m0,
                                           Counts& cnt) {
  __syncwarp();   // every lane is done with the sub-tile before
  if ((threadIdx.x & 31) == 0) wt.t = t;
  const Cam& cam = warp_cam(&wt.cam, a.cams, t.view);
  m0 = 0u;
  if (K <= 0 || K > kCandCap) return;
  const float3 o = make_float3(cam.c[0], cam.c[1], cam.c[2]);
  m0 = stage_candidates<STATS>(a, wt.cand, off, 0, K, o, cnt);
}

// closest hits of S rays of this lane's pixel among the K candidates at `off` (all
// lanes call; `in`: the lane takes part).  Lists of up to kCandCap are in the tile
// (m0 from stage_tile); longer ones go through it in windows.
template <bool STATS, int S>
__device__ __forceinline__ void closest_staged(const RenderArgs& a, WarpTile& wt, int off, int K, unsigned m0,
                                               bool in, const float3 (&d)[S], Hit (&h)[S], Counts& cnt) {
#pragma unroll
  for (int j = 0; j < S; ++j) h[j] = Hit{-1, in ? INFINITY : -1.0f, 0.0f, 0.0f};
  bool done = !in;
  if (K <= kCandCap) {
    if (!done) walk_candidates<STATS, S>(wt.cand, m0, d, h, done, cnt);
    __syncwarp();
    return;
  }
  const float3 o = make_float3(wt.cam.c[0], wt.cam.c[1], wt.cam.c[2]);
  for (int w = 0; w < K; w += kCandCap) {
    if (!__any_sync(0xffffffffu, !done)) break;
    m0 = stage_candidates<STATS>(a, wt.cand, off, w, min(kCandCap, K - w), o, cnt);
    if (!done) walk_candidates<STATS, S>(wt.cand, m0, d, h, done, cnt);
    __syncwarp();   // every lane is done with the window
  }
}

// Radiance of samples [s0, s0 + S) of this lane's pixel, traced together (all lanes
// call it); added to the sums in sample order.
template <bool STATS, int S, bool TRACE = true>
__device__ __forceinline__ void shade_samples(const RenderArgs& a, WarpTile& wt, int off, int K, unsigned m0,
                                              int s0, float3& acc, int& misses, Counts& cnt) {
  const int lane = threadIdx.x & 31;
  const int px = wt.t.x0 + (lane % kSubW), py = wt.t.y0 + (lane / kSubW);
  const bool valid = px < wt.t.W && py < wt.t.H;
  float3 d[S];
  Hit h[S];
#pragma unroll
  for (int j = 0; j < S; ++j) {
    float u1, u2;
    jitter(a, wt.t.ctr1, wt.t.W, px, py, s0 + j, u1, u2);
    d[j] = primary_dir(wt.cam, __fadd_rn((float)px, u1), __fadd_rn((float)py, u2));
    if (STATS && valid) {
      ++cnt.samples;
      ++cnt.rays;
    }
  }
  if (K > 0) {
    closest_staged<STATS, S>(a, wt, off, K, m0, valid, d, h, cnt);
  } else {
    const float3 o = make_float3(wt.cam.c[0], wt.cam.c[1], wt.cam.c[2]);
#pragma unroll
    for (int j = 0; j < S; ++j) {
      h[j] = Hit{-1, INFINITY, 0.0f, 0.0f};
      // K < 0: no usable candidate list, per-ray traversal (only the overflow kernel
      // meets such sub-tiles; the shaders are built without it)
      if (TRACE && valid) h[j] = trace<STATS>(a.nodes, a.tris, o, d[j], a.status, cnt, a.max_visits);
    }
  }
#pragma unroll
  for (int j = 0; j < S; ++j) {
    if (!valid) continue;
    if (h[j].tri >= 0) {
      if (STATS) ++cnt.hits;
      float k;
      const float3 f = shade(a, h[j], k);
      acc.x = __fmaf_rn(f.x, k, acc.x);
      acc.y = __fmaf_rn(f.y, k, acc.y);
      acc.z = __fmaf_rn(f.z, k, acc.z);
    } else {
      ++misses;
    }
  }
}

__device__ __forceinline__ void write_pixel(const RenderArgs& a, const SubTile& t, float3 acc, int misses,
                                            float* __restrict__ image) {
  const int lane = threadIdx.x & 31;
  const int px = t.x0 + (lane % kSubW), py = t.y0 + (lane / kSubW);
  if (px >= t.W || py >= t.H) return;
  // misses contribute background * (misses / spp): a pixel whose samples all miss is
  // exactly its background value
  const size_t pix = t.pix0 + (size_t)py * t.W + px;
  const float fm = __fdiv_rn((float)misses, (float)t.spp);
  const float inv_spp = 1.0f / (float)t.spp;
  float3 bgc = misses ? ld3(a.bg + 3 * pix) : make_float3(0.0f, 0.0f, 0.0f);
  image[3 * pix] = mul_add2(acc.x, inv_spp, bgc.x, fm);
  image[3 * pix + 1] = mul_add2(acc.y, inv_spp, bgc.y, fm);
  image[3 * pix + 2] = mul_add2(acc.z, inv_spp, bgc.z, fm);
}

// Where a backward's vertex sums go: vertex i's dL/dv and dL/dn, added with atomics
// whose result is not read.  Float sums lie as [V][8] (dv, 0, dn, 0), so that a vertex
// takes two 16-byte reductions instead of six of four bytes; float64 and fixed-point
// sums as [V][3] then [V][3].
struct SumF32 {
  float* p;
  __device__ __forceinline__ unsigned sharing(int) const { return 0u; }
  __device__ __forceinline__ void add(int V, int i, float3 dv, float3 dn, unsigned) const {
    float* q = p + 8 * (size_t)i;
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q), "f"(dv.x), "f"(dv.y), "f"(dv.z), "f"(0.0f)
                 : "memory");
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q + 4), "f"(dn.x), "f"(dn.y), "f"(dn.z), "f"(0.0f)
                 : "memory");
  }
};
struct SumF64 {
  double* p;
  __device__ __forceinline__ unsigned sharing(int) const { return 0u; }
  __device__ __forceinline__ void add(int V, int i, float3 dv, float3 dn, unsigned) const {
    add3(p, i, dv.x, dv.y, dv.z);
    add3(p + 3 * V, i, dn.x, dn.y, dn.z);
  }
};
// Fixed point: one copy of the sums for all SMs, so lanes that differentiate one triangle
// side by side, twelve or more of them, are summed first (whole numbers: the sums' bits are
// the same).  Without, large triangles at few samples waited for their vertices' atomics: one
// view of 2048^2 (4096^2) at 1 spp 165 -> 102 (724 -> 188) us; below twelve the lanes' sums
// cost more than the atomics (8 x 512x384 at 16 spp: 188, with groups from six lanes 198).
constexpr int kShared = 12;
struct SumFixed {
  unsigned long long* p;
  // the lanes here that are on this triangle, when there are enough of them
  __device__ __forceinline__ unsigned sharing(int tri) const {
    const unsigned lanes = __match_any_sync(__activemask(), tri);
    return __popc(lanes) >= kShared ? lanes : 0u;
  }
  __device__ __forceinline__ void add(int V, int i, float3 dv, float3 dn, unsigned lanes) const {
    if (!lanes) {
      add3(p, i, dv.x, dv.y, dv.z);
      add3(p + 3 * V, i, dn.x, dn.y, dn.z);
      return;
    }
    const float x[6] = {dv.x, dv.y, dv.z, dn.x, dn.y, dn.z};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      // in pieces of 26, 26 and 12 bits, whose sums over 32 lanes fit a word
      const unsigned long long f = to_fixed(x[c]);
      const unsigned lo = __reduce_add_sync(lanes, (unsigned)f & 0x3ffffffu);
      const unsigned mid = __reduce_add_sync(lanes, (unsigned)(f >> 26) & 0x3ffffffu);
      const unsigned hi = __reduce_add_sync(lanes, (unsigned)(f >> 52));
      if ((threadIdx.x & 31) == __ffs(lanes) - 1)
        atomicAdd(p + (c < 3 ? 3 * i + c : 3 * V + 3 * i + c - 3), lo + ((unsigned long long)mid << 26) + ((unsigned long long)hi << 52));
    }
  }
};

// Value arithmetic of the backward, every contraction spelled out: a window's sums are
// the same in every kernel that differentiates it (HR_DETERMINISTIC relies on it).
__device__ __forceinline__ float3 sub3(float3 a, float3 b) {
  return make_float3(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z));
}
__device__ __forceinline__ float vdot(float3 a, float3 b) {
  return __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)));
}
__device__ __forceinline__ void addmul(float& s, float a, float b) { s = __fmaf_rn(a, b, s); }
__device__ __forceinline__ void addmul(float3& s, float a, float3 b) {
  addmul(s.x, a, b.x);
  addmul(s.y, a, b.y);
  addmul(s.z, a, b.z);
}
// a x + b y (+ c z)
__device__ __forceinline__ float3 comb(float a, float3 x, float b, float3 y) {
  return make_float3(__fmaf_rn(a, x.x, __fmul_rn(b, y.x)), __fmaf_rn(a, x.y, __fmul_rn(b, y.y)),
                     __fmaf_rn(a, x.z, __fmul_rn(b, y.z)));
}
__device__ __forceinline__ float lerp_rn(float a, float b, float t) { return __fmaf_rn(t, __fsub_rn(b, a), a); }

// Samples whose hits are differentiated together.  Within a window a lane's hits are
// taken triangle by triangle, whatever their order among the samples: the triangle's
// record is read and its sums are added to memory once per window instead of once per
// run of consecutive hits (64 random samples of a pixel that shows three triangles
// change triangle two times out of three).
constexpr int kGradWin = 16;
struct GradTile {
  WarpTile w;
  float4 hit[kGradWin][32];   // (triangle, u, v, -); with a texture then (cell, fx, fy, k)
  __device__ __forceinline__ WarpTile& tile() { return w; }
  __device__ __forceinline__ float4& at(int j) { return hit[j][threadIdx.x & 31]; }
};
// the same with each lane's hits in its own (local) memory: the shaders' 41 KB of shared
// memory per block would leave the tree's traversal (k_overflow) a quarter of the SM's L1
struct OverflowTile {
  WarpTile& w;
  float4 hit[kGradWin];
  __device__ __forceinline__ explicit OverflowTile(WarpTile& t) : w(t) {}
  __device__ __forceinline__ WarpTile& tile() { return w; }
  __device__ __forceinline__ float4& at(int j) { return hit[j]; }
};

// direction of sample s of this lane's pixel
__device__ __forceinline__ float3 sample_dir(const RenderArgs& a, const WarpTile& wt, int s) {
  const int lane = threadIdx.x & 31, px = wt.t.x0 + (lane % kSubW), py = wt.t.y0 + (lane / kSubW);
  float u1, u2;
  jitter(a, wt.t.ctr1, wt.t.W, px, py, s, u1, u2);
  return primary_dir(wt.cam, __fadd_rn((float)px, u1), __fadd_rn((float)py, u2));
}

// Differentiation of one window (any lanes), samples s0 ..: `pend` = those of this lane
// with a hit in gt.at(), G = upstream gradient x light colour.
//
// At a fixed ray, moving corner k by dp moves the hit's (u, v, t) by -M^-1 (w_k dp) with
// M = [e1, e2, -d] and weights w = (1 - u - v, u, v), so
//   dL/dp_k = -w_k (gu (d x e2) + gv (e1 x d)) / (e1 . (d x e2)),
// which does not depend on d's length: with d = -s + u e1 + v e2 (s = centre - v0) it is
//   dL/dp_k = -w_k (gu A + gv B + (gu u + gv v) N) / D,
//   A = e2 x s, B = s x e1, N = e1 x e2, D = s . N,
// vectors of the triangle alone.  So per triangle only the nine sums of w_k gu, w_k gv
// and w_k (gu u + gv v) are kept, and no ray direction.  The albedo enters through its
// dot products with G.
//
// Their float32 errors are common to all of a triangle's samples, and seen nearly
// edge-on they are small differences of large products (and the gradient is large): a
// triangle whose |cos| to the view is below kGrazing takes the first form, with each
// sample's own direction (made again) and so its own rounding.  Against 64 bits the two
// forms are equally far off, at 1 / 30 2.3e-5 of a 20 mm triangle's gradient and facing
// 8.5e-7, the rounding of the hits' own u and v; at the same float32 rays they differ by
// 1.1e-6 at 1 / 30.
constexpr float kGrazing = 1.0f / 32;
template <bool STATS, class Sum, class Tile>
__device__ __forceinline__ void grad_window(const RenderArgs& a, Tile& gt, unsigned pend, int s0, float3 G, Sum sum,
                                            Counts& cnt) {
  const unsigned all = pend;
  const float3 o = make_float3(gt.tile().cam.c[0], gt.tile().cam.c[1], gt.tile().cam.c[2]);
  while (pend) {
    const int tri = __float_as_int(gt.at(__ffs(pend) - 1).x);
    const float4* rec = a.frec + (size_t)kFaceRec * tri;
    const float4 r0 = __ldg(rec), r1 = __ldg(rec + 1), r2 = __ldg(rec + 2), r3 = __ldg(rec + 3), r4 = __ldg(rec + 4),
                 r5 = __ldg(rec + 5), r6 = __ldg(rec + 6), r8 = __ldg(rec + 8);
    // this triangle's samples
    unsigned m = 0u;
    for (unsigned q = pend; q; q &= q - 1u) {
      const int j = __ffs(q) - 1;
      if (__float_as_int(gt.at(j).x) == tri) m |= 1u << j;
    }
    pend &= ~m;
    const float3 n0 = xyz(r0), n1 = xyz(r1), n2 = xyz(r2);
    const float c0 = vdot(G, xyz(r3)), cu = vdot(G, sub3(xyz(r4), xyz(r3))), cv = vdot(G, sub3(xyz(r5), xyz(r3)));
    float4 t01 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.tex) t01 = __ldg(rec + 7);
    const float3 e1 = make_float3(r3.w, r4.w, r5.w), e2 = xyz(r6);
    const float3 s = dsub(o, make_float3(r6.w, r8.z, r8.w)), nn = dcross(e1, e2);
    const float D = vdot(s, nn);
    const bool grazing = __fmul_rn(D, D) < __fmul_rn(kGrazing * kGrazing, __fmul_rn(vdot(s, s), vdot(nn, nn)));
    // grazing: the sums of w_k q, q = (gu (d x e2) + gv (e1 x d)) / (e1 . (d x e2)),
    // component by component
    float su[3] = {0.f, 0.f, 0.f}, sv[3] = {0.f, 0.f, 0.f}, sn[3] = {0.f, 0.f, 0.f};
    float3 dn[3] = {make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f)};
    while (m) {
      const int j = __ffs(m) - 1;
      m &= m - 1u;
      const float4 hj = gt.at(j);
      if (STATS) ++cnt.hits;
      const float u = hj.y, v = hj.z, w[3] = {__fsub_rn(__fsub_rn(1.0f, u), v), u, v};
      const float3 nm = interp_normal(u, v, n0, n1, n2);
      const bool lit = ddot(nm, a.sh.l) > 0.0f;
      const float inv_len = rsqrtf(vdot(nm, nm));
      const float3 nh = make_float3(__fmul_rn(nm.x, inv_len), __fmul_rn(nm.y, inv_len), __fmul_rn(nm.z, inv_len));
      const float sigma = lit ? vdot(nh, a.sh.l) : 0.0f;
      const float k = __fmaf_rn(a.sh.kd, sigma, a.sh.ka);
      float gu, gv, galb;   // dL/du, dL/dv through the albedo; G . albedo
      if (a.tex) {
        // albedo = bilinear(texture, uv(u, v)); its texel gradients are added below
        const TexSample ts = tex_coords(a, t01, r8, u, v);
        const float t00 = vdot(G, tex_texel(a, ts.i0, ts.j0)), t10 = vdot(G, tex_texel(a, ts.i1, ts.j0));
        const float t0y = vdot(G, tex_texel(a, ts.i0, ts.j1)), t1y = vdot(G, tex_texel(a, ts.i1, ts.j1));
        const float dx = lerp_rn(__fsub_rn(t10, t00), __fsub_rn(t1y, t0y), ts.fy);
        const float dy = lerp_rn(__fsub_rn(t0y, t00), __fsub_rn(t1y, t10), ts.fx);
        const float dux = __fmul_rn(__fmul_rn(dx, k), (float)a.tex_w), duy = __fmul_rn(__fmul_rn(dy, k), (float)a.tex_h);
        gu = __fmaf_rn(dux, __fsub_rn(t01.z, t01.x), __fmul_rn(duy, __fsub_rn(t01.w, t01.y)));
        gv = __fmaf_rn(dux, __fsub_rn(r8.x, t01.x), __fmul_rn(duy, __fsub_rn(r8.y, t01.y)));
        galb = lerp_rn(lerp_rn(t00, t10, ts.fx), lerp_rn(t0y, t1y, ts.fx), ts.fy);
        if (a.d_tex) gt.at(j) = make_float4(__int_as_float(ts.cell), ts.fx, ts.fy, k);
      } else {
        gu = __fmul_rn(k, cu);
        gv = __fmul_rn(k, cv);
        galb = __fmaf_rn(v, cv, __fmaf_rn(u, cu, c0));
      }
      if (lit) {
        // through the normal: dL/dn of the interpolated n = kd galb (l - nh (nh . l)) / |n|
        const float f = __fmul_rn(__fmul_rn(a.sh.kd, galb), inv_len);
        const float3 dnm = make_float3(__fmul_rn(f, __fmaf_rn(-nh.x, sigma, a.sh.l.x)), __fmul_rn(f, __fmaf_rn(-nh.y, sigma, a.sh.l.y)),
                                       __fmul_rn(f, __fmaf_rn(-nh.z, sigma, a.sh.l.z)));
        gu = __fadd_rn(gu, vdot(dnm, sub3(n1, n0)));
        gv = __fadd_rn(gv, vdot(dnm, sub3(n2, n0)));
#pragma unroll
        for (int q = 0; q < 3; ++q) addmul(dn[q], w[q], dnm);
      }
      float gn = __fmaf_rn(gu, u, __fmul_rn(gv, v));
      if (grazing) {
        const WarpTile& wt = gt.tile();
        const float3 d = sample_dir(a, wt, s0 + j);
        const float3 dxe2 = dcross(d, e2), e1xd = dcross(e1, d), q = comb(gu, dxe2, gv, e1xd);
        const float invD = 1.0f / vdot(e1, dxe2);
        gu = __fmul_rn(q.x, invD);
        gv = __fmul_rn(q.y, invD);
        gn = __fmul_rn(q.z, invD);
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        addmul(su[q], w[q], gu);
        addmul(sv[q], w[q], gv);
        addmul(sn[q], w[q], gn);
      }
    }
    float3 A = dcross(e2, s), B = dcross(s, e1), N = nn;
    float inv = -1.0f / D;
    if (grazing) {
      A = make_float3(1.f, 0.f, 0.f);
      B = make_float3(0.f, 1.f, 0.f);
      N = make_float3(0.f, 0.f, 1.f);
      inv = -1.0f;
    }
    const int iv[3] = {__float_as_int(r0.w), __float_as_int(r1.w), __float_as_int(r2.w)};
    const unsigned sharing = sum.sharing(tri);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float3 dv = comb(__fmul_rn(su[k], inv), A, __fmul_rn(sv[k], inv), B);
      addmul(dv, __fmul_rn(sn[k], inv), N);
      sum.add(a.V, iv[k], dv, dn[k], sharing);
    }
  }
  if (!a.d_tex) return;
  // texel gradients, cell by cell: the four corners' sums of weight x k, times G
  for (pend = all; pend;) {
    const int cell = __float_as_int(gt.at(__ffs(pend) - 1).x);
    float wt[4] = {0.f, 0.f, 0.f, 0.f};
    for (unsigned q = pend; q; q &= q - 1u) {
      const int j = __ffs(q) - 1;
      const float4 hj = gt.at(j);
      if (__float_as_int(hj.x) != cell) continue;
      pend &= ~(1u << j);
      const float ky = hj.w * hj.z, k0 = hj.w - ky;
      wt[1] += k0 * hj.y;
      wt[0] += k0 - k0 * hj.y;
      wt[3] += ky * hj.y;
      wt[2] += ky - ky * hj.y;
    }
    TexSample ts;
    ts.cell = cell;
    tex_corners(a, ts);
    const int ii[4] = {ts.i0, ts.i1, ts.i0, ts.i1}, jj[4] = {ts.j0, ts.j0, ts.j1, ts.j1};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      add3(a.d_tex, jj[q] * a.tex_w + ii[q], wt[q] * G.x, wt[q] * G.y, wt[q] * G.z);
  }
}

// hits of samples [s0, s0 + S) of this lane's pixel into window entries j0 .. (all lanes
// call it; `live` lanes take part); returns the lane's entries with a hit
template <bool STATS, int S, class Tile>
__device__ __forceinline__ unsigned trace_samples(const RenderArgs& a, Tile& gt, int off, int K, unsigned m0,
                                                  int s0, int j0, bool live, Counts& cnt) {
  float3 d[S];
  Hit h[S];
#pragma unroll
  for (int j = 0; j < S; ++j) {
    d[j] = sample_dir(a, gt.tile(), s0 + j);
    if (STATS && live) {
      ++cnt.samples;
      ++cnt.rays;
    }
  }
  closest_staged<STATS, S>(a, gt.tile(), off, K, m0, live, d, h, cnt);
  unsigned hits = 0u;
#pragma unroll
  for (int j = 0; j < S; ++j) {
    if (h[j].tri < 0) continue;
    gt.at(j0 + j) = make_float4(__int_as_float(h[j].tri), h[j].u, h[j].v, 0.0f);
    hits |= 1u << (j0 + j);
  }
  return hits;
}

// the same without a candidate list, samples [s0, s0 + n) into window entries 0 ..: a lane
// goes on with its next ray when it is done with one, so that the warp waits for the
// lanes' sums of nodes and not for the longest of 32 traversals n times.  With the hits in
// the lanes' own memory: backward of 5 views of 125 x 336, 52 spp, 6 k triangles 596 -> 509
// us in all, of 14 views of 152 x 256, 57 spp, 24.6 k triangles 1777 -> 1560.
template <bool STATS, class Tile>
__device__ __forceinline__ unsigned traverse_samples(const RenderArgs& a, Tile& gt, int s0, int n, bool live, Counts& cnt) {
  const WarpTile& wt = gt.tile();
  for (int j = 0; j < n; ++j) {   // the directions, in the hits' places
    const float3 d = sample_dir(a, wt, s0 + j);
    gt.at(j) = make_float4(d.x, d.y, d.z, 0.0f);
    if (STATS && live) {
      ++cnt.samples;
      ++cnt.rays;
    }
  }
  const float3 o = make_float3(wt.cam.c[0], wt.cam.c[1], wt.cam.c[2]);
  unsigned hits = 0u;
  Hit h{-1, INFINITY, 0.0f, 0.0f};
  float3 d = o, inv = o;
  int stack[kStack];
  int sp = 0, node = 0, visits = 0, j = live ? -1 : n;
  bool next = true;
  while (j < n) {
    if (next) {
      if (j >= 0 && h.tri >= 0) {
        gt.at(j) = make_float4(__int_as_float(h.tri), h.u, h.v, 0.0f);
        hits |= 1u << j;
      }
      if (++j == n) break;
      d = xyz(gt.at(j));
      inv = slab_inv(d);
      h = Hit{-1, INFINITY, 0.0f, 0.0f};
      sp = node = visits = 0;
    }
    if (visits++ >= a.max_visits) {   // as in trace()
      set_status(a.status, kStatusLimit);
      next = true;
    } else {
      next = !visit_node<STATS>(a.nodes, a.tris, o, d, inv, h, stack, sp, node, a.status, cnt);
    }
  }
  __syncwarp();
  return hits;
}

// Gradient of samples [s0, s1) of this lane's pixel (upstream g, `live` lanes only; all
// lanes call it after stage_tile), traced S at a time, or (TRACE) ray by ray where there
// is no candidate list.  The windows and the order of a window's sums depend on [s0, s1)
// alone.
template <bool STATS, int S, class Sum, bool TRACE, class Tile>
__device__ __forceinline__ void grad_samples(const RenderArgs& a, Tile& gt, int off, int K, unsigned m0,
                                             int s0, int s1, bool live, float3 g, Sum sum, Counts& cnt) {
  const float3 G = make_float3(g.x * a.sh.lrgb.x, g.y * a.sh.lrgb.y, g.z * a.sh.lrgb.z);
  for (int w0 = s0; w0 < s1; w0 += kGradWin) {
    const int n = min(kGradWin, s1 - w0);
    unsigned pend = 0u;
    if (TRACE && K <= 0) {
      pend = traverse_samples<STATS>(a, gt, w0, n, live, cnt);
    } else {
      int j = 0;
      for (; j + S <= n; j += S) pend |= trace_samples<STATS, S>(a, gt, off, K, m0, w0 + j, j, live, cnt);
      if (S > 1)
        for (; j < n; ++j) pend |= trace_samples<STATS, 1>(a, gt, off, K, m0, w0 + j, j, live, cnt);
    }
    grad_window<STATS>(a, gt, pend, w0, G, sum, cnt);
    __syncwarp();
  }
}

// this lane's upstream gradient dL/df / spp; `live` = non-zero adjoint
__device__ __forceinline__ float3 lane_adjoint(const RenderArgs& a, const SubTile& t, const float* __restrict__ adjoint,
                                               bool& live) {
  const int lane = threadIdx.x & 31;
  const int px = t.x0 + (lane % kSubW), py = t.y0 + (lane / kSubW);
  live = false;
  if (px >= t.W || py >= t.H) return make_float3(0.0f, 0.0f, 0.0f);
  float3 g = ld3(adjoint + 3 * (t.pix0 + (size_t)py * t.W + px));
  live = g.x != 0.0f || g.y != 0.0f || g.z != 0.0f;
  const float inv_spp = 1.0f / (float)t.spp;
  return make_float3(g.x * inv_spp, g.y * inv_spp, g.z * inv_spp);
}

// kernels that take a group of consecutive sub-tiles per warp (k_bin_alloc, k_background,
// k_items_bwd): one per lane of the first kGroupSubtiles lanes
constexpr int kGroupThreads = 256;
constexpr int kGroupSubtiles = 8;

// ---------------------------------------------------------------------------------
// forward candidate lists by screen-space binning
// ---------------------------------------------------------------------------------
// A triangle can only be hit in its screen box (project_record: padded by half a pixel,
// unbounded when a vertex is not in front of the camera), so a sub-tile's list holds the
// triangle records whose box meets the sub-tile's sample square [x0, x0 + 8] x [y0, y0 +
// 4], and for each the pixels that the triangle can cover: the shaders test no box, a
// lane takes the candidates whose mask has its pixel.  The forward builds the lists by binning each (view, record) pair into the sub-tiles its
// box meets -- k_bin counts them, k_bin_alloc gives every sub-tile its pool range and
// work items, k_bin in fill mode writes the records, k_bin_sort orders each list by
// nearest depth -- instead of a frustum walk of the BVH per sub-tile.

// sub-tile columns [c0, c1] and rows [r0, r1] of a view (nsx x nsy sub-tiles) whose
// sample squares meet box b: column c meets it iff b.x <= 8c + 8 and b.z >= 8c (rows
// likewise with 4).  The float subtraction rounds monotonically and the scalings by
// 1/8 and 1/4 and the integers are exact, so no column or row that meets the box is
// left out; a NaN bound keeps the whole range.
struct BinRange {
  int c0, c1, r0, r1;
};
__device__ __forceinline__ BinRange bin_range(float4 b, int nsx, int nsy) {
  BinRange r;
  r.c0 = (int)fminf(fmaxf(ceilf(__fmul_rn(__fsub_rn(b.x, (float)kSubW), 1.0f / kSubW)), 0.0f), (float)nsx);
  r.c1 = (int)fmaxf(fminf(floorf(__fmul_rn(b.z, 1.0f / kSubW)), (float)(nsx - 1)), -1.0f);
  r.r0 = (int)fminf(fmaxf(ceilf(__fmul_rn(__fsub_rn(b.y, (float)kSubH), 1.0f / kSubH)), 0.0f), (float)nsy);
  r.r1 = (int)fmaxf(fminf(floorf(__fmul_rn(b.w, 1.0f / kSubH)), (float)(nsy - 1)), -1.0f);
  return r;
}

// the camera depth of record k's three vertices all below -1e-3: no primary ray
// (camera depth t > 0 at parameter t) can meet it
__device__ __forceinline__ bool record_behind(const RenderArgs& a, const Cam& cam, int k) {
  const float4 t0 = __ldg(&a.tris[3 * k]), t1 = __ldg(&a.tris[3 * k + 1]), t2 = __ldg(&a.tris[3 * k + 2]);
  const float3 v[3] = {make_float3(t0.x, t0.y, t0.z), make_float3(t0.x + t0.w, t0.y + t1.x, t0.z + t1.y),
                       make_float3(t0.x + t1.z, t0.y + t1.w, t0.z + t2.x)};
  bool behind = true;
#pragma unroll
  for (int m = 0; m < 3; ++m)
    behind = behind && cam.R[6] * v[m].x + cam.R[7] * v[m].y + cam.R[8] * v[m].z + cam.t[2] < -1e-3f;
  return behind;
}

constexpr int kBinThreads = 256;
constexpr int kBinPairs = 8;   // (view, record) pairs per warp

// one sub-tile of a pair's range: count it, or (FILL) write the record into the
// sub-tile's pool range at the next free slot
template <bool FILL>
__device__ __forceinline__ void bin_visit(const RenderArgs& a, unsigned* __restrict__ bin, int s, int x0, int y0, int k,
                                          float zm, float4 bb, const ScreenTri& tri) {
  if (!FILL) {
    atomicAdd(&bin[s], 1u);
    return;
  }
  const int2 pk = a.wk.st[s];
  if (pk.y <= 0) return;   // no list: background, per-ray traversal, or no pool room
  const int slot = (int)atomicAdd(&bin[s], 1u);
  if (slot >= pk.y || !in_range(a.status, (long long)pk.x + slot, 0, a.wk.pool_cap)) return;
  a.wk.rec[pk.x + slot] = k;
  a.wk.z[pk.x + slot] = zm;
  a.wk.bb[pk.x + slot] = bb;
  a.wk.pm[pk.x + slot] = tri_pixel_mask(bb, tri, x0, y0);
}

// Each warp takes kBinPairs consecutive pairs i = (active view i / F, record i % F),
// one per lane of its first lanes, and projects them; the (pair, sub-tile) visits of
// all its pairs are then spread over the 32 lanes (visit q belongs to the pair whose
// range of prefix sums holds q), so the visits of one warp are in flight together
// whatever the sizes of the pairs' ranges.
template <bool FILL>
__global__ void __launch_bounds__(kBinThreads) k_bin(RenderArgs a0, unsigned* __restrict__ bin) {
  pdl_wait();
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int F = a0.max_visits - 1;
  const long long total = (long long)visit_views(a0) * F;
  const long long nw = (long long)gridDim.x * (kBinThreads / 32);
  for (long long w0 = ((long long)blockIdx.x * (kBinThreads / 32) + (threadIdx.x >> 5)) * kBinPairs; w0 < total;
       w0 += nw * kBinPairs) {
    const long long i = w0 + lane;
    int st0 = 0, nsx = 1, k = 0, area = 0;
    float zm = 0.0f;
    float4 bb = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    ScreenTri tri{};
    BinRange r{0, -1, 0, -1};
    if (lane < kBinPairs && i < total) {
      const int g = visit_view(a0, (int)(i / F));
      k = (int)(i % F);
      SubTile t;
      view_info(a0, g, t, st0, nsx);
      if (in_range(a0.status, t.inst, 0, a0.n_inst) && inst_active(a0, t.inst)) {
        const RenderArgs a = for_inst(a0, t.inst);
        const Cam cam = load_cam(a.cams, g);
        if (!record_behind(a, cam, k)) {
          project_record<FILL>(a, cam, k, bb, zm, &tri);
          r = bin_range(bb, nsx, (t.H + kSubH - 1) / kSubH);
          if (r.c0 <= r.c1 && r.r0 <= r.r1) area = (r.c1 - r.c0 + 1) * (r.r1 - r.r0 + 1);
        }
      }
    }
    // inclusive prefix sums of the ranges' sizes over the pairs
    int incl = area;
#pragma unroll
    for (int o = 1; o < kBinPairs; o <<= 1) {
      const int y = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += y;
    }
    const int T = __shfl_sync(full, incl, kBinPairs - 1);
    for (int q0 = 0; q0 < T; q0 += 32) {
      const int q = q0 + lane;
      // owner: the first pair whose inclusive sum exceeds q
      int lo = 0;
#pragma unroll
      for (int step = kBinPairs / 2; step > 0; step >>= 1) {
        const int v = __shfl_sync(full, incl, lo + step - 1);
        if (v <= q) lo += step;
      }
      const int own = min(lo, kBinPairs - 1);
      const int s0 = __shfl_sync(full, st0, own), n = __shfl_sync(full, nsx, own);
      const int c0 = __shfl_sync(full, r.c0, own), c1 = __shfl_sync(full, r.c1, own);
      const int r0 = __shfl_sync(full, r.r0, own);
      const int kk = __shfl_sync(full, k, own), end = __shfl_sync(full, incl, own);
      const int na = __shfl_sync(full, area, own);
      const float z = __shfl_sync(full, zm, own);
      float4 b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      ScreenTri tv{};
      if (FILL) {
        b.x = __shfl_sync(full, bb.x, own);
        b.y = __shfl_sync(full, bb.y, own);
        b.z = __shfl_sync(full, bb.z, own);
        b.w = __shfl_sync(full, bb.w, own);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          tv.x[m] = __shfl_sync(full, tri.x[m], own);
          tv.y[m] = __shfl_sync(full, tri.y[m], own);
        }
        tv.margin = __shfl_sync(full, tri.margin, own);
      }
      if (q >= T) continue;
      const int w = c1 - c0 + 1, local = q - (end - na);
      const int col = c0 + local % w, row = r0 + local / w;
      bin_visit<FILL>(a0, bin, s0 + row * n + col, col * kSubW, row * kSubH, kk, z, b, tv);
    }
  }
  if (!FILL) {   // the shading records, for the shader three launches later
    write_face_records(a0);
  }
}

// Work items of the sub-tiles held by lanes 0 .. G - 1 (all lanes call): each
// `need` lane's sub-tile st (instance inst, candidate count K) gets C consecutive
// items.  One reservation per instance among the lanes -- heavy items from the front
// of the instance's region, the others from its back -- so the instance's counters
// see one atomic per warp, not one per sub-tile.  Sub-tiles without a candidate list
// (K < 0) are listed for k_overflow's per-ray traversal; when the region has no room
// for a group, its sub-tiles go to k_overflow whole.
template <int G>
__device__ __forceinline__ void place_items(const RenderArgs& a0, bool need, int st, int inst, int K, int C,
                                            bool heavy) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int key = need ? inst : -1;
  int hx = 0, lx = 0, ht = 0, lt = 0, leader = -1;
  const unsigned needs = __ballot_sync(full, need);
  const int first_key = __shfl_sync(full, key, needs ? __ffs(needs) - 1 : 0);
  if (G == 32 && __all_sync(full, !need || key == first_key)) {
    // one instance, as a rule: sums over the lanes, both kinds in one word (C <= 16)
    const int mine = need ? C << (heavy ? 0 : 16) : 0;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += y;
    }
    const int tot = __shfl_sync(full, incl, 31), excl = incl - mine;
    if (need) {
      hx = excl & 0xffff;
      lx = excl >> 16;
      ht = tot & 0xffff;
      lt = tot >> 16;
      leader = __ffs(needs) - 1;
    }
  } else
#pragma unroll 8
  for (int j = 0; j < G; ++j) {
    const int kj = __shfl_sync(full, key, j), cj = __shfl_sync(full, C, j);
    const bool hj = __shfl_sync(full, (int)heavy, j) != 0;
    if (need && kj == key) {
      if (leader < 0) leader = j;
      if (hj) {
        ht += cj;
        if (j < lane) hx += cj;
      } else {
        lt += cj;
        if (j < lane) lx += cj;
      }
    }
  }
  unsigned long long v = 0ull;
  if (need && lane == leader) {
    v = atomicAdd(alloc_word(a0, inst), (unsigned long long)ht | ((unsigned long long)lt << 32));
    const long long front = (long long)(v & 0xffffffffull), back = (long long)(v >> 32);
    if (front + back + ht + lt <= inst_icap(a0, inst)) {
      if (ht) atomicAdd(&a0.wk.ctr[2 + 2 * inst], (unsigned)ht);
      if (lt) atomicAdd(back_count(a0, inst), (unsigned)lt);
    }
  }
  const int src = leader < 0 ? 0 : leader;
  const unsigned vlo = __shfl_sync(full, (unsigned)(v & 0xffffffffull), src);
  const unsigned vhi = __shfl_sync(full, (unsigned)(v >> 32), src);
  if (!need) return;
  const int icap = inst_icap(a0, inst), ibase = inst_ibase(a0, inst);
  const long long front = vlo, back = vhi;
  const bool fits = front + back + ht + lt <= icap;
  const int first = fits ? (heavy ? (int)front + hx : icap - (int)back - lt + lx) : -1;
  if (first >= 0) {
    for (int c = 0; c < C; ++c) a0.wk.items[ibase + first + c] = make_int4(st, c, C, ibase + first);
    if (K < 0) {
      const int tb = (int)atomicAdd(&a0.wk.ctr[ctr_trace(a0.n_inst)], (unsigned)C);
      for (int c = 0; c < C; ++c)
        if (tb + c < a0.wk.item_cap) a0.wk.trace[tb + c] = ibase + first + c;
    }
  } else {
    a0.wk.ovf[atomicAdd(&a0.wk.ctr[2 + 2 * a0.n_inst], 1u)] = st;
  }
}

// Each warp takes G consecutive sub-tiles, one per lane of its first lanes: 8 to spread a
// small call over the SMs, all 32 lanes when there is work for every warp (2.1 M sub-tiles
// of 128 pairs 178 -> 99 us, a batch of 64 hands 222 -> 144 us).
// A sub-tile with no record in its bin sees only the background (k_background writes
// it).  The others get a pool range for their K records (one atomic per warp), the
// work items of their chunks, and an entry in the list k_bin_sort orders; the count
// becomes the fill's slot counter.  A sub-tile with more records than a list holds,
// or whose records find no pool room, is traced ray by ray (K = -1, -(K + 1)).
template <int G>
__global__ void __launch_bounds__(kGroupThreads) k_bin_alloc(RenderArgs a0, unsigned* __restrict__ bin) {
  pdl_wait();
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int total = visit_count(a0);
  const int nw = gridDim.x * (kGroupThreads / 32);
  for (int g0 = (blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5)) * G; g0 < total;
       g0 += nw * G) {
    int st = -1, K = 0;
    bool listed = false;
    SubTile t{};
    if (lane < G && g0 + lane < total) {
      const int s = visit_subtile(a0, g0 + lane);
      if (in_range(a0.status, s, 0, a0.total_st)) {
        t = subtile(a0, s);
        if (in_range(a0.status, t.inst, 0, a0.n_inst)) {
          st = s;
          if (!inst_active(a0, t.inst)) {   // a retired instance: nothing to render
            a0.wk.st[s] = make_int2(0, 0);
          } else {
            K = (int)bin[s];
            bin[s] = 0u;
            if (K == 0) a0.wk.st[s] = make_int2(0, 0);
            else listed = true;
          }
        }
      }
    }
    // pool ranges of the warp's lists: exclusive prefix sums of K over the lanes
    const int want = listed && K <= kLeafCap ? K : 0;
    int incl = want;
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
      const int y = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += y;
    }
    unsigned base = 0u;
    const int tot = __shfl_sync(full, incl, G - 1);
    if (lane == 0 && tot > 0) base = atomicAdd(&a0.wk.ctr[1], (unsigned)tot);
    base = __shfl_sync(full, base, 0);
    bool sorted = false, heavy = false;
    int Kc = 0, C = 0;
    long long off = 0;
    if (listed) {
      off = (long long)base + incl - want;
      Kc = K;
      if (K > kLeafCap) Kc = -1;
      else if (off + K > a0.wk.pool_cap) Kc = -(K + 1);
      sorted = Kc > 0;
      if (Kc < 0) a0.wk.bvh_need[t.inst] = 1;   // traced ray by ray: the BVH boxes must be current
      a0.wk.st[st] = make_int2(sorted ? (int)off : 0, Kc);
      C = chunks_for(a0, Kc, t.spp);
      heavy = heavy_item(a0, Kc, C, t.spp);
    }
    place_items<G>(a0, listed, st, t.inst, Kc, C, heavy);
    const unsigned sm = __ballot_sync(full, sorted);
    int lb = 0;
    if (lane == 0 && sm) lb = (int)atomicAdd(&a0.wk.ctr[ctr_sort(a0.n_inst)], (unsigned)__popc(sm));
    lb = __shfl_sync(full, lb, 0);
    if (sorted) a0.wk.cand_st[lb + __popc(sm & lanemask_lt())] = make_int4(st, (int)off, Kc, 0);
  }
}

// Pixels of the sub-tiles whose bins hold no record: the background (the value
// write_pixel gives a sub-tile whose samples all miss).  Each warp takes kGroupSubtiles
// consecutive sub-tiles, one per lane of its first lanes, then writes the background
// ones, lane = pixel, every background load issued before the first store.  Runs on
// the context's second stream beside the fill and the sort, which touch no pixel.
template <bool STATS>
__global__ void __launch_bounds__(kGroupThreads) k_background(RenderArgs a0, float* __restrict__ image,
                                                             unsigned long long* stats) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  Counts cnt;
  const int total = visit_count(a0);
  const int nw = gridDim.x * (kGroupThreads / 32);
  for (int g0 = (blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5)) * kGroupSubtiles; g0 < total;
       g0 += nw * kGroupSubtiles) {
    bool background = false;
    SubTile t{};
    if (lane < kGroupSubtiles && g0 + lane < total) {
      const int s = visit_subtile(a0, g0 + lane);
      if (in_range(a0.status, s, 0, a0.total_st)) {
        t = subtile(a0, s);
        background = in_range(a0.status, t.inst, 0, a0.n_inst) && inst_active(a0, t.inst) && a0.wk.st[s].y == 0;
      }
    }
    const unsigned cm = __ballot_sync(full, background);
    if (!cm) continue;
    float3 bgv[kGroupSubtiles];
    size_t pix[kGroupSubtiles];
    bool valid[kGroupSubtiles];
#pragma unroll
    for (int j = 0; j < kGroupSubtiles; ++j) {
      const int x0 = __shfl_sync(full, t.x0, j), y0 = __shfl_sync(full, t.y0, j);
      const int W = __shfl_sync(full, t.W, j), H = __shfl_sync(full, t.H, j);
      const long long p0 = __shfl_sync(full, t.pix0, j);
      const int px = x0 + (lane % kSubW), py = y0 + (lane / kSubW);
      valid[j] = ((cm >> j) & 1u) && px < W && py < H;
      pix[j] = (size_t)p0 + (size_t)py * W + px;
      bgv[j] = valid[j] ? ld3(a0.bg + 3 * pix[j]) : make_float3(0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int j = 0; j < kGroupSubtiles; ++j) {
      const int spp = __shfl_sync(full, t.spp, j);
      if (!valid[j]) continue;
      if (STATS) cnt.samples += spp;   // resolved by the binning: no record meets the sub-tile
      const float fm = __fdiv_rn((float)spp, (float)spp);
      const float inv_spp = 1.0f / (float)spp;
      image[3 * pix[j]] = 0.0f * inv_spp + bgv[j].x * fm;
      image[3 * pix[j] + 1] = 0.0f * inv_spp + bgv[j].y * fm;
      image[3 * pix[j] + 2] = 0.0f * inv_spp + bgv[j].z * fm;
    }
  }
  flush_counts<STATS>(cnt, stats);
}

// A list of K <= 32 E records sorted by (depth, place in the list), E per lane in
// registers: the keys by a bitonic network (strides below E within a lane, the others by
// shuffles), then the boxes and the records through the warp's shared memory to their new
// places.  With the keys in shared memory each of the 21 to 45 stages cost two dependent
// accesses and a barrier, and the boxes were projected again: 128 pairs of views 560 -> 235
// us, 64 hands 452 -> 264 us, a 24.6 k-triangle hand 178 -> 57 us, two views of 128 x 128
// (lists of up to 500) 68 -> 15 us.
template <int E>
__device__ __forceinline__ void sort_in_registers(const RenderArgs& a, int off, int K, float4* sm) {
  typedef unsigned long long u64;
  const int lane = threadIdx.x & 31;
  u64 r[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane + 32 * e;
    r[e] = ~0ull;
    if (i < K) {   // unsigned order of the bits = the floats' order
      const unsigned b = __float_as_uint(a.wk.z[off + i]);
      r[e] = (u64)(b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u)) << 32 | (unsigned)i;
    }
  }
  // (loops over the stages: unrolled, 16 keys are 70 KB of instructions, which a warp reads
  // once and waits for)
#pragma unroll 1
  for (int size = 2; size <= 32 * E; size <<= 1) {
#pragma unroll 1
    for (int j = size >> 1; j >= E; j >>= 1) {
      const bool low = !((lane * E) & j) == !((lane * E) & size);   // this lane keeps the smaller keys
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const u64 o = __shfl_xor_sync(0xffffffffu, r[e], j / E);
        if ((o < r[e]) == low) r[e] = o;
      }
    }
#pragma unroll
    for (int j = E / 2; j > 0; j >>= 1) {
      if (j > size >> 1) continue;
#pragma unroll
      for (int e = 0; e < E; ++e) {   // lane's keys E lane .. E lane + E - 1
        if (e & j) continue;
        const bool up = !((lane * E + e) & size), swap = (r[e + j] < r[e]) == up;
        const u64 x = r[e], y = r[e + j];
        r[e] = swap ? y : x;
        r[e + j] = swap ? x : y;
      }
    }
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (lane + 32 * e < K) sm[lane + 32 * e] = a.wk.bb[off + lane + 32 * e];
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane * E + e;
    if (i >= K) continue;
    const unsigned b = (unsigned)(r[e] >> 32);
    a.wk.bb[off + i] = sm[(unsigned)r[e]];
    a.wk.z[off + i] = __uint_as_float(b ^ ((b >> 31) ? 0x80000000u : 0xffffffffu));
  }
  __syncwarp();
  uint2* sr = reinterpret_cast<uint2*>(sm);
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (lane + 32 * e < K) sr[lane + 32 * e] = make_uint2((unsigned)a.wk.rec[off + lane + 32 * e], a.wk.pm[off + lane + 32 * e]);
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane * E + e;
    if (i >= K) continue;
    const uint2 v = sr[(unsigned)r[e]];
    a.wk.rec[off + i] = (int)v.x;
    a.wk.pm[off + i] = v.y;
  }
  __syncwarp();
}

// one warp per listed sub-tile: its K records (in fill order) sorted by nearest depth
// (bitonic, padded with +inf, across the lanes' registers), written back in order
__global__ void __launch_bounds__(kRenderThreads, 7) k_bin_sort(RenderArgs a0) {
  pdl_wait();
  __shared__ float4 staged[kWarps][kLeafCap];
  float4* sm = staged[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int n = (int)min(*reinterpret_cast<volatile unsigned*>(&a0.wk.ctr[ctr_sort(a0.n_inst)]),
                         (unsigned)a0.total_st);
  for (int vi = blockIdx.x * kWarps + (threadIdx.x >> 5); vi < n; vi += gridDim.x * kWarps) {
    const int4 cd = a0.wk.cand_st[vi];
    const int st = cd.x, off = cd.y, K = cd.z;
    if (!in_range(a0.status, st, 0, a0.total_st)) continue;
    if (lane == 0) a0.wk.bin[st] = 0u;   // the fill's slot counter, clear for the next forward
    if (K <= 0 || K > kLeafCap || off < 0 || !in_range(a0.status, (long long)off + K - 1, 0, a0.wk.pool_cap)) continue;
    if (K <= 32) {
      // one record per lane (depth, box and index as the fill wrote them), a bitonic
      // sort of (depth, lane) across the warp; lane c then takes the c-th record's box
      // and index from its lane
      int k = 0;
      unsigned pm = 0u;
      float4 bb = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      float key = INFINITY;
      if (lane < K) {
        k = a0.wk.rec[off + lane];
        pm = a0.wk.pm[off + lane];
        key = a0.wk.z[off + lane];
        bb = a0.wk.bb[off + lane];
      }
      int src = lane;
#pragma unroll
      for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
          const float ok = __shfl_xor_sync(0xffffffffu, key, stride);
          const int os = __shfl_xor_sync(0xffffffffu, src, stride);
          const bool take_min = ((lane & stride) == 0) == ((lane & size) == 0);
          const bool take = take_min ? (ok < key || (ok == key && os < src)) : (ok > key || (ok == key && os > src));
          if (take) {
            key = ok;
            src = os;
          }
        }
      }
      const int kc = __shfl_sync(0xffffffffu, k, src);
      const unsigned pc = __shfl_sync(0xffffffffu, pm, src);
      const float4 bc = make_float4(__shfl_sync(0xffffffffu, bb.x, src), __shfl_sync(0xffffffffu, bb.y, src),
                                    __shfl_sync(0xffffffffu, bb.z, src), __shfl_sync(0xffffffffu, bb.w, src));
      if (lane < K) {
        a0.wk.bb[off + lane] = bc;
        a0.wk.z[off + lane] = key;
        a0.wk.rec[off + lane] = kc;
        a0.wk.pm[off + lane] = pc;
      }
      continue;
    }
    if (K <= 64) sort_in_registers<2>(a0, off, K, sm);
    else if (K <= 128) sort_in_registers<4>(a0, off, K, sm);
    else if (K <= 256) sort_in_registers<8>(a0, off, K, sm);
    else sort_in_registers<16>(a0, off, K, sm);
    static_assert(kLeafCap <= 512, "16 records per lane");
  }
}

// The backward's own candidate lists (without HR_BWD_REUSE_FWD): one warp per
// sub-tile with a non-zero adjoint walks the BVH with the sub-tile's frustum,
// collects the records it meets into the pool sorted by nearest depth, and allocates
// the sub-tile's work items in its instance's region of the item table; sub-tiles
// whose frustum meets nothing have no interior gradient.  When the pool or the item
// region is full the sub-tile is traced ray by ray or done whole by k_overflow.
template <bool STATS>
__global__ void __launch_bounds__(kRenderThreads) k_gather(RenderArgs a_in, const float* __restrict__ adjoint,
                                                          unsigned long long* stats) {
  const RenderArgs a0 = with_iter(a_in);
  __shared__ GatherSmem gsm[kWarps];
  GatherSmem& gs = gsm[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  Counts cnt;
  const int total = visit_count(a0);
  for (;;) {
    int vi = 0;
    if (lane == 0) vi = (int)atomicAdd(&a0.wk.ctr[0], 1u);
    vi = __shfl_sync(0xffffffffu, vi, 0);
    if (vi >= total) break;
    const int st = visit_subtile(a0, vi);
    if (!in_range(a0.status, st, 0, a0.total_st)) continue;
    const SubTile t = subtile(a0, st);
    if (!in_range(a0.status, t.inst, 0, a0.n_inst)) continue;
    if (!inst_active(a0, t.inst)) {   // a retired instance: nothing to render
      if (lane == 0) a0.wk.st[st] = make_int2(0, 0);
      continue;
    }
    const RenderArgs a = for_inst(a0, t.inst);
    bool live;
    lane_adjoint(a, t, adjoint, live);
    if (!__any_sync(0xffffffffu, live)) {
      if (lane == 0) a.wk.st[st] = make_int2(0, 0);
      continue;
    }
    const Cam cam = load_cam(a.cams, t.view);
    int K = frustum_leaves<STATS>(a, cam, t.x0, t.y0, gs, cnt);
    if (K == 0) {
      if (lane == 0) a.wk.st[st] = make_int2(0, 0);
      const int px = t.x0 + (lane % kSubW), py = t.y0 + (lane / kSubW);
      if (STATS && px < t.W && py < t.H && live) cnt.samples += t.spp;   // resolved by the frustum test
      continue;
    }
    int off = 0;
    if (K > 0) {
      // sort the candidates by nearest depth (bitonic, padded with +inf)
      for (int j = lane; j < K; j += 32) {
        float4 bb;
        float zm;
        int k = gs.leaf[j];
        if (!in_range(a.status, k, 0, a.max_visits - 1)) k = 0;
        gs.leaf[j] = k;
        project_record(a, cam, k, bb, zm);
        gs.key[j] = zm;
        gs.idx[j] = j;
      }
      int P = 1;
      while (P < K) P <<= 1;
      for (int j = K + lane; j < P; j += 32) {
        gs.key[j] = INFINITY;
        gs.idx[j] = 0;
      }
      __syncwarp();
      for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
          for (int i = lane; i < P; i += 32) {
            int ixj = i ^ j;
            if (ixj > i) {
              float zi = gs.key[i], zj = gs.key[ixj];
              bool up = (i & k) == 0;
              if ((zi > zj) == up) {
                gs.key[i] = zj;
                gs.key[ixj] = zi;
                int q = gs.idx[i];
                gs.idx[i] = gs.idx[ixj];
                gs.idx[ixj] = q;
              }
            }
          }
          __syncwarp();
        }
      }
      if (lane == 0) off = (int)atomicAdd(&a.wk.ctr[1], (unsigned)K);
      off = __shfl_sync(0xffffffffu, off, 0);
      if (off + K <= a.wk.pool_cap) {
        for (int c = lane; c < K; c += 32) {
          int j = gs.idx[c];
          if (!in_range(a.status, j, 0, K)) j = 0;
          const int k = gs.leaf[j];
          float4 bb;
          float zm;
          project_record(a, cam, k, bb, zm);
          a.wk.bb[off + c] = bb;
          a.wk.z[off + c] = zm;
          a.wk.rec[off + c] = k;
          a.wk.pm[off + c] = box_pixel_mask(bb, t.x0, t.y0);
        }
      } else {
        // pool full: per-ray traversal for this sub-tile, with K's count kept as
        // -(K + 1) so that its work items are split as they would be with the list
        K = -(K + 1);
      }
    }
    const int C = chunks_for(a, K, t.spp);
    const int ibase = inst_ibase(a, t.inst), icap = inst_icap(a, t.inst);
    int first = 0;
    if (lane == 0) first = alloc_items(a, t.inst, C, heavy_item(a, K, C, t.spp), icap);
    first = __shfl_sync(0xffffffffu, first, 0);
    if (lane == 0) a.wk.st[st] = make_int2(off, K);
    if (first >= 0) {
      for (int c = lane; c < C; c += 32) a.wk.items[ibase + first + c] = make_int4(st, c, C, ibase + first);
      if (K < 0) note_trace_items(a, ibase + first, C);
    } else if (lane == 0) {
      // item region full: the whole sub-tile goes to k_overflow
      a.wk.ovf[atomicAdd(&a.wk.ctr[2 + 2 * a.n_inst], 1u)] = st;
    }
    __syncwarp();
  }
  flush_counts<STATS>(cnt, stats);
}

// The backward's work items from the forward's candidate lists (HR_BWD_REUSE_FWD).
// Each warp takes kGroupSubtiles consecutive sub-tiles, one per lane of its first lanes;
// only sub-tiles with a candidate list (or per-ray traversal) read the adjoint, the
// whole warp loading all of them first (lane = pixel), and those with a non-zero
// adjoint get their work items (place_items).
template <bool STATS>
__global__ void __launch_bounds__(kGroupThreads, 4) k_items_bwd(RenderArgs a0, const float* __restrict__ adjoint,
                                                               unsigned long long* stats) {
  pdl_wait();
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  Counts cnt;
  const int total = visit_count(a0);
  const int nw = gridDim.x * (kGroupThreads / 32);
  for (int g0 = (blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5)) * kGroupSubtiles; g0 < total;
       g0 += nw * kGroupSubtiles) {
    int st = -1;
    int2 pk = make_int2(0, 0);
    bool ok = false;
    SubTile t{};
    if (lane < kGroupSubtiles && g0 + lane < total) {
      const int s = visit_subtile(a0, g0 + lane);
      if (in_range(a0.status, s, 0, a0.total_st)) {
        t = subtile(a0, s);
        if (in_range(a0.status, t.inst, 0, a0.n_inst) && inst_active(a0, t.inst)) {
          st = s;
          ok = true;
          pk = a0.wk.st[s];
          if (pk.y > 0 && !in_range(a0.status, (long long)pk.x + pk.y - 1, 0, a0.wk.pool_cap)) pk.y = -1;
        }
      }
    }
    // sub-tile j's pixels: lane = pixel; every adjoint load issued before the tests
    const unsigned look = __ballot_sync(full, ok && (STATS || pk.y != 0));
    if (!look) continue;
    float3 g[kGroupSubtiles];
    bool valid[kGroupSubtiles];
#pragma unroll
    for (int j = 0; j < kGroupSubtiles; ++j) {
      const int x0 = __shfl_sync(full, t.x0, j), y0 = __shfl_sync(full, t.y0, j);
      const int W = __shfl_sync(full, t.W, j), H = __shfl_sync(full, t.H, j);
      const long long p0 = __shfl_sync(full, t.pix0, j);
      const int px = x0 + (lane % kSubW), py = y0 + (lane / kSubW);
      valid[j] = ((look >> j) & 1u) && px < W && py < H;
      g[j] = valid[j] ? ld3(adjoint + 3 * ((size_t)p0 + (size_t)py * W + px)) : make_float3(0.0f, 0.0f, 0.0f);
    }
    unsigned live = 0u;
#pragma unroll
    for (int j = 0; j < kGroupSubtiles; ++j) {
      const bool lj = valid[j] && (g[j].x != 0.0f || g[j].y != 0.0f || g[j].z != 0.0f);
      if (__ballot_sync(full, lj)) live |= 1u << j;
      const int kj = __shfl_sync(full, pk.y, j), sppj = __shfl_sync(full, t.spp, j);
      if (STATS && lj && kj == 0) cnt.samples += sppj;   // no ray of the sub-tile can hit
    }
    const bool need = ok && ((live >> lane) & 1u) && pk.y != 0;
    const int C = need ? chunks_for(a0, pk.y, t.spp) : 0;
    const bool heavy = need && heavy_item(a0, pk.y, C, t.spp);
    place_items<kGroupSubtiles>(a0, need, st, t.inst, pk.y, C, heavy);
  }
  write_face_records(a0);   // for the shader that follows
  flush_counts<STATS>(cnt, stats);
}

// items of an instance's region that the gather filled (front and back)
__device__ __forceinline__ int front_count(const RenderArgs& a, int inst) {
  return (int)min(*reinterpret_cast<volatile unsigned*>(&a.wk.ctr[2 + 2 * inst]), (unsigned)inst_icap(a, inst));
}
__device__ __forceinline__ int item_count(const RenderArgs& a, int inst) {
  const unsigned b = *reinterpret_cast<volatile unsigned*>(back_count(a, inst));
  return (int)min((unsigned)front_count(a, inst) + b, (unsigned)inst_icap(a, inst));
}
// region slot of the instance's i-th item (0 <= i < item_count): the front items,
// heavy, first; then the back items from the region's end
__device__ __forceinline__ int item_slot(const RenderArgs& a, int inst, int i, int nfront) {
  return i < nfront ? i : inst_icap(a, inst) - 1 - (i - nfront);
}

__device__ __forceinline__ void item_samples(int c, int C, int spp, int& s0, int& s1) {
  s0 = (int)((long long)c * spp / C);
  s1 = (int)((long long)(c + 1) * spp / C);
}

// A warp's place in the work items.  Each instance's items are handed out from one
// counter, in runs of `run` consecutive items (several per warp are left to balance the
// load): consecutive items are mostly of one sub-tile, whose candidates the shaders
// then stage once.  A run is asked for when the one before is done: asked for with the
// run's last item, so that the counter's round trip passed beside the shading, it made a
// warp with a long item hold the next one too (paper step, forward 76 -> 58 us, backward
// 88 -> 70; 5 views of 125 x 336, 52 spp, 6 k triangles 265 -> 162 and 250 -> 157).  The blocks of an SM
// start on one instance (its triangles stay in the SM's L1) and the instances are
// spread over the SMs; a warp whose instance has run out looks for one with items left,
// 32 at a time.
struct Cursor {
  int inst;            // instance, -1 before the first
  int n, nf, run;      // its items, front items and run length
  int pos, end;        // the rest of the current run
};
constexpr int kMaxRun = 16;

__device__ __forceinline__ void enter_instance(const RenderArgs& a, Cursor& c, int inst) {
  c.inst = inst;
  c.n = item_count(a, inst);
  c.nf = front_count(a, inst);
  // about eight runs per warp if every warp had its share of the instances
  const long long warps = max(1LL, (long long)gridDim.x * (blockDim.x / 32) / a.n_inst);
  c.run = (int)min((long long)kMaxRun, max(1LL, c.n / (8 * warps)));
  c.pos = c.end = 0;
}

__device__ __forceinline__ Cursor start_items(const RenderArgs& a) {
  Cursor c;
  // the blocks an SM holds at once differ by the number of SMs
  const int sms = max(1, a.num_sms), home = (int)((long long)(blockIdx.x % sms) * a.n_inst / sms);
  enter_instance(a, c, home);
  return c;
}

// the next item (region slot in `slot`, without the instance's base); false at the end
__device__ __forceinline__ bool next_item(const RenderArgs& a, Cursor& c, int& slot) {
  const unsigned full = 0xffffffffu;
  for (;;) {
    if (c.pos < c.end) {
      slot = item_slot(a, c.inst, c.pos++, c.nf);
      return true;
    }
    if (c.n > 0) {
      int first = 0;
      if ((threadIdx.x & 31) == 0) first = (int)atomicAdd(&a.wk.ctr[3 + 2 * c.inst], (unsigned)c.run);
      c.pos = __shfl_sync(full, first, 0);
      if (c.pos < c.n) {   // (a negative position could only come from a wrapped counter)
        c.pos = max(c.pos, 0);
        c.end = min(c.pos + c.run, c.n);
        continue;
      }
      c.pos = c.end = 0;
    }
    int found = -1;
    for (int base = 1; base < a.n_inst && found < 0; base += 32) {
      const int k = base + (threadIdx.x & 31);
      int inst = c.inst + k;
      if (inst >= a.n_inst) inst -= a.n_inst;
      bool left = false;
      if (k < a.n_inst) {
        const unsigned taken = *reinterpret_cast<volatile unsigned*>(&a.wk.ctr[3 + 2 * inst]);
        left = taken < (unsigned)item_count(a, inst);
      }
      const unsigned b = __ballot_sync(full, left);
      if (b) found = __shfl_sync(full, inst, __ffs(b) - 1);
    }
    if (found < 0) return false;
    enter_instance(a, c, found);
  }
}

// the sub-tile and candidate list of an item; false for a blanked or corrupt item
__device__ __forceinline__ bool load_item(const RenderArgs& a, const int4& item, SubTile& t, int2& pk) {
  if (item.x < 0) return false;   // a blanked slot
  if (!in_range(a.status, item.x, 0, subtile_count(a))) return false;
  t = subtile(a, item.x);
  if (!in_range(a.status, t.inst, 0, a.n_inst)) return false;
  pk = a.wk.st[item.x];
  if (pk.y > 0 && !in_range(a.status, (long long)pk.x + pk.y - 1, 0, a.wk.pool_cap)) pk.y = -1;
  return true;
}

// A forward work item is done (all lanes call): a sub-tile with one item writes its
// pixels at once; otherwise the item's radiance sums go to its slot of the partials,
// and the warp that finishes the sub-tile's last item (a per-sub-tile counter) adds
// the C partials in item order and writes the pixels -- the same sums, in the same
// order, whichever warps traced the items.
__device__ __forceinline__ void finish_item(const RenderArgs& a, const SubTile& t, const int4& item, int slot,
                                            float3 acc, int misses, float* __restrict__ image) {
  const int lane = threadIdx.x & 31;
  if (item.z == 1) {
    write_pixel(a, t, acc, misses, image);
    return;
  }
  a.wk.part[(size_t)slot * 32 + lane] = make_float4(acc.x, acc.y, acc.z, (float)misses);
  // every lane's sums are visible device-wide before lane 0 counts the item (the fence
  // orders each lane's own store; the warp barrier puts all of them before the count)
  __threadfence();
  __syncwarp();
  unsigned prev = 0;
  if (lane == 0) prev = atomicAdd(&a.wk.st_done[item.x], 1u);
  prev = __shfl_sync(0xffffffffu, prev, 0);
  if (prev != (unsigned)item.z - 1u) return;
  __threadfence();
  if (!in_range(a.status, (long long)item.w + item.z - 1, 0, a.wk.item_cap)) return;
  float3 tot = make_float3(0.0f, 0.0f, 0.0f);
  float tmiss = 0.0f;
  for (int c = 0; c < item.z; ++c) {
    const float4 p = __ldcg(&a.wk.part[(size_t)(item.w + c) * 32 + lane]);   // written on other SMs
    tot.x += p.x;
    tot.y += p.y;
    tot.z += p.z;
    tmiss += p.w;
  }
  write_pixel(a, t, tot, (int)tmiss, image);
  if (lane == 0) a.wk.st_done[item.x] = 0u;   // ready for the next launch
}

// warps take work items; S samples per lane at a time.  The sub-tile's description, its
// camera and its candidates are kept in the warp's shared memory from item to item.
// Bound by instruction issue (50 % active, 20 of 32 lanes, 31 M warp instructions on 8 x
// 512x384 at 16 spp) with the latency of the items' chains beside it.  Against a walk that
// took every candidate's box and record through shuffles and global loads for each group
// of samples: 106 -> 59 us there; 64 hands, 612 views: 6.45 -> 2.99 ms; 1024 views of 256^2
// at 4 spp, whose items hold one sample: 2.52 -> 0.90 ms.
template <bool STATS, int S>
__global__ void __launch_bounds__(kRenderThreads, kFwdMinBlocks) k_shade_fwd(RenderArgs a_in, float* __restrict__ image,
                                                                             unsigned long long* stats) {
  pdl_wait();
  __shared__ WarpTile tiles[kWarps];
  WarpTile& wt = tiles[threadIdx.x >> 5];
  const RenderArgs a0 = with_iter(a_in);
  Counts cnt;
  Cursor cur = start_items(a0);
  int at = -1, K = 0, off = 0, slot;   // the sub-tile staged
  unsigned m0 = 0u;
  while (next_item(a0, cur, slot)) {
    const int gi = inst_ibase(a0, cur.inst) + slot;
    const int4 item = a0.wk.items[gi];
    if (item.x != at) {
      SubTile t;
      int2 pk;
      at = -1;
      if (!load_item(a0, item, t, pk) || t.inst != cur.inst) continue;
      if (pk.y < 0) continue;   // no candidate list: k_overflow traces this item
      at = item.x;
      off = pk.x;
      K = pk.y;
      const RenderArgs a = for_inst(a0, cur.inst);
      stage_tile<STATS>(a, wt, t, off, K, m0, cnt);
    }
    const RenderArgs a = for_inst(a0, cur.inst);
    int s0, s1;
    item_samples(item.y, item.z, wt.t.spp, s0, s1);
    float3 acc = make_float3(0.0f, 0.0f, 0.0f);
    int misses = 0;
    for (; s0 + S <= s1; s0 += S) shade_samples<STATS, S, false>(a, wt, off, K, m0, s0, acc, misses, cnt);
    if (S > 1)
      for (; s0 < s1; ++s0) shade_samples<STATS, 1, false>(a, wt, off, K, m0, s0, acc, misses, cnt);
    finish_item(a, wt.t, item, gi, acc, misses, image);
  }
  flush_counts<STATS>(cnt, stats);
}

template <bool STATS>
__device__ __forceinline__ void overflow_grad(const RenderArgs& a, OverflowTile& gt, int inst, int off, int K, unsigned m0,
                                              int s0, int s1, bool live, float3 g, Counts& cnt) {
  if (a.wk.det) {
    grad_samples<STATS, 1, SumFixed, true>(a, gt, off, K, m0, s0, s1, live, g, SumFixed{a.wk.fx + (size_t)inst * 6 * a.V}, cnt);
  } else {
    grad_samples<STATS, 1, SumF32, true>(a, gt, off, K, m0, s0, s1, live, g, SumF32{a.wk.extra + (size_t)inst * 8 * a.V}, cnt);
  }
}

// The rare paths, kept out of the gather and the shaders so that their registers are
// sized for their own work: (1) sub-tiles whose work items did not fit their
// instance's region -- one warp does a whole sub-tile, all its samples, in the chunks
// the items would have had (the forward writes its pixels, the backward adds to the
// instance's extra sums); (2) work items of sub-tiles without a usable candidate list
// (more candidates than the gather's list holds, or the pool full), traced ray by ray.
template <bool BWD, bool STATS>
__global__ void __launch_bounds__(kRenderThreads, BWD ? kBwdMinBlocks : 8) k_overflow(RenderArgs a_in,
                                                                                     const float* __restrict__ adjoint,
                                                            float* __restrict__ image, unsigned long long* stats) {
  pdl_wait();
  __shared__ WarpTile tiles[kWarps];
  WarpTile& wt = tiles[threadIdx.x >> 5];
  OverflowTile gt(wt);   // (backward)
  const RenderArgs a0 = with_iter(a_in);
  const int total = subtile_count(a0);
  const int n = (int)min(*reinterpret_cast<volatile unsigned*>(&a0.wk.ctr[2 + 2 * a0.n_inst]), (unsigned)total);
  Counts cnt;
  for (int i = blockIdx.x * kWarps + (threadIdx.x >> 5); i < n; i += gridDim.x * kWarps) {
    const int st = a0.wk.ovf[i];
    if (!in_range(a0.status, st, 0, total)) continue;
    const SubTile t = subtile(a0, st);
    if (!in_range(a0.status, t.inst, 0, a0.n_inst)) continue;
    const RenderArgs a = for_inst(a0, t.inst);
    int2 pk = a.wk.st[st];
    if (pk.y > 0 && !in_range(a.status, (long long)pk.x + pk.y - 1, 0, a.wk.pool_cap)) pk.y = -1;
    if constexpr (BWD) {
      // in the items' chunks too: each chunk's sums are added exactly as its work item
      // would add them, so fixed-point sums do not depend on which sub-tiles overflowed
      bool live;
      const float3 g = lane_adjoint(a, t, adjoint, live);
      const int C = chunks_for(a, pk.y, t.spp);
      unsigned m0;
      stage_tile<STATS>(a, wt, t, pk.x, pk.y, m0, cnt);
      for (int c = 0; c < C; ++c) {
        int s0, s1;
        item_samples(c, C, t.spp, s0, s1);
        overflow_grad<STATS>(a, gt, t.inst, pk.x, pk.y, m0, s0, s1, live, g, cnt);
      }
    } else {
      // the same chunks and the same order of sums as the work items and finish_item
      // would use, so a pixel's value does not depend on which path rendered it
      const int C = chunks_for(a, pk.y, t.spp);
      unsigned m0;
      stage_tile<STATS>(a, wt, t, pk.x, pk.y, m0, cnt);
      float3 tot = make_float3(0.0f, 0.0f, 0.0f);
      float tmiss = 0.0f;
      for (int c = 0; c < C; ++c) {
        int s0, s1;
        item_samples(c, C, t.spp, s0, s1);
        float3 acc = make_float3(0.0f, 0.0f, 0.0f);
        int misses = 0;
        for (; s0 < s1; ++s0) shade_samples<STATS, 1>(a, wt, pk.x, pk.y, m0, s0, acc, misses, cnt);
        tot.x += acc.x;
        tot.y += acc.y;
        tot.z += acc.z;
        tmiss += (float)misses;
      }
      write_pixel(a, t, tot, (int)tmiss, image);
    }
  }
  // work items of sub-tiles without a candidate list (the shaders skip them, the gather
  // lists them): traced ray by ray, the forward finishing each item as the shader
  // would, the backward adding to the instance's extra sums
  const int nt = (int)min(*reinterpret_cast<volatile unsigned*>(&a0.wk.ctr[ctr_trace(a0.n_inst)]),
                          (unsigned)a0.wk.item_cap);
  for (int i = blockIdx.x * kWarps + (threadIdx.x >> 5); i < nt; i += gridDim.x * kWarps) {
    const int slot = a0.wk.trace[i];
    if (!in_range(a0.status, slot, 0, a0.wk.item_cap)) continue;
    int4 item;
    SubTile t;
    int2 pk;
    item = a0.wk.items[slot];
    if (!load_item(a0, item, t, pk) || pk.y >= 0) continue;
    const RenderArgs a = for_inst(a0, t.inst);
    int s0, s1;
    item_samples(item.y, item.z, t.spp, s0, s1);
    if constexpr (BWD) {
      bool live;
      const float3 g = lane_adjoint(a, t, adjoint, live);
      unsigned m0;
      stage_tile<STATS>(a, wt, t, pk.x, pk.y, m0, cnt);
      overflow_grad<STATS>(a, gt, t.inst, pk.x, pk.y, m0, s0, s1, live, g, cnt);
    } else {
      float3 acc = make_float3(0.0f, 0.0f, 0.0f);
      int misses = 0;
      unsigned m0;
      stage_tile<STATS>(a, wt, t, pk.x, pk.y, m0, cnt);
      for (; s0 < s1; ++s0) shade_samples<STATS, 1>(a, wt, pk.x, pk.y, m0, s0, acc, misses, cnt);
      finish_item(a, t, item, slot, acc, misses, image);
    }
  }
  flush_counts<STATS>(cnt, stats);
}

// interior term: warps take work items.  ACC selects where the gradient collects;
// every mode adds with atomic adds whose result is not read, which retire in L2
// without holding up the warp (float adds to shared memory cost a read and a
// compare-and-swap loop each, and made the sums a quarter of this kernel's time):
//   kAccPartials  block b into partial b % nparts of `nparts` partials [V][8]
//                 (L2-resident, zeroed before the launch), summed in partial order by
//                 k_reduce_partials (single instance)
//   kAccDirect    every triangle's sums of a window straight into its instance's
//                 extra [V][8] (batches)
//   kAccGlobal    meshes beyond kPartialMaxV vertices: into the instance's float64
//                 extra64 [6V] (long runs of cancelling contributions)
//   kAccFixed     HR_DETERMINISTIC: into the instance's fixed-point sums fx [6V]
//                 (order-free integer atomics)
// Bound by instruction issue (51 % active, 17 of 32 lanes on 8 x 512x384 at 16 spp) and the
// latency of divergent loads.  With the hits of a window differentiated triangle by
// triangle instead of run by run, the candidates from the tile and vertices summed 16 bytes
// at a time: 120 -> 70 us there; 64 hands, 612 views 7.4 -> 3.9 ms (with the edge kernel
// beside it), textured 16 x 1024^2 at 64 spp 4.5 -> 2.8 ms.
constexpr int kAccPartials = 0, kAccDirect = 1, kAccGlobal = 2, kAccFixed = 3;
template <bool STATS, int ACC, int S>
__global__ void __launch_bounds__(kRenderThreads, kBwdMinBlocks) k_shade_bwd(RenderArgs a_in,
                                                                             const float* __restrict__ adjoint,
                                                                             float* __restrict__ partials, int nparts,
                                                                             unsigned long long* stats) {
  pdl_wait();
  __shared__ GradTile tiles[kWarps];
  GradTile& gt = tiles[threadIdx.x >> 5];
  const RenderArgs a0 = with_iter(a_in);
  Counts cnt;
  Cursor cur = start_items(a0);
  int at = -1, K = 0, off = 0, slot;   // the sub-tile staged
  unsigned m0 = 0u;
  bool live = false;
  float3 g = make_float3(0.0f, 0.0f, 0.0f);
  while (next_item(a0, cur, slot)) {
    const int inst = cur.inst;
    const int4 item = a0.wk.items[inst_ibase(a0, inst) + slot];
    const RenderArgs a = for_inst(a0, inst);
    if (item.x != at) {
      SubTile t;
      int2 pk;
      at = -1;
      if (!load_item(a0, item, t, pk) || t.inst != inst) continue;
      if (pk.y < 0) continue;   // no candidate list: k_overflow traces this item
      at = item.x;
      off = pk.x;
      K = pk.y;
      g = lane_adjoint(a, t, adjoint, live);
      stage_tile<STATS>(a, gt.w, t, off, K, m0, cnt);
    }
    int s0, s1;
    item_samples(item.y, item.z, gt.w.t.spp, s0, s1);
    if constexpr (ACC == kAccGlobal)
      grad_samples<STATS, S, SumF64, false>(a, gt, off, K, m0, s0, s1, live, g,
                                                     SumF64{a0.wk.extra64 + (size_t)inst * 6 * a0.V}, cnt);
    else if constexpr (ACC == kAccFixed)
      grad_samples<STATS, S, SumFixed, false>(
          a, gt, off, K, m0, s0, s1, live, g, SumFixed{a0.wk.fx + (size_t)inst * 6 * a0.V}, cnt);
    else
      grad_samples<STATS, S, SumF32, false>(
          a, gt, off, K, m0, s0, s1, live, g,
          SumF32{ACC == kAccDirect ? a0.wk.extra + (size_t)inst * 8 * a0.V
                                   : partials + (size_t)(blockIdx.x % nparts) * 8 * a0.V},
          cnt);
  }
  flush_counts<STATS>(cnt, stats);
}

// d_verts and dN from the sums: word i of the [V][8] float sums is the float extra plus
// every partial's word (and the float64 or fixed-point sum).  A block covers 32 words
// with 16 groups of threads: group g sums partials g, g + 16, ... in order, then the 16
// group sums are added in group order (a fixed order for every call).  blockIdx.y
// selects the instance (a batch has no partials).
constexpr int kRedEntries = 32, kRedGroups = 16;
__global__ void __launch_bounds__(kRedEntries * kRedGroups) k_reduce_partials(
    const float* __restrict__ partials, const float* __restrict__ extra_all, const double* __restrict__ extra64_all,
    const unsigned long long* __restrict__ fx_all, int nblocks, int V, float* __restrict__ d_verts_all,
    float* __restrict__ dN_all) {
  pdl_wait();
  __shared__ float red[kRedGroups][kRedEntries];
  const int j = threadIdx.x % kRedEntries, g = threadIdx.x / kRedEntries;
  const int i = blockIdx.x * kRedEntries + j;
  float acc = 0.0f;
  if (i < 8 * V) {
#pragma unroll 4
    for (int b = g; b < nblocks; b += kRedGroups) acc += partials[(size_t)b * 8 * V + i];
  }
  red[g][j] = acc;
  __syncthreads();
  const int v = i / 8, c = i % 8;
  if (g != 0 || i >= 8 * V || (c & 3) == 3) return;
  float* d_verts = d_verts_all + (size_t)blockIdx.y * 3 * V;
  float* dN = dN_all + (size_t)blockIdx.y * 3 * V;
  const size_t wide = (size_t)blockIdx.y * 6 * V + (c < 3 ? 3 * v + c : 3 * V + 3 * v + c - 4);
  float tot = extra_all[(size_t)blockIdx.y * 8 * V + i];
  if (extra64_all) tot = (float)(extra64_all[wide] + (double)tot);
  if (fx_all) tot += from_fixed(fx_all[wide]);
  for (int q = 0; q < kRedGroups; ++q) tot += red[q][j];
  if (c < 3) d_verts[3 * v + c] = tot;
  else dN[3 * v + c - 4] = tot;
}

// per view: silhouette flags in edge order, compacted by a block-wide scan.  In a
// batch the view's instance (view table) selects the vertices ([V][3] per instance).
__global__ void k_silhouettes(const float* __restrict__ verts_all, const int* __restrict__ faces,
                              const int* __restrict__ edges, const int* __restrict__ edge_faces, int E,
                              const Cam* __restrict__ cams, const ViewRec* __restrict__ vt, int V,
                              int* __restrict__ lists, int stride, int* __restrict__ counts,
                              const int* __restrict__ active) {
  __shared__ int warp_tot[32];
  __shared__ int base;
  const int view = blockIdx.x;
  if (vt && active && !active[__ldg(&vt[view].inst)]) return;   // a retired instance
  const float* verts = verts_all + (vt ? (size_t)__ldg(&vt[view].inst) * 3 * V : 0);
  Cam cam = load_cam(cams, view);
  float3 c = make_float3(cam.c[0], cam.c[1], cam.c[2]);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int e0 = 0; e0 < E; e0 += blockDim.x) {
    int e = e0 + threadIdx.x;
    bool sil = false;
    if (e < E) {
      int f2 = edge_faces[2 * e + 1];
      if (f2 < 0) {
        sil = true;
      } else {
        float3 w = dsub(ld3(verts + 3 * edges[2 * e]), c);
        int f1 = edge_faces[2 * e];
        bool s[2];
        int fs[2] = {f1, f2};
        for (int k = 0; k < 2; ++k) {
          int f = fs[k];
          float3 p0 = ld3(verts + 3 * faces[3 * f]), p1 = ld3(verts + 3 * faces[3 * f + 1]),
                 p2 = ld3(verts + 3 * faces[3 * f + 2]);
          s[k] = ddot(dcross(dsub(p1, p0), dsub(p2, p0)), w) < 0.0f;
        }
        sil = s[0] != s[1];
      }
    }
    unsigned bal = __ballot_sync(0xffffffffu, sil);
    int within = __popc(bal & ((1u << lane) - 1u));
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    int before = 0, chunk = 0;
    for (int k = 0; k < nw; ++k) {
      int t = warp_tot[k];
      if (k < warp) before += t;
      chunk += t;
    }
    if (sil) lists[(size_t)view * stride + base + before + within] = e;
    __syncthreads();
    if (threadIdx.x == 0) base += chunk;
    __syncthreads();
  }
  if (threadIdx.x == 0) counts[view] = base;
}

// nearer of two hits: smaller t, then the lower triangle id (a miss loses)
__device__ __forceinline__ bool nearer(const Hit& m, const Hit& h) {
  return m.tri >= 0 && (h.tri < 0 || m.t < h.t || (m.t == h.t && m.tri < h.tri));
}

// the nearest hit of a group of L lanes (all 32 lanes call; the result is the same in
// every lane of a group)
template <int L>
__device__ __forceinline__ Hit group_min(Hit m) {
#pragma unroll
  for (int sh = L / 2; sh > 0; sh >>= 1) {
    Hit o;
    o.t = __shfl_xor_sync(0xffffffffu, m.t, sh, L);
    o.tri = __shfl_xor_sync(0xffffffffu, m.tri, sh, L);
    o.u = __shfl_xor_sync(0xffffffffu, m.u, sh, L);
    o.v = __shfl_xor_sync(0xffffffffu, m.v, sh, L);
    if (nearer(o, m)) m = o;
  }
  return m;
}

// boundary term (edge sampling).  A warp takes 32 / L samples, L lanes each: sample i
// of the launch is i % Ne_max of global view i / Ne_max (views with fewer samples skip
// the rest).  The lanes of a group compute the sample's set-up redundantly (same
// values, broadcast loads), then search the depth-sorted candidates of the sub-tile under
// the sample in windows of 32: lane q of the group first tests the boxes of candidates q,
// q + L, ... against the points of both offset rays (f+ and f-), loads that do not wait for
// one another, and only then intersects those that passed, each ray keeping the lane's
// nearest hit (t, then the lower triangle id); the group's nearest is taken once per window.
// Candidate by candidate, box and triangle were a chain of four dependent loads and the
// group's minimum a dozen shuffles per step, and few boxes hold a point.  Bound by latency
// at few samples and by the lanes' unequal numbers of triangles at many: a batch of 64
// hands 3.45 -> 1.40 ms, a 24.6 k-triangle hand 1.08 -> 0.45 ms, a step of two 128 x 128 views
// with 2048 samples 308 -> 255 us in all.  A ray stops at the first window whose nearest
// depth lies beyond its hit: the hits are those of testing the candidates one by one in
// depth order.  The group's lanes add the six results (two endpoints x three coordinates).
__device__ __forceinline__ void add1(float* p, float x) { atomicAdd(p, x); }
__device__ __forceinline__ void add1(unsigned long long* p, float x) { add_fixed(p, x); }

constexpr int kEdgeWin = 32;   // candidates whose boxes are tested before any is intersected
// T: float sums (dedge [n_inst][3V]) or fixed-point sums (fx [n_inst][6V], dV part);
// L: lanes per sample (the tuning's edge_lanes)
template <bool STATS, class T, int L>
__global__ void __launch_bounds__(kRenderThreads) k_edge_samples(RenderArgs a_in, const float* __restrict__ adjoint,
                                                                 const int* __restrict__ edges,
                                                                 const int* __restrict__ lists, int stride,
                                                                 const int* __restrict__ counts, int Ne_max, float eps,
                                                                 T* __restrict__ d_verts_all, long long inst_stride,
                                                                 unsigned long long* stats) {
  static_assert(L == 1 || L == 2 || L == 4 || L == 8 || L == 16 || L == 32, "lanes per edge sample");
  const unsigned full = 0xffffffffu;
  const RenderArgs a0 = with_iter(a_in);
  const int lane = threadIdx.x & 31, q = lane % L;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long i = warp * (32 / L) + lane / L;
  const int nv = visit_views(a0);
  if (warp * (32 / L) >= (long long)nv * Ne_max) return;   // whole warps leave together
  Counts cnt;
  // ---- set-up (group-uniform); `active` groups go on to the search -------------
  bool active = i < (long long)nv * Ne_max;
  const int jv = active ? (int)(i / Ne_max) : 0, k = active ? (int)(i - (long long)jv * Ne_max) : 0;
  const int view = active ? visit_view(a0, jv) : 0;
  active = active && in_range(a0.status, view, 0, a0.nviews);
  SubTile vw;
  int st0 = 0, nsx = 1;
  RenderArgs a = a0;
  T* d_verts = d_verts_all;
  int nsil = 0, ia = 0, ib = 0, K = 0, off = 0, W = 1;
  float ax = 0.f, ay = 0.f, bx = 0.f, by = 0.f, x = 0.f, y = 0.f, xp = 0.f, yp = 0.f, xm = 0.f, ym = 0.f;
  int bxp = 0, byp = 0, bxm = 0, bym = 0;
  float3 A = make_float3(0.f, 0.f, 0.f), va = A, vb = A, dp = A, dm = A, o = A;
  Cam cam;
  if (active) {
    view_info(a0, view, vw, st0, nsx);
    const int Ne = a0.vt ? __ldg(&a0.vt[view].ne) : Ne_max;
    active = k < Ne && in_range(a0.status, vw.inst, 0, a0.n_inst) && inst_active(a0, vw.inst);
    if (active) {
      a = for_inst(a0, vw.inst);
      d_verts = d_verts_all + (size_t)vw.inst * inst_stride;
      nsil = counts[view];
      active = nsil > 0;
    }
    if (active) {
      const uint4 r = philox4x32_10(make_uint4((uint32_t)k, vw.ctr1, 0u, a.iter4 | 1u), a.key);
      const int si = (int)__umulhi(r.x, (uint32_t)nsil);
      const float t = u24(r.y);
      const int e = lists[(size_t)view * stride + si];
      ia = edges[2 * e];
      ib = edges[2 * e + 1];
      cam = load_cam(a.cams, view);
      va = ld3(a.verts + 3 * ia);
      vb = ld3(a.verts + 3 * ib);
      active = project(cam, va, ax, ay) && project(cam, vb, bx, by);
      if (active) {
        x = __fmaf_rn(t, __fsub_rn(bx, ax), ax);
        y = __fmaf_rn(t, __fsub_rn(by, ay), ay);
        const float nx = __fsub_rn(ay, by), ny = __fsub_rn(bx, ax);
        const float len = __fsqrt_rn(__fmaf_rn(nx, nx, __fmul_rn(ny, ny)));
        active = len > 0.0f;
        if (active) {
          const float nhx = __fdiv_rn(nx, len), nhy = __fdiv_rn(ny, len);
          const float fxp = floorf(x), fyp = floorf(y);
          W = vw.W;
          const int H = vw.H;
          active = !(fxp < 0.0f || fyp < 0.0f || fxp >= (float)W || fyp >= (float)H);
          if (active) {
            const int px = (int)fxp, py = (int)fyp;
            A = ld3(adjoint + 3 * (vw.pix0 + (size_t)py * W + px));
            active = A.x != 0.0f || A.y != 0.0f || A.z != 0.0f;
            if (active) {
              xp = __fmaf_rn(eps, nhx, x);
              yp = __fmaf_rn(eps, nhy, y);
              xm = __fmaf_rn(-eps, nhx, x);
              ym = __fmaf_rn(-eps, nhy, y);
              bxp = (int)fminf(fmaxf(floorf(xp), 0.0f), (float)(W - 1));
              byp = (int)fminf(fmaxf(floorf(yp), 0.0f), (float)(H - 1));
              bxm = (int)fminf(fmaxf(floorf(xm), 0.0f), (float)(W - 1));
              bym = (int)fminf(fmaxf(floorf(ym), 0.0f), (float)(H - 1));
              // the candidates of the sub-tile holding the centre pixel serve both
              // offset rays: its frustum is padded by half a pixel and the offsets are
              // far smaller
              const int st = st0 + (py / kSubH) * nsx + (px / kSubW);
              int2 pk = a.wk.st[st];
              if (pk.y > 0 && (!in_range(a.status, pk.x, 0, a.wk.pool_cap) ||
                               !in_range(a.status, (long long)pk.x + pk.y - 1, 0, a.wk.pool_cap)))
                pk.y = -1;
              off = pk.x;
              K = pk.y;
              o = make_float3(cam.c[0], cam.c[1], cam.c[2]);
              dp = primary_dir(cam, xp, yp);
              dm = primary_dir(cam, xm, ym);
              if (STATS && q == 0) {
                cnt.samples += 2;
                cnt.rays += 2;
              }
            }
          }
        }
      }
    }
  }
  Hit hp{-1, INFINITY, 0.0f, 0.0f}, hm{-1, INFINITY, 0.0f, 0.0f};
  // ---- no candidate list: lanes 0 and 1 of the group traverse the BVH -----------
  if (__any_sync(full, active && K < 0)) {
    if constexpr (L == 1) {
      if (active && K < 0) {
        hp = trace<STATS>(a.nodes, a.tris, o, dp, a.status, cnt, a.max_visits);
        hm = trace<STATS>(a.nodes, a.tris, o, dm, a.status, cnt, a.max_visits);
      }
    } else {
      Hit h{-1, INFINITY, 0.0f, 0.0f};
      if (active && K < 0 && q < 2) h = trace<STATS>(a.nodes, a.tris, o, q == 0 ? dp : dm, a.status, cnt, a.max_visits);
      const int g0 = lane - q;
      Hit r0, r1;
      r0.tri = __shfl_sync(full, h.tri, g0);
      r0.t = __shfl_sync(full, h.t, g0);
      r0.u = __shfl_sync(full, h.u, g0);
      r0.v = __shfl_sync(full, h.v, g0);
      r1.tri = __shfl_sync(full, h.tri, g0 + 1);
      r1.t = __shfl_sync(full, h.t, g0 + 1);
      r1.u = __shfl_sync(full, h.u, g0 + 1);
      r1.v = __shfl_sync(full, h.v, g0 + 1);
      if (active && K < 0) {
        hp = r0;
        hm = r1;
      }
    }
  }
  // ---- candidate search, both rays together ---------------------------------------
  const bool listed = active && K > 0;
  for (int base = 0;; base += kEdgeWin) {
    bool go = listed && base < K;
    if (go && base > 0) {   // group-uniform: no candidate from here on can be nearer than the hits
      const float z0 = __ldg(&a.wk.z[off + base]), zl0 = z0 - (1e-4f * fabsf(z0) + 1e-6f);
      go = !(hp.t < zl0 && hm.t < zl0);
    }
    if (!__any_sync(full, go)) break;
    // the lane's candidates base + q, base + q + L, ... whose boxes hold a ray's point
    unsigned bp = 0u, bm = 0u;
    if (go) {
#pragma unroll
      for (int h = 0; h < kEdgeWin / L; h += 8)
#pragma unroll
        for (int n = h; n < min(h + 8, kEdgeWin / L); ++n) {
          const int c = base + n * L + q;
          const float4 bb = __ldg(&a.wk.bb[off + min(c, K - 1)]);
          if (c < K) {
            bp |= (unsigned)(xp >= bb.x && xp <= bb.z && yp >= bb.y && yp <= bb.w) << n;
            bm |= (unsigned)(xm >= bb.x && xm <= bb.z && ym >= bb.y && ym <= bb.w) << n;
          }
        }
    }
    for (unsigned bits = bp | bm; bits; bits &= bits - 1u) {
      const int n = __ffs(bits) - 1, c = base + n * L + q;
      const float zm = __ldg(&a.wk.z[off + c]), zl = zm - (1e-4f * fabsf(zm) + 1e-6f);
      const bool tp = (bp >> n & 1u) && !(hp.t < zl), tm = (bm >> n & 1u) && !(hm.t < zl);
      if (STATS) cnt.cands += (unsigned)tp + (unsigned)tm;
      if (!tp && !tm) continue;
      const int kr = __ldg(&a.wk.rec[off + c]);
      if (!in_range(a.status, kr, 0, a.max_visits - 1)) continue;
      if (tp) isect<STATS>(a.tris, kr, o, dp, hp, cnt);
      if (tm) isect<STATS>(a.tris, kr, o, dm, hm, cnt);
    }
    __syncwarp();
    hp = group_min<L>(hp);
    hm = group_min<L>(hm);
  }
  if (STATS) {
    if (q == 0) cnt.hits += (unsigned)(active && hp.tri >= 0) + (unsigned)(active && hm.tri >= 0);
    unsigned v[kStatsPer] = {cnt.samples, cnt.rays, cnt.nodes, cnt.tris, cnt.hits, cnt.cands};
    for (int s2 = 0; s2 < kStatsPer; ++s2) {
      unsigned long long xq = v[s2];
      for (int o2 = 16; o2 > 0; o2 >>= 1) xq += __shfl_down_sync(full, xq, o2);
      if (lane == 0 && xq) atomicAdd(stats + s2, xq);
    }
  }
  if (!active || q >= 6) return;
  const float3 fp = hp.tri >= 0 ? radiance(a, hp) : ld3(a.bg + 3 * (vw.pix0 + (size_t)byp * W + bxp));
  const float3 fm = hm.tri >= 0 ? radiance(a, hm) : ld3(a.bg + 3 * (vw.pix0 + (size_t)bym * W + bxm));
  const int Ne = a0.vt ? __ldg(&a0.vt[view].ne) : Ne_max;
  const float wgt = (A.x * (fp.x - fm.x) + A.y * (fp.y - fm.y) + A.z * (fp.z - fm.z)) * ((float)nsil / (float)Ne);
  if (wgt == 0.0f) return;
  const float dax = wgt * (by - y), day = wgt * (x - bx), dbx = wgt * (y - ay), dby = wgt * (ax - x);
  // the six results (endpoint ep = j / 3, coordinate j % 3), lanes q, q + L, ... of the
  // group: the projection Jacobian's transpose, J^T g = R^T (gx, gy, gz)
  for (int j = q; j < 6; j += L) {
    const int ep = j / 3, comp = j % 3;
    const float3 p = ep == 0 ? va : vb;
    const float g2x = ep == 0 ? dax : dbx, g2y = ep == 0 ? day : dby;
    const float X = cam.R[0] * p.x + cam.R[1] * p.y + cam.R[2] * p.z + cam.t[0];
    const float Y = cam.R[3] * p.x + cam.R[4] * p.y + cam.R[5] * p.z + cam.t[1];
    const float Z = cam.R[6] * p.x + cam.R[7] * p.y + cam.R[8] * p.z + cam.t[2];
    const float iz = 1.0f / Z;
    const float gx = g2x * cam.fx * iz, gy = g2y * cam.fy * iz;
    const float gz = -(gx * X + gy * Y) * iz;
    add1(&d_verts[3 * (ep == 0 ? ia : ib) + comp], cam.R[comp] * gx + cam.R[3 + comp] * gy + cam.R[6 + comp] * gz);
  }
}

// dm_u = (I - n n^T) dN_u / |m_u|: the adjoint of the unnormalised normal m_u of
// vertex u from that of its unit normal
__device__ __forceinline__ float3 normal_dm(const float* __restrict__ normals, const float* __restrict__ normal_len,
                                           const float* __restrict__ dN, int u) {
  const float len = normal_len[u];
  const float3 n = ld3(normals + 3 * u), g = ld3(dN + 3 * u);
  if (!(len > 0.0f)) return make_float3(0.0f, 0.0f, 0.0f);
  const float pr = dot3(n, g);
  const float il = 1.0f / len;
  return make_float3((g.x - n.x * pr) * il, (g.y - n.y * pr) * il, (g.z - n.z * pr) * il);
}

// d_verts[v] += sum over incident faces of d(e1 x e2)/dv . dc_f, dc_f = sum of dm
// over f's vertices (dm computed here from dN for each of them: no pass of its own);
// plus the edge term's sums when dedge is given.  blockIdx.y selects the instance.
__global__ void k_normal_gather(const float* __restrict__ verts_all, const int* __restrict__ faces,
                                const int* __restrict__ vf_off, const int* __restrict__ vf_faces,
                                const float* __restrict__ normals_all, const float* __restrict__ normal_len_all,
                                const float* __restrict__ dN_all, int V, const float* __restrict__ dedge_all,
                                float* __restrict__ d_verts_all, const int* __restrict__ active) {
  pdl_wait();
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V || (active && !active[blockIdx.y])) return;
  const size_t o = (size_t)blockIdx.y * 3 * V;
  const float *verts = verts_all + o, *normals = normals_all + o, *dN = dN_all + o;
  const float* normal_len = normal_len_all + (size_t)blockIdx.y * V;
  float* d_verts = d_verts_all + o;
  float3 acc = make_float3(0.0f, 0.0f, 0.0f);
  if (dedge_all) acc = ld3(dedge_all + o + 3 * v);
  for (int k = vf_off[v]; k < vf_off[v + 1]; ++k) {
    int f = vf_faces[k];
    int i0 = faces[3 * f], i1 = faces[3 * f + 1], i2 = faces[3 * f + 2];
    float3 dc = normal_dm(normals, normal_len, dN, i0);
    float3 t1 = normal_dm(normals, normal_len, dN, i1), t2 = normal_dm(normals, normal_len, dN, i2);
    dc = make_float3(dc.x + t1.x + t2.x, dc.y + t1.y + t2.y, dc.z + t1.z + t2.z);
    float3 p0 = ld3(verts + 3 * i0), p1 = ld3(verts + 3 * i1), p2 = ld3(verts + 3 * i2);
    float3 e1 = make_float3(p1.x - p0.x, p1.y - p0.y, p1.z - p0.z);
    float3 e2 = make_float3(p2.x - p0.x, p2.y - p0.y, p2.z - p0.z);
    float3 de1 = cross3(e2, dc), de2 = cross3(dc, e1);
    if (v == i1) {
      acc.x += de1.x; acc.y += de1.y; acc.z += de1.z;
    } else if (v == i2) {
      acc.x += de2.x; acc.y += de2.y; acc.z += de2.z;
    } else {
      acc.x -= de1.x + de2.x; acc.y -= de1.y + de2.y; acc.z -= de1.z + de2.z;
    }
  }
  d_verts[3 * v] += acc.x;
  d_verts[3 * v + 1] += acc.y;
  d_verts[3 * v + 2] += acc.z;
}

// d_verts += dedge (the edge term's sums, when the normals' adjoint is off)
__global__ void k_add_edges(const float* __restrict__ dedge, long long n, float* __restrict__ d_verts) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d_verts[i] += dedge[i];
}

__global__ void k_trace(const Node* __restrict__ nodes, const float4* __restrict__ tris, const float* __restrict__ o,
                        const float* __restrict__ d, int n, int* __restrict__ tri, float* __restrict__ tuv, int* status,
                        int max_visits) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  Counts cnt;
  Hit h = trace<false>(nodes, tris, ld3(o + 3 * i), ld3(d + 3 * i), status, cnt, max_visits);
  tri[i] = h.tri;
  tuv[3 * i] = h.t;
  tuv[3 * i + 1] = h.u;
  tuv[3 * i + 2] = h.v;
}


// HR_TIMING: event pair (2 slot, 2 slot + 1) around internal kernel `slot`
struct Timer {
  Context* ctx;
  cudaStream_t s;
  bool on;
  void begin(int slot) {
    if (on) cudaEventRecord(ctx->ev[2 * slot], s);
  }
  void end(int slot) {
    if (on) cudaEventRecord(ctx->ev[2 * slot + 1], s);
  }
};

RenderArgs make_args(Context* ctx, const hr_model* m, const float* verts, const Cam* cams, int N, int H, int W,
                     const float* bg, const hr_render_opts* o) {
  RenderArgs a;
  a.nodes = ctx->nodes;
  a.tris = ctx->tris;
  a.verts = verts;
  a.faces = m->faces;
  a.normals = ctx->normals;
  a.albedo = m->albedo;
  a.frec = ctx->face_rec;
  a.cams = cams;
  a.bg = bg;
  a.N = N;
  a.H = H;
  a.W = W;
  a.spp = o->spp;
  a.V = m->V;
  a.key = make_uint2((uint32_t)(o->seed & 0xffffffffull), (uint32_t)(o->seed >> 32));
  a.ctr1_hi = o->instance << 16;
  a.iter4 = o->iter << 4;
  a.iter_dev = o->iter_dev;
  a.sh.l = make_float3(o->light_dir[0], o->light_dir[1], o->light_dir[2]);
  a.sh.lrgb = make_float3(o->light_rgb[0], o->light_rgb[1], o->light_rgb[2]);
  a.sh.ka = o->ka;
  a.sh.kd = o->kd;
  a.status = ctx->status;
  a.max_visits = ctx->F + 1;
  a.wk.bb = ctx->pool_bb;
  a.wk.z = ctx->pool_z;
  a.wk.rec = ctx->pool_rec;
  a.wk.pm = ctx->pool_pm;
  a.wk.pool_cap = ctx->pool_cap;
  a.wk.st = ctx->st_info;
  a.wk.items = ctx->items;
  a.wk.item_cap = ctx->item_cap;
  a.wk.part = ctx->item_part;
  a.wk.extra = ctx->extra;
  a.wk.extra64 = ctx->extra64;
  a.wk.ctr = ctx->work_ctr;
  a.wk.ovf = ctx->ovf_list;
  a.wk.trace = ctx->trace_list;
  a.wk.st_done = ctx->st_done;
  a.wk.cand_st = ctx->cand_st;
  a.wk.bin = ctx->bin_cnt;
  a.wk.bvh_need = ctx->bvh_need;
  a.wk.fx = ctx->acc_fx;
  a.wk.det = (o->flags & HR_DETERMINISTIC) != 0;
  a.node_stride = ctx->lim.max_F;
  a.num_sms = ctx->num_sms;
  a.cand_per_chunk = ctx->tune.cand_per_chunk;
  a.max_chunks = ctx->tune.max_chunks;
  a.uv = m->uv;
  a.tex = (o->texture && m->uv) ? o->texture : nullptr;
  a.tex_w = o->tex_w;
  a.tex_h = o->tex_h;
  a.d_tex = a.tex ? o->d_texture : nullptr;
  a.active = ctx->vt ? ctx->active : nullptr;
  a.act_off = a.active ? ctx->act_off : nullptr;
  if (ctx->vt) {
    a.vt = ctx->vt;
    a.it = ctx->it;
    a.n_inst = ctx->n_inst;
    a.nviews = ctx->nviews;
    a.total_st = ctx->total_st;
  } else {
    a.vt = nullptr;
    a.it = nullptr;
    a.n_inst = 1;
    a.nviews = N;
    a.total_st = subtiles_for(N, W, H);
  }
  return a;
}

}  // namespace

int render_grid(int device, int* blocks, int* threads, int* num_sms) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return HR_ERR_CUDA;
  *num_sms = sms;
  *threads = kRenderThreads;
  *blocks = sms * kBlocksPerSm;
  return HR_OK;
}

int subtiles_for(int views, int W, int H) { return views * ((W + kSubW - 1) / kSubW) * ((H + kSubH - 1) / kSubH); }
int subtile_columns(int W) { return (W + kSubW - 1) / kSubW; }

int launch_render_fwd(Context* ctx, const hr_model* m, const float* verts, const Cam* cams, int N, int H, int W,
                      const float* bg, const hr_render_opts* o, float* image, cudaStream_t s) {
  RenderArgs a = make_args(ctx, m, verts, cams, N, H, W, bg, o);
  const bool st = o->flags & HR_STATS;
  Timer tm{ctx, s, (o->flags & HR_TIMING) != 0};
  if (cudaMemsetAsync(ctx->work_ctr, 0, ctr_words(a.n_inst) * sizeof(unsigned), s) != cudaSuccess)
    return HR_ERR_CUDA;
  if (a.act_off) {   // a batch with a mask: the active instances' sub-tiles and views
    k_active_layout<<<1, kLayoutThreads, 0, s>>>(ctx->it, ctx->active, ctx->n_inst, ctx->act_off);
    HR_CHECK_LAUNCH();
  }
  const int blocks = ctx->num_sms * ctx->tune.blocks_per_sm;
  tm.begin(kTimeFwdGather);
  // candidate lists: bin the (view, record) pairs into sub-tiles (count), give each
  // sub-tile its pool range and work items, bin again into the ranges (fill), order
  // each list by nearest depth.  The bins are zero between forwards (cleared once at
  // creation, then by k_bin_alloc and k_bin_sort).  The background sub-tiles' pixels
  // are written on the context's second stream beside the fill and the sort (with
  // kernel timing on, on the caller's stream), joined before the call returns.
  const bool fork = !tm.on;
  cudaStream_t bs = fork ? ctx->side : s;
  {
    const long long pairs = (long long)a.nviews * (a.max_visits - 1);
    const long long bin_warps = (pairs + kBinPairs - 1) / kBinPairs;
    const int bin_blocks = (int)std::min<long long>((bin_warps + kBinThreads / 32 - 1) / (kBinThreads / 32), 8LL * ctx->num_sms);
    launch_pdl(k_bin<false>, dim3(std::max(bin_blocks, 1)), dim3(kBinThreads), 0, s, a, ctx->bin_cnt);
    HR_CHECK_LAUNCH();
    const int group_blocks = ctx->num_sms * 8;
    // full warps from 16 of them per SM on (a 24.6 k-triangle hand at 16 x 1024^2, 524 k sub-tiles: 45 -> 30 us)
    launch_pdl(a.total_st >= 32 * 16 * ctx->num_sms ? k_bin_alloc<32> : k_bin_alloc<8>, dim3(group_blocks), dim3(kGroupThreads),
               0, s, a, ctx->bin_cnt);
    HR_CHECK_LAUNCH();
    if (fork && (cudaEventRecord(ctx->ev_fork, s) != cudaSuccess || cudaStreamWaitEvent(bs, ctx->ev_fork, 0) != cudaSuccess))
      return HR_ERR_CUDA;
    const int bg_blocks = ctx->num_sms * 4;   // one wave at k_background's 64 registers
    if (st)
      k_background<true><<<bg_blocks, kGroupThreads, 0, bs>>>(a, image, ctx->stats);
    else
      k_background<false><<<bg_blocks, kGroupThreads, 0, bs>>>(a, image, nullptr);
    HR_CHECK_LAUNCH();
    // the boxes of a tree whose update rewrote only the records, refitted if a sub-tile
    // was listed for per-ray traversal (k_overflow is the first to traverse)
    const int rc = launch_bvh_lazy_refit(ctx, 0, bs);
    if (rc != HR_OK) return rc;
    if (fork && cudaEventRecord(ctx->ev_join, bs) != cudaSuccess) return HR_ERR_CUDA;
    launch_pdl(k_bin<true>, dim3(std::max(bin_blocks, 1)), dim3(kBinThreads), 0, s, a, ctx->bin_cnt);
    HR_CHECK_LAUNCH();
    launch_pdl(k_bin_sort, dim3(blocks), dim3(kRenderThreads), 0, s, a);
    HR_CHECK_LAUNCH();
  }
  tm.end(kTimeFwdGather);
  tm.begin(kTimeFwdShade);
  {
    const int S = ctx->tune.rays_per_lane;
    auto kern = st ? (S == 1 ? k_shade_fwd<true, 1> : (S == 2 ? k_shade_fwd<true, 2> : k_shade_fwd<true, 4>))
                   : (S == 1 ? k_shade_fwd<false, 1> : (S == 2 ? k_shade_fwd<false, 2> : k_shade_fwd<false, 4>));
    launch_pdl(kern, dim3(blocks), dim3(kRenderThreads), 0, s, a, image, st ? ctx->stats : nullptr);
  }
  HR_CHECK_LAUNCH();
  if (fork && cudaStreamWaitEvent(s, ctx->ev_join, 0) != cudaSuccess) return HR_ERR_CUDA;
  if (st)
    launch_pdl(k_overflow<false, true>, dim3(blocks), dim3(kRenderThreads), 0, s, a, nullptr, image, ctx->stats);
  else
    launch_pdl(k_overflow<false, false>, dim3(blocks), dim3(kRenderThreads), 0, s, a, nullptr, image,
               (unsigned long long*)nullptr);
  HR_CHECK_LAUNCH();
  tm.end(kTimeFwdShade);
  // the item sums are combined inside the shaders (finish_item): the slot stays, empty
  tm.begin(kTimeFwdCombine);
  tm.end(kTimeFwdCombine);
  if (tm.on) ctx->ev_ready |= 1;
  ctx->fwd_verts = verts;
  ctx->fwd_cams = cams;
  ctx->fwd_N = N;
  ctx->fwd_H = H;
  ctx->fwd_W = W;
  ctx->fwd_spp = o->spp;
  ctx->fwd_gen = ctx->bvh_gen;
  ctx->fwd_valid = true;
  return HR_OK;
}

int launch_silhouettes(Context* ctx, const hr_model* m, const float* verts, const Cam* cams, int N, int* lists,
                       int list_stride, int* counts, cudaStream_t s) {
  k_silhouettes<<<N, 512, 0, s>>>(verts, m->faces, m->edges, m->edge_faces, m->E, cams, ctx->vt, m->V, lists,
                                  list_stride, counts, ctx->vt ? ctx->active : nullptr);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

int launch_render_bwd(Context* ctx, const hr_model* m, const float* verts, const Cam* cams, int N, int H, int W,
                      const float* bg, const hr_render_opts* o, const float* adjoint, float* d_verts,
                      cudaStream_t s) {
  RenderArgs a = make_args(ctx, m, verts, cams, N, H, W, bg, o);
  a.cand_per_chunk = ctx->tune.bwd_cand_per_chunk;   // the backward's own work-item split
  if (a.act_off) {   // a batch with a mask: the active instances' sub-tiles and views
    k_active_layout<<<1, kLayoutThreads, 0, s>>>(ctx->it, ctx->active, ctx->n_inst, ctx->act_off);
    HR_CHECK_LAUNCH();
  }
  const int V = m->V, ni = a.n_inst, nv = a.nviews;
  const bool batch = ctx->vt != nullptr;
  const int Ne = batch ? ctx->max_ne : o->edge_samples;
  const bool interior = !(o->flags & HR_BWD_NO_INTERIOR);
  const bool edges = !(o->flags & HR_BWD_NO_EDGES) && Ne > 0;
  const bool normals = !(o->flags & HR_BWD_NO_NORMALS) && interior;
  const bool st = o->flags & HR_STATS;
  Timer tm{ctx, s, (o->flags & HR_TIMING) != 0};
  if (interior || edges) {
    // candidates of the sub-tiles with a non-zero adjoint: the interior shader's work
    // items, and the edge rays' candidate lists
    if (cudaMemsetAsync(ctx->work_ctr, 0, ctr_words(ni) * sizeof(unsigned), s) != cudaSuccess ||
        cudaMemsetAsync(ctx->extra, 0, sizeof(float) * 8 * V * ni, s) != cudaSuccess)
      return HR_ERR_CUDA;
    // the forward's candidate lists still describe this scene when it used the same
    // vertices, cameras and sizes after the last build
    const bool reuse = (o->flags & HR_BWD_REUSE_FWD) && ctx->fwd_valid && ctx->fwd_verts == verts &&
                       ctx->fwd_cams == cams && ctx->fwd_N == N && ctx->fwd_H == H && ctx->fwd_W == W &&
                       (batch || ctx->fwd_spp == o->spp) && ctx->fwd_gen == ctx->bvh_gen;
    tm.begin(kTimeBwdGather);
    if (reuse) {
      if (st)
        launch_pdl(k_items_bwd<true>, dim3(ctx->num_sms * 4), dim3(kGroupThreads), 0, s, a, adjoint, ctx->stats + kStatsPer);
      else
        launch_pdl(k_items_bwd<false>, dim3(ctx->num_sms * 4), dim3(kGroupThreads), 0, s, a, adjoint,
                   (unsigned long long*)nullptr);
    } else {
      // its own lists from a frustum walk of the BVH: the boxes must be current
      const int rc = launch_bvh_lazy_refit(ctx, 1, s);
      if (rc != HR_OK) return rc;
      k_face_records<<<ctx->num_sms, kGroupThreads, 0, s>>>(a);
      HR_CHECK_LAUNCH();
      if (st)
        k_gather<true><<<ctx->num_sms * ctx->tune.blocks_per_sm, kRenderThreads, 0, s>>>(a, adjoint,
                                                                            ctx->stats + kStatsPer);
      else
        k_gather<false><<<ctx->num_sms * ctx->tune.blocks_per_sm, kRenderThreads, 0, s>>>(a, adjoint, nullptr);
    }
    HR_CHECK_LAUNCH();
    tm.end(kTimeBwdGather);
  }
  // The edge-sampling term (silhouettes, edge samples into ctx->dedge) needs only the
  // candidate lists made above; it runs on the context's side stream beside the
  // interior shader and joins before the normals' adjoint adds it to d_verts.  With
  // kernel timing on, everything stays on the caller's stream.  HR_DETERMINISTIC:
  // everything stays on the caller's stream, both terms add their vertex sums to the
  // fixed-point array, and one reduction after both turns it into d_verts and dN.
  const bool det = (o->flags & HR_DETERMINISTIC) != 0;
  const bool fork = edges && !tm.on && !det;
  cudaStream_t es = fork ? ctx->side : s;
  if (det && cudaMemsetAsync(ctx->acc_fx, 0, sizeof(unsigned long long) * 6 * V * ni, s) != cudaSuccess)
    return HR_ERR_CUDA;
  if (edges) {
    if (fork && (cudaEventRecord(ctx->ev_fork, s) != cudaSuccess || cudaStreamWaitEvent(es, ctx->ev_fork, 0) != cudaSuccess))
      return HR_ERR_CUDA;
    if (!det && cudaMemsetAsync(ctx->dedge, 0, sizeof(float) * 3 * V * ni, es) != cudaSuccess) return HR_ERR_CUDA;
  }
  const auto reduce = [&](int acc, int nparts) {
    launch_pdl(k_reduce_partials, dim3((8 * V + kRedEntries - 1) / kRedEntries, ni), dim3(kRedEntries * kRedGroups), 0,
               s, (const float*)ctx->partials, (const float*)ctx->extra,
               (const double*)(acc == kAccGlobal ? ctx->extra64 : nullptr),
               (const unsigned long long*)(det ? ctx->acc_fx : nullptr), acc == kAccPartials ? nparts : 0, V, d_verts,
               ctx->dN);
  };
  if (interior) {
    // float sums up to kPartialMaxV vertices (per SM, or per instance in a batch),
    // float64 beyond; fixed-point sums when deterministic
    const bool global_acc = V > kPartialMaxV;
    if (!det && global_acc &&
        (!ctx->extra64 || cudaMemsetAsync(ctx->extra64, 0, sizeof(double) * 6 * V * ni, s) != cudaSuccess))
      return ctx->extra64 ? HR_ERR_CUDA : HR_ERR_UNSUPPORTED;
    const int acc = det ? kAccFixed : (global_acc ? kAccGlobal : (batch ? kAccDirect : kAccPartials));
    // deterministic: one ray per lane, the arithmetic of the overflow kernel, which may
    // trace any sub-tile whose candidates found no room in the pool
    const int S = det ? 1 : ctx->tune.bwd_rays_per_lane;
#define HR_BWD_KERNEL(A_) \
  (st ? (S == 1 ? k_shade_bwd<true, A_, 1> : (S == 2 ? k_shade_bwd<true, A_, 2> : k_shade_bwd<true, A_, 4>)) \
      : (S == 1 ? k_shade_bwd<false, A_, 1> : (S == 2 ? k_shade_bwd<false, A_, 2> : k_shade_bwd<false, A_, 4>)))
    auto kern = acc == kAccFixed    ? HR_BWD_KERNEL(kAccFixed)
                : acc == kAccGlobal ? HR_BWD_KERNEL(kAccGlobal)
                                    : (acc == kAccDirect ? HR_BWD_KERNEL(kAccDirect) : HR_BWD_KERNEL(kAccPartials));
#undef HR_BWD_KERNEL
    // one partial per SM (the blocks of a launch share them round-robin), zeroed first
    const int blocks = ctx->num_sms * ctx->tune.bwd_blocks_per_sm;
    const int nparts = ctx->num_sms;
    if (acc == kAccPartials &&
        cudaMemsetAsync(ctx->partials, 0, sizeof(float) * 8 * V * (size_t)nparts, s) != cudaSuccess)
      return HR_ERR_CUDA;
    tm.begin(kTimeBwdShade);
    launch_pdl(kern, dim3(blocks), dim3(kRenderThreads), 0, s, a, adjoint, ctx->partials, nparts,
               st ? ctx->stats + kStatsPer : nullptr);
    HR_CHECK_LAUNCH();
    if (st)
      launch_pdl(k_overflow<true, true>, dim3(blocks), dim3(kRenderThreads), 0, s, a, adjoint, (float*)nullptr,
                 ctx->stats + kStatsPer);
    else
      launch_pdl(k_overflow<true, false>, dim3(blocks), dim3(kRenderThreads), 0, s, a, adjoint, (float*)nullptr,
                 (unsigned long long*)nullptr);
    HR_CHECK_LAUNCH();
    tm.end(kTimeBwdShade);
    if (!det) {
      tm.begin(kTimeBwdReduce);
      reduce(acc, nparts);
      HR_CHECK_LAUNCH();
      tm.end(kTimeBwdReduce);
    }
  } else if (!det) {
    if (cudaMemsetAsync(d_verts, 0, sizeof(float) * 3 * V * ni, s) != cudaSuccess) return HR_ERR_CUDA;
  }
  if (edges) {
    tm.begin(kTimeBwdSil);
    int rc = launch_silhouettes(ctx, m, verts, cams, nv, ctx->sil, ctx->lim.max_E, ctx->sil_count, es);
    if (rc != HR_OK) return rc;
    tm.end(kTimeBwdSil);
    // At most edge_lanes lanes per edge sample, fewer when the samples alone fill the GPU
    // (about 2.5 times an SM's resident threads at this kernel's registers): the lanes of a
    // sample share its search but each do its set-up.  Whole passes at 4 / 2 / 1 lanes, us:
    // 28 k samples 326 / 326 / 347, 40 k 323 / 329 / 335, 78 k 278 / 267 / 267, 86 k with
    // long lists 1795 / 1692 / 1714; this kernel for a batch of 64 hands 2177 / 1712 / 1404.
    int L = ctx->tune.edge_lanes;
    while (L > 1 && (long long)nv * Ne * L > 1316LL * ctx->num_sms) L >>= 1;
    const long long n = ((long long)nv * Ne + 32 / L - 1) / (32 / L) * 32;
    const unsigned grid = (unsigned)((n + kRenderThreads - 1) / kRenderThreads);
    tm.begin(kTimeBwdEdges);
#define HR_EDGE_KERNEL(T_)                                                                            \
  (st ? (L == 1 ? k_edge_samples<true, T_, 1> : L == 2 ? k_edge_samples<true, T_, 2> : L == 4 ? k_edge_samples<true, T_, 4>                  \
         : L == 8 ? k_edge_samples<true, T_, 8> : L == 16 ? k_edge_samples<true, T_, 16>              \
                                                        : k_edge_samples<true, T_, 32>)               \
      : (L == 1 ? k_edge_samples<false, T_, 1> : L == 2 ? k_edge_samples<false, T_, 2> : L == 4 ? k_edge_samples<false, T_, 4>                \
         : L == 8 ? k_edge_samples<false, T_, 8> : L == 16 ? k_edge_samples<false, T_, 16>            \
                                                         : k_edge_samples<false, T_, 32>))
    if (det) {
      auto kern = HR_EDGE_KERNEL(unsigned long long);
      kern<<<grid, kRenderThreads, 0, es>>>(a, adjoint, m->edges, ctx->sil, ctx->lim.max_E, ctx->sil_count, Ne,
                                            o->edge_eps_px, ctx->acc_fx, 6LL * V, ctx->stats + 2 * kStatsPer);
    } else {
      auto kern = HR_EDGE_KERNEL(float);
      kern<<<grid, kRenderThreads, 0, es>>>(a, adjoint, m->edges, ctx->sil, ctx->lim.max_E, ctx->sil_count, Ne,
                                            o->edge_eps_px, ctx->dedge, 3LL * V, ctx->stats + 2 * kStatsPer);
    }
#undef HR_EDGE_KERNEL
    HR_CHECK_LAUNCH();
    tm.end(kTimeBwdEdges);
    if (fork && (cudaEventRecord(ctx->ev_join, es) != cudaSuccess || cudaStreamWaitEvent(s, ctx->ev_join, 0) != cudaSuccess))
      return HR_ERR_CUDA;
  }
  if (det) {
    tm.begin(kTimeBwdReduce);
    reduce(kAccFixed, 0);
    HR_CHECK_LAUNCH();
    tm.end(kTimeBwdReduce);
  }
  if (normals) {
    tm.begin(kTimeBwdNormals);
    const dim3 g((V + 255) / 256, ni);
    const int* act = batch ? ctx->active : nullptr;
    launch_pdl(k_normal_gather, g, dim3(256), 0, s, verts, m->faces, m->vf_offsets, m->vf_faces,
               (const float*)ctx->normals, (const float*)ctx->normal_len, (const float*)ctx->dN, V,
               (const float*)(edges && !det ? ctx->dedge : nullptr), d_verts, act);
    HR_CHECK_LAUNCH();
    tm.end(kTimeBwdNormals);
  } else if (edges && !det) {
    const long long n3 = 3LL * V * ni;
    k_add_edges<<<(unsigned)((n3 + 255) / 256), 256, 0, s>>>(ctx->dedge, n3, d_verts);
    HR_CHECK_LAUNCH();
  }
  if (tm.on) ctx->ev_ready |= 2 | (interior ? 4 : 0) | (edges ? 8 : 0) | (normals ? 16 : 0);
  return HR_OK;
}

int launch_trace(Context* ctx, const float* o, const float* d, int n, int* tri, float* tuv, cudaStream_t s) {
  const int rc = launch_bvh_lazy_refit(ctx, 1, s);   // traversal reads the boxes
  if (rc != HR_OK) return rc;
  k_trace<<<(n + 127) / 128, 128, 0, s>>>(ctx->nodes, ctx->tris, o, d, n, tri, tuv, ctx->status, ctx->F + 1);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

}  // namespace hr
