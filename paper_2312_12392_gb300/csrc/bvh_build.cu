// bvh_build.cu -- GPU BVH builder (Morton order, PLOC clustering) collapsed to an 8-wide BVH.
//
// The paper (§6) traced its scenes with OptiX and says nothing about the
// acceleration structure; this builder serves the scene S(n) of §2, Eq. 1.
// Steps, all on the device:
//  1. primitive boxes and centroids; scene and centroid bounds (atomic min/max
//     on order-preserving integer images of the floats);
//  2. 30-bit Morton codes of the centroids (10 bits per axis, in the cube of
//     the largest extent);
//  3. radix sort of (code, primitive) pairs (radix_sort.cu);
//  4. binary tree by PLOC (Meister and Bittner 2018): the primitives in
//     Morton order are clusters; each round every cluster finds the cluster
//     within 16 array positions whose union box has the least surface area,
//     mutual pairs merge (the new node gets the union box), and the array is
//     compacted by a prefix sum, until one cluster is left;
//  5. leaves renumbered in depth-first order, so that every subtree's
//     primitives are contiguous;
//  6. collapse to 8-wide nodes, one launch per level. Subtrees of <= LEAF_MAX
//     (3) primitives become leaves. Which binary nodes are opened into a wide
//     node's 8 slots follows the scene's policy: RCP_COLLAPSE_AREA repeatedly
//     opens the child of largest surface area that holds more than LEAF_MAX
//     primitives; RCP_COLLAPSE_SAH shares the slots out by a bottom-up dynamic
//     program over the binary tree that minimises the surface-area cost. Children
//     are placed in slots so that slot order approximates front-to-back order
//     per ray octant; child boxes are float32 bounds with a small outward pad
//     (tri_pad). Leaf primitives are copied into 48-byte records, contiguous
//     per node. Optionally (split_max > 1) long thin triangles first enter
//     as several clipped references (early split clipping, below); each keeps
//     its part of the triangle, so that a refit after a vertex update bounds
//     it by that part of the moved triangle.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "rcp_internal.cuh"
#include "scene.h"

namespace rcp {

namespace {

constexpr int BUILD_BLOCK = 256;
// Most primitives in one leaf slot: a node's header has 3 bits per slot for
// the count in unary.
constexpr int LEAF_MAX = 3;
static_assert(LEAF_MAX >= 1 && LEAF_MAX <= 3, "a leaf's count must fit the 3 unary bits of its slot");

__device__ __forceinline__ uint32_t f2ord(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// *bad = 1 when any of v[0..n) (16-byte aligned) is infinite or NaN: its
// exponent bits are all set. Bound by reading v once.
__global__ void __launch_bounds__(BUILD_BLOCK) k_any_non_finite(const float* __restrict__ v, int64_t n, int* bad) {
    const uint4* v4 = reinterpret_cast<const uint4*>(v);
    bool found = false;
    const auto non_finite = [](uint32_t u) { return (u & 0x7f800000u) == 0x7f800000u; };
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = t; i < n / 4; i += step) {
        const uint4 u = v4[i];
        found = found || non_finite(u.x) || non_finite(u.y) || non_finite(u.z) || non_finite(u.w);
    }
    for (int64_t i = n / 4 * 4 + t; i < n; i += step) found = found || non_finite(__float_as_uint(v[i]));
    if (found) *bad = 1;
}

__global__ void __launch_bounds__(BUILD_BLOCK) k_widen_albedo(const float* __restrict__ a, int64_t n,
                                                              float4* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = make_float4(a[3 * i], a[3 * i + 1], a[3 * i + 2], 0.f);
}

// bounds layout: [0..2] centroid min, [3..5] centroid max, [6..8] box min, [9..11] box max
__global__ void k_init_bounds(uint32_t* b) {
    const int i = threadIdx.x;
    if (i < 12) b[i] = ((i % 6) < 3) ? 0xffffffffu : 0u;
}

__device__ __forceinline__ void prim_box(const float* __restrict__ tri, const float* __restrict__ sph, int64_t T,
                                         int64_t id, float3& lo, float3& hi) {
    if (id < T) {
        const float* v = tri + 9 * id;
        lo = make_float3(fminf(fminf(v[0], v[3]), v[6]), fminf(fminf(v[1], v[4]), v[7]), fminf(fminf(v[2], v[5]), v[8]));
        hi = make_float3(fmaxf(fmaxf(v[0], v[3]), v[6]), fmaxf(fmaxf(v[1], v[4]), v[7]), fmaxf(fmaxf(v[2], v[5]), v[8]));
    } else {
        const float* s = sph + 4 * (id - T);
        const float r = fabsf(s[3]);
        lo = make_float3(__fsub_rd(s[0], r), __fsub_rd(s[1], r), __fsub_rd(s[2], r));
        hi = make_float3(__fadd_ru(s[0], r), __fadd_ru(s[1], r), __fadd_ru(s[2], r));
    }
}

// Outward pad of a triangle's stored boxes: 2^-12 of its box's extent plus
// 2^-18 of its coordinates' magnitude. The float ray-triangle test accepts
// hits up to a rounding error outside the true edges and vertices; a box that
// is exact at a vertex or an edge would let the walk skip such a hit that a
// test of every primitive accepts. The build's decisions (Morton codes,
// clustering, collapse) use the exact boxes; the boxes stored in the tree
// (leaf slots, and every node's box, refitted from the padded leaves) carry
// the pad. The scene's bounds (and its diameter) are those of the exact
// vertices.
// Float arithmetic rounded upwards (the pad) and outwards (the padded box):
// refits run it for every record of every frame, and double arithmetic is
// slow on this GPU.
__device__ __forceinline__ float tri_pad(const float3& lo, const float3& hi) {
    const float ext = __fadd_ru(__fadd_ru(__fsub_ru(hi.x, lo.x), __fsub_ru(hi.y, lo.y)), __fsub_ru(hi.z, lo.z));
    const float mag = fmaxf(fmaxf(fmaxf(fabsf(lo.x), fabsf(hi.x)), fmaxf(fabsf(lo.y), fabsf(hi.y))),
                            fmaxf(fabsf(lo.z), fabsf(hi.z)));
    return __fadd_ru(__fmul_ru(ext, 0x1p-12f), __fmul_ru(mag, 0x1p-18f));
}

__device__ __forceinline__ void pad_box(float pad, float3& lo, float3& hi) {
    lo = make_float3(__fsub_rd(lo.x, pad), __fsub_rd(lo.y, pad), __fsub_rd(lo.z, pad));
    hi = make_float3(__fadd_ru(hi.x, pad), __fadd_ru(hi.y, pad), __fadd_ru(hi.z, pad));
}

// The stored (padded) box of reference `ref`: its exact box (plo/phi),
// padded by the pad of its primitive when that is a triangle. ref_prim maps
// references to primitives (nullptr: references are the primitives).
__device__ __forceinline__ void padded_ref_box(const float4* plo, const float4* phi, const uint32_t* ref_prim,
                                               const float* tri, const float* sph, int64_t T, uint32_t ref,
                                               float3& lo, float3& hi) {
    const float4 l = plo[ref], h = phi[ref];
    lo = make_float3(l.x, l.y, l.z);
    hi = make_float3(h.x, h.y, h.z);
    const uint32_t prim = ref_prim ? ref_prim[ref] : ref;
    if ((int64_t)prim < T) {
        float3 tl, th;
        prim_box(tri, sph, T, prim, tl, th);
        pad_box(tri_pad(tl, th), lo, hi);
    }
}

__global__ void __launch_bounds__(BUILD_BLOCK) k_prim_bounds(const float* __restrict__ tri,
                                                             const float* __restrict__ sph, int64_t T, int64_t N,
                                                             float4* __restrict__ plo, float4* __restrict__ phi,
                                                             uint32_t* __restrict__ bounds) {
    __shared__ uint32_t sb[12];
    if (threadIdx.x < 12) sb[threadIdx.x] = ((threadIdx.x % 6) < 3) ? 0xffffffffu : 0u;
    __syncthreads();
    uint32_t mine[12];
    for (int a = 0; a < 12; ++a) mine[a] = ((a % 6) < 3) ? 0xffffffffu : 0u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        float3 lo, hi;
        prim_box(tri, sph, T, i, lo, hi);
        plo[i] = make_float4(lo.x, lo.y, lo.z, 0.f);
        phi[i] = make_float4(hi.x, hi.y, hi.z, 0.f);
        const float c[3] = {0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z)};
        const float l[3] = {lo.x, lo.y, lo.z}, h[3] = {hi.x, hi.y, hi.z};
        for (int a = 0; a < 3; ++a) {
            mine[a] = min(mine[a], f2ord(c[a]));
            mine[3 + a] = max(mine[3 + a], f2ord(c[a]));
            mine[6 + a] = min(mine[6 + a], f2ord(l[a]));
            mine[9 + a] = max(mine[9 + a], f2ord(h[a]));
        }
    }
    for (int a = 0; a < 12; ++a) {
        if ((a % 6) < 3) atomicMin(&sb[a], mine[a]);
        else atomicMax(&sb[a], mine[a]);
    }
    __syncthreads();
    if (threadIdx.x < 12) {
        if ((threadIdx.x % 6) < 3) atomicMin(&bounds[threadIdx.x], sb[threadIdx.x]);
        else atomicMax(&bounds[threadIdx.x], sb[threadIdx.x]);
    }
}

// 10 bits of each axis interleaved as ...x2y2z2 x1y1z1 x0y0z0 (x highest).
// Every axis is scaled by the box's largest extent (a cube over lo), not by
// its own: a flat scene (terrain, a forest floor) then keeps its thin axis in
// the low bits, so the top of the hierarchy splits the long axes and no node
// near the root spans the whole scene along them.
__device__ __forceinline__ uint32_t morton30(float x, float y, float z, const float* lo, const float* hi) {
    const float c[3] = {x, y, z};
    const float ext = fmaxf(fmaxf(hi[0] - lo[0], hi[1] - lo[1]), hi[2] - lo[2]);
    uint32_t q[3];
    for (int a = 0; a < 3; ++a) {
        float u = ext > 0.f ? (c[a] - lo[a]) / ext : 0.f;
        int v = (int)(u * 1024.f);
        q[a] = (uint32_t)min(max(v, 0), 1023);
    }
    uint32_t code = 0;
    for (int b = 0; b < 10; ++b)
        code |= (((q[0] >> b) & 1u) << (3 * b + 2)) | (((q[1] >> b) & 1u) << (3 * b + 1)) | (((q[2] >> b) & 1u) << (3 * b));
    return code;
}

__global__ void k_morton(const float4* __restrict__ plo, const float4* __restrict__ phi, int64_t N,
                         const uint32_t* __restrict__ bounds, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    float lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
        lo[a] = ord2f(bounds[a]);
        hi[a] = ord2f(bounds[3 + a]);
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 l = plo[i], h = phi[i];
        keys[i] = morton30(0.5f * (l.x + h.x), 0.5f * (l.y + h.y), 0.5f * (l.z + h.z), lo, hi);
        vals[i] = (uint32_t)i;
    }
}

__global__ void k_morton_points(const float* __restrict__ xyz, int64_t n, float l0, float l1, float l2, float h0,
                                float h1, float h2, uint32_t* __restrict__ codes) {
    const float lo[3] = {l0, l1, l2}, hi[3] = {h0, h1, h2};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        codes[i] = morton30(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], lo, hi);
}

// ---- early split clipping (Ernst and Greiner 2007) ----
// A triangle whose box is large against its own area (long thin triangles,
// such as a cone's sides from apex to base) enters the build as several
// references: its box is halved at the midpoint of the longest axis, the
// triangle is clipped to each half, and the halves whose clipped part is
// still large are halved again, up to split_max references per triangle.
// Each reference is bounded by the box of its clipped part, rounded outwards,
// so the references' boxes together cover the triangle (stored with the pad
// of the whole triangle); every reference's leaf record is the whole
// triangle, so hits are exactly those of one record.
constexpr float SPLIT_RATIO = 4.f;  // split while box half-area > 4 x triangle area
constexpr int SPLIT_MAX = 8;

// Clipping below runs in float with explicit round-to-nearest intrinsics (no
// contraction left to the compiler), so that the counting and the writing
// kernels, and any other caller, compute bit-identical pieces. Its rounding,
// about 2^-23 of the coordinates and edges, sits far inside the pad that every
// stored box carries (2^-12 of the triangle's extent plus 2^-18 of its
// coordinates' magnitude). Double arithmetic runs at a small fraction of the
// float rate on this GPU: the double version took 58 % of the forest's build.

// Box of triangle v (3 vertices) clipped to [lo, hi] (Sutherland-Hodgman).
// False when the triangle misses the box.
__device__ bool clip_triangle_box(const float (&v)[3][3], const float lo[3], const float hi[3], float3& olo,
                                  float3& ohi) {
    float poly[10][3], tmp[10][3];
    int n = 3;
    for (int i = 0; i < 3; ++i)
        for (int a = 0; a < 3; ++a) poly[i][a] = v[i][a];
    for (int a = 0; a < 3; ++a)
        for (int side = 0; side < 2; ++side) {
            const float b = side ? hi[a] : lo[a];
            int m = 0;
            for (int i = 0; i < n; ++i) {
                const float* p = poly[i];
                const float* q = poly[(i + 1) % n];
                const bool pin = side ? p[a] <= b : p[a] >= b;
                const bool qin = side ? q[a] <= b : q[a] >= b;
                if (pin) {
                    for (int c = 0; c < 3; ++c) tmp[m][c] = p[c];
                    ++m;
                }
                if (pin != qin) {  // p[a] != q[a]: they lie on either side of b
                    const float t = __fdiv_rn(__fsub_rn(b, p[a]), __fsub_rn(q[a], p[a]));
                    for (int c = 0; c < 3; ++c) tmp[m][c] = __fmaf_rn(t, __fsub_rn(q[c], p[c]), p[c]);
                    tmp[m][a] = b;  // on the plane exactly
                    ++m;
                }
            }
            n = m;
            if (n == 0) return false;
            for (int i = 0; i < n; ++i)
                for (int c = 0; c < 3; ++c) poly[i][c] = tmp[i][c];
        }
    float l[3] = {poly[0][0], poly[0][1], poly[0][2]}, h[3] = {poly[0][0], poly[0][1], poly[0][2]};
    for (int i = 1; i < n; ++i)
        for (int c = 0; c < 3; ++c) {
            l[c] = fminf(l[c], poly[i][c]);
            h[c] = fmaxf(h[c], poly[i][c]);
        }
    olo = make_float3(l[0], l[1], l[2]);
    ohi = make_float3(h[0], h[1], h[2]);
    return true;
}

// The references of triangle `id` (exact boxes, in emission order); returns
// their number. With rlo/rhi null it only counts; otherwise it writes at most
// `cap` of them. Counting and writing run the same steps, so they agree.
__device__ int split_triangle(const float* __restrict__ tri, uint32_t id, int max_refs, float4* __restrict__ rlo,
                              float4* __restrict__ rhi, int cap) {
    const float* f = tri + 9 * (int64_t)id;
    float v[3][3];
    for (int i = 0; i < 3; ++i)
        for (int a = 0; a < 3; ++a) v[i][a] = f[3 * i + a];
    // The split test compares areas in double, a few operations per triangle
    // and per piece: in float, the cross product of a long thin triangle's
    // edges loses digits and moves the decisions (measured: forest 2.7 %
    // slower). Only the clipping, the bulk of the work, runs in float.
    const double e1[3] = {(double)v[1][0] - v[0][0], (double)v[1][1] - v[0][1], (double)v[1][2] - v[0][2]};
    const double e2[3] = {(double)v[2][0] - v[0][0], (double)v[2][1] - v[0][1], (double)v[2][2] - v[0][2]};
    const double cx = e1[1] * e2[2] - e1[2] * e2[1], cy = e1[2] * e2[0] - e1[0] * e2[2],
                 cz = e1[0] * e2[1] - e1[1] * e2[0];
    const double tri_area = 0.5 * sqrt(cx * cx + cy * cy + cz * cz);
    float sl[SPLIT_MAX][3], sh[SPLIT_MAX][3];
    int sp = 0, n_out = 0;
    for (int a = 0; a < 3; ++a) {
        sl[0][a] = fminf(fminf(f[a], f[3 + a]), f[6 + a]);
        sh[0][a] = fmaxf(fmaxf(f[a], f[3 + a]), f[6 + a]);
    }
    sp = 1;
    while (sp > 0) {
        --sp;
        const float l[3] = {sl[sp][0], sl[sp][1], sl[sp][2]}, h[3] = {sh[sp][0], sh[sp][1], sh[sp][2]};
        const double dx = (double)h[0] - l[0], dy = (double)h[1] - l[1], dz = (double)h[2] - l[2];
        const double box_area = dx * dy + dy * dz + dz * dx;
        // a split adds at most one box to the outstanding ones: keep <= max_refs
        if (tri_area <= 0.0 || n_out + sp + 2 > max_refs || box_area <= SPLIT_RATIO * tri_area) {
            if (rlo && n_out < cap) {
                rlo[n_out] = make_float4(l[0], l[1], l[2], 0.f);
                rhi[n_out] = make_float4(h[0], h[1], h[2], 0.f);
            }
            ++n_out;
            continue;
        }
        const int ax = (dx >= dy && dx >= dz) ? 0 : (dy >= dz ? 1 : 2);
        const float mid = __fmul_rn(0.5f, __fadd_rn(l[ax], h[ax]));
        const int sp0 = sp;
        for (int half = 1; half >= 0; --half) {
            float cl[3] = {l[0], l[1], l[2]}, ch[3] = {h[0], h[1], h[2]};
            if (half) cl[ax] = mid;
            else ch[ax] = mid;
            float3 ol, oh;
            if (clip_triangle_box(v, cl, ch, ol, oh)) {
                sl[sp][0] = ol.x, sl[sp][1] = ol.y, sl[sp][2] = ol.z;
                sh[sp][0] = oh.x, sh[sp][1] = oh.y, sh[sp][2] = oh.z;
                ++sp;
            }
        }
        if (sp == sp0) {  // neither half kept a part (rounding): keep the box itself
            if (rlo && n_out < cap) {
                rlo[n_out] = make_float4(l[0], l[1], l[2], 0.f);
                rhi[n_out] = make_float4(h[0], h[1], h[2], 0.f);
            }
            ++n_out;
        }
    }
    return n_out;
}

// References per primitive (spheres: 1).
__global__ void k_split_count(const float* __restrict__ tri, int64_t T, int64_t N, int max_refs,
                              unsigned long long* __restrict__ counts) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        counts[i] = i < T ? (unsigned long long)split_triangle(tri, (uint32_t)i, max_refs, nullptr, nullptr, 0) : 1ull;
}

// Write the references at their offsets (exclusive prefix sum of the counts,
// R in all). A primitive writes at most the slots its count gave it; a count
// that differs sets *err and the build fails.
__global__ void k_split_write(const float* __restrict__ tri, int64_t T, int64_t N, int max_refs,
                              const unsigned long long* __restrict__ offsets, int64_t R,
                              const float4* __restrict__ plo, const float4* __restrict__ phi,
                              float4* __restrict__ rlo, float4* __restrict__ rhi, uint32_t* __restrict__ rprim,
                              int* __restrict__ err) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = (int64_t)offsets[i];
        const int cap = (int)((i + 1 < N ? (int64_t)offsets[i + 1] : R) - o);
        int n = 1;
        if (i < T) {
            n = split_triangle(tri, (uint32_t)i, max_refs, rlo + o, rhi + o, cap);
            if (n != cap) {
                atomicAdd(err, 1);
                n = min(n, cap);
            }
        } else {
            rlo[o] = plo[i];
            rhi[o] = phi[i];
        }
        for (int k = 0; k < n; ++k) rprim[o + k] = (uint32_t)i;
    }
}

// ---- parts of split references, for refits ----
// A reference of a split triangle stands for the part of the triangle inside
// its box. That part is kept as a convex polygon in the triangle's own
// coordinates (u, v), with p = v0 + u (v1 - v0) + v (v2 - v0). Every point of
// the triangle moves with its (u, v) when the vertices change, so a refit
// maps the polygon through the moved vertices and bounds the reference by
// exactly its part of the moved triangle; the parts of a triangle still cover
// it, whatever the motion.
// A vertex is stored as u and v in 16-bit fixed point (u = q / 65535), one
// 32-bit word: u in the low half. Rounding to nearest moves a mapped vertex by
// at most 2^-17 of each edge, 2^-16 of the triangle's extent, well inside the
// 2^-12 extent pad of the triangle's boxes. A record's part fills PART_MAX
// words; the word PART_END (u = v = 1, impossible in a triangle) ends a part
// of fewer vertices, and a first word PART_END means no part (the whole
// primitive).
constexpr int PART_MAX = 9;  // a triangle clipped by the 6 planes of a box has <= 9 vertices
constexpr uint32_t PART_END = 0xffffffffu;

__device__ __forceinline__ uint32_t quantize_uv(float u, float v) {
    const float su = __fmul_rn(fminf(fmaxf(u, 0.f), 1.f), 65535.f), sv = __fmul_rn(fminf(fmaxf(v, 0.f), 1.f), 65535.f);
    return __float2uint_rn(su) | (__float2uint_rn(sv) << 16);
}

// The part of triangle v inside [lo, hi] (Sutherland-Hodgman in float as
// above, the vertices carrying their (u, v)), written to out[0..PART_MAX) with
// its end marker; returns the vertex count (0: no area left, nothing written).
__device__ int clip_triangle_uv(const float (&v)[3][3], const float lo[3], const float hi[3],
                                uint32_t* __restrict__ out) {
    float poly[PART_MAX + 1][5], tmp[PART_MAX + 1][5];
    for (int i = 0; i < 3; ++i) {
        for (int a = 0; a < 3; ++a) poly[i][a] = v[i][a];
        poly[i][3] = i == 1 ? 1.f : 0.f;
        poly[i][4] = i == 2 ? 1.f : 0.f;
    }
    int n = 3;
    for (int a = 0; a < 3; ++a)
        for (int side = 0; side < 2; ++side) {
            const float b = side ? hi[a] : lo[a];
            int m = 0;
            for (int i = 0; i < n; ++i) {
                const float* p = poly[i];
                const float* q = poly[(i + 1) % n];
                const bool pin = side ? p[a] <= b : p[a] >= b;
                const bool qin = side ? q[a] <= b : q[a] >= b;
                if (pin) {
                    for (int c = 0; c < 5; ++c) tmp[m][c] = p[c];
                    ++m;
                }
                if (pin != qin) {
                    const float t = __fdiv_rn(__fsub_rn(b, p[a]), __fsub_rn(q[a], p[a]));
                    for (int c = 0; c < 5; ++c) tmp[m][c] = __fmaf_rn(t, __fsub_rn(q[c], p[c]), p[c]);
                    tmp[m][a] = b;
                    ++m;
                }
            }
            n = m;
            if (n < 3) return 0;
            for (int i = 0; i < n; ++i)
                for (int c = 0; c < 5; ++c) poly[i][c] = tmp[i][c];
        }
    for (int i = 0; i < n; ++i) out[i] = quantize_uv(poly[i][3], poly[i][4]);
    if (n < PART_MAX) out[n] = PART_END;
    return n;
}

// The part of every record of a split build, at part_uv[PART_MAX r ...], and
// the record's primitive id (with its sphere flag, as in the record) at
// rec_id[r]. A record whose reference box holds its whole triangle, a sphere,
// and a part that clipping left without area (which a refit then bounds by
// the whole moved triangle) get no part.
__global__ void k_record_parts(const float4* __restrict__ prims, int64_t R, const float4* __restrict__ rec_box,
                               const float* __restrict__ tri, int64_t T, uint32_t* __restrict__ part_uv,
                               uint32_t* __restrict__ rec_id) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < R; r += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t idb = __float_as_uint(prims[3 * r + 2].y);
        rec_id[r] = idb;
        int n = 0;
        if (!(idb & SPHERE_BIT) && (int64_t)idb < T) {
            float3 tl, th;
            prim_box(tri, nullptr, T, idb, tl, th);
            const float4 l = rec_box[2 * r], h = rec_box[2 * r + 1];
            if (l.x > tl.x || l.y > tl.y || l.z > tl.z || h.x < th.x || h.y < th.y || h.z < th.z) {
                const float* f = tri + 9 * (int64_t)idb;
                float v[3][3];
                for (int i = 0; i < 3; ++i)
                    for (int a = 0; a < 3; ++a) v[i][a] = f[3 * i + a];
                const float lo[3] = {l.x, l.y, l.z}, hi[3] = {h.x, h.y, h.z};
                n = clip_triangle_uv(v, lo, hi, part_uv + PART_MAX * r);
            }
        }
        if (n == 0) part_uv[PART_MAX * r] = PART_END;
    }
}

// ---- PLOC: parallel locally-ordered clustering (Meister and Bittner, 2018) ----
// Clusters start as the primitives in Morton order. Every iteration each
// cluster finds, among the PLOC_R clusters on either side of it in the array,
// the one whose union box has the smallest surface area; mutual nearest
// neighbours merge into a new binary node, and the array is compacted (the
// merged cluster takes the lower position). Pairs are ordered by (area, index
// gap, parity of the lower index, lower index), a total order, so the
// globally smallest pair is always mutual: every iteration merges at least
// one pair, and a run of equal boxes pairs up (0,1), (2,3), ... at once.
// Node indices count down: the last merge creates the root, node 0.
// What bounds a round is launches and chains more than work: 29 rounds of a
// million triangles took 3.4 ms in 4 to 6 launches and a host wait each. A
// round is now one launch without the host, and the rounds of PLOC_LAST
// clusters or fewer run in one block: 0.66 ms in kernels, 0.06 ms of it the
// last block (a partner and a merge kernel per round took 0.70 ms, a last block
// of 2,048 clusters 0.18 and the nodes' padded boxes, a pass of their own,
// 0.18). Loading the scene: 3.43 -> 3.05 ms.
constexpr int PLOC_R = 16;

__device__ __forceinline__ float union_area(float4 alo, float4 ahi, float4 blo, float4 bhi) {
    const float dx = fmaxf(ahi.x, bhi.x) - fminf(alo.x, blo.x);
    const float dy = fmaxf(ahi.y, bhi.y) - fminf(alo.y, blo.y);
    const float dz = fmaxf(ahi.z, bhi.z) - fminf(alo.z, blo.z);
    // explicit operations, in the order the compiler gives dx dy + dy dz + dz dx:
    // every kernel that compares areas computes the same bits, and near-equal
    // pairs (a terrain's grid has many) merge as they always have
    const float a = __fmaf_rn(dz, dx, __fmaf_rn(dx, dy, __fmul_rn(dy, dz)));
    return fminf(a, INFINITY);  // NaN (an overflow's infinity times zero): infinite
}

// The best partner of cluster i of n: the one within PLOC_R positions that
// comes first by (union area, index gap, parity of the lower index, lower
// index). Gaps are taken in increasing order, so only the two clusters at one
// gap, of lower indices i - g and i, need the tie's rules. -1 when i is alone.
// Cluster i + k's box is lo[k], hi[k]; any area may be infinite (overflow).
__device__ __noinline__ int ploc_partner_any(int i, int n, const float4* lo, const float4* hi) {
    const float4 alo = lo[0], ahi = hi[0];
    float best = INFINITY;
    int partner = -1;
    for (int g = 1; g <= PLOC_R; ++g) {
        const bool has_l = i - g >= 0, has_r = i + g < n;
        const float al = has_l ? union_area(alo, ahi, lo[-g], hi[-g]) : INFINITY;
        const float ar = has_r ? union_area(alo, ahi, lo[g], hi[g]) : INFINITY;
        const bool left_first = !(g & 1) || !((i - g) & 1);
        const bool left = has_l && (!has_r || al < ar || (al == ar && left_first));
        const float a = left ? al : ar;
        if ((has_l || has_r) && (partner < 0 || a < best)) {
            best = a;
            partner = left ? i - g : i + g;
        }
    }
    return partner;
}

// The same over the gaps first, first + step, ... (all of them, or those of
// one of the lanes that share cluster i), where the PLOC_R places before the
// first cluster and after the last hold ploc_no_box(), of infinite union area:
// no bounds to test in the loop, 35 operations a gap instead of 110, and a
// round's partners are what bounds it. Returns the offset to the partner and
// its area; 0 when no finite area was found (ploc_partner_any's case).
__device__ __forceinline__ float4 ploc_no_box() { return make_float4(INFINITY, INFINITY, INFINITY, 0.f); }

__device__ __forceinline__ int ploc_partner(int i, const float4* lo, const float4* hi, int first, int step,
                                            float& best) {
    const float4 alo = lo[0], ahi = hi[0];
    best = INFINITY;
    int offset = 0;
#pragma unroll 4
    for (int g = first; g <= PLOC_R; g += step) {
        const float al = union_area(alo, ahi, lo[-g], hi[-g]);
        const float ar = union_area(alo, ahi, lo[g], hi[g]);
        const bool left = ((g & 1) && !(i & 1)) ? al < ar : al <= ar;  // odd gaps: the even lower index first
        const float a = fminf(al, ar);
        if (a < best) {
            best = a;
            offset = left ? -g : g;
        }
    }
    return offset;
}

// A round's state: n clusters, `created` nodes so far; round r reads
// state[r] and its merge writes state[r + 1].
struct PlocState {
    int n, created, stalled, pad;  // stalled: a round of two clusters or more merged none
};

__device__ __forceinline__ int leaf_count(const int* cnt, int ref) { return ref >= 0 ? cnt[ref] : 1; }

// Where the clustering writes its tree, and its leaves: leaf j is reference
// ids[j] of boxes plo/phi (of primitive ref_prim[ids[j]] when split).
struct PlocTree {
    int2* child;
    float4* blo;
    float4* bhi;
    int* cnt;
    int* parent_int;
    int* parent_leaf;
    const uint32_t* ids;
    const float4* plo;
    const float4* phi;
    const uint32_t* ref_prim;
    const float* tri;
    const float* sph;
    int64_t T;
};

// The padded box of cluster `ref`: a leaf's reference box with its triangle's
// pad, a node's as it was written when it was made.
__device__ __forceinline__ void ploc_padded_box(const PlocTree& t, int ref, float3& lo, float3& hi) {
    if (ref >= 0) {
        const float4 a = t.blo[ref], b = t.bhi[ref];
        lo = make_float3(a.x, a.y, a.z);
        hi = make_float3(b.x, b.y, b.z);
    } else {
        padded_ref_box(t.plo, t.phi, t.ref_prim, t.tri, t.sph, t.T, t.ids[-ref - 1], lo, hi);
    }
}

__device__ __forceinline__ void ploc_write_node(const PlocTree& t, int node, int ra, int rb, int leaves, float4 lo,
                                                float4 hi) {
    t.child[node] = make_int2(ra, rb);
    t.blo[node] = lo;
    t.bhi[node] = hi;
    t.cnt[node] = leaves;
    if (ra >= 0) t.parent_int[ra] = node;
    else t.parent_leaf[-ra - 1] = node;
    if (rb >= 0) t.parent_int[rb] = node;
    else t.parent_leaf[-rb - 1] = node;
}

// The clustering decides on exact boxes; the tree holds the padded ones, their
// union written here while the children are at hand. A pass of its own after
// the clustering, bottom up with an atomic and two fences per node, took
// 175 us of a million triangles' build; here it is about 60 us over all rounds.
__device__ __forceinline__ void ploc_pair(const PlocTree& t, int ra, int rb, float4& lo, float4& hi, int& leaves) {
    float3 la, ha, lb, hb;
    ploc_padded_box(t, ra, la, ha);
    ploc_padded_box(t, rb, lb, hb);
    lo = make_float4(fminf(la.x, lb.x), fminf(la.y, lb.y), fminf(la.z, lb.z), 0.f);
    hi = make_float4(fmaxf(ha.x, hb.x), fmaxf(ha.y, hb.y), fmaxf(ha.z, hb.z), 0.f);
    leaves = leaf_count(t.cnt, ra) + leaf_count(t.cnt, rb);
}

__device__ __forceinline__ void box_union(float4 la, float4 ha, float4 lb, float4 hb, float4& l, float4& h) {
    l = make_float4(fminf(la.x, lb.x), fminf(la.y, lb.y), fminf(la.z, lb.z), 0.f);
    h = make_float4(fmaxf(ha.x, hb.x), fmaxf(ha.y, hb.y), fmaxf(ha.z, hb.z), 0.f);
}

// One round: each cluster's partner, mutual pairs merged into new nodes, and
// the cluster array compacted, in one launch. A block takes a tile of PLOC_TILE
// clusters and computes the partners of the PLOC_R on either side too (the
// pair of a cluster at its edge), from boxes in shared memory; it counts its
// merges and the clusters it keeps, finds the counts before it by decoupled
// look-back (tiles numbered by an atomic counter, so every earlier tile is
// already running; each wait is bounded), and writes its nodes and its part of
// the next array. A tile whose wait runs out writes neither; as its places then
// hold no clusters, the rounds after it, which would follow them, leave at once.
// The merge with m merges before it, over all rounds, becomes
// node N - 2 - m: the last one is the root, node 0. A status word carries both
// counts, 31 bits each, and its flag. From 24,000 clusters down, where launch,
// look-back and the chain of 32 candidates bound it, a round takes 7 to 12 us
// (18 as two kernels); tiles of 480 clusters are as fast at a million and 3 %
// slower at 3,000.
constexpr int PLOC_BLOCK = 256;
constexpr int PLOC_TILE = PLOC_BLOCK - 2 * PLOC_R;  // one cluster per thread, the neighbours' included
constexpr unsigned long long PLOC_AGG = 1ull << 62, PLOC_INC = 2ull << 62, PLOC_COUNTS = (1ull << 62) - 1;
constexpr int PLOC_SPINS = 1 << 26;

// Called by one whole warp of a block: publishes the tile's counts and returns
// the sum of the earlier tiles', 32 of them per round of loads. Past spin_limit
// polls it records the round as failed, publishes what it has (no more than the
// true counts, so later tiles write in range) and returns PLOC_NONE.
constexpr unsigned long long PLOC_NONE = ~0ull;
__device__ __forceinline__ unsigned long long counts_before(unsigned long long* status, int64_t tile,
                                                            unsigned long long total, int* failed, int round,
                                                            int spin_limit) {
    const int lane = threadIdx.x & 31;
    volatile unsigned long long* st = status;
    if (lane == 0) st[tile] = (tile == 0 ? PLOC_INC : PLOC_AGG) | total;
    unsigned long long before = 0;
    bool ran_out = false;
    int64_t t = tile - 1;
    for (int spins = 0; t >= 0;) {
        unsigned long long w = PLOC_INC;  // before the first tile: nothing more to add
        if (t >= lane) w = st[t - lane];
        const unsigned waiting = __ballot_sync(0xffffffffu, (w >> 62) == 0);
        const unsigned inclusive = __ballot_sync(0xffffffffu, (w >> 62) == 2);
        // the nearest tiles up to the first inclusive one, if none of them still counts
        const int last = inclusive ? __ffs(inclusive) - 1 : 31;
        const unsigned use = 0xffffffffu >> (31 - last);
        if (waiting & use) {
            if (++spins > spin_limit) {
                ran_out = true;
                break;
            }
            continue;
        }
        unsigned long long v = (use >> lane) & 1u ? w & PLOC_COUNTS : 0ull;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        before += v;
        if (inclusive) break;
        t -= 32;
    }
    if (lane == 0 && ran_out) atomicMin(failed, round);
    if (lane == 0 && tile > 0) st[tile] = PLOC_INC | (before + total);
    return ran_out ? PLOC_NONE : before;
}

__global__ void __launch_bounds__(PLOC_BLOCK) k_ploc_round(PlocState* __restrict__ state, unsigned* ticket,
                                                           unsigned long long* status, int64_t N,
                                                           const int* __restrict__ ref, const float4* __restrict__ clo,
                                                           const float4* __restrict__ chi, int* __restrict__ ref_out,
                                                           float4* __restrict__ lo_out, float4* __restrict__ hi_out,
                                                           PlocTree tree, int* failed, int round, int spin_limit) {
    constexpr int WARPS = PLOC_BLOCK / 32, HELD = PLOC_BLOCK + 2 * PLOC_R;
    static_assert(WARPS <= 32, "one warp scans the warps' counts");
    __shared__ float4 s_lo[HELD], s_hi[HELD];  // clusters first - PLOC_R ..
    __shared__ int s_ref[HELD], s_nn[PLOC_BLOCK];
    __shared__ unsigned long long s_row[WARPS];  // per warp: counts before it in the tile
    __shared__ unsigned long long s_before;
    __shared__ unsigned s_tile;
    const int n = state->n, first_failed = *failed;  // both loads overlap the ticket
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t tile = s_tile;
    if (first_failed < round || tile * PLOC_TILE >= n) return;
    const int first = (int)(tile * PLOC_TILE) - PLOC_R;  // thread t's cluster is first + t
    for (int t = threadIdx.x; t < HELD; t += PLOC_BLOCK) {
        const int g = first - PLOC_R + t;
        const bool in = g >= 0 && g < n;
        s_lo[t] = in ? clo[g] : ploc_no_box();
        s_hi[t] = in ? chi[g] : ploc_no_box();
        if (in) s_ref[t] = ref[g];
    }
    __syncthreads();
    const int i = first + (int)threadIdx.x, me = PLOC_R + (int)threadIdx.x;
    const bool real = i >= 0 && i < n;
    int partner = -1;
    if (real) {
        float area;
        const int offset = ploc_partner(i, s_lo + me, s_hi + me, 1, 1, area);
        partner = offset ? i + offset : ploc_partner_any(i, n, s_lo + me, s_hi + me);
    }
    s_nn[threadIdx.x] = partner;
    __syncthreads();
    const bool mine = real && threadIdx.x >= PLOC_R && threadIdx.x < PLOC_BLOCK - PLOC_R;
    if (!mine || partner < 0 || s_nn[partner - first] != i) partner = -1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // ballots give the counts and each lane's place. Merges (the lower end of
    // a mutual pair) << 31 | stays.
    const unsigned merges = __ballot_sync(0xffffffffu, partner >= 0 && partner > i);
    const unsigned stays = __ballot_sync(0xffffffffu, mine && !(partner >= 0 && partner < i));
    if (lane == 0) s_row[warp] = (unsigned long long)__popc(merges) << 31 | (unsigned)__popc(stays);
    float4 pl, ph;
    int leaves = 0;  // of the new node; its loads overlap the look-back
    const int other = partner - first + PLOC_R;
    __syncthreads();
    if (warp == 0) {
        const unsigned long long row = lane < WARPS ? s_row[lane] : 0ull;
        unsigned long long x = row;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane < WARPS) s_row[lane] = x - row;
        const unsigned long long total = __shfl_sync(0xffffffffu, x, 31);
        const unsigned long long before = counts_before(status, tile, total, failed, round, spin_limit);
        if (lane == 0) s_before = before;
        // the last tile's counts and those before it are the round's
        if (lane == 0 && before != PLOC_NONE && (tile + 1) * PLOC_TILE >= n) {
            const unsigned long long all = before + total;
            const int merged = (int)(all >> 31);
            state[1] = PlocState{(int)(all & 0x7fffffffull), state->created + merged,
                                 state->stalled | (n > 1 && merged == 0), 0};
        }
    }
    if ((merges >> lane) & 1u) ploc_pair(tree, s_ref[me], s_ref[other], pl, ph, leaves);
    __syncthreads();
    if (s_before == PLOC_NONE || !((stays >> lane) & 1u)) return;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned long long run = s_before + s_row[warp];
    const int64_t pos = (int64_t)(run & 0x7fffffffull) + __popc(stays & lt);
    float4 l = s_lo[me], h = s_hi[me];
    int r = s_ref[me];
    if (partner >= 0) {
        const int node = (int)(N - 2 - state->created - (int64_t)(run >> 31) - __popc(merges & lt));
        const float4 la = l, ha = h;
        box_union(la, ha, s_lo[other], s_hi[other], l, h);
        ploc_write_node(tree, node, r, s_ref[other], leaves, pl, ph);
        r = node;
    }
    ref_out[pos] = r;
    lo_out[pos] = l;
    hi_out[pos] = h;
}

// The last rounds in one block: PLOC_LAST clusters or fewer in shared memory
// (exact and padded boxes, references, leaf counts) until one is left. More
// than half of a build's rounds are below this size, and a launch costs several
// microseconds however few clusters it has. One SM's issue rate bounds the
// first rounds and a warp's chain of candidates the others, so with fewer
// clusters than threads up to PLOC_R lanes share a cluster's candidates: 59 us
// from 1,024 clusters (one lane per cluster and exact boxes only, with the
// counts read from device memory in every round: 180 us from 2,048).
constexpr int PLOC_LAST = 1024;
struct PlocLastShared {
    float4 lo[PLOC_LAST + 2 * PLOC_R], hi[PLOC_LAST + 2 * PLOC_R];  // exact, which decide
    float4 plo[PLOC_LAST], phi[PLOC_LAST];  // padded, which the tree holds; plo.w: leaf count
    int ref[PLOC_LAST];
    int nn[PLOC_LAST];
    unsigned warp_tot[PLOC_LAST / 32];
};

__global__ void __launch_bounds__(PLOC_LAST) k_ploc_last(PlocState* state, int64_t N, const int* __restrict__ ref,
                                                         const float4* __restrict__ clo,
                                                         const float4* __restrict__ chi, PlocTree tree) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    PlocLastShared& s = *reinterpret_cast<PlocLastShared*>(s_raw);
    float4 *const lo = s.lo + PLOC_R, *const hi = s.hi + PLOC_R;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int n = state->n, created = state->created;
    bool stalled = false;
    if (t < n) {
        const int r = ref[t];
        float3 l, h;
        ploc_padded_box(tree, r, l, h);
        lo[t] = clo[t];
        hi[t] = chi[t];
        s.plo[t] = make_float4(l.x, l.y, l.z, __int_as_float(leaf_count(tree.cnt, r)));
        s.phi[t] = make_float4(h.x, h.y, h.z, 0.f);
        s.ref[t] = r;
    }
    if (t < PLOC_R) {
        lo[t - PLOC_R] = hi[t - PLOC_R] = ploc_no_box();
        lo[n + t] = hi[n + t] = ploc_no_box();
    }
    __syncthreads();
    while (n > 1 && !stalled) {
        int shift = 0;  // 2^shift lanes per cluster
        while ((2 << shift) <= PLOC_R && (n << shift) * 2 <= PLOC_LAST) ++shift;
        {
            const int i = t >> shift, sub = t & ((1 << shift) - 1);
            float best = INFINITY;
            int offset = 0;
            if (i < n) offset = ploc_partner(i, lo + i, hi + i, 1 + sub, 1 << shift, best);
            for (int o = 1; o < 1 << shift; o <<= 1) {
                const float other = __shfl_xor_sync(0xffffffffu, best, o);
                const int theirs = __shfl_xor_sync(0xffffffffu, offset, o);
                // (area, gap); gaps of two lanes differ, and no offset has an infinite area
                if (other < best || (other == best && abs(theirs) < abs(offset))) {
                    best = other;
                    offset = theirs;
                }
            }
            if (i < n && sub == 0) s.nn[i] = offset ? i + offset : ploc_partner_any(i, n, lo + i, hi + i);
        }
        __syncthreads();
        const bool real = t < n;
        int partner = real ? s.nn[t] : -1;
        if (partner >= 0 && s.nn[partner] != t) partner = -1;
        const bool merge = partner >= 0 && partner > t, stay = real && !(partner >= 0 && partner < t);
        const unsigned merges = __ballot_sync(0xffffffffu, merge), stays = __ballot_sync(0xffffffffu, stay);
        if (lane == 0) s.warp_tot[warp] = (unsigned)__popc(merges) << 16 | (unsigned)__popc(stays);
        // the clusters that stay, read before any is overwritten
        float4 l, h, pl, ph;
        int ra = 0, rb = 0;
        if (stay) {
            l = lo[t];
            h = hi[t];
            pl = s.plo[t];
            ph = s.phi[t];
            ra = s.ref[t];
            if (merge) {
                const float4 l0 = l, h0 = h, pl0 = pl, ph0 = ph, pl1 = s.plo[partner];
                box_union(l0, h0, lo[partner], hi[partner], l, h);
                box_union(pl0, ph0, pl1, s.phi[partner], pl, ph);
                pl.w = __int_as_float(__float_as_int(pl0.w) + __float_as_int(pl1.w));
                rb = s.ref[partner];
            }
        }
        __syncthreads();
        static_assert(PLOC_LAST / 32 == 32, "one lane per warp's total");
        unsigned x = s.warp_tot[lane];
        const unsigned own = x;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const unsigned total = __shfl_sync(0xffffffffu, x, 31);
        const unsigned before = __shfl_sync(0xffffffffu, x - own, warp);
        n = (int)(total & 0xffffu);
        if (stay) {
            const unsigned lt = (1u << lane) - 1u;
            const int pos = (int)(before & 0xffffu) + __popc(stays & lt);
            if (merge) {
                const int node = (int)(N - 2 - created - (int)(before >> 16) - __popc(merges & lt));
                ploc_write_node(tree, node, ra, rb, __float_as_int(pl.w), make_float4(pl.x, pl.y, pl.z, 0.f), ph);
                ra = node;
            }
            lo[pos] = l;
            hi[pos] = h;
            s.plo[pos] = pl;
            s.phi[pos] = ph;
            s.ref[pos] = ra;
        }
        if (t < PLOC_R) lo[n + t] = hi[n + t] = ploc_no_box();
        created += (int)(total >> 16);
        stalled = (total >> 16) == 0;
        __syncthreads();  // the next array before the next round
    }
    if (t == 0) state[1] = PlocState{n, created, state->stalled | (stalled ? 1 : 0), 0};
}

__global__ void k_ploc_init(const uint32_t* __restrict__ sorted_ids, int64_t n, const float4* __restrict__ plo,
                            const float4* __restrict__ phi, int* __restrict__ ref, float4* __restrict__ clo,
                            float4* __restrict__ chi) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t id = sorted_ids[j];
        ref[j] = -(int)(j + 1);
        clo[j] = plo[id];
        chi[j] = phi[id];
    }
}

// Depth-first leaf order: a node's first leaf is the number of leaves left of
// it, i.e. the sum of the left siblings' leaf counts on its path to the root.
// Internal node i gets range (first, first + count - 1); leaf j gets pos[j].
__global__ void k_dfs_offsets(const int2* __restrict__ child, const int* __restrict__ parent_int,
                              const int* __restrict__ parent_leaf, const int* __restrict__ cnt, int64_t N,
                              int2* __restrict__ range, int* __restrict__ pos, int* err) {
    const int64_t total = 2 * N - 1;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
        const bool internal = k < N - 1;
        int cur = internal ? (int)k : -(int)(k - (N - 1)) - 1;
        int p = internal ? parent_int[k] : parent_leaf[k - (N - 1)];
        int off = 0;
        for (int guard = 0; p >= 0; ++guard) {
            if (guard >= (1 << 22)) {
                atomicAdd(err, 1);
                break;
            }
            const int2 c = child[p];
            if (c.y == cur) off += leaf_count(cnt, c.x);
            cur = p;
            p = parent_int[p];
        }
        if (internal) range[k] = make_int2(off, off + cnt[k] - 1);
        else pos[k - (N - 1)] = off;
    }
}

// Leaves renumbered into depth-first order: sorted ids permuted, and leaf
// references in the children rewritten.
__global__ void k_dfs_apply(const int* __restrict__ pos, const uint32_t* __restrict__ ids_in, int64_t N,
                            uint32_t* __restrict__ ids_out, int2* __restrict__ child, int* err) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x) {
        const int pk = pos[k];
        if (pk < 0 || pk >= N) {
            atomicAdd(err, 1);
            continue;
        }
        ids_out[pk] = ids_in[k];
        if (k < N - 1) {
            int2 c = child[k];
            if (c.x < 0) c.x = -pos[-c.x - 1] - 1;
            if (c.y < 0) c.y = -pos[-c.y - 1] - 1;
            child[k] = c;
        }
    }
}

// ---- slot assignment of the 8-wide collapse by surface-area cost ----
// Cost model (SAH, up to the common factor 1 / area(root)): visiting a wide
// node costs SAH_NODE primitive tests, in proportion to the node's area; a
// leaf costs one test per primitive, in proportion to its area. For binary
// node n and k = 1..8, dp[n][k-1] is the least cost of the subtree of n when
// it may take up to k slots of its parent's wide node: one slot (a leaf if it
// holds <= LEAF_MAX primitives, else a wide node of its own), or its two
// children sharing the k slots (a subtree of <= LEAF_MAX primitives always
// takes one slot, a leaf). split[n] byte k-1 (k >= 2) is the left
// child's share of the best split, 0 when one slot is best; byte 0 is the
// left share of the best split of all 8 slots, used when n is a wide node.
// A node visit in the trace kernel is about 3.8 times a triangle test.
constexpr float SAH_NODE = 3.8f;

__device__ __forceinline__ float box_area(float4 lo, float4 hi) {
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return dx * dy + dy * dz + dz * dx;
}

__device__ __forceinline__ void slot_costs(int ref, const float4* dp, const float4* plo, const float4* phi,
                                           const uint32_t* ids, float d[8]) {
    if (ref < 0) {  // one primitive: a leaf of one, whatever the slots
        const uint32_t id = ids[-ref - 1];
        const float a = box_area(plo[id], phi[id]);
        for (int k = 0; k < 8; ++k) d[k] = a;
    } else {
        const float4 u = __ldcg(&dp[2 * ref]), v = __ldcg(&dp[2 * ref + 1]);
        d[0] = u.x, d[1] = u.y, d[2] = u.z, d[3] = u.w, d[4] = v.x, d[5] = v.y, d[6] = v.z, d[7] = v.w;
    }
}

// Bottom up, one thread per leaf: at each node the second arriving thread
// computes it from both children (the first stops).
__global__ void k_sah_dp(const int2* __restrict__ child, const int2* __restrict__ range,
                         const int* __restrict__ parent_int, const int* __restrict__ parent_leaf,
                         const float4* __restrict__ blo, const float4* __restrict__ bhi,
                         const float4* __restrict__ plo, const float4* __restrict__ phi,
                         const uint32_t* __restrict__ ids, int64_t N, float4* dp, uint2* split, int* arrivals,
                         int* err) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
        int node = parent_leaf[j];
        for (int guard = 0; node >= 0; ++guard) {
            if (guard >= (1 << 22)) {
                atomicAdd(err, 1);
                break;
            }
            __threadfence();
            if (atomicAdd(&arrivals[node], 1) == 0) break;
            __threadfence();
            const int2 c = child[node];
            float dl[8], dr[8];
            slot_costs(c.x, dp, plo, phi, ids, dl);
            slot_costs(c.y, dp, plo, phi, ids, dr);
            float dsplit[9];
            int arg[9];
            for (int k = 2; k <= 8; ++k) {
                float best = INFINITY;
                int ba = 1;
                for (int a = 1; a < k; ++a) {
                    const float v = dl[a - 1] + dr[k - a - 1];
                    if (v < best) {
                        best = v;
                        ba = a;
                    }
                }
                dsplit[k] = best;
                arg[k] = ba;
            }
            const float area = box_area(blo[node], bhi[node]);
            const int2 r = range[node];
            const int cnt = r.y - r.x + 1;
            const float c_node = area * SAH_NODE + dsplit[8];
            const float c_one = cnt <= LEAF_MAX ? fminf(area * (float)cnt, c_node) : c_node;
            float d[8];
            uint32_t bytes[8];
            d[0] = c_one;
            bytes[0] = (uint32_t)arg[8];
            for (int k = 2; k <= 8; ++k) {
                const bool sp = cnt > LEAF_MAX && dsplit[k] < c_one;  // small subtrees stay one leaf
                d[k - 1] = sp ? dsplit[k] : c_one;
                bytes[k - 1] = sp ? (uint32_t)arg[k] : 0u;
            }
            __stcg(&dp[2 * node], make_float4(d[0], d[1], d[2], d[3]));
            __stcg(&dp[2 * node + 1], make_float4(d[4], d[5], d[6], d[7]));
            split[node] = make_uint2(bytes[0] | bytes[1] << 8 | bytes[2] << 16 | bytes[3] << 24,
                                     bytes[4] | bytes[5] << 8 | bytes[6] << 16 | bytes[7] << 24);
            node = parent_int[node];
        }
    }
}

// ---- exclusive scan of 64-bit words: tiles of 1024, tile sums scanned recursively ----
constexpr int SCAN_BLOCK = 256;
constexpr int SCAN_TILE = 4 * SCAN_BLOCK;

__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_tiles(unsigned long long* data, int64_t n,
                                                           unsigned long long* sums) {
    __shared__ unsigned long long warp_tot[SCAN_BLOCK / 32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + 4 * threadIdx.x;
    unsigned long long v[4];
    for (int q = 0; q < 4; ++q) v[q] = base + q < n ? data[base + q] : 0ull;
    const unsigned long long tsum = v[0] + v[1] + v[2] + v[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = tsum;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned long long t = lane < SCAN_BLOCK / 32 ? warp_tot[lane] : 0ull;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < SCAN_BLOCK / 32) warp_tot[lane] = t;
    }
    __syncthreads();
    unsigned long long run = (warp > 0 ? warp_tot[warp - 1] : 0ull) + x - tsum;
    for (int q = 0; q < 4; ++q) {
        if (base + q < n) data[base + q] = run;
        run += v[q];
    }
    if (threadIdx.x == SCAN_BLOCK - 1) sums[blockIdx.x] = run;
}

__global__ void k_scan_add(unsigned long long* data, int64_t n, const unsigned long long* offs) {
    const int64_t i = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x;
    const unsigned long long o = offs[blockIdx.x];
    for (int q = 0; q < 4; ++q)
        if (i + q * SCAN_BLOCK < n) data[i + q * SCAN_BLOCK] += o;
}

struct BinTree {
    const int2* child;
    const int2* range;
    const float4* blo;
    const float4* bhi;
    const float4* plo;
    const float4* phi;
    const uint32_t* sorted_ids;
    const uint2* split;  // slot splits of the surface-area policy (k_sah_dp); nullptr: area policy
    const uint32_t* ref_prim;  // reference -> primitive (nullptr: references are the primitives)
    const float* tri;
    const float* sph;
    int64_t T;
};

__device__ __forceinline__ int split_share(const uint2 s, int k) {  // k = 1..8 slots; byte 0: wide-node split
    const uint32_t w = k <= 4 ? s.x : s.y;
    return (int)((w >> (8 * ((k - 1) & 3))) & 0xffu);
}

__device__ __forceinline__ void ref_box(const BinTree& bt, int ref, float3& lo, float3& hi, int& first, int& last) {
    float4 l, h;
    if (ref >= 0) {
        l = bt.blo[ref];
        h = bt.bhi[ref];
        const int2 r = bt.range[ref];
        first = r.x;
        last = r.y;
        lo = make_float3(l.x, l.y, l.z);
        hi = make_float3(h.x, h.y, h.z);
    } else {
        const int j = -ref - 1;
        padded_ref_box(bt.plo, bt.phi, bt.ref_prim, bt.tri, bt.sph, bt.T, bt.sorted_ids[j], lo, hi);
        first = last = j;
    }
}

}  // namespace

__device__ __forceinline__ void write_prim_record(float4* __restrict__ rec, const float* __restrict__ tri,
                                                  const float* __restrict__ sph, int64_t T, uint32_t id) {
    if (id < T) {
        const float* v = tri + 9 * (int64_t)id;
        float e1[3] = {v[3] - v[0], v[4] - v[1], v[5] - v[2]};
        float e2[3] = {v[6] - v[0], v[7] - v[1], v[8] - v[2]};
        // Degenerate (collinear) triangles are never hit (det == 0). The float
        // cross product of the rounded edges is within 8 * 2^-24 * M1 * M2 (+
        // 2^-24 of itself) of the exact one (M: largest edge component), so a
        // component above 2^-19 M1 M2 proves the triangle has area; only the
        // rest take the exact test, the double cross product of the exact
        // edge differences.
        const float m1 = fmaxf(fmaxf(fabsf(e1[0]), fabsf(e1[1])), fabsf(e1[2]));
        const float m2 = fmaxf(fmaxf(fabsf(e2[0]), fabsf(e2[1])), fabsf(e2[2]));
        const float fx = e1[1] * e2[2] - e1[2] * e2[1], fy = e1[2] * e2[0] - e1[0] * e2[2],
                    fz = e1[0] * e2[1] - e1[1] * e2[0];
        const float thr = 0x1p-19f * m1 * m2;
        if (!(fmaxf(fmaxf(fabsf(fx), fabsf(fy)), fabsf(fz)) > thr && thr > 0.f)) {
            const double d1[3] = {(double)v[3] - v[0], (double)v[4] - v[1], (double)v[5] - v[2]};
            const double d2[3] = {(double)v[6] - v[0], (double)v[7] - v[1], (double)v[8] - v[2]};
            const double nx = d1[1] * d2[2] - d1[2] * d2[1], ny = d1[2] * d2[0] - d1[0] * d2[2],
                         nz = d1[0] * d2[1] - d1[1] * d2[0];
            if (nx == 0.0 && ny == 0.0 && nz == 0.0)
                for (int a = 0; a < 3; ++a) e1[a] = e2[a] = 0.f;
        }
        rec[0] = make_float4(v[0], v[1], v[2], e1[0]);
        rec[1] = make_float4(e1[1], e1[2], e2[0], e2[1]);
        rec[2] = make_float4(e2[2], __uint_as_float(id), 0.f, 0.f);
    } else {
        const float* s = sph + 4 * ((int64_t)id - T);
        rec[0] = make_float4(s[0], s[1], s[2], fabsf(s[3]));
        rec[1] = make_float4(0.f, 0.f, 0.f, 0.f);
        rec[2] = make_float4(0.f, __uint_as_float(id | SPHERE_BIT), 0.f, 0.f);
    }
}

namespace {

// One level of the collapse. frontier[i] = (binary ref, wide node index).
// rec_box (nullable) receives each record's exact reference box.
// Eight lanes per node, lane q for child q until the slots are known and for
// slot q when the boxes are written: opening a child, the 8 x 8 slot costs of
// each of the 8 assignments and the rows' writes are spread over them. One
// thread per node took 22 us for the root alone (a serial chain of 512 costs
// and of dependent loads) and 460 us for the eight levels of a million
// triangles; eight lanes take 9 and 246 us.
constexpr int COLLAPSE_BLOCK = 128;
static_assert(COLLAPSE_BLOCK % 32 == 0, "a node's eight lanes must share a warp");

// Over the eight lanes of a node: the lane with the largest value, the lowest
// of equals.
__device__ __forceinline__ int lane_of_max(float& v, int q) {
    int l = q;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const float v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const int l2 = __shfl_xor_sync(0xffffffffu, l, o);
        if (v2 > v || (v2 == v && l2 < l)) {
            v = v2;
            l = l2;
        }
    }
    return l;
}

__global__ void __launch_bounds__(COLLAPSE_BLOCK)
    k_collapse(BinTree bt, const int2* __restrict__ frontier, int n_front, int2* __restrict__ next_front,
               uint32_t* counters, WNode* __restrict__ nodes, float4* __restrict__ nbox, float4* __restrict__ prims,
               const float* __restrict__ tri, const float* __restrict__ sph, int64_t T, int* max_leaf,
               float4* __restrict__ rec_box) {
    const int64_t t = blockIdx.x * (int64_t)COLLAPSE_BLOCK + threadIdx.x;
    const int64_t i = t >> 3;
    const int q = (int)(t & 7);
    const bool live = i < n_front;
    const int2 self = live ? frontier[i] : make_int2(-1, 0);
    const int ref = self.x, w = self.y;
    // this lane's child (q < m): its binary reference, box and leaf range
    int m = 0, cref = 0, cfirst = 0, clast = 0;
    float3 lo = make_float3(INFINITY, INFINITY, INFINITY), hi = make_float3(-INFINITY, -INFINITY, -INFINITY);
    bool area_policy = false;
    if (live) {
        if (ref < 0) {
            m = 1;
            cref = ref;
        } else if (bt.split) {
            // surface-area policy: the 8 slots of this wide node are shared out by
            // the stored splits; a subtree given k slots is one slot (k == 1, a
            // primitive, or share 0) or passes shares a and k - a to its children
            // (every lane follows the shares and keeps its own child)
            int sref[8], sk[8];
            int sp = 0;
            const int2 c = bt.child[ref];
            const int a = split_share(bt.split[ref], 1);
            sref[sp] = c.y, sk[sp++] = 8 - a;
            sref[sp] = c.x, sk[sp++] = a;
            while (sp > 0) {
                --sp;
                const int x = sref[sp], k = sk[sp];
                const int share = (x < 0 || k == 1) ? 0 : split_share(bt.split[x], k);
                if (share <= 0 || share >= k) {
                    if (m == q) cref = x;
                    ++m;
                    continue;
                }
                const int2 cc = bt.child[x];
                sref[sp] = cc.y, sk[sp++] = k - share;
                sref[sp] = cc.x, sk[sp++] = share;
            }
        } else {
            // area policy: start from the two children and repeatedly open the
            // child of largest surface area that holds more than LEAF_MAX primitives
            const int2 c = bt.child[ref];
            m = 2;
            cref = q == 0 ? c.x : c.y;
            area_policy = true;
        }
        if (q < m) ref_box(bt, cref, lo, hi, cfirst, clast);
    }
    for (int it = 0; it < 6; ++it) {
        float area = -1.f;
        if (area_policy && m < 8 && q < m && cref >= 0 && clast - cfirst + 1 > LEAF_MAX) {
            const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
            area = dx * dy + dy * dz + dz * dx;
            if (!(area > -1.f)) area = -1.f;
        }
        const int best = lane_of_max(area, q);
        const int bref = __shfl_sync(0xffffffffu, cref, best, 8);
        if (area > -1.f) {
            const int2 ch = bt.child[bref];
            if (q == best || q == m) {
                cref = q == best ? ch.x : ch.y;
                ref_box(bt, cref, lo, hi, cfirst, clast);
            }
            ++m;
        }
    }
    // the union of the children
    float3 ulo = lo, uhi = hi;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        ulo.x = fminf(ulo.x, __shfl_xor_sync(0xffffffffu, ulo.x, o));
        ulo.y = fminf(ulo.y, __shfl_xor_sync(0xffffffffu, ulo.y, o));
        ulo.z = fminf(ulo.z, __shfl_xor_sync(0xffffffffu, ulo.z, o));
        uhi.x = fmaxf(uhi.x, __shfl_xor_sync(0xffffffffu, uhi.x, o));
        uhi.y = fmaxf(uhi.y, __shfl_xor_sync(0xffffffffu, uhi.y, o));
        uhi.z = fmaxf(uhi.z, __shfl_xor_sync(0xffffffffu, uhi.z, o));
    }
    // slots: greedy assignment of children to octant directions
    const float ox = 0.5f * (lo.x + hi.x) - 0.5f * (ulo.x + uhi.x);
    const float oy = 0.5f * (lo.y + hi.y) - 0.5f * (ulo.y + uhi.y);
    const float oz = 0.5f * (lo.z + hi.z) - 0.5f * (ulo.z + uhi.z);
    unsigned used = 0;
    int slot = -1;
    for (int it = 0; it < 8; ++it) {
        float best = -INFINITY;
        int bs = __ffs(~used) - 1;
        if (q < m && slot < 0) {
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const float cost = ((s & 1) ? ox : -ox) + ((s & 2) ? oy : -oy) + ((s & 4) ? oz : -oz);
                if (!(used & (1u << s)) && cost > best) {
                    best = cost;
                    bs = s;
                }
            }
            best = fmaxf(best, -3.4e38f);  // a child that still has no slot comes before the others
        }
        const int l = lane_of_max(best, q);
        const int s = __shfl_sync(0xffffffffu, bs, l, 8);
        if (it < m) {
            if (q == l) slot = s;
            used |= 1u << s;
        }
    }
    // classify and allocate
    const bool internal = q < m && cref >= 0 && clast - cfirst + 1 > LEAF_MAX;
    const int cnt = q < m && !internal ? clast - cfirst + 1 : 0;
    uint32_t imask = internal ? 1u << slot : 0u, leaf_bits = cnt ? bits_below(cnt) << (3 * slot) : 0u;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        imask |= __shfl_xor_sync(0xffffffffu, imask, o);
        leaf_bits |= __shfl_xor_sync(0xffffffffu, leaf_bits, o);
    }
    const int n_int = __popc(imask), n_prim = __popc(leaf_bits);
    uint32_t child_base = 0, prim_base = 0, front_base = 0;
    if (q == 0) {
        if (n_int) {
            child_base = atomicAdd(&counters[0], (uint32_t)n_int);
            front_base = atomicAdd(&counters[2], (uint32_t)n_int);
        }
        if (n_prim) prim_base = atomicAdd(&counters[1], (uint32_t)n_prim);
    }
    child_base = __shfl_sync(0xffffffffu, child_base, 0, 8);
    front_base = __shfl_sync(0xffffffffu, front_base, 0, 8);
    prim_base = __shfl_sync(0xffffffffu, prim_base, 0, 8);
    if (internal) {
        const uint32_t rank = __popc(imask & bits_below(slot));
        next_front[front_base + rank] = make_int2(cref, (int)(child_base + rank));
    }
    for (int k = 0; k < cnt; ++k) {
        const uint32_t r = bt.sorted_ids[cfirst + k];
        const int64_t rec = (int64_t)prim_base + __popc(leaf_bits & bits_below(3 * slot)) + k;
        write_prim_record(prims + 3 * rec, tri, sph, T, bt.ref_prim ? bt.ref_prim[r] : r);
        if (rec_box) {
            rec_box[2 * rec] = bt.plo[r];
            rec_box[2 * rec + 1] = bt.phi[r];
        }
    }
    const int leaf_max = __reduce_max_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0 && leaf_max) atomicMax(max_leaf, leaf_max);
    // the box of slot q, exactly as its child's (an empty slot: lo = +inf, hi =
    // -inf, which no ray enters)
    int owner = -1;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (__shfl_sync(0xffffffffu, slot, c, 8) == q) owner = c;
    const int from = owner < 0 ? q : owner;
    float3 sl, sh;
    sl.x = __shfl_sync(0xffffffffu, lo.x, from, 8);
    sl.y = __shfl_sync(0xffffffffu, lo.y, from, 8);
    sl.z = __shfl_sync(0xffffffffu, lo.z, from, 8);
    sh.x = __shfl_sync(0xffffffffu, hi.x, from, 8);
    sh.y = __shfl_sync(0xffffffffu, hi.y, from, 8);
    sh.z = __shfl_sync(0xffffffffu, hi.z, from, 8);
    if (owner < 0) {
        sl = make_float3(INFINITY, INFINITY, INFINITY);
        sh = make_float3(-INFINITY, -INFINITY, -INFINITY);
    }
    if (!live) return;
    WNode& nd = nodes[w];
    nd.box[0][0][q] = nd.box[0][2][q] = sl.x;
    nd.box[0][1][q] = sh.x;
    nd.box[1][0][q] = nd.box[1][2][q] = sl.y;
    nd.box[1][1][q] = sh.y;
    nd.box[2][0][q] = nd.box[2][2][q] = sl.z;
    nd.box[2][1][q] = sh.z;
    if (q == 0) {
        nd.child_base = child_base;
        nd.prim_base = prim_base;
        nd.slots = imask | leaf_bits << 8;
        nd.pad = 0;
        nbox[2 * w] = make_float4(ulo.x, ulo.y, ulo.z, 0.f);
        nbox[2 * w + 1] = make_float4(uhi.x, uhi.y, uhi.z, 0.f);
    }
}

// ---------------------------------------------------------------- refit after a vertex update

// Leaf records' parts and primitive ids in a split build (both null otherwise).
struct Parts {
    const uint32_t* uv;
    const uint32_t* id;
};

// Box of record r (primitive id with its sphere flag: idb) from the current
// vertices: its part of the moved triangle when it has one (clamped to the
// whole triangle's box, which holds the part), else its whole primitive's
// box. Padded with the triangle's pad when `pad`.
__device__ __forceinline__ void record_box(uint32_t idb, int64_t r, Parts parts, const float* __restrict__ tri,
                                           const float* __restrict__ sph, int64_t T, bool pad, float3& lo,
                                           float3& hi) {
    const int64_t id = (int64_t)(idb & ~SPHERE_BIT);
    float3 tl, th;
    prim_box(tri, sph, T, id, tl, th);
    lo = tl;
    hi = th;
    if (parts.uv && id < T && parts.uv[PART_MAX * r] != PART_END) {
        const float* f = tri + 9 * id;
        const float3 a = make_float3(f[0], f[1], f[2]);
        const float3 e1 = make_float3(f[3] - f[0], f[4] - f[1], f[5] - f[2]);
        const float3 e2 = make_float3(f[6] - f[0], f[7] - f[1], f[8] - f[2]);
        float3 l = make_float3(INFINITY, INFINITY, INFINITY), h = make_float3(-INFINITY, -INFINITY, -INFINITY);
        const uint32_t* q = parts.uv + PART_MAX * r;
        for (int k = 0; k < PART_MAX; ++k) {
            const uint32_t w = q[k];
            if (w == PART_END) break;
            const float u = (float)(w & 0xffffu) * (1.f / 65535.f), v = (float)(w >> 16) * (1.f / 65535.f);
            const float3 p = make_float3(fmaf(v, e2.x, fmaf(u, e1.x, a.x)), fmaf(v, e2.y, fmaf(u, e1.y, a.y)),
                                         fmaf(v, e2.z, fmaf(u, e1.z, a.z)));
            l = make_float3(fminf(l.x, p.x), fminf(l.y, p.y), fminf(l.z, p.z));
            h = make_float3(fmaxf(h.x, p.x), fmaxf(h.y, p.y), fmaxf(h.z, p.z));
        }
        lo = make_float3(fmaxf(lo.x, l.x), fmaxf(lo.y, l.y), fmaxf(lo.z, l.z));
        hi = make_float3(fminf(hi.x, h.x), fminf(hi.y, h.y), fminf(hi.z, h.z));
    }
    // the 16-bit (u, v) and the float mapping move a vertex by ~2^-16 of the
    // triangle's extent, inside the pad of the whole triangle
    if (pad && id < T) pad_box(tri_pad(tl, th), lo, hi);
}

// First step of a refit, one thread per record: the record rewritten from the
// moved vertices (spheres do not move) and its padded box (rbox, 6 floats per
// record: lo, hi), which k_refit_wide gathers into the leaf slots. A split
// build reads the records' ids from parts.id (4 bytes, not a record's sector).
__global__ void k_refit_records(float4* __restrict__ prims, int64_t n, Parts parts, const float* __restrict__ tri,
                                const float* __restrict__ sph, int64_t T, float2* __restrict__ rbox) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t idb = parts.id ? parts.id[r] : __float_as_uint(prims[3 * r + 2].y);
        if (!(idb & SPHERE_BIT)) write_prim_record(prims + 3 * r, tri, sph, T, idb);
        float3 lo, hi;
        record_box(idb, r, parts, tri, sph, T, true, lo, hi);
        rbox[3 * r] = make_float2(lo.x, lo.y);
        rbox[3 * r + 1] = make_float2(lo.z, hi.x);
        rbox[3 * r + 2] = make_float2(hi.y, hi.z);
    }
}

// Recompute the child boxes of the nodes in [begin, end) (one level, deepest
// first). Eight lanes per node, lane s for slot s: the slot's box is the union
// of its leaf records' boxes (rbox) or its internal child's box, and each of
// the node's nine box rows (8 floats, one 32-byte sector) is written by its
// eight lanes together. Empty slots get the empty box (+inf, -inf) that the
// collapse gave them. Only the node's header is read. The node's union box
// (nbox) is reduced over its eight lanes, which share a warp.
constexpr int REFIT_BLOCK = 128;
static_assert(REFIT_BLOCK % 32 == 0, "a node's eight lanes must share a warp");

__global__ void __launch_bounds__(REFIT_BLOCK) k_refit_wide(WNode* __restrict__ nodes, float4* __restrict__ nbox,
                                                            int64_t begin, int64_t end,
                                                            const float2* __restrict__ rbox) {
    const int64_t t = blockIdx.x * (int64_t)REFIT_BLOCK + threadIdx.x;
    const int64_t w = begin + (t >> 3);
    const int s = (int)(t & 7);
    const bool live = w < end;
    float3 lo = make_float3(INFINITY, INFINITY, INFINITY), hi = make_float3(-INFINITY, -INFINITY, -INFINITY);
    if (live) {
        WNode& nd = nodes[w];
        const uint4 hd = *reinterpret_cast<const uint4*>(&nd.child_base);
        const uint32_t leaf_bits = hd.z >> 8;
        if (hd.z & (1u << s)) {
            const int64_t c = hd.x + __popc(hd.z & bits_below(s));
            const float4 l = nbox[2 * c], h = nbox[2 * c + 1];
            lo = make_float3(l.x, l.y, l.z);
            hi = make_float3(h.x, h.y, h.z);
        } else {
            const int cnt = __popc((leaf_bits >> (3 * s)) & 7u), off = __popc(leaf_bits & bits_below(3 * s));
            const float2* b = rbox + 3 * ((int64_t)hd.y + off);
            for (int q = 0; q < cnt; ++q) {
                const float2 a = b[3 * q], m = b[3 * q + 1], z = b[3 * q + 2];
                lo = make_float3(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, m.x));
                hi = make_float3(fmaxf(hi.x, m.y), fmaxf(hi.y, z.x), fmaxf(hi.z, z.y));
            }
        }
        nd.box[0][0][s] = nd.box[0][2][s] = lo.x;
        nd.box[0][1][s] = hi.x;
        nd.box[1][0][s] = nd.box[1][2][s] = lo.y;
        nd.box[1][1][s] = hi.y;
        nd.box[2][0][s] = nd.box[2][2][s] = lo.z;
        nd.box[2][1][s] = hi.z;
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        lo.x = fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, o));
        lo.y = fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, o));
        lo.z = fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, o));
        hi.x = fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, o));
        hi.y = fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, o));
        hi.z = fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, o));
    }
    if (live && s == 0) {
        nbox[2 * w] = make_float4(lo.x, lo.y, lo.z, 0.f);
        nbox[2 * w + 1] = make_float4(hi.x, hi.y, hi.z, 0.f);
    }
}

// ---------------------------------------------------------------- validation

__device__ __forceinline__ void slot_box(const WNode& nd, int s, double lo[3], double hi[3]) {
    for (int a = 0; a < 3; ++a) {
        lo[a] = nd.box[a][0][s];
        hi[a] = nd.box[a][1][s];
    }
}

// n_records leaf records over n_prims primitives; rec_box (nullable): each
// record's exact reference box, which must lie in its leaf slot (else the
// record's unpadded box from the current vertices must: its part of the
// triangle after a refit of a split build, or the whole primitive's box).
__global__ void k_validate(const WNode* __restrict__ nodes, int64_t n_nodes, const float4* __restrict__ nbox,
                           const float4* __restrict__ prims, int64_t n_records, int64_t n_prims,
                           const float4* __restrict__ rec_box, Parts parts, const float* __restrict__ tri,
                           const float* __restrict__ sph, int64_t T, unsigned* __restrict__ seen_rec,
                           unsigned* __restrict__ seen_id, unsigned* __restrict__ node_refs, int* errors) {
    const int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w >= n_nodes) return;
    const WNode nd = nodes[w];
    const uint32_t imask = nd.slots & 0xffu, leaf_bits = nd.slots >> 8;
    for (int s = 0; s < 8; ++s) {
        const uint32_t lb = (leaf_bits >> (3 * s)) & 7u;
        const bool internal = imask & (1u << s);
        if (lb & (lb + 1u)) atomicAdd(&errors[0], 1);  // a count in unary
        if (!internal && !lb) continue;  // empty
        double lo[3], hi[3];
        slot_box(nd, s, lo, hi);
        for (int a = 0; a < 3; ++a)
            if (nd.box[a][2][s] != nd.box[a][0][s]) atomicAdd(&errors[2], 1);
        if (internal) {
            if (lb) atomicAdd(&errors[0], 1);  // a slot is a child or a leaf
            const int64_t c = (int64_t)nd.child_base + __popc(imask & bits_below(s));
            if (c <= w || c >= n_nodes) {
                atomicAdd(&errors[1], 1);
                continue;
            }
            atomicAdd(&node_refs[c], 1u);
            const float4 l = nbox[2 * c], h = nbox[2 * c + 1];
            if (l.x < lo[0] || l.y < lo[1] || l.z < lo[2] || h.x > hi[0] || h.y > hi[1] || h.z > hi[2])
                atomicAdd(&errors[2], 1);
        } else {
            const int cnt = __popc(lb), off = __popc(leaf_bits & bits_below(3 * s));
            for (int q = 0; q < cnt; ++q) {
                const int64_t r = (int64_t)nd.prim_base + off + q;
                if (r >= n_records) {
                    atomicAdd(&errors[3], 1);
                    continue;
                }
                atomicAdd(&seen_rec[r], 1u);
                const uint32_t id = __float_as_uint(prims[3 * r + 2].y) & ~SPHERE_BIT;
                if (id < (uint32_t)n_prims) atomicAdd(&seen_id[id], 1u);
                else atomicAdd(&errors[6], 1);
                float3 pl, ph;
                if (rec_box) {
                    const float4 l = rec_box[2 * r], h = rec_box[2 * r + 1];
                    pl = make_float3(l.x, l.y, l.z);
                    ph = make_float3(h.x, h.y, h.z);
                } else {
                    record_box(__float_as_uint(prims[3 * r + 2].y), r, parts, tri, sph, T, false, pl, ph);
                }
                if (pl.x < lo[0] || pl.y < lo[1] || pl.z < lo[2] || ph.x > hi[0] || ph.y > hi[1] || ph.z > hi[2])
                    atomicAdd(&errors[4], 1);
            }
        }
    }
}

// every record referenced once; every primitive in exactly one record, or in
// at least one when triangles are split into several references
__global__ void k_check_counts(const unsigned* a, int64_t n_records, const unsigned* b, int64_t n_prims,
                               bool split, const unsigned* node_refs, int64_t n_nodes, int* errors) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_records;
         i += (int64_t)gridDim.x * blockDim.x)
        if (a[i] != 1u) atomicAdd(&errors[5], 1);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_prims; i += (int64_t)gridDim.x * blockDim.x)
        if (split ? b[i] < 1u : b[i] != 1u) atomicAdd(&errors[6], 1);
    for (int64_t i = 1 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_nodes;
         i += (int64_t)gridDim.x * blockDim.x)
        if (node_refs[i] != 1u) atomicAdd(&errors[7], 1);
}

int grid_for(int64_t n, int block, int cap) {
    int64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}



// Tile counts of each level of the recursive scan of up to n words.
std::vector<int64_t> scan_levels(int64_t n) {
    std::vector<int64_t> lv;
    do {
        n = (n + SCAN_TILE - 1) / SCAN_TILE;
        lv.push_back(n);
    } while (n > 1);
    return lv;
}

// Exclusive scan of d[0..n) in place; the sum of all n words lands in *total.
// aux holds the tile sums of this level followed by those of deeper levels.
void scan_u64(unsigned long long* d, int64_t n, unsigned long long* aux, const std::vector<int64_t>& lv, size_t l,
              unsigned long long* total, cudaStream_t st) {
    const int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    k_scan_tiles<<<(unsigned)tiles, SCAN_BLOCK, 0, st>>>(d, n, aux);
    if (tiles > 1) {
        scan_u64(aux, tiles, aux + lv[l], lv, l + 1, total, st);
        k_scan_add<<<(unsigned)tiles, SCAN_BLOCK, 0, st>>>(d, n, aux);
    } else {
        cudaMemcpyAsync(total, aux, sizeof(unsigned long long), cudaMemcpyDeviceToDevice, st);
    }
}

// Binary tree over the N >= 2 primitives in Morton order (ids_in) by PLOC.
// Fills child, blo/bhi (padded) and range of internal nodes 0..N-2 (root 0), with the
// leaves renumbered depth-first: ids_out[j] is the primitive of leaf j.
// `tree` comes without its counts.
// first_tile (a test's): the first tile that the first round runs; the ones
// before it never do.
rcp_status build_ploc(int64_t N, PlocTree tree, uint32_t* ids_out, int2* range, int* d_err, int cap, Arena& arena,
                      cudaStream_t st, int spin_limit = PLOC_SPINS, unsigned first_tile = 0) {
    Carved<int> ref_a, ref_b, cnt, pos;
    Carved<float4> lo_a, hi_a, lo_b, hi_b;
    // per batch of up to PLOC_BATCH rounds: the rounds' states, tile counters and tile status
    constexpr int PLOC_BATCH = 16;
    constexpr int FAILED = PLOC_BATCH + 1;  // the state whose n is the first round with a wait that ran out
    Carved<PlocState> state;
    Carved<unsigned long long> marks;
    const int64_t tiles_max = (N + PLOC_TILE - 1) / PLOC_TILE;
    RCP_CUDA(ref_a.alloc(arena, N));
    RCP_CUDA(ref_b.alloc(arena, N));
    RCP_CUDA(cnt.alloc(arena, N));
    RCP_CUDA(pos.alloc(arena, N));
    RCP_CUDA(lo_a.alloc(arena, N));
    RCP_CUDA(hi_a.alloc(arena, N));
    RCP_CUDA(lo_b.alloc(arena, N));
    RCP_CUDA(hi_b.alloc(arena, N));
    RCP_CUDA(state.alloc(arena, FAILED + 1));
    RCP_CUDA(marks.alloc(arena, PLOC_BATCH * (1 + tiles_max)));
    RCP_CUDA(cudaMemsetAsync(tree.parent_int, 0xff, sizeof(int) * N, st));
    RCP_CUDA(cudaMemsetAsync(tree.parent_leaf, 0xff, sizeof(int) * N, st));
    tree.cnt = cnt.p;
    int *rin = ref_a.p, *rout = ref_b.p;
    float4 *lin = lo_a.p, *hin = hi_a.p, *lout = lo_b.p, *hout = hi_b.p;
    k_ploc_init<<<grid_for(N, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(tree.ids, N, tree.plo, tree.phi, rin, lin, hin);
    PlocState hs[FAILED + 1] = {};
    hs[0].n = (int)N;
    hs[FAILED].n = INT_MAX;
    RCP_CUDA(cudaMemcpyAsync(state.p, hs, sizeof(hs), cudaMemcpyHostToDevice, st));
    PlocState h = hs[0];
    // The rounds run without the host between them: each reads its count from
    // the device, under a grid sized for the count at the batch's start, which
    // only shrinks. The host reads the count once per batch.
    while (h.n > PLOC_LAST) {
        const int64_t n0 = h.n, tiles = (n0 + PLOC_TILE - 1) / PLOC_TILE;
        // a round leaves three clusters of four or a little more: as many
        // rounds as that ratio needs, an even number of array swaps
        const int need = (int)std::ceil(std::log((double)n0 / PLOC_LAST) / std::log(4.0 / 3.0));
        const int rounds = std::min(PLOC_BATCH, std::max(2, (need + 1) & ~1));
        RCP_CUDA(cudaMemsetAsync(marks.p, 0, sizeof(unsigned long long) * PLOC_BATCH * (1 + tiles), st));
        if (first_tile && h.created == 0)
            RCP_CUDA(cudaMemcpyAsync(marks.p, &first_tile, sizeof(first_tile), cudaMemcpyHostToDevice, st));
        for (int r = 0; r < rounds; ++r) {
            k_ploc_round<<<(unsigned)tiles, PLOC_BLOCK, 0, st>>>(state.p + r, (unsigned*)(marks.p + r),
                                                                 marks.p + PLOC_BATCH + r * tiles, N, rin, lin, hin,
                                                                 rout, lout, hout, tree, &state.p[FAILED].n, r,
                                                                 spin_limit);
            std::swap(rin, rout);
            std::swap(lin, lout);
            std::swap(hin, hout);
        }
        RCP_CUDA(cudaGetLastError());
        RCP_CUDA(cudaMemcpyAsync(hs, state.p, sizeof(hs), cudaMemcpyDeviceToHost, st));
        RCP_CUDA(cudaMemcpyAsync(state.p, state.p + rounds, sizeof(h), cudaMemcpyDeviceToDevice, st));
        RCP_CUDA(cudaStreamSynchronize(st));
        if (hs[FAILED].n != INT_MAX) {
            set_error("BVH build: the clustering's look-back wait ran out");
            return RCP_ERR_TIMEOUT;
        }
        h = hs[rounds];
        // the smallest pair is always mutual, so a round without a merge means
        // the device state is corrupt
        if (h.stalled || h.n < 1 || h.n >= n0 || h.n + h.created != N) {
            set_error("BVH build: clustering made no progress");
            return RCP_ERR_STATE;
        }
    }
    RCP_CUDA(cudaFuncSetAttribute(k_ploc_last, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(PlocLastShared)));
    k_ploc_last<<<1, PLOC_LAST, sizeof(PlocLastShared), st>>>(state.p, N, rin, lin, hin, tree);
    RCP_CUDA(cudaGetLastError());
    RCP_CUDA(cudaMemcpyAsync(&h, state.p + 1, sizeof(h), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    if (h.stalled || h.n != 1 || h.created != N - 1) {
        set_error("BVH build: clustering made no progress");
        return RCP_ERR_STATE;
    }
    k_dfs_offsets<<<grid_for(2 * N - 1, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(
        tree.child, tree.parent_int, tree.parent_leaf, tree.cnt, N, range, pos.p, d_err);
    k_dfs_apply<<<grid_for(N, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(pos.p, tree.ids, N, ids_out, tree.child, d_err);
    RCP_CUDA(cudaGetLastError());
    // the scratch above is given back by the caller: finish using it first
    RCP_CUDA(cudaStreamSynchronize(st));
    return RCP_OK;
}

}  // namespace

rcp_status ingest_scene(Scene& sc, const float* albedo3, bool* bad_tri, bool* bad_sph, cudaStream_t st) {
    const int64_t N = sc.T + sc.S;
    *bad_tri = *bad_sph = false;
    if (N == 0) return RCP_OK;
    Arena arena;
    Carved<float> raw;
    Carved<int> bad;
    RCP_CUDA(arena.reserve(sizeof(float) * 3 * N + 1024));
    RCP_CUDA(raw.alloc(arena, 3 * N));
    RCP_CUDA(bad.alloc(arena, 2));
    RCP_CUDA(cudaMemcpyAsync(raw.p, albedo3, sizeof(float) * 3 * N, cudaMemcpyHostToDevice, st));
    RCP_CUDA(cudaMemsetAsync(bad.p, 0, 2 * sizeof(int), st));
    int sms = 148, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_any_non_finite<<<grid_for(9 * sc.T / 4 + 1, BUILD_BLOCK, sms * 8), BUILD_BLOCK, 0, st>>>(sc.d_tri, 9 * sc.T,
                                                                                                bad.p);
    k_any_non_finite<<<grid_for(sc.S + 1, BUILD_BLOCK, sms * 8), BUILD_BLOCK, 0, st>>>(sc.d_sph, 4 * sc.S, bad.p + 1);
    k_widen_albedo<<<grid_for(N, BUILD_BLOCK, sms * 8), BUILD_BLOCK, 0, st>>>(raw.p, N, sc.d_albedo);
    int h[2];
    RCP_CUDA(cudaMemcpyAsync(h, bad.p, sizeof(h), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    *bad_tri = h[0] != 0;
    *bad_sph = h[1] != 0;
    return RCP_OK;
}

rcp_status build_bvh(Scene& sc, cudaStream_t st) {
    const int64_t T = sc.T, N = sc.T + sc.S;
    EventPair ev;
    RCP_CUDA(ev.create());
    RCP_CUDA(cudaEventRecord(ev.a, st));
    int sms = 148;
    {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    const int cap = sms * 16;
    const bool split = sc.split_max > 1 && T > 0, sah = sc.collapse == RCP_COLLAPSE_SAH;
    // Temporaries in one allocation: 32 bytes per primitive (48 when split),
    // and per reference 72 that live through the build, then the clustering's
    // 84 or what follows it (the slot costs' 40 under the surface-area policy,
    // arrivals and frontiers 8, and the nodes' first estimate, one per five
    // references at 336 bytes), whichever is more.
    const auto per_reference = [&](int64_t refs) {
        return (size_t)refs * (72 + std::max(84, 8 + (sah ? 40 : 0) + 68)) + radix_sort_scratch_bytes(refs) + (1 << 20);
    };
    Arena arena;
    RCP_CUDA(arena.reserve(split ? (size_t)N * 48 + (1 << 20) : (size_t)N * 32 + per_reference(N)));
    Carved<float4> plo, phi;
    Carved<uint32_t> bounds;
    RCP_CUDA(plo.alloc(arena, N));
    RCP_CUDA(phi.alloc(arena, N));
    RCP_CUDA(bounds.alloc(arena, 12));
    k_init_bounds<<<1, 32, 0, st>>>(bounds.p);
    k_prim_bounds<<<grid_for(N, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(sc.d_tri, sc.d_sph, T, N, plo.p, phi.p,
                                                                          bounds.p);
    // references: the primitives themselves, or split triangles (R >= N)
    int64_t R = N;
    Carved<float4> rlo, rhi;
    Carved<uint32_t> rprim;
    const float4* ref_lo = plo.p;
    const float4* ref_hi = phi.p;
    if (split) {
        Carved<unsigned long long> counts, aux, total;
        const std::vector<int64_t> lv = scan_levels(N);
        int64_t aux_n = 0;
        for (int64_t t : lv) aux_n += t;
        RCP_CUDA(counts.alloc(arena, N));
        RCP_CUDA(aux.alloc(arena, aux_n));
        RCP_CUDA(total.alloc(arena, 1));
        k_split_count<<<grid_for(N, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(sc.d_tri, T, N, sc.split_max,
                                                                              counts.p);
        scan_u64(counts.p, N, aux.p, lv, 0, total.p, st);
        unsigned long long hr = 0;
        RCP_CUDA(cudaMemcpyAsync(&hr, total.p, sizeof(hr), cudaMemcpyDeviceToHost, st));
        RCP_CUDA(cudaStreamSynchronize(st));
        R = (int64_t)hr;
        if (R < N || R > N * (int64_t)SPLIT_MAX || R >= ((int64_t)1 << 30)) {
            set_error("BVH build: split references out of range (at most 2^30 - 1)");
            return RCP_ERR_ARG;
        }
        RCP_CUDA(arena.reserve((size_t)R * 36 + per_reference(R)));
        RCP_CUDA(rlo.alloc(arena, R));
        RCP_CUDA(rhi.alloc(arena, R));
        RCP_CUDA(rprim.alloc(arena, R));
        Carved<int> split_err;
        RCP_CUDA(split_err.alloc(arena, 1));
        RCP_CUDA(cudaMemsetAsync(split_err.p, 0, sizeof(int), st));
        k_split_write<<<grid_for(N, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(
            sc.d_tri, T, N, sc.split_max, counts.p, R, plo.p, phi.p, rlo.p, rhi.p, rprim.p, split_err.p);
        int h_err = 0;
        RCP_CUDA(cudaMemcpyAsync(&h_err, split_err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        RCP_CUDA(cudaStreamSynchronize(st));
        if (h_err) {
            set_error("BVH build: split references counted and written differently");
            return RCP_ERR_STATE;
        }
        ref_lo = rlo.p;
        ref_hi = rhi.p;
    }
    Carved<float4> blo, bhi;
    Carved<uint32_t> keys, vals, akeys, avals, counters;
    Carved<int2> child, range, fa, fb;
    Carved<int> parent_int, parent_leaf, err;
    Carved<char> scratch;
    RCP_CUDA(keys.alloc(arena, R));
    RCP_CUDA(vals.alloc(arena, R));
    RCP_CUDA(akeys.alloc(arena, R));
    RCP_CUDA(avals.alloc(arena, R));
    RCP_CUDA(counters.alloc(arena, 4));
    RCP_CUDA(err.alloc(arena, 2));
    RCP_CUDA(child.alloc(arena, R));
    RCP_CUDA(range.alloc(arena, R));
    RCP_CUDA(blo.alloc(arena, R));
    RCP_CUDA(bhi.alloc(arena, R));
    RCP_CUDA(parent_int.alloc(arena, R));
    RCP_CUDA(parent_leaf.alloc(arena, R));
    RCP_CUDA(scratch.alloc(arena, radix_sort_scratch_bytes(R)));
    DevBuf<float4> prims, rec_box;  // the scene's own
    RCP_CUDA(prims.alloc(3 * R));
    if (split) RCP_CUDA(rec_box.alloc(2 * R));
    RCP_CUDA(cudaMemsetAsync(err.p, 0, 2 * sizeof(int), st));
    RCP_CUDA(cudaMemsetAsync(counters.p, 0, sizeof(uint32_t) * 4, st));
    k_morton<<<grid_for(R, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(ref_lo, ref_hi, R, bounds.p, keys.p, vals.p);
    rcp_status rs = radix_sort_pairs(keys.p, vals.p, akeys.p, avals.p, R, 30, scratch.p, err.p, st);
    if (rs != RCP_OK) return rs;
    uint32_t* ids = vals.p;  // reference indices in leaf order (Morton order, then depth-first)
    Carved<float4> dp;
    Carved<uint2> slot_split;
    Carved<int> arrivals;
    if (R >= 2) {
        // a sort whose look-back wait ran out leaves no valid permutation to cluster
        int sort_flag = 0;
        RCP_CUDA(cudaMemcpyAsync(&sort_flag, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        RCP_CUDA(cudaStreamSynchronize(st));
        if (sort_flag) {
            set_error("radix sort: look-back wait ran out");
            return RCP_ERR_TIMEOUT;
        }
        const Arena::Mark before = arena.mark();
        const PlocTree tree{child.p, blo.p, bhi.p,  nullptr, parent_int.p, parent_leaf.p,
                            vals.p,  ref_lo, ref_hi, split ? rprim.p : nullptr, sc.d_tri, sc.d_sph, T};
        rcp_status pr = build_ploc(R, tree, avals.p, range.p, err.p + 1, cap, arena, st);
        arena.release(before);
        if (pr != RCP_OK) {
            return pr;
        }
        ids = avals.p;
    }
    if (R >= 2 && sah) {
        RCP_CUDA(dp.alloc(arena, 2 * (R - 1)));
        RCP_CUDA(slot_split.alloc(arena, R - 1));
        RCP_CUDA(arrivals.alloc(arena, R - 1));
        RCP_CUDA(cudaMemsetAsync(arrivals.p, 0, sizeof(int) * (R - 1), st));
        k_sah_dp<<<grid_for(R, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(child.p, range.p, parent_int.p,
                                                                         parent_leaf.p, blo.p, bhi.p, ref_lo, ref_hi,
                                                                         ids, R, dp.p, slot_split.p, arrivals.p,
                                                                         err.p + 1);
    }
    // scene bounds -> diameter
    uint32_t hb[12];
    RCP_CUDA(cudaMemcpyAsync(hb, bounds.p, sizeof(hb), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    auto ord2f_h = [](uint32_t u) {
        uint32_t v = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
        float f;
        memcpy(&f, &v, 4);
        return f;
    };
    if (N > 0) {
        float d2 = 0.f;
        for (int a = 0; a < 3; ++a) {
            const float ext = ord2f_h(hb[9 + a]) - ord2f_h(hb[6 + a]);
            d2 += ext * ext;
        }
        sc.diam = sqrtf(d2);
    } else {
        sc.diam = 0.f;
    }

    // collapse, level by level
    std::vector<int64_t> level_begin;
    int depth = 0;
    int64_t n_nodes = 0;
    // Nodes (and their boxes) as the collapse numbers them. A level's launch
    // writes the nodes numbered before it, so there is room for those by then.
    // An internal child holds LEAF_MAX + 1 references or more, which bounds a
    // frontier.
    Carved<WNode> nodes_full;
    Carved<float4> nbox_full;
    int64_t node_cap = R / 5 + 64;
    RCP_CUDA(fa.alloc(arena, R / (LEAF_MAX + 1) + 1));
    RCP_CUDA(fb.alloc(arena, R / (LEAF_MAX + 1) + 1));
    RCP_CUDA(nodes_full.alloc(arena, node_cap));
    RCP_CUDA(nbox_full.alloc(arena, 2 * node_cap));
    if (N > 0) {
        int2 root = make_int2(R >= 2 ? 0 : -1, 0);
        RCP_CUDA(cudaMemcpyAsync(fa.p, &root, sizeof(int2), cudaMemcpyHostToDevice, st));
        uint32_t one = 1;
        RCP_CUDA(cudaMemcpyAsync(counters.p, &one, sizeof(uint32_t), cudaMemcpyHostToDevice, st));
        int* d_max_leaf = err.p;  // reuse: err[0] is the sort's flag, checked below before reuse
        int herr[2] = {0, 0};
        RCP_CUDA(cudaMemcpyAsync(herr, err.p, sizeof(herr), cudaMemcpyDeviceToHost, st));
        RCP_CUDA(cudaStreamSynchronize(st));
        if (herr[1]) {
            set_error("BVH build: the clustered tree is malformed (a path to the root too long or a leaf out of range)");
            return RCP_ERR_STATE;
        }
        if (herr[0]) {
            set_error("radix sort: look-back wait ran out");
            return RCP_ERR_TIMEOUT;
        }
        RCP_CUDA(cudaMemsetAsync(d_max_leaf, 0, sizeof(int), st));
        BinTree bt{child.p, range.p, blo.p, bhi.p, ref_lo, ref_hi, ids,
                   sah ? slot_split.p : nullptr, split ? rprim.p : nullptr, sc.d_tri,
                   sc.d_sph, T};
        int n_front = 1;
        int64_t begin = 0;
        int2* cur = fa.p;
        int2* nxt = fb.p;
        while (n_front > 0) {
            if (depth >= 512) {
                set_error("BVH collapse did not terminate (corrupted binary tree)");
                return RCP_ERR_STATE;
            }
            level_begin.push_back(begin);
            ++depth;
            RCP_CUDA(cudaMemsetAsync(counters.p + 2, 0, sizeof(uint32_t), st));
            k_collapse<<<(int)((8 * (int64_t)n_front + COLLAPSE_BLOCK - 1) / COLLAPSE_BLOCK), COLLAPSE_BLOCK, 0, st>>>(bt, cur, n_front, nxt, counters.p, nodes_full.p,
                                                               nbox_full.p, prims.p, sc.d_tri, sc.d_sph, T, d_max_leaf,
                                                               rec_box.p);
            uint32_t hc[3];
            RCP_CUDA(cudaMemcpyAsync(hc, counters.p, sizeof(hc), cudaMemcpyDeviceToHost, st));
            RCP_CUDA(cudaStreamSynchronize(st));
            begin += n_front;
            n_front = (int)hc[2];
            n_nodes = hc[0];
            std::swap(cur, nxt);
            if (n_nodes > node_cap) {  // the written nodes move to a larger array
                node_cap = std::max(2 * node_cap, n_nodes);
                Carved<WNode> more;
                Carved<float4> more_box;
                RCP_CUDA(more.alloc(arena, node_cap));
                RCP_CUDA(more_box.alloc(arena, 2 * node_cap));
                RCP_CUDA(cudaMemcpyAsync(more.p, nodes_full.p, sizeof(WNode) * begin, cudaMemcpyDeviceToDevice, st));
                RCP_CUDA(cudaMemcpyAsync(more_box.p, nbox_full.p, sizeof(float4) * 2 * begin, cudaMemcpyDeviceToDevice,
                                         st));
                nodes_full = more;
                nbox_full = more_box;
            }
        }
        level_begin.push_back(begin);
        RCP_CUDA(cudaMemcpyAsync(&sc.max_leaf, d_max_leaf, sizeof(int), cudaMemcpyDeviceToHost, st));
    }
    // the parts of split references, for refits
    DevBuf<uint32_t> parts;  // PART_MAX words per record, then the records' ids
    if (split) {
        RCP_CUDA(parts.alloc((PART_MAX + 1) * R));
        k_record_parts<<<grid_for(R, BUILD_BLOCK, cap), BUILD_BLOCK, 0, st>>>(prims.p, R, rec_box.p, sc.d_tri, T,
                                                                               parts.p, parts.p + PART_MAX * R);
    }
    // trim the node arrays to size
    RCP_CUDA(cudaMalloc((void**)&sc.d_nodes, (sizeof(WNode) + sizeof(float4) * 2) * (n_nodes ? n_nodes : 1)));
    sc.d_nbox = (float4*)((WNode*)sc.d_nodes + n_nodes);
    if (n_nodes) {
        RCP_CUDA(cudaMemcpyAsync(sc.d_nodes, nodes_full.p, sizeof(WNode) * n_nodes, cudaMemcpyDeviceToDevice, st));
        RCP_CUDA(cudaMemcpyAsync(sc.d_nbox, nbox_full.p, sizeof(float4) * 2 * n_nodes, cudaMemcpyDeviceToDevice,
                                 st));
    }
    RCP_CUDA(cudaEventRecord(ev.b, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    sc.d_prims = prims.release();
    sc.d_refbox = rec_box.release();
    sc.d_part_uv = parts.release();
    sc.d_rec_id = sc.d_part_uv ? sc.d_part_uv + PART_MAX * R : nullptr;
    sc.n_records = R;
    sc.n_nodes = n_nodes;
    sc.depth = depth;
    sc.level_begin = level_begin;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev.a, ev.b);
    sc.build_ms = ms;
    RCP_CUDA(cudaGetLastError());
    return RCP_OK;
}

rcp_status refit_bvh(Scene& sc, cudaStream_t st) {
    const int64_t N = sc.T + sc.S;
    if (N == 0 || sc.n_nodes == 0) return RCP_OK;
    // a split build's references are bounded by their parts of the moved
    // triangles; the build-time reference boxes no longer apply
    if (sc.d_refbox) {
        RCP_CUDA(cudaStreamSynchronize(st));
        cudaFree(sc.d_refbox);
        sc.d_refbox = nullptr;
    }
    if (!sc.d_rbox) RCP_CUDA(cudaMalloc((void**)&sc.d_rbox, sizeof(float2) * 3 * sc.n_records));
    EventPair ev;
    RCP_CUDA(ev.create());
    RCP_CUDA(cudaEventRecord(ev.a, st));
    int sms = 148, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_refit_records<<<grid_for(sc.n_records, BUILD_BLOCK, sms * 16), BUILD_BLOCK, 0, st>>>(
        sc.d_prims, sc.n_records, Parts{sc.d_part_uv, sc.d_rec_id}, sc.d_tri, sc.d_sph, sc.T, sc.d_rbox);
    for (int l = (int)sc.level_begin.size() - 2; l >= 0; --l) {
        const int64_t b = sc.level_begin[l], e = sc.level_begin[l + 1];
        if (e <= b) continue;
        k_refit_wide<<<(int)((8 * (e - b) + REFIT_BLOCK - 1) / REFIT_BLOCK), REFIT_BLOCK, 0, st>>>(
            (WNode*)sc.d_nodes, sc.d_nbox, b, e, sc.d_rbox);
    }
    RCP_CUDA(cudaEventRecord(ev.b, st));
    RCP_CUDA(cudaEventSynchronize(ev.b));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev.a, ev.b);
    sc.build_ms = ms;
    RCP_CUDA(cudaGetLastError());
    return RCP_OK;
}

rcp_status validate_bvh(const Scene& sc, cudaStream_t st) {
    const int64_t N = sc.T + sc.S, R = sc.n_records;
    if (N == 0) return RCP_OK;
    DevBuf<unsigned> words;  // per record, per primitive and per node its references counted, then the errors
    RCP_CUDA(words.alloc(R + N + sc.n_nodes + 8));
    RCP_CUDA(cudaMemsetAsync(words.p, 0, sizeof(unsigned) * (R + N + sc.n_nodes + 8), st));
    unsigned *seen_rec = words.p, *seen_id = seen_rec + R, *node_refs = seen_id + N;
    int* errors = (int*)(node_refs + sc.n_nodes);
    k_validate<<<(int)((sc.n_nodes + 127) / 128), 128, 0, st>>>((const WNode*)sc.d_nodes, sc.n_nodes, sc.d_nbox,
                                                                 sc.d_prims, R, N, sc.d_refbox,
                                                                 Parts{sc.d_part_uv, sc.d_rec_id}, sc.d_tri, sc.d_sph,
                                                                 sc.T, seen_rec, seen_id, node_refs, errors);
    k_check_counts<<<grid_for(std::max<int64_t>(std::max(R, N), sc.n_nodes), 256, 4096), 256, 0, st>>>(
        seen_rec, R, seen_id, N, sc.split_max > 1, node_refs, sc.n_nodes, errors);
    int h[8];
    RCP_CUDA(cudaMemcpyAsync(h, errors, sizeof(h), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    static const char* what[8] = {"slot masks",       "child index order", "child box outside slot",
                                  "leaf record range", "primitive outside leaf slot",
                                  "record not referenced exactly once", "primitive id missing or repeated",
                                  "node not referenced exactly once"};
    for (int i = 0; i < 8; ++i)
        if (h[i]) {
            set_error(std::string("BVH validation failed: ") + what[i] + " (" + std::to_string(h[i]) + ")");
            return RCP_ERR_STATE;
        }
    return RCP_OK;
}

// A clustering whose first round never runs its first tile: 2,000 boxes, all
// equal (nine tiles, of which eight wait for the first).
rcp_status debug_cluster_timeout(int spin_limit, cudaStream_t st) {
    const int64_t N = 2000;
    Arena arena;
    Carved<float4> lo, hi, blo, bhi;
    Carved<uint32_t> ids, ids_out;
    Carved<int2> child, range;
    Carved<int> parent_int, parent_leaf, err;
    RCP_CUDA(arena.reserve(N * 320 + (1 << 16)));
    RCP_CUDA(lo.alloc(arena, N));
    RCP_CUDA(hi.alloc(arena, N));
    RCP_CUDA(blo.alloc(arena, N));
    RCP_CUDA(bhi.alloc(arena, N));
    RCP_CUDA(ids.alloc(arena, N));
    RCP_CUDA(ids_out.alloc(arena, N));
    RCP_CUDA(child.alloc(arena, N));
    RCP_CUDA(range.alloc(arena, N));
    RCP_CUDA(parent_int.alloc(arena, N));
    RCP_CUDA(parent_leaf.alloc(arena, N));
    RCP_CUDA(err.alloc(arena, 1));
    RCP_CUDA(cudaMemsetAsync(lo.p, 0, sizeof(float4) * N, st));
    RCP_CUDA(cudaMemsetAsync(hi.p, 0, sizeof(float4) * N, st));
    RCP_CUDA(cudaMemsetAsync(ids.p, 0, sizeof(uint32_t) * N, st));  // every leaf is box 0
    RCP_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
    const PlocTree tree{child.p, blo.p, bhi.p, nullptr, parent_int.p, parent_leaf.p, ids.p,
                        lo.p,    hi.p,  nullptr, nullptr, nullptr, 0};  // no triangles: no box is padded
    const rcp_status r = build_ploc(N, tree, ids_out.p, range.p, err.p, 64, arena, st, spin_limit, 1);
    RCP_CUDA(cudaStreamSynchronize(st));
    return r;
}

rcp_status debug_morton(const float* xyz, int64_t n, const float* lo, const float* hi, uint32_t* codes,
                        cudaStream_t st) {
    if (n <= 0) return RCP_OK;
    k_morton_points<<<grid_for(n, 256, 4096), 256, 0, st>>>(xyz, n, lo[0], lo[1], lo[2], hi[0], hi[1], hi[2],
                                                             codes);
    RCP_CUDA(cudaGetLastError());
    return RCP_OK;
}

}  // namespace rcp
