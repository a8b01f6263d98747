// rcp_internal.cuh -- shared device types of the renderer (not part of the ABI).
//
// Layout in device memory (all 16-byte aligned):
//  * WNode: one 8-wide BVH node with float child boxes, 304 bytes = 19 x float4.
//  * Prim records: 3 x float4 = 48 bytes per primitive, in leaf order:
//      triangle  w0 = (v0.xyz, e1.x)  w1 = (e1.yz, e2.xy)  w2 = (e2.z, id, 0, 0)
//      sphere    w0 = (centre, r)     w1 = 0               w2 = (0, id | SPHERE_BIT, 0, 0)
//    with e1 = v1 - v0, e2 = v2 - v0 (float32), id = the caller's primitive id.
//  * Albedo: float4 per primitive, indexed by id.
//  * Images: float4 per pixel (RGB, hit distance), row-major.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/rcp.h"

namespace rcp {

constexpr uint32_t SPHERE_BIT = 0x80000000u;
constexpr int MAX_STACK = 64;  // traversal stack entries (>= BVH depth)

// One 8-wide node, 19 rows of 16 bytes. Child slot s (0..7) has the float
// box box[a][0][s]..box[a][1][s] per axis a (an empty slot: lo = +inf, hi =
// -inf); box[a][2] repeats the low planes behind the high ones, so that a ray
// finds its near planes at box[a][n] and its far planes right behind them, n =
// 0 or 1 by the sign of its direction: one address per axis instead of two
// (rows 6a + 2n .. 6a + 2n + 3). A ray reads 13 of the rows, whichever its
// octant: the copies cost memory (304 bytes against 208), not traffic.
// slots: bit s set = slot s holds an internal child, node child_base + the
// number of internal slots below s; bits 8 + 3 s .. 10 + 3 s hold a leaf
// slot's record count (1..3) in unary, and the records of a node's leaves lie
// from prim_base on in slot order, so the record of leaf bit j is prim_base +
// the number of leaf bits below j. The header is row 18.
struct __align__(16) WNode {
    float box[3][3][8];
    uint32_t child_base;
    uint32_t prim_base;
    uint32_t slots;  // internal mask | leaf record bits << 8
    uint32_t pad;
};
constexpr int NODE_ROWS = 19;
static_assert(sizeof(WNode) == 16 * NODE_ROWS, "WNode must be 19 rows of 16 bytes");

// Bits below bit b of a mask's slot or leaf bit b (b <= 24).
__host__ __device__ __forceinline__ uint32_t bits_below(uint32_t b) { return (1u << b) - 1u; }

struct LightDev {
    int type;
    float x, y, z;
    float ambient;
};

// Device-resident scene: BVH, primitive records and shading data.
struct SceneDev {
    const float4* nodes;   // n_nodes * NODE_ROWS
    const float4* prims;   // n_records * 3
    const float4* albedo;  // n_prims
    int64_t n_prims;
    int64_t n_records;     // leaf records (more than n_prims when triangles are split)
    int64_t n_nodes;
    LightDev light;
    float tmin;  // 1e-6 * diameter
    float eps;   // 1e-4 * diameter (shadow-ray offset)
};

// Pass n of a multi-sample render of several passes: what it needs to leave
// out the tiles whose values repeat (flags_out null: it traces every tile). A tile's flags of a pass: bit 0 = every
// pixel equals the pass before, bit 1 = every pixel equals the pass before that
// (all four lanes, bit for bit).
struct MsRepeat {
    const uint8_t* flags_in;  // pass n-1's flags per tile, nullptr in pass 1
    uint8_t* flags_out;       // pass n's
    int has_two_ago;          // out held I_{n-2} before this pass (n >= 3, not the last pass)
    const float4* two_ago;    // I_{n-2} (n >= 3); the pass's own out unless it is the last pass
    const int32_t* ids_two_ago;  // hit ids of passes n-2 and n-1 (null unless the render returns ids)
    const int32_t* ids_before;
    const unsigned* shadow_before;  // per tile, shadow rays of pass n-1
    unsigned* shadow;               // per tile, of pass n-2 on entry, of pass n afterwards
};

// One view (camera + image) of a batched pass. The camera terms are
// precomputed on the host in double and rounded once:
//   g(x, y) = fF + (2x + 1 - W) fR + (H - 2y - 1) fU  (eye -> focal-plane point)
//   V(c)    = (2c.r - 1) kR + (2c.g - 1) kU + (2c.b - 1) kF
struct ViewDev {
    const struct SceneDev* scene;  // the view's scene (launches over views of several scenes)
    int* status;                   // set to 1 when a walk of this view overflowed its stack (device or host memory)
    float E[3];
    float fF[3], fR[3], fU[3];
    float kR[3], kU[3], kF[3];
    float Fw[3];  // unit view axis F: the z-depth of a hit is t (d . F)
    int W, H;
    int mapping;
    float z0;
    float kpx;  // IMAGE: displacement in pixels; NORMAL: k in world units
    int passes;  // passes a chained launch runs for this view (in: its first input, out: its last output)
    const float4* in;    // previous image, nullptr = I_0
    const float4* base;  // image-space passes: the frame's traced image
    float4* out;         // this pass's image
    int32_t* prim;     // nullable hit ids
    float* rgb;        // nullable: this pass also writes R, G, B (3 floats per pixel, row-major) here,
                       // host memory that the device reads and writes coherently
    int2* hint;        // nullable: per pixel, the record of its latest primary hit and of its latest
                       // shadow occluder (-1 none); tested first, rewritten by every traced pass
    int64_t pix_begin;  // first global pixel index of this view
    int64_t chunk_begin;  // first work chunk (8x4 tile) of this view
    int tiles_x;
    int spp;              // samples per pixel, 0 = one at the centre
    float jit[2 * RCP_MAX_SPP];
    MsRepeat repeat;
    int* done_count;  // nullable: tiles of this view still to finish in the launch (device)
    int* done_flag;   // set to 1 (host-visible) once they have all finished
};

// Host-side owner of a built scene.
struct Scene;

struct Counters {
    unsigned long long rays, primary, shadow, nodes, boxes, tris, spheres;
};

// thread-local error message
void set_error(const std::string& msg);
rcp_status cuda_fail(cudaError_t e, const char* what);

// Owner of one device array, freed on every return path.
template <class T>
struct DevBuf {
    T* p = nullptr;
    DevBuf() = default;
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
    ~DevBuf() {
        if (p) cudaFree(p);
    }
    cudaError_t alloc(size_t n) { return cudaMalloc((void**)&p, sizeof(T) * (n ? n : 1)); }
    T* release() {
        T* q = p;
        p = nullptr;
        return q;
    }
};

// Device memory for the temporaries of one call, carved from one allocation
// (more where the first estimate falls short) and freed on every return path.
// A driver allocation or free costs 20-60 us whatever its size, and a scene
// build has about forty temporaries.
class Arena {
  public:
    Arena() = default;
    Arena(const Arena&) = delete;
    Arena& operator=(const Arena&) = delete;
    ~Arena() {
        for (char* c : chunks_) cudaFree(c);
    }
    // Make room for `bytes` more in one piece.
    cudaError_t reserve(size_t bytes) {
        if (off_ + bytes <= cap_) return cudaSuccess;
        char* c = nullptr;
        const cudaError_t e = cudaMalloc((void**)&c, bytes);
        if (e != cudaSuccess) return e;
        chunks_.push_back(c);
        cap_ = bytes;
        off_ = 0;
        return cudaSuccess;
    }
    template <class T>
    cudaError_t take(T** out, size_t n) {
        const size_t bytes = (sizeof(T) * (n ? n : 1) + 255) & ~(size_t)255;
        const cudaError_t e = reserve(bytes);
        if (e != cudaSuccess) return e;
        *out = reinterpret_cast<T*>(chunks_.back() + off_);
        off_ += bytes;
        return cudaSuccess;
    }
    // What is taken between mark and release is given back by release.
    struct Mark {
        size_t chunks, off;
    };
    Mark mark() const { return Mark{chunks_.size(), off_}; }
    void release(Mark m) {
        if (m.chunks == chunks_.size()) off_ = m.off;
    }

  private:
    std::vector<char*> chunks_;
    size_t cap_ = 0, off_ = 0;  // of the newest chunk
};

// One array carved from an Arena.
template <class T>
struct Carved {
    T* p = nullptr;
    cudaError_t alloc(Arena& a, size_t n) { return a.take(&p, n); }
};

// Two timing events, destroyed on every return path.
struct EventPair {
    cudaEvent_t a = nullptr, b = nullptr;
    EventPair() = default;
    EventPair(const EventPair&) = delete;
    EventPair& operator=(const EventPair&) = delete;
    ~EventPair() {
        if (a) cudaEventDestroy(a);
        if (b) cudaEventDestroy(b);
    }
    cudaError_t create() {
        cudaError_t e = cudaEventCreate(&a);
        return e == cudaSuccess ? cudaEventCreate(&b) : e;
    }
};

#define RCP_CUDA(call)                                          \
    do {                                                        \
        cudaError_t e_ = (call);                                \
        if (e_ != cudaSuccess) return rcp::cuda_fail(e_, #call); \
    } while (0)

// The radix sort (radix_sort.cu): n pairs in place on the low `bits` bits of the
// keys. alt_keys/alt_vals are n-element buffers, scratch has
// radix_sort_scratch_bytes(n). resident_tiles: the most tiles that one launch
// for all passes is tried with (negative: as many as the device has SMs).
size_t radix_sort_scratch_bytes(int64_t n);
rcp_status radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* alt_keys, uint32_t* alt_vals, int64_t n, int bits,
                            void* scratch, int* d_error, cudaStream_t stream, int64_t resident_tiles = -1);

}  // namespace rcp
