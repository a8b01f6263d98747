// radix_sort.cu -- LSD radix sort of (uint32 key, uint32 value) pairs, 8 bits a pass.
//
// Used by the BVH builder to order primitives by 30-bit Morton code, and by
// the allocation-free sort below. A pass ranks a tile of keys in shared memory
// (warp ballots + per-warp counters, stable), finds the tile's place per digit
// among all tiles, and scatters through shared memory so that writes of one
// digit run are contiguous.
//  * While the tiles fit the GPU at once (one per SM, 1.09 million pairs on
//    152 SMs), one cooperative launch runs every pass (k_sort_resident).
//  * Beyond that, or where the device does not run that many blocks at once,
//    onesweep: one histogram kernel counts all digit passes at
//    once (its last block scans the counts), then one launch per digit finds a
//    tile's place by decoupled look-back over earlier tiles (numbered in launch
//    order by an atomic counter, so every earlier tile is already running).
//
// What bounds it up to about a million pairs is latency: 16 MB a pass moves
// through L2 in a few microseconds, and each block's chain of load, rank,
// place and scatter is serial (9 us a pass for a single tile, of which about
// 3.5 us are shared-memory bank conflicts of random digits and 3 us the two
// barriers). So: tiles of 7,168 pairs over 1,024 threads, which put a million
// pairs on the SMs in one wave; in onesweep a look-back that polls eight
// earlier tiles at once, where one at a time is a chain of L2 round trips, the
// tile's own scan done by other warps meanwhile, one memset for every pass's
// status words, and programmatic launches, so that a pass's blocks are
// resident when the pass before ends. 1,000,003 pairs on 30 bits, the whole
// call with its last read-back: 170 us (four passes of 25 us and a histogram),
// onesweep as here 99-101 us, resident 96-98 us (52 us in the kernel).
//
// Every wait on another tile's status is bounded: after spin_limit polls
// (SPIN_LIMIT in a sort) the kernel records an error flag and proceeds, so a
// fault in the protocol shows up as an error status instead of a hang.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "rcp_internal.cuh"

namespace rcp {

namespace {

constexpr int RADIX = 256;
constexpr int PASSES_MAX = 4;
constexpr int SORT_BLOCK = 1024;
constexpr int SORT_WARPS = SORT_BLOCK / 32;
constexpr int ITEMS = 7;
constexpr int TILE = SORT_BLOCK * ITEMS;  // 7168 pairs
constexpr int LOOK = 8;                   // earlier tiles polled at once
constexpr int GROUPS = SORT_BLOCK / RADIX;  // of one thread per digit each
static_assert(SORT_BLOCK % RADIX == 0 && GROUPS >= 2, "one group looks back while another scans the tile's counts");
constexpr uint32_t FLAG_AGG = 1u << 30;
constexpr uint32_t FLAG_INC = 2u << 30;
constexpr uint32_t COUNT_MASK = (1u << 30) - 1;
constexpr long long SPIN_LIMIT = 1ll << 26;

// Scratch words: the passes' digit counts (bucket starts once scanned), then
// one tile counter per pass and the histogram's block counter, then the
// passes' tile status, RADIX words per tile.
constexpr int COUNTERS = 8;
constexpr size_t scratch_words(int64_t tiles, int passes) {
    return (size_t)PASSES_MAX * RADIX + COUNTERS + (size_t)passes * (size_t)tiles * RADIX;
}

constexpr int HIST_BLOCK = 1024;  // one block per SM: each adds its counts to the global ones once
constexpr int HIST_KEYS = 8;      // keys a thread holds at a time

// Digit counts of all passes; the last block to finish turns each pass's 256
// counts into exclusive prefix sums.
__global__ void __launch_bounds__(HIST_BLOCK) k_histogram(const uint32_t* __restrict__ keys, int64_t n, int passes,
                                                          uint32_t* hist, uint32_t* blocks_done) {
    __shared__ uint32_t h[PASSES_MAX][RADIX];
    __shared__ uint32_t s_warp[RADIX / 32];
    __shared__ bool s_last;
    for (int i = threadIdx.x; i < PASSES_MAX * RADIX; i += HIST_BLOCK) (&h[0][0])[i] = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * HIST_BLOCK;
    for (int64_t i = blockIdx.x * (int64_t)HIST_BLOCK + threadIdx.x; i < n; i += HIST_KEYS * step) {
        uint32_t k[HIST_KEYS];
#pragma unroll
        for (int q = 0; q < HIST_KEYS; ++q) k[q] = i + q * step < n ? keys[i + q * step] : 0u;
#pragma unroll
        for (int q = 0; q < HIST_KEYS; ++q)
            if (i + q * step < n)
                for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(k[q] >> (8 * p)) & 0xff], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * RADIX; i += HIST_BLOCK) {
        const uint32_t v = (&h[0][0])[i];
        if (v) atomicAdd(&hist[i], v);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(blocks_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool scans = threadIdx.x < RADIX;  // one thread per digit
    for (int p = 0; p < passes; ++p) {
        const uint32_t v = scans ? __ldcg(&hist[p * RADIX + threadIdx.x]) : 0u;
        uint32_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (scans && lane == 31) s_warp[warp] = x;
        __syncthreads();
        if (scans) {
            for (int w = 0; w < warp; ++w) x += s_warp[w];
            hist[p * RADIX + threadIdx.x] = x - v;
        }
        __syncthreads();
    }
}

// The lanes whose digit equals this lane's, by one ballot per digit bit (as fast
// as a warp match here).
__device__ __forceinline__ unsigned same_digit(uint32_t d) {
    unsigned peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (d >> b) & 1u;
        const unsigned with = __ballot_sync(0xffffffffu, set);
        peers &= set ? with : ~with;
    }
    return peers;
}

struct SortShared {
    uint32_t keys[TILE];
    uint32_t vals[TILE];
    uint32_t wcnt[SORT_WARPS][RADIX];
    uint32_t tile_off[RADIX];
    uint32_t global[RADIX];
    uint32_t warp_tot[2][RADIX / 32];
    uint32_t tile;
};

// Rank a tile's keys by digit: rank[j] is key j's place among its warp's keys
// of the digit, s.wcnt[w][d] the warps' counts (zeroed before).
__device__ __forceinline__ void rank_keys(SortShared& s, const uint32_t (&k)[ITEMS], uint32_t (&rank)[ITEMS],
                                          int shift) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t d = (k[j] >> shift) & 0xff;
        const unsigned peers = same_digit(d);
        const uint32_t before = s.wcnt[warp][d];
        rank[j] = before + __popc(peers & lt);
        __syncwarp();
        if ((peers >> lane) == 1u) s.wcnt[warp][d] = before + __popc(peers);  // highest lane of the group
        __syncwarp();
    }
}

// Digit d's count in the tile; s.wcnt becomes its exclusive scan over the warps.
__device__ __forceinline__ uint32_t scan_warp_counts(SortShared& s, int d) {
    uint32_t count = 0;
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) {
        const uint32_t c = s.wcnt[w][d];
        s.wcnt[w][d] = count;
        count += c;
    }
    return count;
}

// Exclusive scan of one value per digit over 256 threads of the block (d: the
// thread's digit), which meet at named barrier `bar`.
__device__ __forceinline__ uint32_t scan_digits(uint32_t (&warp_tot)[RADIX / 32], uint32_t c, int d, int bar) {
    const int lane = threadIdx.x & 31;
    uint32_t x = c;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[d >> 5] = x;
    asm volatile("bar.sync %0, 256;" ::"r"(bar) : "memory");
    for (int w = 0; w < d >> 5; ++w) x += warp_tot[w];
    return x - c;
}

// The tile's pairs into shared memory in digit order, then to their places.
__device__ __forceinline__ void scatter_tile(SortShared& s, const uint32_t (&k)[ITEMS], const uint32_t (&v)[ITEMS],
                                             const uint32_t (&rank)[ITEMS], int shift, int valid,
                                             uint32_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out) {
    const int warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t d = (k[j] >> shift) & 0xff;
        const uint32_t r = s.tile_off[d] + s.wcnt[warp][d] + rank[j];
        s.keys[r] = k[j];
        s.vals[r] = v[j];
    }
    __syncthreads();
    for (int pos = threadIdx.x; pos < valid; pos += SORT_BLOCK) {
        const uint32_t key = s.keys[pos];
        const uint32_t d = (key >> shift) & 0xff;
        const uint32_t dst = s.global[d] + (pos - s.tile_off[d]);
        keys_out[dst] = key;
        vals_out[dst] = s.vals[pos];
    }
}

__global__ void __launch_bounds__(SORT_BLOCK, 1) k_onesweep(const uint32_t* __restrict__ keys_in,
                                                            const uint32_t* __restrict__ vals_in,
                                                            uint32_t* __restrict__ keys_out,
                                                            uint32_t* __restrict__ vals_out, int64_t n, int shift,
                                                            const uint32_t* __restrict__ bucket_base, uint32_t* status,
                                                            uint32_t* tile_counter, int* error_flag,
                                                            long long spin_limit) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    SortShared& s = *reinterpret_cast<SortShared*>(s_raw);
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < SORT_WARPS * RADIX; i += SORT_BLOCK) (&s.wcnt[0][0])[i] = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the pass (or histogram) before has finished
    asm volatile("griddepcontrol.launch_dependents;");
    if (tid == 0) s.tile = atomicAdd(tile_counter, 1u);
    __syncthreads();
    const uint32_t tile = s.tile;
    const int64_t base = (int64_t)tile * TILE + warp * (32 * ITEMS) + lane;

    uint32_t k[ITEMS], v[ITEMS], rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)  // past the end: ranks after every real key of its digit
        k[j] = base + 32 * j < n ? keys_in[base + 32 * j] : 0xffffffffu;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) v[j] = base + 32 * j < n ? vals_in[base + 32 * j] : 0u;
    rank_keys(s, k, rank, shift);
    __syncthreads();

    const int d = tid & (RADIX - 1);
    uint32_t count = 0;
    if (tid < RADIX) {
        count = scan_warp_counts(s, d);
        // publish this tile's count (tile 0's is already inclusive); a status
        // word carries flag and count together, so no fence orders anything
        volatile uint32_t* st = status + (size_t)tile * RADIX;
        st[d] = (tile == 0 ? FLAG_INC : FLAG_AGG) | count;
        s.tile_off[d] = count;
    }
    __syncthreads();
    if (tid < RADIX) {
        // look back over earlier tiles, LOOK of them per round of loads
        uint32_t prefix = 0;
        int64_t t = (int64_t)tile - 1;
        long long spins = 0;
        while (t >= 0) {
            uint32_t sv[LOOK];
#pragma unroll
            for (int q = 0; q < LOOK; ++q) {
                sv[q] = FLAG_INC;  // before the first tile: nothing more to add
                if (t >= q) sv[q] = ((volatile uint32_t*)status)[(size_t)(t - q) * RADIX + d];
            }
            bool found = false, waiting = false;
            int taken = 0;
#pragma unroll
            for (int q = 0; q < LOOK; ++q) {
                const uint32_t flag = sv[q] & ~COUNT_MASK;
                waiting = waiting || flag == 0;
                if (!found && !waiting) {
                    prefix += sv[q] & COUNT_MASK;
                    found = flag == FLAG_INC;
                    ++taken;
                }
            }
            if (found) break;
            t -= taken;
            if (taken == 0 && ++spins > spin_limit) {
                atomicExch(error_flag, 1);
                break;
            }
        }
        if (tile > 0) ((volatile uint32_t*)status)[(size_t)tile * RADIX + d] = FLAG_INC | (prefix + count);
        s.global[d] = bucket_base[d] + prefix;
    } else if (tid < 2 * RADIX) {
        s.tile_off[d] = scan_digits(s.warp_tot[0], s.tile_off[d], d, 1);
    }
    __syncthreads();
    const int64_t left = n - (int64_t)tile * TILE;
    scatter_tile(s, k, v, rank, shift, left < TILE ? (int)left : TILE, keys_out, vals_out);
}

// ---- all passes in one launch, while the tiles fit the GPU at once ----
// Up to one tile per SM, a block keeps its tile's place through every pass: it
// ranks its keys, publishes its 256 digit counts, and after a grid-wide barrier
// adds up every tile's counts itself (all tiles' and the earlier tiles'), where
// separate passes need a histogram beforehand and look back tile by tile; the
// pairs go to the other buffer and a second barrier ends the pass. The launch is
// cooperative, so that every block that a barrier waits for runs; each wait is bounded all the same, and as the
// counts are zero beforehand, one that runs out leaves sums too small: the pairs
// still go to places in range.
struct ResidentShared {
    SortShared t;
    uint32_t part[GROUPS][2][RADIX];  // per group: all tiles' counts, earlier tiles' counts
};

__device__ __forceinline__ void grid_barrier(uint32_t* arrived, uint32_t target, int* error_flag,
                                             long long spin_limit) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(arrived, 1u);
        long long spins = 0;
        while (*(volatile uint32_t*)arrived < target)
            if (++spins > spin_limit) {
                atomicExch(error_flag, 1);
                break;
            }
        __threadfence();
    }
    __syncthreads();
}

__global__ void __launch_bounds__(SORT_BLOCK, 1) k_sort_resident(uint32_t* keys, uint32_t* vals, uint32_t* alt_keys,
                                                                 uint32_t* alt_vals, int64_t n, int passes,
                                                                 uint32_t* counts, uint32_t* arrived, int* error_flag,
                                                                 long long spin_limit) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    ResidentShared& rs = *reinterpret_cast<ResidentShared*>(s_raw);
    SortShared& s = rs.t;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tiles = gridDim.x, tile = blockIdx.x;
    const int64_t base = (int64_t)tile * TILE + warp * (32 * ITEMS) + lane;
    const int64_t left = n - (int64_t)tile * TILE;
    const int valid = left < TILE ? (int)left : TILE;
    const int d = tid & (RADIX - 1), group = tid / RADIX;
    uint32_t barriers = 0;
    for (int p = 0; p < passes; ++p) {
        const uint32_t *ki = p & 1 ? alt_keys : keys, *vi = p & 1 ? alt_vals : vals;
        const int shift = 8 * p;
        for (int i = tid; i < SORT_WARPS * RADIX; i += SORT_BLOCK) (&s.wcnt[0][0])[i] = 0;
        uint32_t k[ITEMS], v[ITEMS], rank[ITEMS];
        // other blocks wrote these in the pass before: past this SM's L1
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)  // past the end: ranks after every real key of its digit
            k[j] = base + 32 * j < n ? __ldcg(ki + base + 32 * j) : 0xffffffffu;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) v[j] = base + 32 * j < n ? __ldcg(vi + base + 32 * j) : 0u;
        __syncthreads();
        rank_keys(s, k, rank, shift);
        __syncthreads();
        uint32_t* cnt = counts + (size_t)p * tiles * RADIX;
        if (tid < RADIX) {
            const uint32_t c = scan_warp_counts(s, d);
            s.tile_off[d] = c;
            __stcg(cnt + (size_t)tile * RADIX + d, c);
        }
        grid_barrier(arrived, ++barriers * tiles, error_flag, spin_limit);
        // each group adds up its share of the tiles
        uint32_t all = 0, earlier = 0;
        const int t0 = group * tiles / GROUPS, t1 = (group + 1) * tiles / GROUPS;
#pragma unroll 8
        for (int t = t0; t < t1; ++t) {
            const uint32_t c = __ldcg(cnt + (size_t)t * RADIX + d);
            all += c;
            if (t < tile) earlier += c;
        }
        rs.part[group][0][d] = all;
        rs.part[group][1][d] = earlier;
        __syncthreads();
        if (group == 0) {
            all = earlier = 0;
            for (int g = 0; g < GROUPS; ++g) {
                all += rs.part[g][0][d];
                earlier += rs.part[g][1][d];
            }
            s.global[d] = scan_digits(s.warp_tot[1], all, d, 1) + earlier;
        } else if (group == 1) {
            s.tile_off[d] = scan_digits(s.warp_tot[0], s.tile_off[d], d, 2);
        }
        __syncthreads();
        scatter_tile(s, k, v, rank, shift, valid, p & 1 ? keys : alt_keys, p & 1 ? vals : alt_vals);
        if (p + 1 < passes) grid_barrier(arrived, ++barriers * tiles, error_flag, spin_limit);
    }
}

// One digit pass: launched programmatically behind the kernel before it.
rcp_status launch_onesweep(const uint32_t* ki, const uint32_t* vi, uint32_t* ko, uint32_t* vo, int64_t n, int shift,
                           const uint32_t* bucket_base, uint32_t* status, uint32_t* tile_counter, int64_t blocks,
                           int* d_error, long long spin_limit, cudaStream_t stream) {
    RCP_CUDA(cudaFuncSetAttribute(k_onesweep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(SORT_BLOCK);
    cfg.dynamicSmemBytes = sizeof(SortShared);
    cfg.stream = stream;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    RCP_CUDA(cudaLaunchKernelEx(&cfg, k_onesweep, ki, vi, ko, vo, n, shift, bucket_base, status, tile_counter, d_error,
                                spin_limit));
    return RCP_OK;
}

cudaError_t launch_resident(uint32_t* keys, uint32_t* vals, uint32_t* alt_keys, uint32_t* alt_vals, int64_t n, int passes,
                            uint32_t* counts, uint32_t* arrived, int64_t tiles, int* d_error, long long spin_limit,
                            cudaStream_t stream) {
    cudaError_t e = cudaFuncSetAttribute(k_sort_resident, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(ResidentShared));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles);
    cfg.blockDim = dim3(SORT_BLOCK);
    cfg.dynamicSmemBytes = sizeof(ResidentShared);
    cfg.stream = stream;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_sort_resident, keys, vals, alt_keys, alt_vals, n, passes, counts, arrived,
                              d_error, spin_limit);
}

// The sorted pairs, if they lie elsewhere, back to the caller's arrays.
rcp_status copy_back(uint32_t* keys, uint32_t* vals, const uint32_t* ki, const uint32_t* vi, int64_t n,
                     cudaStream_t stream) {
    if (ki == keys) return RCP_OK;
    RCP_CUDA(cudaMemcpyAsync(keys, ki, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, stream));
    RCP_CUDA(cudaMemcpyAsync(vals, vi, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, stream));
    return RCP_OK;
}

}  // namespace

size_t radix_sort_scratch_bytes(int64_t n) {
    return sizeof(uint32_t) * scratch_words(std::max<int64_t>((n + TILE - 1) / TILE, 1), PASSES_MAX);
}

rcp_status radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* alt_keys, uint32_t* alt_vals, int64_t n, int bits,
                            void* scratch, int* d_error, cudaStream_t stream, int64_t resident_tiles) {
    if (n <= 1) return RCP_OK;
    if (n >= (int64_t)COUNT_MASK) {
        set_error("radix sort: too many keys (limit 2^30)");
        return RCP_ERR_ARG;
    }
    const int passes = (bits + 7) / 8;
    const int64_t tiles = (n + TILE - 1) / TILE;
    uint32_t* hist = (uint32_t*)scratch;
    uint32_t* counters = hist + PASSES_MAX * RADIX;
    uint32_t* status = counters + COUNTERS;
    RCP_CUDA(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * scratch_words(tiles, passes), stream));
    int sms = 0, dev = 0;
    RCP_CUDA(cudaGetDevice(&dev));
    RCP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    uint32_t *ki = keys, *vi = vals, *ko = alt_keys, *vo = alt_vals;
    // One tile per SM at most: one launch for all passes. The call on 1,000,003
    // pairs takes 96-98 us, onesweep 99-101; at 1,000 to 600,000 pairs the two
    // are within 2 % of each other (the same chain of loads, ranks and barriers
    // or look-backs, and the call's read-back).
    if (tiles <= (resident_tiles < 0 ? sms : resident_tiles)) {
        const cudaError_t e = launch_resident(keys, vals, alt_keys, alt_vals, n, passes, status, counters, tiles, d_error,
                                              SPIN_LIMIT, stream);
        if (e == cudaSuccess) {
            if (passes & 1) {
                std::swap(ki, ko);
                std::swap(vi, vo);
            }
            return copy_back(keys, vals, ki, vi, n, stream);
        }
        // fewer SMs to be had at once than the device has (a partition of it):
        // the passes one by one need no tiles to run together
        if (e != cudaErrorCooperativeLaunchTooLarge) return cuda_fail(e, "cooperative sort launch");
        cudaGetLastError();
    }
    int64_t hblocks = (n + HIST_BLOCK * HIST_KEYS - 1) / (HIST_BLOCK * HIST_KEYS);
    if (hblocks > sms) hblocks = sms;
    k_histogram<<<(int)hblocks, HIST_BLOCK, 0, stream>>>(keys, n, passes, hist, counters + PASSES_MAX);
    RCP_CUDA(cudaGetLastError());
    for (int p = 0; p < passes; ++p) {
        rcp_status r = launch_onesweep(ki, vi, ko, vo, n, 8 * p, hist + p * RADIX, status + (size_t)p * tiles * RADIX,
                                       counters + p, tiles, d_error, SPIN_LIMIT, stream);
        if (r != RCP_OK) return r;
        std::swap(ki, ko);
        std::swap(vi, vo);
    }
    return copy_back(keys, vals, ki, vi, n, stream);
}

}  // namespace rcp

// ---------------------------------------------------------------- allocation-free variant
//
// rcp_sort_pairs_static: the same sort with every scratch buffer (ping-pong
// keys and values, digit histograms, tile status, tile counters, the look-back
// error flag) carved out of one file-scope device array, so the call never
// allocates device memory.

namespace rcp {
namespace {

constexpr int64_t STATIC_MAX = RCP_SORT_STATIC_MAX_PAIRS;
constexpr int64_t STATIC_TILES = (STATIC_MAX + TILE - 1) / TILE;
constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t OFF_KEYS = 0;
constexpr size_t OFF_VALS = align256(OFF_KEYS + sizeof(uint32_t) * STATIC_MAX);
constexpr size_t OFF_SCRATCH = align256(OFF_VALS + sizeof(uint32_t) * STATIC_MAX);
constexpr size_t SCRATCH_BYTES = sizeof(uint32_t) * scratch_words(STATIC_TILES, PASSES_MAX);
constexpr size_t OFF_ERROR = align256(OFF_SCRATCH + SCRATCH_BYTES);
constexpr size_t STATIC_BYTES = align256(OFF_ERROR + sizeof(int));

}  // namespace
}  // namespace rcp

// Held by every device that loads the library, for the life of the process.
static __device__ __align__(256) unsigned char g_sort_static_scratch[rcp::STATIC_BYTES];

namespace rcp {
namespace {

constexpr int MAX_DEVICES = 64;
std::mutex g_static_mu;
void* g_static_ptr[MAX_DEVICES] = {};

// Device address of the static scratch on the current device, looked up once
// per device (host code cannot use the array's name as a device pointer).
rcp_status static_scratch(unsigned char** out) {
    int dev = 0;
    RCP_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) {
        set_error("rcp_sort_pairs_static: device ordinal out of range");
        return RCP_ERR_STATE;
    }
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_sort_static_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_sort_static_scratch)");
        g_static_ptr[dev] = p;
    }
    *out = (unsigned char*)g_static_ptr[dev];
    return RCP_OK;
}

}  // namespace
}  // namespace rcp

extern "C" int64_t rcp_sort_static_capacity(void) { return rcp::STATIC_MAX; }

extern "C" rcp_status rcp_sort_pairs_static(uint32_t* keys, uint32_t* values, int64_t n, int bits, void* stream) {
    using namespace rcp;
    if (n < 0 || bits < 1 || bits > 32 || (n > 0 && (!keys || !values))) {
        set_error("rcp_sort_pairs_static: bad argument");
        return RCP_ERR_ARG;
    }
    if (n > STATIC_MAX) {
        set_error("rcp_sort_pairs_static: n = " + std::to_string(n) +
                  " exceeds the static scratch capacity of RCP_SORT_STATIC_MAX_PAIRS (" + std::to_string(STATIC_MAX) +
                  ") pairs");
        return RCP_ERR_ARG;
    }
    if (n <= 1) return RCP_OK;
    unsigned char* base = nullptr;
    rcp_status r = static_scratch(&base);
    if (r != RCP_OK) return r;
    cudaStream_t st = (cudaStream_t)stream;
    int* d_err = (int*)(base + OFF_ERROR);
    RCP_CUDA(cudaMemsetAsync(d_err, 0, sizeof(int), st));  // the array keeps the last call's contents
    r = radix_sort_pairs(keys, values, (uint32_t*)(base + OFF_KEYS), (uint32_t*)(base + OFF_VALS), n, bits,
                         base + OFF_SCRATCH, d_err, st);
    if (r != RCP_OK) return r;
    int h = 0;
    RCP_CUDA(cudaMemcpyAsync(&h, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    if (h) {
        set_error("rcp_sort_pairs_static: look-back wait ran out");
        return RCP_ERR_TIMEOUT;
    }
    return RCP_OK;
}

// ---------------------------------------------------------------- test of the bounded wait
//
// rcp_debug_sort_lookback_timeout: one onesweep block takes tile 1 of a
// two-tile pass while tile 0 never runs, so every one of its look-back waits
// polls a status that nothing publishes. After spin_limit polls each wait
// gives up and sets the error flag, and the block finishes its tile with a
// partial offset. With every key 0 all of the block's keys go to digit 0,
// whose bucket starts at 0, so its writes land at indices [0, TILE) of the
// 2 TILE-element output arrays.

extern "C" rcp_status rcp_debug_sort_lookback_timeout(int64_t spin_limit, void* stream) {
    using namespace rcp;
    if (spin_limit < 1 || spin_limit > (1ll << 20)) {
        set_error("rcp_debug_sort_lookback_timeout: spin_limit outside [1, 2^20]");
        return RCP_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = 2 * (int64_t)TILE;
    DevBuf<uint32_t> keys, vals, ko, vo, scratch;
    DevBuf<int> err;
    RCP_CUDA(keys.alloc(n));
    RCP_CUDA(vals.alloc(n));
    RCP_CUDA(ko.alloc(n));
    RCP_CUDA(vo.alloc(n));
    RCP_CUDA(scratch.alloc(scratch_words(2, 1)));
    RCP_CUDA(err.alloc(1));
    uint32_t* hist = scratch.p;
    uint32_t* counter = hist + PASSES_MAX * RADIX;
    uint32_t* status = counter + COUNTERS;
    RCP_CUDA(cudaMemsetAsync(keys.p, 0, sizeof(uint32_t) * n, st));
    RCP_CUDA(cudaMemsetAsync(vals.p, 0, sizeof(uint32_t) * n, st));
    RCP_CUDA(cudaMemsetAsync(scratch.p, 0, sizeof(uint32_t) * scratch_words(2, 1), st));
    RCP_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
    k_histogram<<<2, HIST_BLOCK, 0, st>>>(keys.p, n, 1, hist, counter + PASSES_MAX);
    const uint32_t one = 1;  // the block claims tile 1; tile 0 is never claimed
    RCP_CUDA(cudaMemcpyAsync(counter, &one, sizeof(one), cudaMemcpyHostToDevice, st));
    rcp_status r = launch_onesweep(keys.p, vals.p, ko.p, vo.p, n, 0, hist, status, counter, 1, err.p,
                                   (long long)spin_limit, st);
    if (r != RCP_OK) return r;
    int h = 0;
    RCP_CUDA(cudaMemcpyAsync(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    if (h) {
        set_error("radix sort: look-back wait ran out");
        return RCP_ERR_TIMEOUT;
    }
    return RCP_OK;
}

// rcp_debug_sort_barrier_timeout: one tile sorted in one launch, the barriers'
// counter one short of what they expect, so each of the three of two digit passes
// runs out.

extern "C" rcp_status rcp_debug_sort_barrier_timeout(int64_t spin_limit, void* stream) {
    using namespace rcp;
    if (spin_limit < 1 || spin_limit > (1ll << 20)) {
        set_error("rcp_debug_sort_barrier_timeout: spin_limit outside [1, 2^20]");
        return RCP_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = TILE;
    DevBuf<uint32_t> pairs, scratch;  // keys, values and their alternates
    DevBuf<int> err;
    RCP_CUDA(pairs.alloc(4 * n));
    RCP_CUDA(scratch.alloc(scratch_words(1, 2)));
    RCP_CUDA(err.alloc(1));
    uint32_t* counter = scratch.p + PASSES_MAX * RADIX;
    RCP_CUDA(cudaMemsetAsync(pairs.p, 0, sizeof(uint32_t) * 4 * n, st));
    RCP_CUDA(cudaMemsetAsync(scratch.p, 0, sizeof(uint32_t) * scratch_words(1, 2), st));
    RCP_CUDA(cudaMemsetAsync(counter, 0xff, sizeof(uint32_t), st));  // -1
    RCP_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
    const cudaError_t e = launch_resident(pairs.p, pairs.p + n, pairs.p + 2 * n, pairs.p + 3 * n, n, 2, counter + COUNTERS,
                                          counter, 1, err.p, (long long)spin_limit, st);
    if (e != cudaSuccess) return cuda_fail(e, "rcp_debug_sort_barrier_timeout");
    int h = 0;
    RCP_CUDA(cudaMemcpyAsync(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    RCP_CUDA(cudaStreamSynchronize(st));
    if (h) {
        set_error("radix sort: barrier wait ran out");
        return RCP_ERR_TIMEOUT;
    }
    return RCP_OK;
}
