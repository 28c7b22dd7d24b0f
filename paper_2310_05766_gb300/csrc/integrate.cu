// Per-scan TSDF integration kernels (FeatSense, Section "TSDF Map Generation").
//
// rays (K-A): one thread per point, coalesced float4 loads. Transforms the
//   point by the pose, sets up the ray (range r, unit direction d, unit
//   interpolation direction int = d x (d x up) with up the sensor z axis) and
//   appends it (two float4) to a compacted list of live rays: a ray whose whole
//   march (+-tau around the hit, widened by the fill height of Eq. 4 and a
//   safety margin) stays outside the window box is dropped, since none of its
//   samples could land in the window. Order is kept within a CTA, so
//   neighbouring rays stay neighbours. On the plain path the list is split:
//   rays whose fill reaches a voxel each side (delta_z r >= vs) are appended
//   from its front, the others from its end.
// contrib (K-B): persistent; a warp takes work items (32 consecutive live
//   rays, a group of KPT steps k of k = -K..K), one ray per lane. For each of its steps the
//   thread walks the fill samples j = -J..J (Eq. 3 / Eq. 4) in warp lock-step.
//   A sample inside the window yields (voxel, q), q the int16 code of the
//   truncated projective distance of the voxel centre, and issues one
//   fire-and-forget 64-bit reduction into the per-scan accumulator:
//     WSUM    : acc += (count << 40) + sum(q)   (two's-complement packing; exact
//               while count < 2^24 and |sum| < 2^39)
//     MIN_ABS : acc = max(acc, 65536 - key), key = (|q| << 1) | (q < 0)
//   so acc == 0 means "untouched". Optionally (MERGE) lanes that hit the same
//   voxel in the same iteration are first combined with match.any +
//   redux.sync so that one lane per distinct voxel issues the reduction. The
//   issuing lane marks the voxel's brick in a byte-per-brick flag array with
//   a plain store (idempotent, nothing to wait for), filtered by a per-CTA
//   shared-memory cache of the bricks the CTA has marked. The items of the
//   list's front (the costly rays) come first. Integer accumulation makes the
//   result independent of the order of the atomics.
// scan: rays and contrib in one kernel, for small scans (scan_fused).
// compact (large windows, sort reduction): turns the brick flags into a list of
//   touched bricks (4 flags per thread, one list atomic per warp) and clears
//   the flags.
// apply (K-C): one CTA per SM; each reads the brick flags itself (windows of
//   up to 2^16 bricks; the compaction kernel lists the bricks of larger ones),
//   takes its share of the touched bricks and works on quarter-brick warp
//   tasks staged through shared memory: Eq. 1 in exact integers with one
//   rounding (half away from zero) and Eq. 2 with the weight cap for every
//   touched voxel (non-zero accumulator), changed pairs written back and their
//   accumulators reset. Each CTA publishes its share of the scan's counters:
//   touched voxels and, in WSUM mode, the contributions too (the sum of the
//   decoded weights).
// finish (sort reduction): the last apply CTA to retire sums the per-scan
//   counters into the published ones and clears the per-scan state.
//
// Sort reduction (an alternative to the accumulator atomics, same results):
// rays also reserve each live ray's pair slots (one per march sample); emit is
// the contrib march writing (voxel word, code) to the sample's slot instead of
// reducing it (no atomics; samples beyond the capacity fall back to the
// accumulators); count adds each brick's pairs (warp-merged per brick);
// scan turns counts into segment starts; scatter moves every pair to its
// brick's segment as a 32-bit (offset, code); sort_apply reduces each brick's
// segment per voxel in shared memory and applies Eq. 1 / Eq. 2. Together
// count, scan and scatter are a counting sort of the contributions by brick.
//
// Kernels may be launched with programmatic stream serialisation: each may be
// scheduled while its predecessor drains, and waits (griddepcontrol.wait) for
// the predecessor's completion before touching its results.
//
// Every float operation on the geometry path is an explicit round-to-nearest
// intrinsic (no contraction into FMA), in the same order as the CPU oracle, so
// voxel indices and codes agree bit for bit.
#include <algorithm>
#include <mutex>
#include <set>
#include <unordered_map>
#include <utility>

#include "integrate_device.cuh"

// Minimum resident CTAs per SM requested for the scan kernel: 4 caps it at 64
// registers (no spills), 32 resident warps per SM.
#ifndef TSDF_SCAN_MIN_CTAS
#define TSDF_SCAN_MIN_CTAS 4
#endif
// The same for the contribution kernel.
#ifndef TSDF_CONTRIB_MIN_CTAS
#define TSDF_CONTRIB_MIN_CTAS 4
#endif
// Largest scan of the one-kernel path (points). Drawn when the other path was
// four kernels (one kernel / ray list, us a pass: room 16x360 17.9 / 26.2 and
// 64x512 17.2 / 18.1; outdoor 16x512 21.1 / 33.1, 32x512 18.6 / 24.6, 64x1024
// 31.3 / 29.4; corridor 32x512 38.5 / 49.5, 64x1024 41.9 / 44.9). With the ray
// set-up beside the previous scan's apply the list has become the faster one for
// most scans that follow one another: room 16x360 14.2 / 14.4 and 64x512 14.0 /
// 14.4; outdoor 16x512 29.2 / 26.0, 32x512 25.8 / 23.1, 32x1024 31.2 / 26.7,
// 64x1024 29.6 / 24.7, 128x1024 27.6 / 23.2; corridor 32x512 32.3 / 28.7, 32x1024
// 37.1 / 33.9, 64x1024 35.6 / 34.3, 128x2048 46.2 / 41.6. Scans alone (wall time
// of the call and its end): room 16x360 31.1 / 31.1, outdoor 32x512 44.5 / 43.7,
// corridor 32x512 50.8 / 49.4; the static entry 21.3-23.8 / 22.6. The one-kernel
// path needs no ray buffers.
#ifndef TSDF_SCAN_FUSED_MAX
#define TSDF_SCAN_FUSED_MAX 32768
#endif
// Tiles wanted of a scan (six per SM: with three, outdoor 32x512 20.3 instead
// of 18.6 us, 32x1024 42.1 instead of 34.3), and the largest tile.
#ifndef TSDF_SCAN_TILES
#define TSDF_SCAN_TILES 912
#endif
#ifndef TSDF_SCAN_MAX_TILE
#define TSDF_SCAN_MAX_TILE 256
#endif
// The same for the sort reduction's emit kernel (no cap).
#ifndef TSDF_EMIT_MIN_CTAS
#define TSDF_EMIT_MIN_CTAS 1
#endif
// CTAs per SM launched by the contribution kernels, which walk their work with
// a grid stride; 0 = as many as are resident at once.
#ifndef TSDF_CONTRIB_CTAS_PER_SM
#define TSDF_CONTRIB_CTAS_PER_SM 8
#endif

namespace tsdf {
namespace {

using namespace dev;

// Threads per CTA of the ray set-up kernel (one list atomic per CTA and list end).
#ifndef TSDF_RAYS_THREADS
#define TSDF_RAYS_THREADS 256
#endif
constexpr int kRaysThreads = TSDF_RAYS_THREADS;

template <bool SORT>
__global__ void __launch_bounds__(kRaysThreads) rays_kernel(const ScanArgs a, const MapDev m) {
    __shared__ RaysSmemT<kRaysThreads / 32> sm;
    if constexpr (SORT)
        rays_task_sort<true, kRaysThreads / 32>(a, m, (int)(blockIdx.x * blockDim.x), blockIdx.x, &sm);
    else
        rays_task_ppt<true, kRaysThreads / 32, kRaysPPT>(a, m, (int)(blockIdx.x * blockDim.x) * kRaysPPT,
                                                                blockIdx.x, &sm);
}

template <bool POOL>
__device__ __forceinline__ void cache_init(uint32_t* btab) {
    for (int i = threadIdx.x; i < (POOL ? kSlotCacheWords : kBrickCache); i += blockDim.x) btab[i] = kNoVoxel;
}

// The CTA's cache for a march: of marked bricks, or (pool reduction) of claimed
// slots; `btab` filled with ones is empty as either.
template <bool POOL>
__device__ __forceinline__ BrickCache march_cache(uint32_t* btab) {
    BrickCache bc{btab, 32u - kBrickCacheLog2};
    bc.slots = POOL ? reinterpret_cast<unsigned long long*>(btab) : nullptr;
    return bc;
}

// Contribution work items: (block of 32 consecutive live rays, group of KPT
// steps). Each warp walks the items with a grid stride and loads the next
// item's rays while it processes the current one. The grid is
// TSDF_CONTRIB_CTAS_PER_SM CTAs per SM, more than are resident at once, so the
// hardware hands the CTAs of later waves to the SMs that finish first. The
// warps of one CTA take consecutive items (the step groups of the same 32
// rays and of their neighbours), so they mark the same bricks and the CTA's
// brick cache absorbs most marks: giving a CTA's warps unrelated items, or
// handing out items through counters, made the kernel about 30 % slower, the
// extra time in brick-flag stores.
constexpr int kContribThreads = 256;

template <int MODE, bool MERGE, bool POOL>
__global__ void __launch_bounds__(kContribThreads, TSDF_CONTRIB_MIN_CTAS) contrib_kernel(const ScanArgs a,
                                                                                        const MapDev m,
                                                                                        const int kpt_max) {
    __shared__ unsigned long long red[kContribThreads / 32];
    __shared__ __align__(8) uint32_t btab[POOL ? kSlotCacheWords : kBrickCache];   // POOL: the slot cache
    const unsigned lane = threadIdx.x & 31u;
    const unsigned gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
    __shared__ unsigned s_counts[3];   // rays from the front, from the end, steps per item
    pdl_trigger();
    cache_init<POOL>(btab);
    pdl_wait();   // ray list and live count come from the rays kernel
    // A coherent load after the wait (a read-only __ldg could be hoisted above
    // it and see a count from before the rays kernel finished), one per CTA:
    // every CTA of the grid reads the same line, so per-warp reads would make
    // it a hot spot. The ray list may be split (heavy rays from the front,
    // light ones from the end): the blocks of the front come first, so the
    // costly items are taken by the first wave of CTAs and the CTAs that start
    // late get light ones.
    // Steps per item: an item of long steps (high fill columns) is cut while the
    // items are too few to even out over the warps. A 33 k-point corridor scan
    // of 18 lines (some hundred samples a step): 52 -> 28 us; corridor 64x1024
    // 24.6 -> 23.2, outdoor 64x1024 19.1 -> 18.4. Items of short steps stay
    // whole (one of 256^3 voxels at 0.1 m, no fill: 10.5 us with four steps, 12.3
    // with one), as do those of larger scans (corridor 128x2048: 29.2 and 33.3).
    // By one thread and without divisions: after an L2 flush, with the kernel's
    // code out of cache too, each line of it counts (outdoor 128x1024: 17.6 us,
    // done by every warp with divisions 17.8, the march a second time for a
    // constant four steps 17.6, only that march and no choice 17.1).
    const unsigned steps = (unsigned)(2 * a.K + 1);
    if (threadIdx.x == 0) {
        const unsigned f = __ldcg(&m.ctr->live[m.parity].front), b = __ldcg(&m.ctr->live[m.parity].back);
        const unsigned fill = __ldcg(&m.ctr->live[m.parity].fill);
        const unsigned blocks = (f + 31u) / 32u + (b + 31u) / 32u;
        const float rays = (float)(f + b), samples = rays + 2.f * (float)fill;   // of one step
        unsigned k = (unsigned)kpt_max;   // 1, 2 or 4
        while (k > 1u && (float)k * samples > 14.f * rays && blocks * ((steps + k - 1u) >> (k >> 1)) < 2u * nwarps) k >>= 1;
        s_counts[0] = f;
        s_counts[1] = b;
        s_counts[2] = k;
    }
    __syncthreads();   // (also orders the brick cache initialisation)
    const unsigned nf = s_counts[0], nb = s_counts[1];
    const unsigned bf = (nf + 31u) / 32u, bb = (nb + 31u) / 32u;
    const int kpt = (int)s_counts[2];
    const unsigned ngrp = (steps + kpt - 1) / kpt;
    const unsigned nitems = (bf + bb) * ngrp;
    // first ray of block `blk` and the end of its part of the list
    auto block_ray = [&](unsigned blk, unsigned& end) {
        if (blk < bf) {
            end = nf;
            return blk * 32u;
        }
        end = m.ray_cap;
        return m.ray_cap - nb + (blk - bf) * 32u;
    };
    unsigned hits = 0;
    unsigned last_brick = kNoVoxel;
    uint32_t last_slot = kPoolEmpty;
    const BrickCache bc = march_cache<POOL>(btab);
    float4 A, B;
    {
        unsigned end;
        const unsigned r0 = block_ray(gwarp / ngrp, end);
        load_rays(m, gwarp < nitems ? end : 0u, r0 + lane, A, B);
    }
    for (unsigned item = gwarp; item < nitems; item += nwarps) {   // warp-uniform
        float4 An, Bn;
        const unsigned next = item + nwarps;
        unsigned end;
        const unsigned r0 = block_ray(next / ngrp, end);
        load_rays(m, next < nitems ? end : 0u, r0 + lane, An, Bn);   // prefetch
        contrib_item<MODE, MERGE, false, POOL>(a, m, item % ngrp, kpt, A, B, hits, last_brick, kNoSlot, nullptr,
                                               &last_slot, bc);
        A = An;
        B = Bn;
    }
    if (MODE == 1) {
        // MIN_ABS keeps no contribution count per voxel: count them here
        const unsigned long long total = cta_sum<kContribThreads / 32>((unsigned long long)hits, red);
        if (threadIdx.x == 0 && total) atomicAdd(&m.ctr->part[blockIdx.x % kParts].hits, total);
    }
}

constexpr int kScanWarps = 8;
constexpr int kScanThreads = kScanWarps * 32;

// scan: ray set-up and contributions of one tile of `tile` points (a power of
// two, 32 .. 256) per CTA; `parts` CTAs share a tile's march steps when the
// scan has too few tiles for the chip (part p takes every parts-th item, and
// each of them sets the tile's rays up again).
//
// For small scans, which are bound by the chain of kernels and not by work:
// the rays stay in shared memory, so there is no ray list in memory, no list
// atomic and one kernel boundary less (the set-up runs before the wait for the
// previous scan). The tile shrinks with the scan and the work items with the
// tile, so that a scan of a few thousand points still occupies every SM (a
// 5760-point scan: 180 CTAs of one 32-ray block, nine steps over eight warps;
// through the ray list 14.3 us of contributions, here 12.0 with the set-up,
// and 17.9 instead of 26.2 us for the whole scan).
template <int MODE, bool MERGE, bool POOL>
__global__ void __launch_bounds__(kScanThreads, TSDF_SCAN_MIN_CTAS) scan_kernel(const ScanArgs a, const MapDev m,
                                                                               const int tile, const int parts,
                                                                               const int kpt_max) {
    __shared__ float4 s_a[kScanThreads], s_b[kScanThreads];
    __shared__ __align__(8) uint32_t btab[POOL ? kSlotCacheWords : kBrickCache];   // POOL: the slot cache
    __shared__ unsigned s_heavy[kScanWarps], s_light[kScanWarps], s_valid[kScanWarps];
    __shared__ unsigned s_next;
    __shared__ unsigned long long red[kScanWarps];
    const unsigned lane = threadIdx.x & 31u;
    const unsigned warp = threadIdx.x >> 5;
    const unsigned part = parts > 1 ? blockIdx.x % (unsigned)parts : 0u;
    const int first = (int)(parts > 1 ? blockIdx.x / (unsigned)parts : blockIdx.x) * tile;
    // ---- the tile's rays, compacted into shared memory
    const int i = first + (int)threadIdx.x;
    const bool in = (int)threadIdx.x < tile && i < a.n;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) p = __ldg(a.pts + i);   // the caller's points: no dependency on earlier grids
    pdl_trigger();
    cache_init<POOL>(btab);
    if (threadIdx.x == 0) s_next = kScanWarps;
    unsigned nlive, nheavy;
    {
        float4 ra, rb;
        bool valid, live;
        ray_setup(a, p, in, ra, rb, valid, live);
        const bool heavy = live && rb.w != 0.f && fm(fm(a.dz, ra.w), a.inv_vs) >= 1.f;
        const unsigned hmask = __ballot_sync(kFull, heavy);
        const unsigned lmask = __ballot_sync(kFull, live && !heavy);
        const unsigned vmask = __ballot_sync(kFull, valid);
        if (lane == 0) {
            s_heavy[warp] = __popc(hmask);
            s_light[warp] = __popc(lmask);
            s_valid[warp] = __popc(vmask);
        }
        __syncthreads();
        unsigned hb = 0, lb = 0, ht = 0, lt = 0;
#pragma unroll
        for (int w = 0; w < kScanWarps; ++w) {
            const unsigned h = s_heavy[w], l = s_light[w];
            if (w < (int)warp) {
                hb += h;
                lb += l;
            }
            ht += h;
            lt += l;
        }
        nheavy = ht;
        nlive = ht + lt;
        const unsigned below = (1u << lane) - 1u;
        if (live) {
            const unsigned off = heavy ? hb + __popc(hmask & below) : ht + lb + __popc(lmask & below);
            s_a[off] = ra;
            s_b[off] = rb;
        }
        __syncthreads();
    }
    pdl_wait();   // the previous scan's apply resets the counters, flags and accumulators
    if (part == 0u && threadIdx.x < 32) {
        const unsigned v = __reduce_add_sync(kFull, lane < kScanWarps ? s_valid[lane] : 0u);
        if (lane == 0 && v) atomicAdd(&m.ctr->live[m.parity].valid, v);
    }
    if (nlive == 0u) return;   // CTA-uniform
    // ---- march: items (32 rays of the tile, kpt steps), claimed by the warps
    const unsigned steps = (unsigned)(2 * a.K + 1);
    const unsigned blocks = (nlive + 31u) / 32u;
    int kpt = kpt_max;
    while (kpt > 1 && blocks * ((steps + kpt - 1) / kpt) < 2u * kScanWarps * (unsigned)parts) kpt >>= 1;
    const unsigned ngrp = (steps + kpt - 1) / kpt;
    const unsigned nitems = blocks * ngrp;
    unsigned hits = 0;
    unsigned last_brick = kNoVoxel;
    uint32_t last_slot = kPoolEmpty;
    const BrickCache bc = march_cache<POOL>(btab);
    unsigned claim = warp;
    for (;;) {
        const unsigned item = claim * (unsigned)parts + part;
        if (item >= nitems) break;
        const unsigned ray = (item / ngrp) * 32u + lane;
        float4 A = make_float4(0.f, 0.f, 0.f, -1.f), B = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ray < nlive) {
            A = s_a[ray];
            B = s_b[ray];
        }
        contrib_item<MODE, MERGE, false, POOL>(a, m, item % ngrp, kpt, A, B, hits, last_brick, kNoSlot, nullptr,
                                               &last_slot, bc);
        if (lane == 0) claim = atomicAdd(&s_next, 1u);
        claim = __shfl_sync(kFull, claim, 0);
    }
    if (MODE == 1) {
        // MIN_ABS keeps no contribution count per voxel: count them here
        const unsigned long long total = cta_sum<kScanWarps>((unsigned long long)hits, red);
        if (threadIdx.x == 0 && total) atomicAdd(&m.ctr->part[blockIdx.x % kParts].hits, total);
    }
}

// Sort reduction: the contribution march writing pairs (same work items).
template <int MODE, int KPT>
__global__ void __launch_bounds__(256, TSDF_EMIT_MIN_CTAS) emit_kernel(const ScanArgs a, const MapDev m) {
    __shared__ unsigned long long red[8];
    __shared__ uint32_t btab[kBrickCache];
    const unsigned lane = threadIdx.x & 31u;
    const unsigned gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
    pdl_trigger();
    brick_cache_init(btab);
    __syncthreads();
    pdl_wait();
    unsigned nlive = 0;
    if (lane == 0) nlive = __ldcg(&m.ctr->live_count);
    nlive = __shfl_sync(kFull, nlive, 0);
    const unsigned ngrp = (unsigned)(2 * a.K + KPT) / KPT;
    const unsigned nitems = (nlive + 31u) / 32u * ngrp;
    unsigned hits = 0;
    unsigned last_brick = kNoVoxel;
    bool ovf = false;
    for (unsigned item = gwarp; item < nitems; item += nwarps) {   // warp-uniform
        const unsigned ray = (item / ngrp) * 32u + lane;
        float4 A, B;
        load_rays(m, nlive, ray, A, B);
        const uint32_t sslot = ray < nlive ? m.ray_slot[ray] : kNoSlot;
        contrib_item<MODE, false, true>(a, m, item % ngrp, KPT, A, B, hits, last_brick, sslot, &ovf, nullptr,
                                             BrickCache{btab, 32u - kBrickCacheLog2});
    }
    if (ovf) m.ctr->overflow = 1u;
    if (MODE == 1) {
        const unsigned long long total = cta_sum<8>((unsigned long long)hits, red);
        if (threadIdx.x == 0 && total) atomicAdd(&m.ctr->part[blockIdx.x % kParts].hits, total);
    }
}

__global__ void __launch_bounds__(256) sort_count_kernel(const MapDev m) {
    pdl_trigger();
    pdl_wait();   // pairs come from emit, brick slots from compact
    const uint32_t n = sort_nslots(m);
    const uint32_t w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t w = w0; w * 128u < n; w += nw) sort_count_warp(m, w * 128u, n);
}

__global__ void __launch_bounds__(1024) sort_scan_kernel(const MapDev m) {
    __shared__ uint32_t smem[33];
    __shared__ uint32_t nb;
    pdl_trigger();
    pdl_wait();
    if (threadIdx.x == 0) nb = __ldcg(&m.ctr->brick_count);
    __syncthreads();
    sort_scan_cta(m, nb, smem);
}

__global__ void __launch_bounds__(256) sort_scatter_kernel(const MapDev m) {
    pdl_trigger();
    pdl_wait();
    const uint32_t n = sort_nslots(m);
    const uint32_t w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t w = w0; w * 128u < n; w += nw) sort_scatter_warp(m, w * 128u, n);
}

__global__ void __launch_bounds__(256) compact_kernel(const MapDev m, const uint32_t nwords) {
    pdl_trigger();
    pdl_wait();   // flags come from the contrib kernel
    compact_words(m, blockIdx.x * blockDim.x + threadIdx.x, nwords);
}

constexpr int kApplyWarps = 4;   // CTA size of the sort reduction's apply kernel

// ---- apply of the plain path: one CTA per SM.
//
// Flags (windows of at most kFlagBricks bricks): every CTA reads ALL brick
// flags (64 KB for 512x512x128 voxels, from L2), ranks the touched bricks with
// one CTA-wide prefix sum and takes every gridDim-th of them, so there is no
// compaction kernel, no list in memory and no list read before each task. The
// flags are cleared when all CTAs have read them: the last one to say so has
// one warp do it while the others work on. Larger windows: the compaction
// kernel lists the bricks, and each CTA takes every gridDim-th entry. Pool
// reduction: the claimed slots are the list; their table entries are reset,
// and when the pool was full the scan is dropped (accumulators cleared only).
//
// The CTA's bricks are cut into quarter-brick warp tasks. What bounds them is
// the latency of their loads (1.5 KB a task), so each warp keeps kApplyStages
// tasks in flight with cp.async into shared memory: at the outdoor scan (4.4 k
// bricks, 3.6 tasks per warp) that is all of them at once.
//
// Counters are published CTA by CTA (see kPubWords): no CTA waits for the
// others at the end (a fence, a returning atomic and the last CTA's reads were
// 3 us of every scan).
//
// 512 threads and four stages: 1024 threads leave no registers for the next
// scan's ray set-up beside them (outdoor pass 25.2 us, with four stages), 768
// threads 23.6, 512 threads 23.1, 384 threads 24.1; fewer than three stages of
// 512 threads are too little in flight for the corridor (53.9 against 46.2 us).
// Before (compaction kernel, four CTAs of 128 threads per SM and more, no
// staging, counters through the last CTA): outdoor 26.8, corridor 51.4, box room
// 17.9 us a pass; so staged: 23.1, 46.2, 14.4; with the exact quotient of
// apply_voxel_fast in place of an integer division 22.2, 45.5, 14.3. Its 36.9 k
// registers find no room beside three CTAs of 128 threads of a batched launch;
// with 64 registers a thread it would, but then two CTAs fit an SM and land on
// it (outdoor 27, corridor 52), and with 384 threads at 25.3 and 52.
constexpr int kApplyThreads = 512;
constexpr int kApplyWarpsPlain = kApplyThreads / 32;
constexpr int kApplyStages = 4;
constexpr int kApplyPairs = 2;                    // voxel pairs per lane in one task: a quarter brick
constexpr unsigned kApplyParts = 8u / kApplyPairs;
constexpr int kStageBytes = 128 * (8 + 4);        // accumulators and grid words of a quarter brick
constexpr int kApplySmem = kApplyWarpsPlain * kApplyStages * kStageBytes;
constexpr int kApplyList = 1024;                  // bricks of one CTA listed at a time
// Windows whose flags every CTA reads itself; larger ones go through the
// compaction kernel. Flags / list, us a pass: 2^16 bricks 23.5 / 24.5 (outdoor
// 128x1024) and 29.2 / 30.0 (16x512), 2^17 bricks 26.1 / 24.4 and 32.3 / 30.4;
// with flags up to 2^17 a thread holds 16 vectors of them and windows of 2^15
// take 18.8 instead of 17.3.
constexpr uint32_t kFlagBricks = 1u << 16;
constexpr int kFlagVecs = (int)(kFlagBricks / 16) / kApplyThreads;   // 16-flag vectors per thread, at most
static_assert(kFlagVecs * kApplyThreads * 16 == (int)kFlagBricks && kFlagVecs % 2 == 0, "flags per thread");

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Ranks the bricks whose flags are set and puts the CTA's own (ranks c, c + G,
// c + 2G, ...) into s_list; returns the number of touched bricks. ginv =
// ceil(2^32 / G): (rank * ginv) >> 32 is rank / G for rank <= 2^16.
__device__ __forceinline__ unsigned list_own_bricks(const uint8_t* flag, uint32_t bricks, unsigned c, unsigned G,
                                                    unsigned ginv, uint32_t* s_list, unsigned* s_warp) {
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint4* fv = reinterpret_cast<const uint4*>(flag);
    const unsigned nvec = bricks / 16u;   // 0: a window of 1 .. 8 bricks
    uint4 f[kFlagVecs];
#pragma unroll
    for (int j = 0; j < kFlagVecs; ++j) {
        const unsigned v = (unsigned)j * kApplyThreads + threadIdx.x;
        f[j] = make_uint4(0u, 0u, 0u, 0u);
        if (v < nvec) f[j] = __ldcg(fv + v);
    }
    if (nvec == 0u && threadIdx.x == 0) {
        for (uint32_t k = 0; k < bricks; ++k) (k < 4 ? f[0].x : f[0].y) |= (uint32_t)__ldcg(flag + k) << (8u * (k & 3u));
    }
    // this thread's touched bricks: a 16-bit mask per vector
    auto bits4 = [](uint32_t w) { return ((w & 0x01010101u) * 0x01020408u) >> 24 & 0xFu; };   // byte k -> bit k
    uint32_t mask[kFlagVecs / 2] = {};
    unsigned cnt = 0;
#pragma unroll
    for (int j = 0; j < kFlagVecs; ++j) {
        if ((f[j].x | f[j].y | f[j].z | f[j].w) == 0u) continue;   // most are empty
        const uint32_t b = bits4(f[j].x) | bits4(f[j].y) << 4 | bits4(f[j].z) << 8 | bits4(f[j].w) << 12;
        mask[j / 2] |= b << (16 * (j & 1));
        cnt += __popc(b);
    }
    unsigned incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, incl, o);
        if (lane >= (unsigned)o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();   // (every thread of the CTA has read its flags)
    const unsigned t = lane < (unsigned)kApplyWarpsPlain ? s_warp[lane] : 0u;
    unsigned ti = t;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, ti, o);
        if (lane >= (unsigned)o) ti += y;
    }
    const unsigned total = __shfl_sync(kFull, ti, 31);
    const unsigned rank = __shfl_sync(kFull, ti - t, warp) + incl - cnt;   // touched bricks before this thread's
    if (cnt) {
        unsigned q = __umulhi(rank, ginv);   // rank / G
        if (rank - q * G > c) ++q;
        for (unsigned r = q * G + c; r < rank + cnt; r += G, ++q) {
            unsigned skip = r - rank;
            int j = 0;
            uint32_t b = 0;
#pragma unroll
            for (int k = 0; k < kFlagVecs; ++k) {
                const uint32_t bk = mask[k / 2] >> (16 * (k & 1)) & 0xFFFFu;
                const unsigned n = __popc(bk);
                if (b == 0u) {
                    if (skip < n) {
                        b = bk;
                        j = k;
                    } else {
                        skip -= n;
                    }
                }
            }
            for (; skip; --skip) b &= b - 1u;
            s_list[q] = ((unsigned)j * kApplyThreads + threadIdx.x) * 16u + (unsigned)(__ffs(b) - 1);
        }
    }
    __syncthreads();
    return total;
}

enum ApplySource { kFromFlags, kFromList, kFromPool };

template <int MODE, int SRC>
__global__ void __launch_bounds__(kApplyThreads, 1) apply_kernel(const MapDev m, const uint32_t bricks,
                                                                const unsigned ginv, const int32_t w_max,
                                                                const int32_t flags) {
    extern __shared__ __align__(16) unsigned char stages[];
    __shared__ uint32_t s_list[kApplyList];
    __shared__ unsigned s_warp[kApplyWarpsPlain];
    __shared__ unsigned long long red_u[kApplyWarpsPlain], red_h[kApplyWarpsPlain];
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const unsigned G = gridDim.x, c = blockIdx.x;
    pdl_wait();      // flags or list, and accumulators, come from the earlier kernels
    pdl_trigger();   // (after the wait: the next scan's ray set-up writes the ray list)
    unsigned nb;
    bool dropped = false;   // pool: some brick found it full, the scan only clears up after itself
    if (SRC == kFromFlags) {
        nb = list_own_bricks(m.brick_flag, bricks, c, G, ginv, s_list, s_warp);
    } else {
        if (threadIdx.x == 0) {
            s_warp[0] = __ldcg(SRC == kFromList ? &m.ctr->brick_count : &m.ctr->pool_count);
            s_warp[1] = SRC == kFromPool ? __ldcg(&m.ctr->pool_overflow) : 0u;
        }
        __syncthreads();
        nb = s_warp[0];
        if (SRC == kFromPool) {
            nb = min(nb, m.pool_cap);
            dropped = s_warp[1] != 0u;
        }
    }
    long long* pub = m.host_last ? m.host_last : m.ctr->pub;
    if (warp == kApplyWarpsPlain - 1) {
        unsigned last = 0;
        if (lane == 0) {
            __threadfence();
            last = atomicAdd(&m.ctr->flags_read, 1u) == G - 1u ? 1u : 0u;
            __threadfence();
        }
        if (__shfl_sync(kFull, last, 0)) {   // all CTAs have read the flags (the list's length): clear them
            if (SRC != kFromFlags) {
                if (lane == 0) m.ctr->brick_count = m.ctr->pool_count = m.ctr->pool_overflow = 0u;
            } else if (bricks < 16u) {
                if (lane < bricks) m.brick_flag[lane] = 0;
            } else {
                for (unsigned v = lane; v < bricks / 16u; v += 32u)
                    reinterpret_cast<uint4*>(m.brick_flag)[v] = make_uint4(0u, 0u, 0u, 0u);
            }
            if (lane == 0) m.ctr->flags_read = 0u;
        }
    } else if (warp == kApplyWarpsPlain - 2 && c == 0u) {
        // the scan's own counters: valid rays, and in MIN_ABS mode the
        // contributions that the march counted; both start the next scan at 0
        LiveCounts* lc = &m.ctr->live[m.parity];
        unsigned long long h = 0;
        if (MODE == 1) {
            h = __ldcg(&m.ctr->part[lane].hits);
            m.ctr->part[lane].hits = 0ull;
            for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(kFull, h, o);
        }
        if (lane == 0) {
            pub[0] = (long long)__ldcg(&lc->valid);
            pub[1] = dropped ? 0 : (long long)h;
            pub[2] = 0;
            pub[3] = dropped ? kStatusCapacity : 0;
            pub[4] = (long long)G;
            lc->front = lc->back = lc->valid = lc->fill = 0u;
        }
    }
    // ---- warp tasks: quarters of the CTA's bricks, kApplyStages in flight
    const unsigned mine = c < nb ? (nb - c + G - 1u) / G : 0u;
    unsigned char* const ring = stages + (size_t)warp * (kApplyStages * kStageBytes);
    unsigned long long touched = 0, hits = 0;
    for (unsigned b0 = 0; b0 < mine; b0 += kApplyList) {   // CTA-uniform; one round unless a list is very long
        const unsigned nl = min(mine - b0, (unsigned)kApplyList);
        if (SRC != kFromFlags) {
            __syncthreads();
            for (unsigned i = threadIdx.x; i < nl; i += kApplyThreads) {
                const size_t at = c + (size_t)(b0 + i) * G;
                const uint32_t brick = __ldcg((SRC == kFromList ? m.brick_list : m.pool_brick) + at);
                s_list[i] = brick;
                if (SRC == kFromPool) m.pool_table[brick] = kPoolEmpty;
            }
            __syncthreads();
        }
        // accumulators of task t: the brick's own, or its pool slot's
        auto acc_word = [&](unsigned t, size_t v) {
            if (SRC != kFromPool) return v;
            return ((size_t)(c + (size_t)(b0 + t / kApplyParts) * G) << 9) + (t % kApplyParts) * 128u;
        };
        unsigned long long* const accs = SRC == kFromPool ? m.pool_acc : m.acc;
        const unsigned ntask = nl * kApplyParts;
        auto fetch = [&](unsigned t, unsigned stage) {
            if (t < ntask) {
                const size_t v = ((size_t)s_list[t / kApplyParts] << 9) + (t % kApplyParts) * 128u;
                ulonglong2* sa = reinterpret_cast<ulonglong2*>(ring + stage * kStageBytes);
                uint2* sg = reinterpret_cast<uint2*>(ring + stage * kStageBytes + 1024);
                const ulonglong2* ga = reinterpret_cast<const ulonglong2*>(accs + acc_word(t, v));
                const uint2* gg = reinterpret_cast<const uint2*>(m.grid + v);
                cp_async16(sa + lane, ga + lane);
                cp_async16(sa + 32 + lane, ga + 32 + lane);
                cp_async8(sg + lane, gg + lane);
                cp_async8(sg + 32 + lane, gg + 32 + lane);
            }
            cp_async_commit();
        };
#pragma unroll
        for (unsigned k = 0; k < kApplyStages; ++k) fetch(warp + k * kApplyWarpsPlain, k);
        unsigned stage = 0;
        for (unsigned t = warp; t < ntask; t += kApplyWarpsPlain) {   // warp-uniform
            cp_async_wait<kApplyStages - 1>();   // (a lane reads only what it copied itself)
            const size_t v = ((size_t)s_list[t / kApplyParts] << 9) + (t % kApplyParts) * 128u;
            const ulonglong2* sa = reinterpret_cast<const ulonglong2*>(ring + stage * kStageBytes);
            const uint2* sg = reinterpret_cast<const uint2*>(ring + stage * kStageBytes + 1024);
            ulonglong2 acc[kApplyPairs] = {sa[lane], sa[32 + lane]};
            uint2 g[kApplyPairs] = {sg[lane], sg[32 + lane]};
            if (!dropped) apply_pairs<MODE, kApplyPairs>(w_max, flags, acc, g, sg, touched, hits);   // (else the grid words as they were)
            fetch(t + kApplyStages * kApplyWarpsPlain, stage);
            store_pairs<kApplyPairs>(reinterpret_cast<uint2*>(m.grid + v),
                                     reinterpret_cast<ulonglong2*>(accs + acc_word(t, v)), acc, g);
            stage = stage + 1u == kApplyStages ? 0u : stage + 1u;
        }
        cp_async_wait<0>();
    }
    for (int o = 16; o > 0; o >>= 1) {
        touched += __shfl_xor_sync(kFull, touched, o);
        hits += __shfl_xor_sync(kFull, hits, o);
    }
    if (lane == 0) {
        red_u[warp] = touched;
        red_h[warp] = hits;
    }
    __syncthreads();
    if (warp == 0) {
        touched = lane < (unsigned)kApplyWarpsPlain ? red_u[lane] : 0ull;
        hits = lane < (unsigned)kApplyWarpsPlain ? red_h[lane] : 0ull;
        for (int o = 16; o > 0; o >>= 1) {
            touched += __shfl_xor_sync(kFull, touched, o);
            hits += __shfl_xor_sync(kFull, hits, o);
        }
        // (in MIN_ABS mode the contributions are the march's count)
        if (lane == 0) *reinterpret_cast<longlong2*>(pub + 8 + 2 * c) = make_longlong2((long long)touched, MODE == 0 ? (long long)hits : 0);
    }
}

// Sort reduction: one warp per listed brick (as apply_kernel, and likewise
// the last CTA publishes the counters).
template <int MODE>
__global__ void __launch_bounds__(kApplyWarps * 32) sort_apply_kernel(const MapDev m, const int32_t w_max,
                                                                       const int32_t flags) {
    __shared__ uint32_t s_grid[kApplyWarps][kBrickVoxels];
    __shared__ unsigned long long s_acc[kApplyWarps][kBrickVoxels];
    __shared__ uint16_t s_off[kApplyWarps][kBrickVoxels];
    __shared__ unsigned long long red_u[kApplyWarps], red_h[kApplyWarps];
    __shared__ unsigned s_last;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned w = threadIdx.x >> 5;
    const unsigned gwarp = blockIdx.x * kApplyWarps + w;
    const unsigned nwarps = gridDim.x * kApplyWarps;
    pdl_wait();
    pdl_trigger();   // (after the wait: the next scan's ray set-up writes the ray list)
    unsigned nb = 0, ovf = 0;
    if (lane == 0) {
        nb = __ldcg(&m.ctr->brick_count);
        ovf = __ldcg(&m.ctr->overflow);
    }
    nb = __shfl_sync(kFull, nb, 0);
    ovf = __shfl_sync(kFull, ovf, 0);
    unsigned long long touched = 0, hits = 0;
    for (unsigned i = gwarp; i < nb; i += nwarps)
        sort_apply_brick<MODE>(m, w_max, flags, i, ovf != 0u, s_grid[w], s_acc[w], s_off[w], touched, hits);
    for (int o = 16; o > 0; o >>= 1) {
        touched += __shfl_xor_sync(kFull, touched, o);
        hits += __shfl_xor_sync(kFull, hits, o);
    }
    if (lane == 0) {
        red_u[w] = touched;
        red_h[w] = hits;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long bu = 0, bh = 0;
        for (int k = 0; k < kApplyWarps; ++k) {
            bu += red_u[k];
            bh += red_h[k];
        }
        if (bu) atomicAdd(&m.ctr->part[blockIdx.x % kParts].touched, bu);
        if (bh) atomicAdd(&m.ctr->part[blockIdx.x % kParts].hits, bh);
    }
    finish_if_last(m, &s_last);
}

// Launch with `smem` bytes of dynamic shared memory, with programmatic stream
// serialisation when `pdl` is set.
template <typename... KArgs, typename... Args>
cudaError_t launch_smem(size_t smem, void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, bool pdl,
                        Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, bool pdl, Args&&... args) {
    return launch_smem(0, kernel, grid, block, s, pdl, std::forward<Args>(args)...);
}

// Allows `kernel` `bytes` of dynamic shared memory on the current device (once
// per kernel and device).
cudaError_t allow_smem(const void* kernel, int bytes) {
    static std::mutex mu;
    static std::set<std::pair<const void*, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({kernel, dev})) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.insert({kernel, dev});
    return e;
}

// CTAs of `kernel` (launched with `threads` threads and static shared memory
// only) that the current device holds at once: SMs x resident CTAs per SM.
// Persistent kernels launch exactly this many, so no CTA waits for a second
// wave. Cached per kernel and device.
int resident_ctas(const void* kernel, int threads) {
    static std::mutex mu;
    static std::unordered_map<unsigned long long, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long key = (unsigned long long)(uintptr_t)kernel * 1024ull + (unsigned long long)dev;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int sms = 1, per_sm = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int n = (sms > 0 ? sms : 1) * per_sm;
    cache[key] = n;
    return n;
}

template <typename... KArgs>
dim3 resident_grid(void (*kernel)(KArgs...), int threads, int per_sm = 0) {
    if (per_sm > 0) {
        static int sms[64] = {};
        int dev = 0;
        cudaGetDevice(&dev);
        const int d = dev >= 0 && dev < 64 ? dev : 0;
        if (sms[d] == 0) {
            int v = 1;
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
            sms[d] = v > 0 ? v : 1;
        }
        return dim3((unsigned)(sms[d] * per_sm));
    }
    return dim3((unsigned)resident_ctas(reinterpret_cast<const void*>(kernel), threads));
}

template <int MODE, int KPT>
cudaError_t launch_emit_k(const ScanArgs& a, const MapDev& m, bool pdl, cudaStream_t s) {
    auto* k = emit_kernel<MODE, KPT>;
    return launch(k, resident_grid(k, 256, TSDF_CONTRIB_CTAS_PER_SM), dim3(256), s, pdl, a, m);
}

}  // namespace

// Tile and parts of a scan of n points with K march steps each side of the hit.
// The largest tile that gives every SM work (several CTAs for each, so that
// uneven tiles even out); with the smallest tile, several CTAs per tile while
// each still has an item for every warp.
bool scan_fused(int64_t n) { return n <= TSDF_SCAN_FUSED_MAX; }

ScanShape scan_shape(int64_t n, int K) {
    const int64_t want = TSDF_SCAN_TILES;
    ScanShape g{TSDF_SCAN_MAX_TILE, 1, 0};
    while (g.tile > 32 && (n + g.tile - 1) / g.tile < want) g.tile >>= 1;
    const int64_t tiles = (n + g.tile - 1) / g.tile;
    if (tiles > 0 && tiles < want) {
        const int64_t items = (int64_t)(g.tile / 32) * (2 * (int64_t)K + 1);
        g.parts = (int)std::max<int64_t>(1, std::min<int64_t>((want + tiles - 1) / tiles, items / kScanWarps));
    }
    g.grid = (unsigned)(tiles * g.parts);
    return g;
}

// The kernel of the given mode, merge and pool reduction among a template's instances.
#define TSDF_PICK(kernel, reduce, merge, pool)                                         \
    ((pool) ? ((reduce) == 0 ? kernel<0, false, true> : kernel<1, false, true>)        \
            : (merge) ? ((reduce) == 0 ? kernel<0, true, false> : kernel<1, true, false>) \
                      : ((reduce) == 0 ? kernel<0, false, false> : kernel<1, false, false>))

const void* scan_kernel_fn(int32_t reduce, bool merge) {
    return reinterpret_cast<const void*>(TSDF_PICK(scan_kernel, reduce, merge, false));
}

cudaError_t launch_scan(const ScanArgs& a, const MapDev& m, int32_t reduce, bool merge, bool pool, int kpt, bool pdl,
                        cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    const ScanShape g = scan_shape(a.n, a.K);
    return launch(TSDF_PICK(scan_kernel, reduce, merge, pool), dim3(g.grid), dim3(kScanThreads), s, pdl, a, m, g.tile,
                  g.parts, kpt);
}

const void* rays_kernel_fn(bool sort) {
    return sort ? reinterpret_cast<const void*>(rays_kernel<true>) : reinterpret_cast<const void*>(rays_kernel<false>);
}

const void* contrib_kernel_fn(int32_t reduce, bool merge) {
    return reinterpret_cast<const void*>(TSDF_PICK(contrib_kernel, reduce, merge, false));
}

unsigned rays_grid(int64_t n, bool sort) {
    const int64_t per_cta = (int64_t)kRaysThreads * (sort ? 1 : kRaysPPT);
    return (unsigned)((n + per_cta - 1) / per_cta);
}

cudaError_t launch_rays(const ScanArgs& a, const MapDev& m, bool sort, bool pdl, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    return launch(sort ? rays_kernel<true> : rays_kernel<false>, dim3(rays_grid(a.n, sort)), dim3(kRaysThreads), s,
                  pdl, a, m);
}

cudaError_t launch_contrib(const ScanArgs& a, const MapDev& m, int32_t reduce, bool merge, bool pool, int kpt,
                           bool pdl, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    auto* k = TSDF_PICK(contrib_kernel, reduce, merge, pool);
    return launch(k, resident_grid(k, kContribThreads, TSDF_CONTRIB_CTAS_PER_SM), dim3(kContribThreads), s, pdl, a, m,
                  kpt);
}

cudaError_t launch_emit(const ScanArgs& a, const MapDev& m, int32_t reduce, int kpt, bool pdl, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    if (reduce == 0) {
        switch (kpt) {
            case 2: return launch_emit_k<0, 2>(a, m, pdl, s);
            case 4: return launch_emit_k<0, 4>(a, m, pdl, s);
            default: return launch_emit_k<0, 1>(a, m, pdl, s);
        }
    }
    switch (kpt) {
        case 2: return launch_emit_k<1, 2>(a, m, pdl, s);
        case 4: return launch_emit_k<1, 4>(a, m, pdl, s);
        default: return launch_emit_k<1, 1>(a, m, pdl, s);
    }
}

cudaError_t launch_sort_count(const MapDev& m, bool pdl, cudaStream_t s) {
    return launch(sort_count_kernel, resident_grid(sort_count_kernel, 256), dim3(256), s, pdl, m);
}

cudaError_t launch_sort_scan(const MapDev& m, bool pdl, cudaStream_t s) {
    return launch(sort_scan_kernel, dim3(1), dim3(1024), s, pdl, m);
}

cudaError_t launch_sort_scatter(const MapDev& m, bool pdl, cudaStream_t s) {
    return launch(sort_scatter_kernel, resident_grid(sort_scatter_kernel, 256), dim3(256), s, pdl, m);
}

cudaError_t launch_sort_apply(const MapDev& m, int32_t reduce, int32_t w_max, int32_t flags, bool pdl,
                              cudaStream_t s) {
    auto* k = reduce == 0 ? sort_apply_kernel<0> : sort_apply_kernel<1>;
    return launch(k, resident_grid(k, kApplyWarps * 32), dim3(kApplyWarps * 32), s, pdl, m,
                  w_max, flags);
}

cudaError_t launch_compact(const MapDev& m, uint32_t bricks, bool pdl, cudaStream_t s) {
    const uint32_t nwords = (bricks + 3u) / 4u;
    return launch(compact_kernel, dim3((nwords + 255u) / 256u), dim3(256), s, pdl, m, nwords);
}

cudaError_t launch_apply(const MapDev& m, uint32_t bricks, bool pool, int32_t reduce, int32_t w_max, int32_t flags,
                         bool pdl, cudaStream_t s) {
    const unsigned sms = resident_grid(apply_kernel<0, kFromFlags>, kApplyThreads, 1).x;
    const unsigned G = std::min(sms, (unsigned)kMaxApplyCtas);
    const bool by_flags = !pool && bricks <= kFlagBricks && (bricks + G - 1) / G <= (uint32_t)kApplyList;
    if (!pool && !by_flags) {
        const cudaError_t e = launch_compact(m, bricks, pdl, s);
        if (e != cudaSuccess) return e;
    }
    auto* k = pool ? (reduce == 0 ? apply_kernel<0, kFromPool> : apply_kernel<1, kFromPool>)
              : by_flags ? (reduce == 0 ? apply_kernel<0, kFromFlags> : apply_kernel<1, kFromFlags>)
                         : (reduce == 0 ? apply_kernel<0, kFromList> : apply_kernel<1, kFromList>);
    const cudaError_t e = allow_smem(reinterpret_cast<const void*>(k), kApplySmem);
    if (e != cudaSuccess) return e;
    const unsigned ginv = (unsigned)(((1ull << 32) + G - 1) / G);
    return launch_smem(kApplySmem, k, dim3(G), dim3(kApplyThreads), s, pdl, m, bricks, ginv, w_max, flags);
}

}  // namespace tsdf
