// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

struct tsdf_map;     // host-side map object (defined in api.cu)
struct tsdf_batch;   // batch object (defined in batch.cu)

namespace tsdf {

constexpr int32_t kQMax = 32767;
constexpr int kBrick = 8;                 // bricks are 8 x 8 x 8 voxels, stored contiguously
constexpr int kBrickVoxels = 512;

constexpr int32_t kFlagStepValue = 1;    // TSDF_FLAG_STEP_VALUE
constexpr int32_t kFlagScanWeight = 2;   // TSDF_FLAG_SCAN_WEIGHT

constexpr int kParts = 32;        // counters are spread over 32 slots, one 128-byte line each

// Per-map device counters (one instance per map, in device memory). The
// counters of the scan in flight are split over kParts slots so that CTAs
// add to different L2 lines; the finish kernel sums them.
struct CounterPart {
    unsigned long long valid;       // valid rays
    unsigned long long hits;        // in-window contributions
    unsigned long long touched;     // voxels updated
    unsigned long long pad[13];
};

// Published counters of the last completed scan, in device memory and, when
// the map has it, mapped host memory: words 0..3 are valid rays, contributions,
// touched voxels and status (0, or TSDF_ERR_CAPACITY when the scan was dropped:
// pool full); word 4 is the number of CTAs whose own (touched voxels,
// contributions) follow from word 8 on and are still to be added
// (sum_counters): the plain path's apply publishes them CTA by CTA, so that no
// CTA waits for another.
constexpr int kMaxApplyCtas = 160;
constexpr int kPubWords = 8 + 2 * kMaxApplyCtas;

// Rays of a plain scan (split ray list): heavy ones from the list's front,
// light ones from its end, valid points, and the sum of the rays' fill heights
// (voxels each side at the hit, 255 at most). Two of them, used in turn by
// consecutive scans (MapDev::parity): the ray set-up counts into one while the
// previous scan's apply still reads and clears the other.
struct LiveCounts {
    unsigned int front, back, valid, fill;
};

struct MapCounters {
    CounterPart part[kParts];
    long long pub[kPubWords];
    LiveCounts live[2];
    unsigned int live_count;        // rays of the scan in flight that can reach the window (compacted)
    unsigned int brick_count;       // length of the touched-brick list of the scan in flight
    unsigned long long slot_count;  // sort reduction: pair slots reserved by the scan in flight
    unsigned int overflow;          // sort reduction: 1 if some contribution went to the accumulators
    unsigned int apply_done;        // CTAs of the apply kernel that have finished (the last one publishes)
    unsigned long long surface_count;   // points found by the last surface extraction
    unsigned int pool_count;        // pool reduction: slots claimed by the scan in flight (may exceed the capacity)
    unsigned int pool_overflow;     // pool reduction: 1 if a brick found the pool full (the scan is dropped)
    unsigned int flags_read;        // CTAs of the plain apply that have read the brick flags or the list length
    unsigned int pad_;
};

constexpr uint32_t kPoolEmpty = 0xFFFFFFFFu;      // pool table entry of a brick without a slot
constexpr long long kStatusCapacity = -8;        // TSDF_ERR_CAPACITY

constexpr uint32_t kNoSlot = 0xFFFFFFFFu;        // ray without pair slots (all its samples overflow)
constexpr uint32_t kRaySlotLimit = 1u << 20;      // rays with more samples than this overflow
constexpr uint32_t kPairCapMax = 1u << 28;        // largest pair capacity of a map

// Device-side view of one map. The window is bricked and ring addressed:
// global voxel g lives in brick ((g >> 3) mod (dims / 8)) at offset
// ((g.z & 7) * 8 + (g.y & 7)) * 8 + (g.x & 7).
struct MapDev {
    uint32_t* grid;                 // value (low 16) | weight (high 16), 512 words per brick
    unsigned long long* acc;        // packed per-scan accumulators, same layout; all zero between scans
    uint8_t* brick_flag;            // one byte per brick (padded to 4): 1 = touched by the scan in flight
    uint32_t* brick_list;           // touched bricks of the scan in flight, built by the compaction kernel
    float4* ray_a;                  // per live ray (compacted): (dir.x, dir.y, dir.z, r)
    float4* ray_b;                  // per live ray (compacted): (int.x, int.y, int.z, fill ? 1 : 0)
    uint32_t ray_cap;               // entries of ray_a / ray_b (the split list fills them from both ends)
    MapCounters* ctr;
    long long* host_last;           // mapped pinned host memory for the published counters (kPubWords), or null
    uint32_t parity;                // which LiveCounts the plain scan in flight uses
    uint32_t wait_first;            // 1: its ray set-up counts only when the previous scan is over (graphs)
    // sort reduction (null / 0 when the map has no sort buffers)
    uint32_t* brick_slot;           // per brick: its position in the brick list (touched bricks only)
    uint32_t* seg_count;            // per list position: pair count, then the scatter cursor; zero between scans
    uint32_t* seg_start;            // per list position: first entry of the brick's segment in `sorted`
    uint32_t* ray_slot;             // per live ray: first pair slot, or kNoSlot
    uint2* pairs;                   // emitted (voxel word, code) per sample; word kNoVoxel = outside the window
    uint32_t* sorted;               // (offset in brick << 16) | (code & 0xFFFF), grouped by brick
    uint32_t pair_cap;              // capacity of `pairs` and `sorted`
    // pool reduction (null / 0 when the map has no pool)
    uint32_t* pool_table;           // per brick: its slot in the pool, kPoolEmpty between scans
    uint32_t* pool_brick;           // per slot: the brick that claimed it
    unsigned long long* pool_acc;   // per slot: 512 packed accumulators, all zero between scans
    uint32_t pool_cap;              // slots
};

// Everything the kernels need about one scan, passed by value.
struct ScanArgs {
    const float4* pts;
    int32_t n;
    int32_t K;                      // march steps on each side of the hit
    float R[9];                     // row-major rotation, sensor -> world
    float t[3];                     // sensor position in the world
    float vs, inv_vs, tau, qs, dz, rmin, rmax;
    int32_t fill;                   // delta_z > 0
    float win_lo[3], win_hi[3];     // window box in metres (rounded outward), for ray culling
    float fo[3];                    // window origin as float (exact: |origin| <= 2^23)
    float fe[3];                    // origin + dims as float (exact)
    uint32_t cmask[3];              // dims / 8 - 1 per axis
    uint32_t lcx, lcxy;             // log2(dims.x / 8), log2(dims.x / 8 * dims.y / 8)
    uint32_t dmask[3];              // dims - 1 per axis
    uint32_t omod[3];               // origin mod dims per axis (ring offset of the window origin)
    int32_t flags;                  // TSDF_FLAG_* bits
    // Derived constants of the lean contribution march (set by fill_lean_args).
    float2 l_nt;                    // (-t.x, -t.y)
    float2 l_m;                     // 1.5 * 2^23 - origin, x and y (exact: origins are multiples of 8)
    float l_mz;                     // the same for z
    float l_ntz;                    // -t.z
    uint32_t l_omb[3];              // (origin mod dims) - 0x4B400000 per axis, modulo 2^32
    uint32_t l_cy, l_cz;            // 2^(lcx + 9) - 64 and 2^(lcxy + 9) - 512 (brick strides in the word index)
};

// Fill the lean-march constants of `a` from its other fields (host side,
// after t, vs, inv_vs, fo, dmask, omod, lcx and lcxy are set).
inline void fill_lean_args(ScanArgs& a) {
    a.l_nt = make_float2(-a.t[0], -a.t[1]);
    a.l_m = make_float2(12582912.0f - a.fo[0], 12582912.0f - a.fo[1]);
    a.l_mz = 12582912.0f - a.fo[2];
    a.l_ntz = -a.t[2];
    for (int i = 0; i < 3; ++i) a.l_omb[i] = a.omod[i] - 0x4B400000u;
    a.l_cy = (1u << (a.lcx + 9u)) - 64u;
    a.l_cz = (1u << (a.lcxy + 9u)) - 512u;
}

// One brick slot that changes owner during a shift.
struct ShiftItem {
    uint32_t brick;                 // ring brick index
    uint32_t pad0;
    unsigned long long out_ptr;     // address of the shift's candidate slot with this item's index
    unsigned long long in_ptr;      // store address of the entering brick, 0 = zero fill
    unsigned long long pad1;
};

// One 2048-byte chunk copy (device addresses).
struct ChunkCopy {
    unsigned long long dst;
    unsigned long long src;
};

struct WindowGeom {
    uint32_t dims[3];
    uint32_t cmask[3];
    uint32_t lcx, lcxy;
};

// One scan of a batch: everything the batched kernel needs about it.
struct BatchItem {
    ScanArgs a;
    MapDev m;
    int32_t reduce;
    int32_t w_max;
    uint32_t bricks;
    int32_t flags;
};


// Host helpers implemented in api.cu for the batched path: validate a scan for
// `map`, grow its ray buffers if needed and fill the batch item.
int prepare_batch_item(::tsdf_map* map, const float* points_dev, int64_t n, const float pose[12], BatchItem* out);
int map_device(const ::tsdf_map* map);
// Device address of the map's published counters (kPubWords words).
const long long* map_last_counters(const ::tsdf_map* map);
// Host address of the mapped pinned copy of those counters, which every
// integration (per-map or batched) writes; null when the map has none.
const volatile long long* map_host_counters(const ::tsdf_map* map);
// Valid rays, contributions and touched voxels from published counters.
inline void sum_counters(const volatile long long* pub, long long out[3]) {
    out[0] = pub[0];
    out[1] = pub[1];
    out[2] = pub[2];
    const long long n = pub[4];
    for (long long c = 0; c < n; ++c) {
        out[2] += pub[8 + 2 * c];
        out[1] += pub[8 + 2 * c + 1];
    }
}
// Grow the map's per-ray buffers to hold n points (synchronous allocation).
int map_reserve_points(::tsdf_map* map, int64_t n);

// Grow the map's ray and sort-reduction buffers for scans of n points
// (synchronous allocation on first use or growth).
int map_reserve_sort(::tsdf_map* map, int64_t n);

// tsdf_batch_integrate; beside: a small launch that has to run beside another
// batch object's share of the device (in the shape that fits beside any, and
// without a say in the autotuner's choice).
int batch_integrate(::tsdf_batch* batch, ::tsdf_map* const* maps, const float* const* points_dev, const int64_t* n,
                    const float* poses, int32_t count, bool beside, void* stream);

// Launchers (return the cudaError_t of the launch).
// Ray set-up into the map's ray list. sort: pair slots per ray too (sort
// reduction); otherwise heavy rays (fill of at least one voxel each side) from
// the list's front, the others from its end (the contribution kernel takes
// heavy work first).
cudaError_t launch_rays(const ScanArgs& a, const MapDev& m, bool sort, bool pdl, cudaStream_t s);
// Plain atomic path up to the list of touched bricks: one kernel over tiles
// of points for small scans, else ray set-up and the contribution kernel
// (scan_fused tells which; the ray list is needed only by the latter).
bool scan_fused(int64_t n);
struct ScanShape {
    int tile;                       // points per CTA
    int parts;                      // CTAs that share a tile's march steps
    unsigned grid;                  // CTAs
};
ScanShape scan_shape(int64_t n, int K);
// CTAs of the ray set-up kernel for a scan of n points.
unsigned rays_grid(int64_t n, bool sort);
// The kernel functions that these launchers launch for these arguments (to
// find their nodes in a captured graph).
const void* scan_kernel_fn(int32_t reduce, bool merge);
const void* rays_kernel_fn(bool sort);
const void* contrib_kernel_fn(int32_t reduce, bool merge);
// (pool: contributions into claimed pool slots)
cudaError_t launch_scan(const ScanArgs& a, const MapDev& m, int32_t reduce, bool merge, bool pool, int kpt, bool pdl,
                        cudaStream_t s);
cudaError_t launch_contrib(const ScanArgs& a, const MapDev& m, int32_t reduce, bool merge, bool pool, int kpt,
                           bool pdl, cudaStream_t s);
cudaError_t launch_compact(const MapDev& m, uint32_t bricks, bool pdl, cudaStream_t s);
// Eq. 1 / Eq. 2 on the bricks whose flags are set, or (pool) that have slots;
// the flags' or slots' reset, and the scan's counters.
cudaError_t launch_apply(const MapDev& m, uint32_t bricks, bool pool, int32_t reduce, int32_t w_max, int32_t flags,
                         bool pdl, cudaStream_t s);
// Sort reduction: emit pairs, count per brick, prefix, scatter, reduce + apply.
cudaError_t launch_emit(const ScanArgs& a, const MapDev& m, int32_t reduce, int kpt, bool pdl, cudaStream_t s);
cudaError_t launch_sort_count(const MapDev& m, bool pdl, cudaStream_t s);
cudaError_t launch_sort_scan(const MapDev& m, bool pdl, cudaStream_t s);
cudaError_t launch_sort_scatter(const MapDev& m, bool pdl, cudaStream_t s);
cudaError_t launch_sort_apply(const MapDev& m, int32_t reduce, int32_t w_max, int32_t flags, bool pdl,
                              cudaStream_t s);
// The leaving brick of each item that holds a non-zero voxel claims the next
// candidate slot (*claimed counts them, from 0) and is copied to
// items[claim].out_ptr; claim[item] is that index or -1 (the brick held no
// data). claim may point to mapped host memory.
cudaError_t launch_shift(uint32_t* grid, const ShiftItem* items, int count, unsigned* claimed, int* claim,
                         cudaStream_t s);
cudaError_t launch_copy_chunks(const ChunkCopy* items, int count, cudaStream_t s);
// Registration: device memory for the CTAs' sums (32 doubles each) and their
// arrival counter (0 between calls), and the device-visible address of the 29
// sums of the normal equations (mapped host memory, or device memory): 32
// doubles, the last of which gets the evaluation's serial number when the sums
// are complete.
constexpr int kRegisterCtasPerSm = 1;
constexpr int kRegisterMaxCtas = 512;
struct RegisterBuffers {
    double* part;
    unsigned* done;
    double* out;
};
cudaError_t launch_register(const float* pts_dev, int n, const float pose[12], const uint32_t* grid,
                            const WindowGeom& geo, const long long origin[3], float vs, float inv_vs, float tau,
                            int min_w, int sms, const RegisterBuffers& buf, double serial, cudaStream_t s);
bool register_step(const double sys[29], float pose[12], double* step_norm);
cudaError_t launch_mesh(const uint32_t* grid, const WindowGeom& geo, const long long origin[3], int min_w, float vs,
                        float* out, unsigned long long cap, unsigned long long* count, cudaStream_t s);
cudaError_t launch_surface(const uint32_t* grid, const WindowGeom& geo, const long long origin[3], int min_w, float vs,
                           float4* out, unsigned long long cap, unsigned long long* count, cudaStream_t s);
cudaError_t launch_read_box(const uint32_t* grid, const long long lo[3], const uint32_t box[3],
                            const WindowGeom& g, int16_t* v, int16_t* w, cudaStream_t s);
cudaError_t launch_write_box(uint32_t* grid, const long long lo[3], const uint32_t box[3], const WindowGeom& g,
                             const int16_t* v, const int16_t* w, cudaStream_t s);

}  // namespace tsdf
