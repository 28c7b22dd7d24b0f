// Consumers of the map's zero level set (the paper's outlook puts mesh
// extraction and TSDF-based registration after the map generation).
//
// Both kernels work brick by brick, as the window is stored: a warp takes a
// brick (8^3 voxels, 2 KiB contiguous), loads it with four 16-byte loads per
// lane and goes on to the next one unless some voxel has been observed often
// enough; only then are the voxels of the neighbouring bricks that its pairs or
// cubes reach fetched too, and the 9^3 voxels put into shared memory. So the
// window is read once (134 MB for 512x512x128 voxels, 20 us at the memory
// rate), with no division or ring arithmetic per voxel, and the work of the few
// bricks with a surface is done from shared memory. Output is appended with
// one atomic per brick, so its order is unspecified.
//
// Surface points: for every pair of 6-connected window voxels a and b = a +
// e_axis with both weights >= min_weight and values of different sign
// ((v_a < 0) != (v_b < 0)), one point where the linear interpolation of the
// stored codes between the two voxel centres is zero:
//   t = v_a / (v_a - v_b)                       (one IEEE division, round to nearest)
//   p_axis = ((float)g_axis + 0.5 + t) * vs      (the other two: ((float)g + 0.5) * vs)
// in world metres, with the axis index in the fourth component.
//
// Measured on a map of six outdoor scans (512x512x128): surface 209 us with a
// thread per window voxel, mesh 1830 us with a thread per window cube.
#include "tsdf_internal.cuh"

namespace tsdf {
namespace {

constexpr unsigned kFullMask = 0xFFFFFFFFu;
constexpr int kWarps = 8;              // warps per CTA
constexpr int kTile = 9 * 9 * 9;       // a brick's voxels and one layer of its upper neighbours'

__device__ __forceinline__ int value_of(uint32_t w) { return (int)(int16_t)(w & 0xFFFFu); }
__device__ __forceinline__ int weight_of(uint32_t w) { return (int)w >> 16; }

struct BrickWindow {
    WindowGeom geo;
    uint32_t bricks;
    uint32_t slot[3];    // ring slot of the window's first chunk, per axis
    int origin[3];       // window origin in voxels
};

// One warp: brick `b` (ring index) into `tile` (voxel (x, y, z) at 81 z + 9 y +
// x) with the layers x = 8, y = 8, z = 8 of its neighbours (EDGES: also where
// two or three of them meet), zero beyond the window. g0: the brick's first
// voxel in global coordinates. False when no voxel of the brick has weight >=
// min_w: then nothing was staged.
template <bool EDGES>
__device__ __forceinline__ bool load_tile(const uint32_t* __restrict__ grid, const BrickWindow& wd, uint32_t b,
                                          int min_w, uint32_t* tile, int g0[3]) {
    const unsigned lane = threadIdx.x & 31u;
    const uint4* bp = reinterpret_cast<const uint4*>(grid + ((size_t)b << 9));
    uint4 w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = __ldg(bp + 32 * j + lane);
    bool seen = false;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        seen = seen || weight_of(w[j].x) >= min_w || weight_of(w[j].y) >= min_w || weight_of(w[j].z) >= min_w ||
               weight_of(w[j].w) >= min_w;
    if (!__any_sync(kFullMask, seen)) return false;
    __syncwarp();   // the warp is done with the previous brick's tile
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned o = 4u * (32u * j + lane);   // four voxels of one x row
        uint32_t* t = tile + (o >> 6) * 81u + ((o >> 3) & 7u) * 9u + (o & 7u);
        t[0] = w[j].x;
        t[1] = w[j].y;
        t[2] = w[j].z;
        t[3] = w[j].w;
    }
    const WindowGeom& g = wd.geo;
    const uint32_t s[3] = {b & g.cmask[0], (b >> g.lcx) & g.cmask[1], b >> g.lcxy};
    uint32_t next[3];    // ring slot of the upper neighbour
    bool inside[3];      // it belongs to the window
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const uint32_t r = (s[a] - wd.slot[a]) & g.cmask[a];   // chunk position in the window
        g0[a] = wd.origin[a] + 8 * (int)r;
        next[a] = (s[a] + 1u) & g.cmask[a];
        inside[a] = r < g.cmask[a];
    }
    constexpr unsigned kHalo = EDGES ? 217u : 192u;
    for (unsigned i = lane; i < kHalo; i += 32u) {
        unsigned x, y, z;
        if (EDGES) {
            if (i < 81u) {             // z = 8: 9 x 9
                z = 8u;
                y = i / 9u;
                x = i - 9u * y;
            } else if (i < 153u) {     // y = 8, z < 8: 9 x 8
                y = 8u;
                z = (i - 81u) / 9u;
                x = i - 81u - 9u * z;
            } else {                   // x = 8, y < 8, z < 8
                x = 8u;
                y = (i - 153u) & 7u;
                z = (i - 153u) >> 3;
            }
        } else {
            const unsigned u = i & 7u, v = (i >> 3) & 7u, f = i >> 6;
            x = f == 0u ? 8u : u;
            y = f == 1u ? 8u : (f == 0u ? u : v);
            z = f == 2u ? 8u : v;
        }
        const bool ox = x == 8u, oy = y == 8u, oz = z == 8u;
        uint32_t word = 0u;
        if ((!ox || inside[0]) && (!oy || inside[1]) && (!oz || inside[2])) {
            const size_t nb = ((size_t)(oz ? next[2] : s[2]) << g.lcxy) | ((oy ? next[1] : s[1]) << g.lcx) |
                              (ox ? next[0] : s[0]);
            word = __ldg(grid + (nb << 9) + ((z & 7u) * 8u + (y & 7u)) * 8u + (x & 7u));
        }
        tile[z * 81u + y * 9u + x] = word;
    }
    __syncwarp();
    return true;
}

__global__ void __launch_bounds__(kWarps * 32) surface_kernel(const uint32_t* __restrict__ grid, const BrickWindow wd,
                                                             int min_w, float vs, float4* __restrict__ out,
                                                             unsigned long long cap,
                                                             unsigned long long* __restrict__ count) {
    __shared__ uint32_t s_tile[kWarps][kTile];
    const unsigned lane = threadIdx.x & 31u;
    uint32_t* tile = s_tile[threadIdx.x >> 5];
    const uint32_t stride = gridDim.x * kWarps;
    for (uint32_t b = blockIdx.x * kWarps + (threadIdx.x >> 5); b < wd.bricks; b += stride) {   // warp-uniform
        int g0[3];
        if (!load_tile<false>(grid, wd, b, min_w, tile, g0)) continue;
        // crossings of this lane's voxels: bit 3 i + axis for voxel 32 i + lane
        constexpr unsigned kNext[3] = {1u, 9u, 81u};
        unsigned long long found = 0ull;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const unsigned v = 32u * i + lane;
            const uint32_t* t = tile + (v >> 6) * 81u + ((v >> 3) & 7u) * 9u + (v & 7u);
            const uint32_t wa = t[0];
            if (weight_of(wa) < min_w) continue;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                const uint32_t wb = t[kNext[ax]];
                if (weight_of(wb) >= min_w && ((wa ^ wb) & 0x8000u)) found |= 1ull << (3 * i + ax);
            }
        }
        const unsigned n = (unsigned)__popcll(found);
        unsigned incl = n;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFullMask, incl, o);
            if (lane >= (unsigned)o) incl += y;
        }
        const unsigned tot = __shfl_sync(kFullMask, incl, 31);
        if (tot == 0u) continue;
        unsigned long long at = 0;
        if (lane == 31) at = atomicAdd(count, (unsigned long long)tot);
        at = __shfl_sync(kFullMask, at, 31) + (incl - n);
        for (; found; found &= found - 1ull, ++at) {
            if (at >= cap) break;
            const unsigned bit = (unsigned)__ffsll((long long)found) - 1u;
            const unsigned i = bit / 3u, ax = bit - 3u * i, v = 32u * i + lane;
            const unsigned x = v & 7u, y = (v >> 3) & 7u, z = v >> 6;
            const uint32_t* t = tile + z * 81u + y * 9u + x;
            const int va = value_of(t[0]), vb = value_of(t[ax == 0u ? 1u : ax == 1u ? 9u : 81u]);
            const float f[3] = {__fadd_rn((float)(g0[0] + (int)x), 0.5f), __fadd_rn((float)(g0[1] + (int)y), 0.5f),
                                __fadd_rn((float)(g0[2] + (int)z), 0.5f)};
            const float d = __fdiv_rn((float)va, (float)(va - vb));
            out[at] = make_float4(__fmul_rn(ax == 0u ? __fadd_rn(f[0], d) : f[0], vs),
                                  __fmul_rn(ax == 1u ? __fadd_rn(f[1], d) : f[1], vs),
                                  __fmul_rn(ax == 2u ? __fadd_rn(f[2], d) : f[2], vs), (float)ax);
        }
    }
}

// ---- marching tetrahedra (see tsdf_extract_mesh in the public header).
// Corners of a dual cube are numbered by their offsets, x + 2 y + 4 z; the
// cube's sign mask has a bit per negative corner. Tetrahedron tt is 000, e_i,
// e_i + e_j, 111 for the tt-th axis order (i, j, k) in lexicographic order; its
// corners as four 4-bit numbers:
__device__ __forceinline__ unsigned tet_codes(unsigned tt) {
    const unsigned i = tt >> 1, j = (i == 0u) ? 1u + (tt & 1u) : (i == 1u ? 2u * (tt & 1u) : (tt & 1u));
    const unsigned c1 = 1u << i, c2 = c1 | (1u << j);
    return (c1 << 4) | (c2 << 8) | (7u << 12);
}
// Signs of its corners (bit k: corner k is negative) in a cube's sign mask.
__device__ __forceinline__ unsigned tet_signs(unsigned codes, unsigned mask) {
    return (mask & 1u) | ((mask >> ((codes >> 4) & 15u)) & 1u) << 1 | ((mask >> ((codes >> 8) & 15u)) & 1u) << 2 |
           ((mask >> 7) & 1u) << 3;
}
// Triangles of a tetrahedron with `neg` negative corners: 0, 1, 2, 1, 0.
__device__ __forceinline__ unsigned tet_triangles(unsigned neg) { return (0x64u >> (2u * neg)) & 3u; }

// Whether the triangle's normal points away from the positive corners
// (n . dir < 0), with dir = mean of the positive corners - mean of the negative
// ones: in binary32 where that decides it, else in binary64, as the vertices
// are (a sliver's sign can hang on the rounding of its vertices). The
// binary32 value is off by less than 8 roundings of the terms' absolute sum.
__device__ __forceinline__ bool mt_flip(const float (&p)[3], const float (&q)[3], const float (&r)[3], unsigned codes,
                                        unsigned signs) {
    const unsigned neg = __popc(signs);
    const float wn = neg == 1u ? -1.0f : neg == 2u ? -0.5f : -1.0f / 3.0f;
    const float wp = neg == 3u ? 1.0f : neg == 2u ? 0.5f : 1.0f / 3.0f;
    float d[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if ((codes >> (4 * k + a)) & 1u) d[a] += (signs >> k) & 1u ? wn : wp;
    const float e1[3] = {q[0] - p[0], q[1] - p[1], q[2] - p[2]};
    const float e2[3] = {r[0] - p[0], r[1] - p[1], r[2] - p[2]};
    const float t[6] = {e1[1] * e2[2] * d[0], e1[2] * e2[1] * d[0], e1[2] * e2[0] * d[1],
                        e1[0] * e2[2] * d[1], e1[0] * e2[1] * d[2], e1[1] * e2[0] * d[2]};
    const float s = (t[0] - t[1]) + (t[2] - t[3]) + (t[4] - t[5]);
    const float m = (fabsf(t[0]) + fabsf(t[1])) + (fabsf(t[2]) + fabsf(t[3])) + (fabsf(t[4]) + fabsf(t[5]));
    if (fabsf(s) > 4e-6f * m) return s < 0.f;
    double dir[3] = {0.0, 0.0, 0.0};
    for (unsigned k = 0; k < 4; ++k)
        for (unsigned a = 0; a < 3; ++a)
            dir[a] += ((signs >> k) & 1u ? -1.0 / (int)neg : 1.0 / (4 - (int)neg)) * (double)((codes >> (4 * k + a)) & 1u);
    const double f1[3] = {(double)q[0] - p[0], (double)q[1] - p[1], (double)q[2] - p[2]};
    const double f2[3] = {(double)r[0] - p[0], (double)r[1] - p[1], (double)r[2] - p[2]};
    const double nx = f1[1] * f2[2] - f1[2] * f2[1], ny = f1[2] * f2[0] - f1[0] * f2[2],
                 nz = f1[0] * f2[1] - f1[1] * f2[0];
    return nx * dir[0] + ny * dir[1] + nz * dir[2] < 0.0;
}

__device__ __forceinline__ void mt_store(float* o, const float (&p)[3], const float (&q)[3], const float (&r)[3],
                                         bool flip) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o[a] = p[a];
        o[3 + a] = flip ? r[a] : q[a];
        o[6 + a] = flip ? q[a] : r[a];
    }
}

__global__ void __launch_bounds__(kWarps * 32) mesh_kernel(const uint32_t* __restrict__ grid, const BrickWindow wd,
                                                          int min_w, float vs, float* __restrict__ out,
                                                          unsigned long long cap,
                                                          unsigned long long* __restrict__ count) {
    __shared__ uint32_t s_tile[kWarps][kTile];
    __shared__ uint32_t s_cube[kWarps][512];   // cubes with triangles: number | sign mask << 9 | first triangle << 17
    __shared__ uint16_t s_pack[256];           // per sign mask: two bits per tetrahedron, its triangles
    static_assert(kWarps * 32 == 256, "one sign mask per thread");
    {
        unsigned pack = 0;
        for (unsigned tt = 0; tt < 6; ++tt)
            pack |= tet_triangles(__popc(tet_signs(tet_codes(tt), threadIdx.x))) << (2u * tt);
        s_pack[threadIdx.x] = (uint16_t)pack;
    }
    __syncthreads();
    // triangles of the first `fields` tetrahedra of a packed word (12 at most in all)
    auto sum_fields = [](unsigned pack, unsigned fields) {
        unsigned x = pack & ((1u << (2u * fields)) - 1u);
        x = (x & 0x333u) + ((x >> 2) & 0x333u);
        return (x + (x >> 4) + (x >> 8)) & 15u;
    };
    const unsigned lane = threadIdx.x & 31u;
    uint32_t* tile = s_tile[threadIdx.x >> 5];
    uint32_t* cubes = s_cube[threadIdx.x >> 5];
    const uint32_t stride = gridDim.x * kWarps;
    for (uint32_t b = blockIdx.x * kWarps + (threadIdx.x >> 5); b < wd.bricks; b += stride) {   // warp-uniform
        int g0[3];
        if (!load_tile<true>(grid, wd, b, min_w, tile, g0)) continue;
        // ---- the cubes whose corners are all observed and differ in sign
        unsigned nc = 0, nt = 0;
        for (unsigned i = 0; i < 16u; ++i) {
            const unsigned v = 32u * i + lane;
            const uint32_t* t = tile + (v >> 6) * 81u + ((v >> 3) & 7u) * 9u + (v & 7u);
            bool ok = true;
            unsigned mask = 0;
#pragma unroll
            for (unsigned c = 0; c < 8u; ++c) {
                const uint32_t w = t[(c & 1u) + 9u * ((c >> 1) & 1u) + 81u * (c >> 2)];
                ok = ok && weight_of(w) >= min_w;
                mask |= ((w >> 15) & 1u) << c;
            }
            const unsigned n = ok ? sum_fields(s_pack[mask], 6u) : 0u;
            const unsigned act = __ballot_sync(kFullMask, n != 0u);
            if (act == 0u) continue;
            unsigned incl = n;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(kFullMask, incl, o);
                if (lane >= (unsigned)o) incl += y;
            }
            if (n) cubes[nc + __popc(act & ((1u << lane) - 1u))] = v | mask << 9 | (nt + incl - n) << 17;
            nc += __popc(act);
            nt += __shfl_sync(kFullMask, incl, 31);
        }
        if (nt == 0u) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(count, (unsigned long long)nt);
        at = __shfl_sync(kFullMask, at, 0);
        __syncwarp();
        // ---- a lane per tetrahedron
        for (unsigned e = lane; e < 6u * nc; e += 32u) {
            const uint32_t cw = cubes[e / 6u];
            const unsigned tt = e % 6u, v = cw & 511u, mask = (cw >> 9) & 255u;
            const unsigned codes = tet_codes(tt), signs = tet_signs(codes, mask);
            const unsigned n = tet_triangles(__popc(signs));
            const unsigned long long slot = at + (cw >> 17) + sum_fields(s_pack[mask], tt);
            if (n == 0u || slot >= cap) continue;
            const unsigned x = v & 7u, y = (v >> 3) & 7u, z = v >> 6;
            const uint32_t* t = tile + z * 81u + y * 9u + x;
            // Edges (negative corner, positive corner) of the triangle's or
            // quadrilateral's vertices, as corner numbers k: one corner against
            // three, the three in order; two against two, a < b negative and
            // c < d positive: ac, ad, bd, bc.
            unsigned pk, qk;   // four 2-bit numbers each
            if (n == 1u) {
                const bool one_neg = __popc(signs) == 1;
                const unsigned lone = (unsigned)__ffs(one_neg ? signs : ~signs & 15u) - 1u;
                unsigned rest = 0;
                unsigned shift = 0;
#pragma unroll
                for (unsigned k = 0; k < 4u; ++k)
                    if (k != lone) {
                        rest |= k << shift;
                        shift += 2u;
                    }
                const unsigned same = lone * 0x15u;
                pk = one_neg ? same : rest;
                qk = one_neg ? rest : same;
            } else {
                const unsigned a = (unsigned)__ffs(signs) - 1u, bb = 31u - (unsigned)__clz(signs);
                const unsigned inv = ~signs & 15u;
                const unsigned c = (unsigned)__ffs(inv) - 1u, d = 31u - (unsigned)__clz(inv);
                pk = a | a << 2 | bb << 4 | bb << 6;
                qk = c | d << 2 | d << 4 | c << 6;
            }
            auto vertex = [&](unsigned u, float (&o)[3]) {
                const unsigned cp = (codes >> (4u * ((pk >> (2u * u)) & 3u))) & 15u;
                const unsigned cq = (codes >> (4u * ((qk >> (2u * u)) & 3u))) & 15u;
                const int vp = value_of(t[(cp & 1u) + 9u * ((cp >> 1) & 1u) + 81u * (cp >> 2)]);
                const int vq = value_of(t[(cq & 1u) + 9u * ((cq >> 1) & 1u) + 81u * (cq >> 2)]);
                const float s = __fdiv_rn((float)vp, (float)(vp - vq));
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int bp = (int)((cp >> a) & 1u), bq = (int)((cq >> a) & 1u);
                    const int gp = g0[a] + (int)(a == 0 ? x : a == 1 ? y : z) + bp;
                    o[a] = __fmul_rn(__fadd_rn(__fadd_rn((float)gp, 0.5f), __fmul_rn(s, (float)(bq - bp))), vs);
                }
            };
            float p[3], q[3], r[3];
            vertex(0u, p);
            vertex(1u, q);
            vertex(2u, r);
            mt_store(out + 9ull * slot, p, q, r, mt_flip(p, q, r, codes, signs));
            if (n == 2u && slot + 1ull < cap) {
                vertex(3u, q);
                mt_store(out + 9ull * (slot + 1ull), p, r, q, mt_flip(p, r, q, codes, signs));
            }
        }
    }
}

BrickWindow brick_window(const WindowGeom& geo, const long long origin[3]) {
    BrickWindow w;
    w.geo = geo;
    w.bricks = (geo.cmask[0] + 1u) * (geo.cmask[1] + 1u) * (geo.cmask[2] + 1u);
    for (int a = 0; a < 3; ++a) {
        w.slot[a] = (uint32_t)((unsigned long long)(origin[a] >> 3) & geo.cmask[a]);
        w.origin[a] = (int)origin[a];   // |origin| <= 2^23
    }
    return w;
}

unsigned brick_grid(uint32_t bricks) {
    const uint32_t ctas = (bricks + kWarps - 1) / kWarps;
    return ctas < 8192u ? ctas : 8192u;
}

}  // namespace

cudaError_t launch_mesh(const uint32_t* grid, const WindowGeom& geo, const long long origin[3], int min_w, float vs,
                        float* out, unsigned long long cap, unsigned long long* count, cudaStream_t s) {
    const BrickWindow w = brick_window(geo, origin);
    mesh_kernel<<<brick_grid(w.bricks), kWarps * 32, 0, s>>>(grid, w, min_w, vs, out, cap, count);
    return cudaGetLastError();
}

cudaError_t launch_surface(const uint32_t* grid, const WindowGeom& geo, const long long origin[3], int min_w, float vs,
                           float4* out, unsigned long long cap, unsigned long long* count, cudaStream_t s) {
    const BrickWindow w = brick_window(geo, origin);
    surface_kernel<<<brick_grid(w.bricks), kWarps * 32, 0, s>>>(grid, w, min_w, vs, out, cap, count);
    return cudaGetLastError();
}

}  // namespace tsdf
