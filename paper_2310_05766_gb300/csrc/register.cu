// Scan-to-map registration on the TSDF (a consumer of the map; the paper's
// outlook names registration against the TSDF map). Gauss-Newton on
//   E(T) = sum_i d(T p_i)^2,
// d the trilinear interpolation of the stored truncated distances at a point,
// with the pose update q' = Exp(w) q + v (w, v in the world frame).
//
// The kernel evaluates, for the current pose, the normal equations of all
// points: a thread computes q = R p + t and u = q / vs - 0.5 of its points in
// binary32 (explicit round-to-nearest, the ray set-up's order), takes the 8
// voxels i0 + {0,1}^3 with i0 = floor(u), and if all lie in the window with
// weights >= min_w and |d| < tau adds J = [q x grad d, grad d] (binary64) to
// H = sum J J^T, g = sum J d, the cost and the count. The host solves
// H xi = -g (Cholesky) and updates the pose.
//
// What bounds it is the binary64 rate (2 fused multiply-adds per cycle and SM),
// so the binary64 work is cut to what the sums need: codes stay unscaled (the
// scale and the voxel size are factors of the 28 sums, applied once at the
// end), the interpolation and its gradient share their differences, products
// are fused into their sums, a warp's sums go through a transposing butterfly
// (31 additions a lane instead of 140), and a thread adds up several points
// first. About 80 instead of 375 binary64 instructions per point.
// The CTAs' sums are added by the last CTA to finish, in a fixed order, which
// writes the system to mapped host memory: one launch per evaluation, no
// clearing, no copy.
#include <cmath>
#include <cstring>

#include "tsdf_internal.cuh"

namespace tsdf {
namespace {

constexpr unsigned kFullMaskR = 0xFFFFFFFFu;
constexpr int kSysN = 29;      // 21 (H upper triangle) + 6 (g) + cost + count
constexpr int kRegWarps = 6;

struct RegArgs {
    const float4* pts;
    int n;
    float R[9];
    float t[3];
    float inv_vs;
    float lo[3], hi[3];      // window origin, and the last voxel that has an upper neighbour (exact)
    int min_w;
    double scale;            // tau / 32767
    double tau;
    double f_h, f_g, f_c;    // factors of H, g and the cost
    double serial;           // written behind the system, for a host that watches it
    WindowGeom geo;
};

// d of a point as its eight scaled codes interpolate it, in the order of the
// definition: decides |d| < tau where all corners are next to the truncation.
__device__ __noinline__ bool truncated(const int (&c)[8], double fx, double fy, double fz, double scale, double tau) {
    double x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = (double)c[2 * k] * scale * (1 - fx) + (double)c[2 * k + 1] * scale * fx;
    const double y0 = x[0] * (1 - fy) + x[1] * fy, y1 = x[2] * (1 - fy) + x[3] * fy;
    return !(fabs(y0 * (1 - fz) + y1 * fz) < tau);
}

// Contribution of point p to the system (codes per voxel and codes; count in
// `used`).
__device__ __forceinline__ void reg_point(const RegArgs& a, const uint32_t* __restrict__ grid, const float4& p,
                                          double (&acc)[28], unsigned& used) {
    float q[3], f[3];
    unsigned i0[3];
    bool in = isfinite(p.x) && isfinite(p.y) && isfinite(p.z);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        q[r] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(a.R[3 * r], p.x), __fmul_rn(a.R[3 * r + 1], p.y)),
                                   __fmul_rn(a.R[3 * r + 2], p.z)),
                         a.t[r]);
        const float u = __fsub_rn(__fmul_rn(q[r], a.inv_vs), 0.5f);
        const float fl = floorf(u);
        f[r] = __fsub_rn(u, fl);
        in = in && fl >= a.lo[r] && fl <= a.hi[r];   // both voxels of the axis in the window
        i0[r] = in ? (unsigned)(int)fl : 0u;
    }
    if (!in) return;
    // word index of a voxel = the sum of one term per axis
    size_t w[3][2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const unsigned x = i0[0] + k, y = i0[1] + k, z = i0[2] + k;
        w[0][k] = ((size_t)((x >> 3) & a.geo.cmask[0]) << 9) | (x & 7u);
        w[1][k] = ((size_t)((y >> 3) & a.geo.cmask[1]) << (a.geo.lcx + 9u)) | ((y & 7u) << 3);
        w[2][k] = ((size_t)((z >> 3) & a.geo.cmask[2]) << (a.geo.lcxy + 9u)) | ((z & 7u) << 6);
    }
    uint32_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = __ldg(grid + (w[0][k & 1] + w[1][(k >> 1) & 1] + w[2][k >> 2]));
    int c[8];
    bool seen = true;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        seen = seen && ((int)v[k] >> 16) >= a.min_w;
        c[k] = (int)(int16_t)(v[k] & 0xFFFFu);
    }
    if (!seen) return;
    const double fx = (double)f[0], fy = (double)f[1], fz = (double)f[2];
    // interpolate along x, y, z, keeping the derivative along each axis
    double dx[4], cx[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        dx[k] = (double)(c[2 * k + 1] - c[2 * k]);
        cx[k] = fma(fx, dx[k], (double)c[2 * k]);
    }
    const double dy0 = cx[1] - cx[0], dy1 = cx[3] - cx[2];
    const double cy0 = fma(fy, dy0, cx[0]), cy1 = fma(fy, dy1, cx[2]);
    const double gx0 = fma(fy, dx[1] - dx[0], dx[0]), gx1 = fma(fy, dx[3] - dx[2], dx[2]);
    const double g[3] = {fma(fz, gx1 - gx0, gx0), fma(fz, dy1 - dy0, dy0), cy1 - cy0};
    const double d = fma(fz, g[2], cy0);
    if (fabs(d) >= 32766.99 && truncated(c, fx, fy, fz, a.scale, a.tau)) return;
    const double qd[3] = {(double)q[0], (double)q[1], (double)q[2]};
    const double J[6] = {fma(qd[1], g[2], -(qd[2] * g[1])), fma(qd[2], g[0], -(qd[0] * g[2])),
                         fma(qd[0], g[1], -(qd[1] * g[0])), g[0], g[1], g[2]};
    int k = 0;
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int cc = r; cc < 6; ++cc, ++k) acc[k] = fma(J[r], J[cc], acc[k]);
#pragma unroll
    for (int r = 0; r < 6; ++r) acc[21 + r] = fma(J[r], d, acc[21 + r]);
    acc[27] = fma(d, d, acc[27]);
    ++used;
}

__global__ void __launch_bounds__(kRegWarps * 32) register_kernel(const RegArgs a, const uint32_t* __restrict__ grid,
                                                                 double* __restrict__ part,
                                                                 unsigned* __restrict__ done,
                                                                 double* __restrict__ out) {
    __shared__ double red[kRegWarps][32];
    __shared__ unsigned s_last;
    double acc[28];
    unsigned used = 0;
#pragma unroll
    for (int k = 0; k < 28; ++k) acc[k] = 0.0;
    const int stride = (int)(gridDim.x * blockDim.x);
    int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < a.n) p = __ldg(a.pts + i);
    while (i < a.n) {
        const int next = i + stride;
        float4 pn = p;
        if (next < a.n) pn = __ldg(a.pts + next);   // in flight while this point is worked on
        reg_point(a, grid, p, acc, used);
        p = pn;
        i = next;
    }
    // transposing butterfly: lane l ends with the warp's sum of entry l
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    double v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = k < 28 ? acc[k] : 0.0;
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const bool up = (lane & (unsigned)h) != 0u;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double keep = up ? v[k + h] : v[k], give = up ? v[k] : v[k + h];
            v[k] = keep + __shfl_xor_sync(kFullMaskR, give, h);
        }
    }
    const unsigned n_used = __reduce_add_sync(kFullMaskR, used);
    red[warp][lane] = lane == 28u ? (double)n_used : v[0];
    __syncthreads();
    if (warp == 0) {
        double s = red[0][lane];
#pragma unroll
        for (int w = 1; w < kRegWarps; ++w) s += red[w][lane];
        part[(size_t)blockIdx.x * 32u + lane] = s;
        __threadfence();
        __syncwarp();
        if (lane == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1u ? 1u : 0u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double s = 0.0;
    for (unsigned b = warp; b < gridDim.x; b += kRegWarps) s += __ldcg(part + (size_t)b * 32u + lane);
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        s = red[0][lane];
#pragma unroll
        for (int w = 1; w < kRegWarps; ++w) s += red[w][lane];
        if (lane < (unsigned)kSysN)
            out[lane] = s * (lane < 21u ? a.f_h : lane < 27u ? a.f_g : lane < 28u ? a.f_c : 1.0);
        if (lane == 0) *done = 0u;   // before the fence: a host that sees the serial may launch on another stream
        __threadfence_system();
        __syncwarp();
        if (lane == 0) *reinterpret_cast<volatile double*>(out + 31) = a.serial;   // the system above is complete
    }
}

}  // namespace

// CTAs of the kernel: one of six warps per SM. The binary64 unit is full with
// that, and a thread of a 128 x 1024 scan adds up four or five points before
// the warp's sums (six evaluations and one more: 239 us, 234-255 since the two
// calls synchronise; eight warps 250, two CTAs per SM 262-273 us; 720 us before).
cudaError_t launch_register(const float* pts_dev, int n, const float pose[12], const uint32_t* grid,
                            const WindowGeom& geo, const long long origin[3], float vs, float inv_vs, float tau,
                            int min_w, int sms, const RegisterBuffers& buf, double serial, cudaStream_t s) {
    RegArgs a{};
    a.pts = reinterpret_cast<const float4*>(pts_dev);
    a.n = n;
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c) a.R[3 * r + c] = pose[4 * r + c];
        a.t[r] = pose[4 * r + 3];
        a.lo[r] = (float)origin[r];
        a.hi[r] = (float)(origin[r] + (long long)geo.dims[r] - 2);
    }
    a.inv_vs = inv_vs;
    a.scale = (double)tau / 32767.0;
    a.tau = (double)tau;
    const double k = a.scale / (double)vs;   // d and its gradient from codes and codes per voxel
    a.f_h = k * k;
    a.f_g = k * a.scale;
    a.f_c = a.scale * a.scale;
    a.serial = serial;
    a.min_w = min_w;
    a.geo = geo;
    int blocks = (n + kRegWarps * 32 - 1) / (kRegWarps * 32);
    const int most = sms * kRegisterCtasPerSm < kRegisterMaxCtas ? sms * kRegisterCtasPerSm : kRegisterMaxCtas;
    if (blocks > most) blocks = most;
    if (blocks < 1) blocks = 1;
    register_kernel<<<blocks, kRegWarps * 32, 0, s>>>(a, grid, buf.part, buf.done, buf.out);
    return cudaGetLastError();
}

// One Gauss-Newton step on the host: solve H xi = -g by Cholesky (binary64),
// then R' = Exp(w) R, t' = Exp(w) t + v. Returns false if H is not positive
// definite.
bool register_step(const double sys[29], float pose[12], double* step_norm) {
    double H[6][6];
    int k = 0;
    for (int r = 0; r < 6; ++r)
        for (int c = r; c < 6; ++c) H[r][c] = H[c][r] = sys[k++];
    double L[6][6] = {};
    for (int j = 0; j < 6; ++j) {
        double s = H[j][j];
        for (int p = 0; p < j; ++p) s -= L[j][p] * L[j][p];
        if (!(s > 0.0)) return false;
        L[j][j] = std::sqrt(s);
        for (int i = j + 1; i < 6; ++i) {
            double t = H[i][j];
            for (int p = 0; p < j; ++p) t -= L[i][p] * L[j][p];
            L[i][j] = t / L[j][j];
        }
    }
    double y[6], xi[6];
    for (int i = 0; i < 6; ++i) {
        double t = -sys[21 + i];
        for (int p = 0; p < i; ++p) t -= L[i][p] * y[p];
        y[i] = t / L[i][i];
    }
    for (int i = 5; i >= 0; --i) {
        double t = y[i];
        for (int p = i + 1; p < 6; ++p) t -= L[p][i] * xi[p];
        xi[i] = t / L[i][i];
    }
    const double w[3] = {xi[0], xi[1], xi[2]};
    const double th = std::sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    const double K[3][3] = {{0, -w[2], w[1]}, {w[2], 0, -w[0]}, {-w[1], w[0], 0}};
    double K2[3][3];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            K2[r][c] = 0.0;
            for (int p = 0; p < 3; ++p) K2[r][c] += K[r][p] * K[p][c];
        }
    const double a = th < 1e-12 ? 1.0 : std::sin(th) / th;
    const double b = th < 1e-12 ? 0.0 : (1.0 - std::cos(th)) / (th * th);
    double E[3][3];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) E[r][c] = (r == c ? 1.0 : 0.0) + a * K[r][c] + b * K2[r][c];
    double P[3][4];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 4; ++c) P[r][c] = (double)pose[4 * r + c];
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c) {
            double v = 0.0;
            for (int p = 0; p < 3; ++p) v += E[r][p] * P[p][c];
            pose[4 * r + c] = (float)v;
        }
        double v = xi[3 + r];
        for (int p = 0; p < 3; ++p) v += E[r][p] * P[p][3];
        pose[4 * r + 3] = (float)v;
    }
    double n2 = 0.0;
    for (int i = 0; i < 6; ++i) n2 += xi[i] * xi[i];
    *step_norm = std::sqrt(n2);
    return true;
}

}  // namespace tsdf
