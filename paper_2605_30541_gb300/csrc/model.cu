// Velocity-model builder warps (App. "Model builder modules"): the
// pull-sample steps of Squish (Alg. squish), Fault (Alg. fault) and a
// simplified Deposit (Alg. deposit) on (nz, ny, nx) row-major device grids,
// ny = 1 for a 2D slice. One thread per output voxel, x fastest, so reads of
// the source grid by neighbouring threads fall in the same lines.
//
// Interpolation (the paper says "sinc"): an 8-tap Lanczos-windowed sinc per
// axis, sinc(x) sinc(x/4) on |x| < 4, weights normalised to sum 1, taps
// beyond the grid taking the edge value; labels by nearest neighbour (round
// half to even). A voxel whose pulled depth lies outside [0, nz) (depths
// down to -1e-6 counting as 0) takes the fill velocity and label. Source
// positions are computed in FP64, weights and sums in FP32.
#include <algorithm>
#include <cmath>

#include "sim_internal.h"

namespace gsim {
namespace {

constexpr int kTaps = 8;
constexpr int kMaxBeds = 128;

// Normalised weights of the 8 taps at x_k = fr + 3 - k, fr in [0, 1], of the
// windowed sinc sin(pi x) sin(pi x / 4) / x^2 (up to a constant). Every
// |sin(pi x_k)| is sin(pi fr), which cancels in the normalisation, and the
// angles pi x_k / 4 lie 45 degrees apart: with a = pi fr / 4 and b = pi / 4 - a
// their sines are sin b, cos a, cos b, sin a, -sin b, -cos a, -cos b, -sin a
// for k = 0 .. 7. Two sine-cosine pairs and eight reciprocals in place of
// sixteen sines and sixteen quotients. A hair above a sample, where 1 / fr^2
// would overflow (fr below 5.4e-20) and every other weight is below 2^-40, the
// sample itself is taken.
__device__ __forceinline__ void tap_weights(float fr, float *w) {
    if (fr <= 0x1p-40f || fr >= 1.f) {  // on a sample (fr rounds to 1 just below the next one); not for NaN
#pragma unroll
        for (int k = 0; k < kTaps; k++) w[k] = k == (fr < 1.f ? 3 : 4) ? 1.f : 0.f;
        return;
    }
    float sa, ca, sb, cb;
    sincospif(0.25f * fr, &sa, &ca);
    sincospif(0.25f * (1.f - fr), &sb, &cb);
    const float v[kTaps] = {-sb, ca, -cb, sa, sb, -ca, cb, -sa};
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < kTaps; k++) {
        const float r = __frcp_rn(fr + (float)(3 - k));
        w[k] = v[k] * (r * r);
        sum += w[k];
    }
    const float inv = 1.f / sum;
#pragma unroll
    for (int k = 0; k < kTaps; k++) w[k] *= inv;
}
// First tap index and weights of the 8 taps around s. The index is held to
// [-far, far] - 3 so that the sums formed with it do not overflow for positions
// of any size; one that is no number reads some cell of the grid.
__device__ __forceinline__ int taps(double s, int far, float *w) {
    const double f = floor(s);
    tap_weights((float)(s - f), w);
    return max(-far, min(far, (int)f)) - 3;
}
constexpr int kFarPoint = 0x7fffffff - kTaps;  // positions
constexpr int kFarShift = 1 << 30;             // displacements and offsets of depths below 2^30

__device__ __forceinline__ int clampi(int i, int n) { return i < 0 ? 0 : (i >= n ? n - 1 : i); }

__device__ __forceinline__ bool filled(double sz, int nz) { return sz < -1e-6 || sz >= (double)nz; }

__device__ __forceinline__ int nearest(double s, int n) { return clampi((int)rint(s), n); }

// ---------------------------------------------------------------- Squish
// A column's displacement is one number, so its 8 weights are the same at
// every depth: a thread computes them once and walks down kSquishRows rows
// of its column with a sliding window of the 8 taps (each input value read
// once per chunk). Threads: x fastest (coalesced rows), then y, then chunks.
constexpr int kSquishRows = 32;

__global__ void k_squish(int nz, int ny, int nx, const float *__restrict__ v, const int *__restrict__ lab,
                         const float *__restrict__ dz, float fill_v, int fill_label, float *__restrict__ vo,
                         int *__restrict__ lo) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= nx) return;
    const int z0 = blockIdx.z * kSquishRows, z1 = min(nz, z0 + kSquishRows);
    const long long col = (long long)y * nx + x, plane = (long long)ny * nx;
    const float d = dz[col];
    float w[kTaps];
    const int s0 = taps((double)d, kFarShift, w);  // taps of row z: z + s0 .. z + s0 + 7
    // the pulled depth z + d = (z + di) + fr with di = floor(d), fr in [0, 1)
    // exact in FP32, so the fill test and the nearest row are integer logic
    const int di = s0 + 3;
    const float fr = d - floorf(d);
    const int up = fr > 0.5f ? 1 : (fr < 0.5f ? 0 : -1);  // -1: a tie, rounded to even
    float win[kTaps];
#pragma unroll
    for (int k = 0; k < kTaps - 1; k++) win[k + 1] = v[clampi(z0 + s0 + k, nz) * plane + col];
#pragma unroll 4
    for (int z = z0; z < z1; z++) {
#pragma unroll
        for (int k = 0; k < kTaps - 1; k++) win[k] = win[k + 1];
        win[kTaps - 1] = v[clampi(z + s0 + kTaps - 1, nz) * plane + col];
        const long long o = z * plane + col;
        const int zk = z + di;
        // outside [0, nz) (depths down to -1e-6 count as 0)
        if (zk >= nz || zk <= -2 || (zk == -1 && fr < 1.f - 1e-6f)) {
            vo[o] = fill_v;
            if (lo) lo[o] = fill_label;
            continue;
        }
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < kTaps; k++) acc += w[k] * win[k];
        vo[o] = acc;
        if (lo) lo[o] = lab[clampi(zk + (up >= 0 ? up : (zk & 1)), nz) * plane + col];
    }
}

// ---------------------------------------------------------------- Fault
//
// FP64 issue bounds this warp: an SM issues two FP64 lanes per clock, and the
// positions need FP64. So (1) a warp looks at up to 32 segments of 32 voxels
// at once, one per lane, and copies those that lie wholly outside the die-off
// region (a segment's centre, half its length from its voxels, tells; the
// region is a band of a few tens of cells round the fault); (2) the moved
// voxels use the rotation of their offset from the axis by the small slip
// angle (no angle is turned back into a position), and short series for the
// functions on the ranges they meet here. 619 x 64 x 1000 voxels with labels,
// a band of 50 cells either side: 6.24 ms with every voxel in full, 2.82 ms now.
constexpr int kAtan = 16;  // base angles of the arc tangent: j pi / (4 kAtan)
struct FaultK {
    double ct[3];      // cylinder centre (z, y, x)
    double ed[3], es[3];
    double R, th0, shift, dir, d_die, d_perp, th_die;
    double i_die, i_perp, i_th;                   // reciprocals
    double base_c[kAtan + 1], base_s[kAtan + 1];  // cosine and sine of the base angles
};

// cos(pi x / 2) for 0 <= x <= 1: 1 - 2 sin^2(pi x / 4), the sine by its Taylor
// series (next term below 6e-17 at x = 1)
__device__ __forceinline__ double cos_half_pi(double x) {
    const double a = 0.78539816339744830962 * x, y = a * a;
    double p = -1.0 / 1307674368000.0;           // -1 / 15!
    p = fma(p, y, 1.0 / 6227020800.0);           // 1 / 13!
    p = fma(p, y, -1.0 / 39916800.0);            // -1 / 11!
    p = fma(p, y, 1.0 / 362880.0);               // 1 / 9!
    p = fma(p, y, -1.0 / 5040.0);                // -1 / 7!
    p = fma(p, y, 1.0 / 120.0);
    p = fma(p, y, -1.0 / 6.0);
    const double s = fma(a * y, p, a);
    return fma(-2.0 * s, s, 1.0);
}

// sin d and cos d - 1 for |d| <= 1/4 by their Taylor series (next terms below 1e-19)
__device__ __forceinline__ void small_rotation(double d, double *sn, double *cs1) {
    const double y = d * d;
    double p = 1.0 / 6227020800.0;
    p = fma(p, y, -1.0 / 39916800.0);
    p = fma(p, y, 1.0 / 362880.0);
    p = fma(p, y, -1.0 / 5040.0);
    p = fma(p, y, 1.0 / 120.0);
    p = fma(p, y, -1.0 / 6.0);
    *sn = fma(d * y, p, d);
    double q = -1.0 / 87178291200.0;             // -1 / 14!
    q = fma(q, y, 1.0 / 479001600.0);            // 1 / 12!
    q = fma(q, y, -1.0 / 3628800.0);             // -1 / 10!
    q = fma(q, y, 1.0 / 40320.0);
    q = fma(q, y, -1.0 / 720.0);
    q = fma(q, y, 1.0 / 24.0);
    q = fma(q, y, -0.5);
    *cs1 = q * y;
}

// The angle of (u, w), in (-pi, pi]. The point (m, n), m >= n >= 0, of the
// first half quadrant is turned back by the base angle nearest its FP32
// angle; what is left is at most pi / (8 kAtan) plus FP32 rounding, where the
// series of the arc tangent needs six terms (next term below 1e-19). The
// quotient is the FP32 reciprocal after two Newton steps and a residual step.
__device__ __forceinline__ double angle_of(const FaultK &F, double w, double u) {
    const double aw = fabs(w), au = fabs(u);
    const double m = fmax(aw, au), n = fmin(aw, au);
    if (!(m > 0.0)) return 0.0;
    const float mf = (float)m;
    if (!(mf > 1e-30f && mf < 1e30f)) return atan2(w, u);
    const int j = (int)rintf(atanf((float)n / mf) * (kAtan * 1.2732395447f));
    const double c = F.base_c[j], s = F.base_s[j];
    const double num = fma(n, c, -(m * s)), den = fma(m, c, n * s);
    double r = (double)__frcp_rn((float)den);
    r = fma(r, fma(-den, r, 1.0), r);
    r = fma(r, fma(-den, r, 1.0), r);
    double q = num * r;
    q = fma(r, fma(-den, q, num), q);
    const double y = q * q;
    double p = -1.0 / 11.0;
    p = fma(p, y, 1.0 / 9.0);
    p = fma(p, y, -1.0 / 7.0);
    p = fma(p, y, 0.2);
    p = fma(p, y, -1.0 / 3.0);
    double t = fma(0.78539816339744830962 / kAtan, (double)j, fma(q * y, p, q));
    if (aw > au) t = 1.57079632679489661923 - t;
    if (u < 0.0) t = 3.14159265358979323846 - t;
    return w < 0.0 ? -t : t;
}

__device__ __forceinline__ void fault_voxel(int nz, int ny, int nx, const float *__restrict__ v,
                                            const int *__restrict__ lab, const FaultK &F, float fill_v, int fill_label,
                                            float *__restrict__ vo, int *__restrict__ lo, int z, int y, int x) {
    const long long i = ((long long)z * ny + y) * nx + x;
    // cylindrical coordinates about the axis through ct along e_s
    const double wz = z - F.ct[0], wy = y - F.ct[1], wx = x - F.ct[2];
    const double u = wy * F.ed[1] + wx * F.ed[2];
    const double as = wy * F.es[1] + wx * F.es[2];
    const double r = sqrt(fma(u, u, wz * wz));
    const double rr = fabs(r - F.R) * F.i_die, rs = fabs(as) * F.i_perp;
    double rt = 2.0;
    if (rr < 1.0 && rs < 1.0) rt = fabs(angle_of(F, wz, u) - F.th0) * F.i_th;
    if (!(rr < 1.0 && rs < 1.0 && rt < 1.0)) {  // outside the die-off region: the voxel does not move
        vo[i] = v[i];
        if (lo) lo[i] = lab[i];
        return;
    }
    const double taper = cos_half_pi(rr) * cos_half_pi(rt) * cos_half_pi(rs);
    const double chi = r >= F.R ? 1.0 : -1.0;
    const double d = -chi * F.dir * taper * F.shift;
    double sn, c1;
    if (fabs(F.shift) <= 0.25) {
        small_rotation(d, &sn, &c1);
    } else {
        double cs;
        sincos(d, &sn, &cs);
        c1 = cs - 1.0;
    }
    // pulled from 2 p - p_rotated = p - (the offset's change under the rotation)
    const double du = fma(u, c1, -(wz * sn));
    const double sz = z - fma(wz, c1, u * sn), sy = y - du * F.ed[1], sx = x - du * F.ed[2];
    if (filled(sz, nz)) {
        vo[i] = fill_v;
        if (lo) lo[i] = fill_label;
        return;
    }
    float wzt[kTaps], wxt[kTaps];
    const int iz0 = taps(sz, kFarPoint, wzt), ix0 = taps(sx, kFarPoint, wxt);
    int xs[kTaps];
#pragma unroll
    for (int c = 0; c < kTaps; c++) xs[c] = clampi(ix0 + c, nx);
    float acc = 0.f;
    if (ny == 1) {
#pragma unroll
        for (int a = 0; a < kTaps; a++) {
            const float *row = v + (long long)clampi(iz0 + a, nz) * nx;
            float ra = 0.f;
#pragma unroll
            for (int c = 0; c < kTaps; c++) ra += wxt[c] * row[xs[c]];
            acc += wzt[a] * ra;
        }
    } else {
        float wyt[kTaps];
        const int iy0 = taps(sy, kFarPoint, wyt);
        for (int a = 0; a < kTaps; a++) {
            const long long pz = (long long)clampi(iz0 + a, nz) * ny;
            float pa = 0.f;
#pragma unroll
            for (int b = 0; b < kTaps; b++) {
                const float *row = v + (pz + clampi(iy0 + b, ny)) * nx;
                float rb = 0.f;
#pragma unroll
                for (int c = 0; c < kTaps; c++) rb += wxt[c] * row[xs[c]];
                pa += wyt[b] * rb;
            }
            acc += wzt[a] * pa;
        }
    }
    vo[i] = acc;
    if (lo) lo[i] = lab[((long long)nearest(sz, nz) * ny + nearest(sy, ny)) * nx + nearest(sx, nx)];
}

// A warp takes QX segments of 32 voxels of ROWS rows (z) of one y: lane l
// judges segment (row l / QX, place l % QX). 8 x 4 where the grid has warps
// enough that the few that meet the region spread over the SMs; a warp walks
// its near segments one after another, so smaller grids take 1 x 4 or 1 x 1
// (with 8 x 4 a 472 x 23 x 107 volume took 0.43 ms for three warps, against
// 0.33 with a thread per voxel in full and 0.24 with 1 x 1).
constexpr int kFaultWarps = 4;

template <int ROWS, int QX>
__global__ void __launch_bounds__(kFaultWarps * 32) k_fault(int nz, int ny, int nx, const float *__restrict__ v,
                                                            const int *__restrict__ lab, const __grid_constant__ FaultK F,
                                                            float fill_v, int fill_label, float *__restrict__ vo,
                                                            int *__restrict__ lo) {
    const int lane = threadIdx.x & 31;
    const int x0 = (blockIdx.x * kFaultWarps + (threadIdx.x >> 5)) * 32 * QX, y = blockIdx.y, z0 = blockIdx.z * ROWS;
    if (x0 >= nx) return;
    bool near;
    {
        const int z = z0 + lane / QX;
        const double wz = z - F.ct[0], wy = y - F.ct[1], wx = x0 + 32 * (lane % QX) + 15.5 - F.ct[2];
        const double u = wy * F.ed[1] + wx * F.ed[2], as = wy * F.es[1] + wx * F.es[2];
        // 15.5 cells to the furthest voxel; the rest covers the rounding of r and as
        const double slack = 16.5 + 1e-12 * (F.R + fabs(as));
        const bool away = fabs(sqrt(fma(u, u, wz * wz)) - F.R) >= F.d_die + slack || fabs(as) >= F.d_perp + slack;
        near = lane < ROWS * QX && z < nz && !away;
    }
    unsigned mask = __ballot_sync(0xffffffffu, near);
    const int rows = min(ROWS, nz - z0);
    const long long pl = (long long)ny * nx, i0 = ((long long)z0 * ny + y) * nx + x0;
    if (QX == 4 && mask == 0 && nx % 4 == 0 &&
        ((reinterpret_cast<size_t>(v) | reinterpret_cast<size_t>(vo) | reinterpret_cast<size_t>(lab) |
          reinterpret_cast<size_t>(lo)) & 15) == 0) {
        if (x0 + 4 * lane >= nx) return;
        const long long i = i0 + 4 * lane;
        float4 a[ROWS];
        int4 b[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; r++)
            if (r < rows) {
                a[r] = *reinterpret_cast<const float4 *>(v + i + r * pl);
                if (lo) b[r] = *reinterpret_cast<const int4 *>(lab + i + r * pl);
            }
#pragma unroll
        for (int r = 0; r < ROWS; r++)
            if (r < rows) {
                *reinterpret_cast<float4 *>(vo + i + r * pl) = a[r];
                if (lo) *reinterpret_cast<int4 *>(lo + i + r * pl) = b[r];
            }
        return;
    }
    for (int k = 0; k < QX; k++) {  // the segments outside the region
        if (x0 + 32 * k + lane >= nx) break;
        const long long i = i0 + 32 * k + lane;
        float a[ROWS];
        int b[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; r++)
            if (r < rows && !(mask >> (QX * r + k) & 1u)) {
                a[r] = v[i + r * pl];
                if (lo) b[r] = lab[i + r * pl];
            }
#pragma unroll
        for (int r = 0; r < ROWS; r++)
            if (r < rows && !(mask >> (QX * r + k) & 1u)) {
                vo[i + r * pl] = a[r];
                if (lo) lo[i + r * pl] = b[r];
            }
    }
    for (; mask; mask &= mask - 1) {
        const int q = __ffs(mask) - 1, x = x0 + 32 * (q % QX) + lane;
        if (x < nx) fault_voxel(nz, ny, nx, v, lab, F, fill_v, fill_label, vo, lo, z0 + q / QX, y, x);
    }
}

// ---------------------------------------------------------------- Deposit
struct DepositK {
    int t, nbeds, nzt, label0;
    float beta, a_eta, f_top, f_base, vbar;
    float vbed[kMaxBeds];
    int off[kMaxBeds];
};

__global__ void k_deposit(int nz, int ny, int nx, const float *__restrict__ v, const int *__restrict__ lab,
                          const DepositK P, const float *__restrict__ bounds, const float *__restrict__ eta,
                          float *__restrict__ vo, int *__restrict__ lo) {
    const long long plane = (long long)ny * nx;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= nx) return;
    const long long col = (long long)y * nx + x, i = z * plane + col;
    {
        if (z >= P.t) {  // the model below, pushed down by the slab
            vo[i] = v[i - (long long)P.t * plane];
            if (lo) lo[i] = lab[i - (long long)P.t * plane];
            return;
        }
        int ell = 0;
        float start = 0.f;
        for (int b = 0; b < P.nbeds - 1; b++) {  // beds whose boundary lies above z
            const float h = bounds[b * plane + col];
            if (h < (float)z) {
                ell++;
                start = fmaxf(start, h);
            }
        }
        const float top = P.f_top > 0.f ? fminf((float)z / (P.f_top * P.t), 1.f) : 1.f;
        const float base = P.f_base > 0.f ? fminf((float)(P.t - z) / (P.f_base * P.t), 1.f) : 1.f;
        const float tau = top * base;
        const int zt = clampi(z - (int)floorf(start) + P.off[ell], P.nzt);
        const float tex = eta ? eta[zt * plane + col] : 0.f;
        vo[i] = (P.vbar + P.beta * z) + tau * ((P.vbed[ell] - P.vbar) + P.a_eta * tex);
        if (lo) lo[i] = P.label0 + ell;
    }
}

sim_status finish(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return SIM_OK;
    cudaGetLastError();
    set_thread_error((std::string(what) + ": " + cudaGetErrorString(e)).c_str());
    return SIM_ERR_CUDA;
}

bool bad_grid(int nz, int ny, int nx, const float *v, const float *vo, const int *lab, const int *lo) {
    return nz < 1 || ny < 1 || nx < 1 || !v || !vo || v == vo || (!lab) != (!lo) || (lab && lab == lo);
}

}  // namespace
}  // namespace gsim

using namespace gsim;

extern "C" sim_status sim_model_squish(int nz, int ny, int nx, const float *v_in, const int *lab_in, const float *dz,
                                       float fill_v, int fill_label, float *v_out, int *lab_out, void *stream) {
    if (bad_grid(nz, ny, nx, v_in, v_out, lab_in, lab_out) || !dz) {
        set_thread_error("sim_model_squish: need positive sizes, distinct input and output grids, a displacement "
                         "field, and labels on both sides or neither");
        return SIM_ERR_ARG;
    }
    if (ny > 65535 || (nz + kSquishRows - 1) / kSquishRows > 65535) {
        set_thread_error("sim_model_squish: ny and nz / 32 must stay below 65536");
        return SIM_ERR_ARG;
    }
    const dim3 grid((nx + 127) / 128, ny, (nz + kSquishRows - 1) / kSquishRows);
    k_squish<<<grid, 128, 0, static_cast<cudaStream_t>(stream)>>>(nz, ny, nx, v_in, lab_in, dz, fill_v, fill_label,
                                                                  v_out, lab_out);
    return finish(cudaGetLastError(), "sim_model_squish");
}

extern "C" sim_status sim_model_fault(int nz, int ny, int nx, const float *v_in, const int *lab_in,
                                      const sim_fault *f, float fill_v, int fill_label, float *v_out, int *lab_out,
                                      void *stream) {
    if (bad_grid(nz, ny, nx, v_in, v_out, lab_in, lab_out) || !f || !(f->radius > 0) || !(f->d_die > 0) ||
        !(f->d_perp > 0) || !(f->theta_die > 0) || (f->direction != 1 && f->direction != -1)) {
        set_thread_error("sim_model_fault: need positive sizes, distinct grids, labels on both sides or neither, "
                         "radius and die-off extents > 0 and direction +1 or -1");
        return SIM_ERR_ARG;
    }
    FaultK K{};
    K.ed[0] = 0.0;
    K.ed[1] = std::cos(f->azimuth);
    K.ed[2] = std::sin(f->azimuth);
    K.es[0] = 0.0;
    K.es[1] = -std::sin(f->azimuth);
    K.es[2] = std::cos(f->azimuth);
    const double dz = f->radius * std::sin(f->dip), daz = f->radius * std::cos(f->dip);
    K.ct[0] = f->cz - dz;
    K.ct[1] = f->cy - daz * K.ed[1];
    K.ct[2] = f->cx - daz * K.ed[2];
    K.th0 = std::atan2(dz, daz);
    K.R = f->radius;
    K.shift = f->slip / f->radius;
    K.dir = f->direction;
    K.d_die = f->d_die;
    K.d_perp = f->d_perp;
    K.th_die = f->theta_die;
    K.i_die = 1.0 / f->d_die;
    K.i_perp = 1.0 / f->d_perp;
    K.i_th = 1.0 / f->theta_die;
    for (int j = 0; j <= kAtan; j++) {
        K.base_c[j] = std::cos(j * (0.78539816339744830962 / kAtan));
        K.base_s[j] = std::sin(j * (0.78539816339744830962 / kAtan));
    }
    if (ny > 65535 || nz > 65535) {
        set_thread_error("sim_model_fault: ny and nz must stay below 65536");
        return SIM_ERR_ARG;
    }
    // the most segments per warp that leave 16384 warps (152 SMs x 16 warps x 7:
    // about a seventh of the tiles meet the region)
    const long long segs = (long long)((nx + 31) / 32) * ny * nz;
    auto go = [&](auto kernel, int rows, int qx) {
        const dim3 grid((nx + 32 * qx * kFaultWarps - 1) / (32 * qx * kFaultWarps), ny, (nz + rows - 1) / rows);
        kernel<<<grid, kFaultWarps * 32, 0, static_cast<cudaStream_t>(stream)>>>(nz, ny, nx, v_in, lab_in, K, fill_v,
                                                                                 fill_label, v_out, lab_out);
    };
    if (segs >= 32 * 16384LL) go(k_fault<8, 4>, 8, 4);
    else if (segs >= 4 * 16384LL) go(k_fault<1, 4>, 1, 4);
    else go(k_fault<1, 1>, 1, 1);
    return finish(cudaGetLastError(), "sim_model_fault");
}

extern "C" sim_status sim_model_deposit(int nz, int ny, int nx, const float *v_in, const int *lab_in,
                                        const sim_deposit *p, const float *bounds, const float *vbed,
                                        const int *offsets, const float *eta, float *v_out, int *lab_out,
                                        void *stream) {
    if (bad_grid(nz, ny, nx, v_in, v_out, lab_in, lab_out) || !p || p->t < 1 || p->t > nz || p->nbeds < 1 ||
        p->nbeds > kMaxBeds || (p->nbeds > 1 && !bounds) || !vbed || !offsets || (eta && p->nzt < 1) ||
        p->f_top < 0 || p->f_base < 0) {
        set_thread_error("sim_model_deposit: need positive sizes, distinct grids, labels on both sides or neither, "
                         "1 <= t <= nz, 1 <= nbeds <= 128, bed boundaries when nbeds > 1, bed velocities and "
                         "offsets, and non-negative taper fractions");
        return SIM_ERR_ARG;
    }
    DepositK K{};
    K.t = p->t;
    K.nbeds = p->nbeds;
    K.nzt = eta ? p->nzt : 1;
    K.label0 = p->label0;
    K.beta = p->beta;
    K.a_eta = eta ? p->a_eta : 0.f;
    K.f_top = p->f_top;
    K.f_base = p->f_base;
    double sum = 0.0;
    for (int b = 0; b < p->nbeds; b++) {
        K.vbed[b] = vbed[b];
        K.off[b] = std::max(-kFarShift, std::min(kFarShift, offsets[b]));  // z - start + offset does not overflow
        sum += vbed[b];
    }
    K.vbar = (float)(sum / p->nbeds);
    if (ny > 65535 || nz > 65535) {
        set_thread_error("sim_model_deposit: ny and nz must stay below 65536");
        return SIM_ERR_ARG;
    }
    const dim3 grid((nx + 127) / 128, ny, nz);
    k_deposit<<<grid, 128, 0, static_cast<cudaStream_t>(stream)>>>(nz, ny, nx, v_in, lab_in, K, bounds, eta, v_out,
                                                                   lab_out);
    return finish(cudaGetLastError(), "sim_model_deposit");
}
