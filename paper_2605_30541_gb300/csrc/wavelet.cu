// Band-passed Ricker source wavelet of the paper's production runs (Sec.
// "Source Wavelet", Tab. bands): a Ricker pulse of peak frequency f0 centred
// at t0 = 1/f0, filtered by a Butterworth band-pass at [f_lo, f_hi] forward
// and then backward in time (zero phase), divided by its l2 norm and
// multiplied by sqrt((f_hi - f_lo) / 24 Hz).
//
// The filter is designed on the host from the Butterworth definition:
// analog low-pass prototype poles exp(i pi (2k + N + 1) / (2N)), the
// low-pass to band-pass map around w0 = sqrt(w_lo w_hi) with bandwidth
// w_hi - w_lo (edges prewarped, w = 2 fs tan(pi f / fs)), then the bilinear
// map z = (2 fs + s) / (2 fs - s), grouped into second-order sections (each
// a conjugate pole pair with two zeros; gain on the first section). The half of
// the pairs with the lower frequencies takes the zeros at z = 1, two each, the
// other half those at z = -1 (an odd order's middle pair one of each), low ones
// first: high-passes, then low-passes.
// Forward-backward filtering follows the usual zero-phase recipe: the signal
// is extended at both ends by its odd reflection about the end samples
// (3 (2 S + 1) samples for S sections; the record must be longer than that),
// each pass starts every section in the steady state of a constant input
// equal to the first sample it sees (the first section passes no constant, so
// only it has a state to start from), and the extension is
// dropped at the end. The recursion runs in FP64 as a scan over chunks of
// the record (k_bandpass_ricker); the result is written in the requested
// precision.
//
// What keeps the rounding small. With a zero at 1 and one at -1 in every section
// the low ones answer a step, such as the start of a chunk, by 1 / theta each
// (theta = 2 pi f dt), which a wide band's other sections do not undo: the
// chunks' shares of a state then cancel to a small part of themselves. As
// high-passes and low-passes they answer by no more than they pass. And a
// section in transposed direct form, y = v + z1, z1' = z2 + b1 v - a1 y,
// z2' = b2 v - a2 y, whose poles lie within theta of z = 1, has z1 and z2 that
// nearly cancel: every rounding grows by 1 / theta^2. With e = z2 + t z1 in place
// of z2, t = 1 (a1 <= 0) or -1 (poles nearer z = -1), the same recursion is
//     y = v + z1,  z1' = k y + (p v + e),  e' = q v + t e - d y,
//     k = -(t + a1),  d = 1 + t a1 + a2,  p = t + b1,  q = 1 + t b1 + b2
// (p = -1, 1, 3 or -3; q = 0 or 4; k and d exact for |a1| > 1/2), whose
// roundings do not grow. Error of the two passes against 113-bit arithmetic with
// the same coefficients, of the peak (a host model; the first two columns in
// direct form with zeros at 1 and -1 in every section):
//   order, band, dt, samples      | serial  | scan    | scan, this form
//   4, 3-6 Hz, 1 ms, 8001         | 6e-14   | 2.9e-13 | 5e-15
//   4, 3-25 Hz, 1 ms, 8001        | 2e-14   | 1.6e-13 | 1e-15
//   4, 3-6 Hz, 0.1 ms, 40001      | 2.0e-12 | 2.2e-11 | 1.9e-14
//   4, 2-1500 Hz, 0.25 ms, 4777   | 8e-13   | 1.6e-11 | 1.5e-15
//   8, 2-1500 Hz, 0.25 ms, 4777   | 5e-10   | 3.5e-6  | 2e-15
//   16, 3-25 Hz, 1 ms, 8001       | 3.2e-10 | 4.2e-9  | 3e-15
//   16, 5-400 Hz, 1 ms, 4000      | 2.8e-5  | > 1     | 1.5e-15
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <complex>
#include <vector>

#include "sim_internal.h"

namespace gsim {
namespace {

using cd = std::complex<double>;

struct Sos {
    double b0, b1, b2, a1, a2;  // b0 (1 + b1 z^-1 + b2 z^-2) / (1 + a1 z^-1 + a2 z^-2)
};

// Digital Butterworth band-pass of order N (2N poles) at [f_lo, f_hi], fs = 1/dt.
std::vector<Sos> butter_bandpass(int N, double f_lo, double f_hi, double fs) {
    const double pi = 3.14159265358979323846;
    const double wl = 2.0 * fs * std::tan(pi * f_lo / fs), wh = 2.0 * fs * std::tan(pi * f_hi / fs);
    const double bw = wh - wl, w0 = std::sqrt(wl * wh);
    std::vector<cd> poles;  // analog band-pass poles
    for (int k = 0; k < N; k++) {
        const cd p = std::exp(cd(0.0, pi * (2.0 * k + N + 1) / (2.0 * N)));  // left half plane, |p| = 1
        const cd a = p * (bw / 2.0), r = std::sqrt(a * a - w0 * w0);
        poles.push_back(a + r);
        poles.push_back(a - r);
    }
    // analog gain bw^N (N zeros at s = 0); bilinear map
    cd gain(std::pow(bw, N), 0.0);
    std::vector<cd> zp;
    for (const cd &p : poles) {
        zp.push_back((2.0 * fs + p) / (2.0 * fs - p));
        gain /= (2.0 * fs - p);
    }
    gain *= std::pow(2.0 * fs, N);  // prod over the N finite zeros (s = 0) of (2 fs - 0)
    // zeros: N at z = 1 (from s = 0), N at z = -1 (from s = infinity);
    // sections: conjugate pairs of poles (upper half plane ones)
    std::vector<cd> up;
    for (const cd &z : zp)
        if (z.imag() > 0) up.push_back(z);
    std::sort(up.begin(), up.end(), [](const cd &a, const cd &b) { return std::arg(a) < std::arg(b); });
    const int n = (int)up.size(), half = n / 2;
    // within a kind the sharpest first (of the orders tried the smallest error)
    auto sharp = [](const cd &a, const cd &b) { return std::norm(a) > std::norm(b); };
    std::sort(up.begin(), up.begin() + half, sharp);
    std::sort(up.end() - half, up.end(), sharp);
    std::vector<Sos> s;
    for (int i = 0; i < n; i++) {
        Sos q{};
        q.b0 = i == 0 ? gain.real() : 1.0;
        q.b1 = i < half ? -2.0 : (i >= n - half ? 2.0 : 0.0);
        q.b2 = i < half || i >= n - half ? 1.0 : -1.0;
        q.a1 = -2.0 * up[i].real();
        q.a2 = std::norm(up[i]);
        s.push_back(q);
    }
    return s;
}

constexpr int kMaxSections = 16;

// ---------------------------------------------------------------- scan plan (host)
//
// The cascade of N sections with zero input maps its state (two values per
// section) linearly; P[l] is that map over 2^l chunks of C samples, block
// lower triangular (section i depends on sections j <= i only), block (i, j)
// at i (i + 1) / 2 + j, its four values row by row.
struct Block {
    double v[4];
};
using Tri = std::vector<Block>;  // N (N + 1) / 2 blocks

Tri tri_mul(const Tri &a, const Tri &b, int N) {
    Tri r(a.size());
    for (int i = 0; i < N; i++)
        for (int j = 0; j <= i; j++) {
            Block o{};
            for (int k = j; k <= i; k++) {
                const Block &x = a[i * (i + 1) / 2 + k], &y = b[k * (k + 1) / 2 + j];
                for (int p = 0; p < 2; p++)
                    for (int q = 0; q < 2; q++)
                        o.v[2 * p + q] = std::fma(x.v[2 * p + 1], y.v[2 + q], std::fma(x.v[2 * p], y.v[q], o.v[2 * p + q]));
            }
            r[i * (i + 1) / 2 + j] = o;
        }
    return r;
}

// NS: sections the plan holds. Four is the production order; the other
// orders share one instance that loops over its sections.
template <int NS>
struct Scan {
    static constexpr int MAXS = NS ? NS : kMaxSections;
    static constexpr int CTAS = NS ? 8 : 4;               // one cluster
    static constexpr int WPC = NS ? 4 : 1;                // warps per CTA
    static constexpr int WARPS = CTAS * WPC;
    static constexpr int T = 32 * WARPS;                  // threads = chunks
    static constexpr int LEV = NS ? 10 : 7;               // (an order-16 plan of 8 would pass 32 KB of parameters)
    static_assert(T == 1 << LEV, "levels of the scan");
    int nsec, C;
    double g;
    double k[MAXS], d[MAXS], p[MAXS], q[MAXS];  // a section's constants
    int flip[MAXS];                             // sign bit of its t in the high word
    double e0;                                  // first section's e at rest under a unit input
    double P[LEV][MAXS * (MAXS + 1) / 2 * 4];
};

// map of one sample: the recursion from v = 0; state values (z1, e)
template <int NS>
void plan_scan(Scan<NS> &F, int C) {
    const int N = F.nsec;
    F.C = C;
    Tri one((size_t)N * (N + 1) / 2), m = one;
    for (int k = 0; k < N; k++) m[k * (k + 1) / 2 + k].v[0] = m[k * (k + 1) / 2 + k].v[3] = 1.0;
    for (int j = 0; j < N; j++)
        for (int c = 0; c < 2; c++) {  // column of state value c of section j
            double v = 0.0;
            for (int i = j; i < N; i++) {
                const double z1 = i == j && c == 0 ? 1.0 : 0.0, e = i == j && c == 1 ? 1.0 : 0.0, y = v + z1;
                Block &b = one[i * (i + 1) / 2 + j];
                b.v[c] = std::fma(F.k[i], y, std::fma(F.p[i], v, e));
                b.v[2 + c] = std::fma(-F.d[i], y, std::fma(F.q[i], v, F.flip[i] ? -e : e));
                v = y;
            }
        }
    for (int c = C; c; c >>= 1) {
        if (c & 1) m = tri_mul(one, m, N);
        if (c > 1) one = tri_mul(one, one, N);
    }
    for (int l = 0; l < Scan<NS>::LEV; l++) {
        for (size_t b = 0; b < m.size(); b++)
            for (int q = 0; q < 4; q++) F.P[l][4 * b + q] = m[b].v[q];
        if (l + 1 < Scan<NS>::LEV) m = tri_mul(m, m, N);
    }
}

// ---------------------------------------------------------------- kernel
__device__ double ricker_at(double f0, double t) {
    const double pi = 3.14159265358979323846;
    const double a = (pi * f0 * t) * (pi * f0 * t);
    return (1.0 - 2.0 * a) * exp(-a);
}

// The recursion of 2 N states over n = nt + 2 pad samples is a chain of n
// dependent steps: one thread walked it in 22.4 ms for the production record
// (8001 samples, order 4). Here T = 1024 threads own C = ceil(n / T)
// consecutive samples each: every chunk runs from a zero state, the end
// states are combined by a scan with the chunk map (within each warp, then
// over the warps' totals, read through distributed shared memory), and every
// chunk runs again from its true start, in place. The backward pass is
// the same with the chunks in reverse order, on the thread's own samples, so
// a sample never leaves its thread until it is written out. What is left is
// the latency of the FP64 chains (about C samples four times over, 30 chunk
// maps, C exponentials), which the four warps of each SM overlap: with one
// warp per SM (256 chunks) the kernel took 167 us, with four 105 us (both in
// direct form). 8001 samples, launch and host plan included: 22.4 ms before,
// 128 us in direct form, 134 us in the present form.
template <int NS>
__global__ void __launch_bounds__(32 * Scan<NS>::WPC) k_bandpass_ricker(const __grid_constant__ Scan<NS> F, int nt,
                                                                            double dt, double f0, int pad, double scale,
                                                                            double *work, void *out, int fp64) {
    using S = Scan<NS>;
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ double chunk[];  // C samples of each thread of the CTA (work: in global memory instead)
    __shared__ double tot[2][S::WPC][2 * S::MAXS];  // the warps' totals of each pass
    __shared__ double part[S::WPC];
    const int N = NS ? NS : F.nsec;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, rank = (int)cl.block_rank(), C = F.C;
    const int warp = rank * S::WPC + wib, t = warp * 32 + lane;
    const long long n = nt + 2LL * pad, j0 = (long long)t * C;
    const int m = (int)max(0LL, min((long long)C, n - j0));  // the thread's samples
    double *const x = work ? work + t : chunk + threadIdx.x;
    const int ld = work ? S::T : 32 * S::WPC;

    // the extended record: odd reflections about the end samples
    for (int i = 0; i < m; i++) {
        const long long k = j0 + i - pad;
        double v;
        if (k < 0) v = 2.0 * ricker_at(f0, -1.0 / f0) - ricker_at(f0, -k * dt - 1.0 / f0);
        else if (k < nt) v = ricker_at(f0, k * dt - 1.0 / f0);
        else v = 2.0 * ricker_at(f0, (nt - 1) * dt - 1.0 / f0) - ricker_at(f0, (2LL * (nt - 1) - k) * dt - 1.0 / f0);
        x[(long long)i * ld] = v;
    }

    for (int dir = 1; dir >= -1; dir -= 2) {
        const bool first = m > 0 && (dir > 0 ? t == 0 : j0 + C >= n);
        double z1[S::MAXS], z2[S::MAXS], s1[S::MAXS], s2[S::MAXS];  // z2: the state value e
        auto start = [&]() {  // the first chunk: the steady state of its first sample
#pragma unroll
            for (int k = 0; k < S::MAXS; k++) {
                if (NS == 0 && k >= N) break;
                const double v = k == 0 && first ? F.g * x[(long long)(dir > 0 ? 0 : m - 1) * ld] : 0.0;
                z1[k] = -v;
                z2[k] = F.e0 * v;
            }
        };
        auto run = [&](bool store) {
            for (int i = 0; i < m; i++) {
                double *p = x + (long long)(dir > 0 ? i : m - 1 - i) * ld;
                double v = F.g * *p;
#pragma unroll
                for (int k = 0; k < S::MAXS; k++) {
                    if (NS == 0 && k >= N) break;
                    const double y = v + z1[k], e = z2[k];
                    z1[k] = fma(F.k[k], y, fma(F.p[k], v, e));
                    double u = __hiloint2double(__double2hiint(e) ^ F.flip[k], __double2loint(e));  // t e
                    if (F.q[k] != 0.0) u = fma(F.q[k], v, u);
                    z2[k] = fma(-F.d[k], y, u);
                    v = y;
                }
                if (store) *p = v;
            }
        };
        start();
        run(false);
        // apply the map over 2^l chunks: (s1, s2) mapped and added to (o1, o2)
        auto map_add = [&](int l, const double *q1, const double *q2, double *o1, double *o2) {
#pragma unroll
            for (int i = 0; i < S::MAXS; i++) {
                if (NS == 0 && i >= N) break;
#pragma unroll
                for (int j = 0; j <= i; j++) {
                    const double *b = F.P[l] + 4 * (i * (i + 1) / 2 + j);
                    o1[i] = fma(b[0], q1[j], fma(b[1], q2[j], o1[i]));
                    o2[i] = fma(b[2], q1[j], fma(b[3], q2[j], o2[i]));
                }
            }
        };
        auto each = [&](auto f) {
#pragma unroll
            for (int k = 0; k < S::MAXS; k++) {
                if (NS == 0 && k >= N) break;
                f(k);
            }
        };
        auto back = [&](double v, int d) {  // v of the lane d places earlier in this pass
            return dir > 0 ? __shfl_up_sync(0xffffffffu, v, d) : __shfl_down_sync(0xffffffffu, v, d);
        };
        // inclusive scan of the end states over the warp's chunks, in this pass's order
        const int place = dir > 0 ? lane : 31 - lane;
#pragma unroll
        for (int l = 0; l < 5; l++) {
            each([&](int k) { s1[k] = back(z1[k], 1 << l), s2[k] = back(z2[k], 1 << l); });
            if (place >= 1 << l) map_add(l, s1, s2, z1, z2);
        }
        // scan of the warps' totals: lane j takes the j-th warp's (the others repeat the last)
        double(*const mine)[2 * S::MAXS] = tot[dir > 0 ? 0 : 1];
        if (place == 31) each([&](int k) { mine[wib][2 * k] = z1[k], mine[wib][2 * k + 1] = z2[k]; });
        cl.sync();
        const int nth = dir > 0 ? warp : S::WARPS - 1 - warp;  // the warp's place in this pass
        double t1[S::MAXS], t2[S::MAXS];
        {
            const int j = min(lane, S::WARPS - 1), from_w = dir > 0 ? j : S::WARPS - 1 - j;
            const double *const from = cl.map_shared_rank(&mine[from_w % S::WPC][0], from_w / S::WPC);
            each([&](int k) { t1[k] = from[2 * k], t2[k] = from[2 * k + 1]; });
        }
#pragma unroll
        for (int l = 5; l < S::LEV; l++) {
            const int d = 1 << (l - 5);
            each([&](int k) {
                s1[k] = __shfl_up_sync(0xffffffffu, t1[k], d);
                s2[k] = __shfl_up_sync(0xffffffffu, t2[k], d);
            });
            if (lane >= d && lane < S::WARPS) map_add(l, s1, s2, t1, t2);
        }
        // the state entering the warp's first chunk, carried over the earlier chunks of the warp
        each([&](int k) {
            const double v1 = __shfl_sync(0xffffffffu, t1[k], max(nth - 1, 0));
            const double v2 = __shfl_sync(0xffffffffu, t2[k], max(nth - 1, 0));
            t1[k] = nth > 0 ? v1 : 0.0;
            t2[k] = nth > 0 ? v2 : 0.0;
        });
#pragma unroll
        for (int l = 0; l < 5; l++)
            if (place >> l & 1) {
                each([&](int k) { s1[k] = s2[k] = 0.0; });
                map_add(l, t1, t2, s1, s2);
                each([&](int k) { t1[k] = s1[k], t2[k] = s2[k]; });
            }
        // each chunk's true start: the state after the chunk before it
        each([&](int k) { s1[k] = back(z1[k], 1), s2[k] = back(z2[k], 1); });
        start();
        if (!first)
            each([&](int k) {
                z1[k] = t1[k] + (place > 0 ? s1[k] : 0.0);
                z2[k] = t2[k] + (place > 0 ? s2[k] : 0.0);
            });
        run(true);
    }

    // l2 norm over the record, in a fixed order
    double ss = 0.0;
    for (int i = 0; i < m; i++) {
        const long long k = j0 + i - pad;
        const double v = x[(long long)i * ld];
        if (k >= 0 && k < nt) ss += v * v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) part[wib] = ss;
    cl.sync();
    ss = 0.0;
    for (int r = 0; r < S::WARPS; r++) ss += *cl.map_shared_rank(&part[r % S::WPC], r / S::WPC);
    const double c = ss > 0.0 ? scale / sqrt(ss) : 0.0;
    // the CTA's samples [32 WPC C rank, 32 WPC C (rank + 1)), written in order
    double *const x0 = x - threadIdx.x;
    for (int i = threadIdx.x; i < 32 * S::WPC * C; i += 32 * S::WPC) {
        const long long k = 32LL * S::WPC * C * rank + i - pad;
        const int h = i / C;
        if (k < 0 || k >= nt) continue;
        const double v = c * x0[(long long)(i - h * C) * ld + h];
        if (fp64) static_cast<double *>(out)[k] = v;
        else static_cast<float *>(out)[k] = (float)v;
    }
    cl.sync();  // no CTA leaves while another reads its shared memory
}

// Most chunk bytes kept in shared memory; longer records (over 200 000
// samples at order 4) keep their samples in a global workspace.
constexpr size_t kChunkSmem = 200 * 1024;

template <int NS>
cudaError_t launch_bandpass(const std::vector<Sos> &s, int nt, double dt, double f0, int pad, double scale, void *out,
                            int fp64, double **work, cudaStream_t st) {
    using S = Scan<NS>;
    S F{};
    F.nsec = (int)s.size();
    F.g = s[0].b0;
    for (int k = 0; k < F.nsec; k++) {
        const double t = s[k].a1 <= 0.0 ? 1.0 : -1.0;
        F.flip[k] = t > 0.0 ? 0 : INT_MIN;
        F.k[k] = -(t + s[k].a1);
        F.d[k] = (1.0 + t * s[k].a1) + s[k].a2;
        F.p[k] = t + s[k].b1;
        F.q[k] = 1.0 + t * s[k].b1 + s[k].b2;
        if (k == 0) F.e0 = s[k].b2 - t;
    }
    const long long n = nt + 2LL * pad;
    plan_scan<NS>(F, (int)((n + S::T - 1) / S::T));
    size_t smem = (size_t)F.C * 32 * S::WPC * sizeof(double);
    cudaError_t e = cudaSuccess;
    if (smem > kChunkSmem) {
        smem = 0;
        e = cudaMalloc(work, (size_t)F.C * S::T * sizeof(double));
    } else {
        e = cudaFuncSetAttribute(k_bandpass_ricker<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChunkSmem);
    }
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S::CTAS);
    cfg.blockDim = dim3(32 * S::WPC);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S::CTAS;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_bandpass_ricker<NS>, F, nt, dt, f0, pad, scale, *work, out, fp64);
}

}  // namespace
}  // namespace gsim

extern "C" sim_status sim_wavelet_bandpass(int nt, double dt, double f0, double f_lo, double f_hi, int order,
                                           int precision, void *out, void *stream) {
    using namespace gsim;
    if (nt < 2 || !(dt > 0) || !(f0 > 0) || !out || order < 1 || order > kMaxSections ||
        !(f_lo > 0) || !(f_hi > f_lo) || !(f_hi < 0.5 / dt) || (precision != SIM_FP32 && precision != SIM_FP64)) {
        set_thread_error("sim_wavelet_bandpass: need nt >= 2, dt > 0, f0 > 0, 0 < f_lo < f_hi < 1/(2 dt), "
                         "1 <= order <= 16, a known precision and an output array");
        return SIM_ERR_ARG;
    }
    const std::vector<Sos> s = butter_bandpass(order, f_lo, f_hi, 1.0 / dt);
    if ((int)s.size() != order) {
        set_thread_error("sim_wavelet_bandpass: the band-pass has real poles (band too wide for this design)");
        return SIM_ERR_ARG;
    }
    const int pad = 3 * (2 * (int)s.size() + 1);
    if (nt <= pad) {
        set_thread_error("sim_wavelet_bandpass: the record must be longer than the reflection at its ends");
        return SIM_ERR_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaPointerAttributes attr{};
    const bool dev_out = cudaPointerGetAttributes(&attr, out) == cudaSuccess && attr.type == cudaMemoryTypeDevice;
    cudaGetLastError();
    const size_t esz = precision == SIM_FP64 ? 8 : 4;
    double *work = nullptr;
    void *dout = out;
    cudaError_t e = cudaSuccess;
    if (!dev_out) e = cudaMalloc(&dout, esz * nt);
    if (e == cudaSuccess) {
        const double scale = std::sqrt((f_hi - f_lo) / 24.0);
        const int fp64 = precision == SIM_FP64;
        e = order == 4 ? launch_bandpass<4>(s, nt, dt, f0, pad, scale, dout, fp64, &work, st)
                       : launch_bandpass<0>(s, nt, dt, f0, pad, scale, dout, fp64, &work, st);
    }
    if (e == cudaSuccess && !dev_out) e = cudaMemcpyAsync(out, dout, esz * nt, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (work) cudaFree(work);
    if (!dev_out && dout) cudaFree(dout);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_thread_error(cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? SIM_ERR_OOM : SIM_ERR_CUDA;
    }
    return SIM_OK;
}
