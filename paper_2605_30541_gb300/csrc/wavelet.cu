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
// a conjugate pole pair with two zeros; gain on the first section).
// Forward-backward filtering follows the usual zero-phase recipe: the signal
// is extended at both ends by its odd reflection about the end samples
// (3 (2 S + 1) samples for S sections; the record must be longer than that),
// each pass starts every section in the steady state of a constant input
// equal to the first sample it sees (a band-pass section passes no constant,
// so only the first section has a state to start from), and the extension is
// dropped at the end. The recursion runs in FP64 as a scan over chunks of
// the record (k_bandpass_ricker); the result is written in the requested
// precision.
//
// A section's state. In transposed direct form, y = v + z1, z1' = z2 - a1 y,
// z2' = -v - a2 y, the poles lie within theta = 2 pi f dt of z = 1, z1 and z2
// nearly cancel, and every rounding grows by 1 / theta^2. With the sum e = z1 +
// z2, which is small, in place of z2 the same recursion is
//     y = v + z1,  z1' = k y + (e + v),  e' = e - d y,  k = -(1 + a1),  d = 1 + a1 + a2,
// whose roundings do not grow (k and d are exact for a1 < -1/2). Sections with
// a1 > 0, whose poles lie nearer z = -1, take e = z2 - z1 likewise: t is the
// sign, 1 or -1, in z1' = k y + (e + t v), e' = t e - d y, k = -(t + a1),
// d = 1 + t a1 + a2.
#include <cooperative_groups.h>

#include <climits>
#include <cmath>
#include <complex>
#include <vector>

#include "sim_internal.h"

namespace gsim {
namespace {

using cd = std::complex<double>;

struct Sos {
    double b0, b1, b2, a1, a2;  // a0 = 1
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
    // zeros: N at z = 1 (from s = 0), N at z = -1 (from s = infinity)
    // sections: conjugate pairs of poles (upper half plane ones), zeros (1, -1) each
    std::vector<cd> up;
    for (const cd &z : zp)
        if (z.imag() > 0) up.push_back(z);
    std::vector<Sos> s;
    for (size_t i = 0; i < up.size(); i++) {
        Sos q{};
        q.b0 = 1.0;
        q.b1 = 0.0;  // (z - 1)(z + 1) = z^2 - 1
        q.b2 = -1.0;
        q.a1 = -2.0 * up[i].real();
        q.a2 = std::norm(up[i]);
        s.push_back(q);
    }
    if (s.empty()) return s;
    const double g = gain.real();
    s[0].b0 *= g;
    s[0].b1 *= g;
    s[0].b2 *= g;
    return s;
}

constexpr int kMaxSections = 16;

// ---------------------------------------------------------------- scan plan (host)
//
// The cascade of N sections with zero input maps its state (two values per
// section) linearly; P[l] is that map over 2^l chunks of C samples, block
// lower triangular (section i depends on sections j <= i only), block (i, j)
// at i (i + 1) / 2 + j, its four values row by row.
//
// The powers are formed in pairs of doubles (an unevaluated sum hi + lo,
// Dekker's and Knuth's error-free sum and product) and rounded once: in FP64
// alone their own errors are several times those of the recursion. Error of the
// two passes against 113-bit arithmetic with the same coefficients, of the peak
// (a host model; direct form is the transposed one above):
//   order, band, dt, samples       | serial, direct | scan, direct | scan, this
//   4, 3-6 Hz, 1 ms, 8001          | 6e-14          | 2.9e-13      | 5e-16
//   4, 3-25 Hz, 1 ms, 8001         | 2e-14          | 1.6e-13      | 4e-16
//   4, 3-6 Hz, 0.1 ms, 40001       | 2.0e-12        | 2.2e-11      | 1.4e-15
//   12, 3-25 Hz, 1 ms, 8001        | 2.0e-11        | 7.4e-11      | 1.3e-13
//   16, 3-25 Hz, 1 ms, 8001        | 3.2e-10        | 4.2e-9       | 4e-12
struct Dd {
    double hi, lo;
};
Dd dd_fma(const Dd &a, const Dd &b, const Dd &c) {  // a b + c
    const volatile double prod = a.hi * b.hi;  // volatile: the compiler may not fuse it into the sum below
    const double p = prod, pe = std::fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi);
    const double s = p + c.hi, t = s - p;
    const double se = ((p - (s - t)) + (c.hi - t)) + (pe + c.lo);
    const double h = s + se;
    return {h, se - (h - s)};
}
struct Block {
    Dd v[4];
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
                        o.v[2 * p + q] = dd_fma(x.v[2 * p + 1], y.v[2 + q], dd_fma(x.v[2 * p], y.v[q], o.v[2 * p + q]));
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
    double k[MAXS], d[MAXS], t[MAXS];  // a section's k, d and t
    int flip[MAXS];                    // sign bit of t in the high word
    double P[LEV][MAXS * (MAXS + 1) / 2 * 4];
};

// map of one sample: the recursion from v = 0; state values (z1, e)
template <int NS>
void plan_scan(Scan<NS> &F, int C) {
    const int N = F.nsec;
    F.C = C;
    Tri one((size_t)N * (N + 1) / 2), m = one;
    for (int k = 0; k < N; k++) m[k * (k + 1) / 2 + k].v[0].hi = m[k * (k + 1) / 2 + k].v[3].hi = 1.0;
    for (int j = 0; j < N; j++)
        for (int q = 0; q < 2; q++) {  // column of state value q of section j
            Dd v{0.0, 0.0};
            for (int i = j; i < N; i++) {
                const Dd z1{i == j && q == 0 ? 1.0 : 0.0, 0.0}, e{i == j && q == 1 ? 1.0 : 0.0, 0.0};
                const Dd y = dd_fma({1.0, 0.0}, v, z1), t{F.t[i], 0.0};
                Block &b = one[i * (i + 1) / 2 + j];
                b.v[q] = dd_fma({F.k[i], 0.0}, y, dd_fma(t, v, e));
                b.v[2 + q] = dd_fma({-F.d[i], 0.0}, y, dd_fma(t, e, {0.0, 0.0}));
                v = y;
            }
        }
    for (int c = C; c; c >>= 1) {
        if (c & 1) m = tri_mul(one, m, N);
        if (c > 1) one = tri_mul(one, one, N);
    }
    for (int l = 0; l < Scan<NS>::LEV; l++) {
        for (size_t b = 0; b < m.size(); b++)
            for (int q = 0; q < 4; q++) F.P[l][4 * b + q] = m[b].v[q].hi;
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
// 127 us in direct form, 130 us in the form with the sum e.
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
                z2[k] = -v - F.t[k] * v;
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
                    z1[k] = fma(F.k[k], y, fma(F.t[k], v, e));
                    z2[k] = fma(-F.d[k], y, __hiloint2double(__double2hiint(e) ^ F.flip[k], __double2loint(e)));  // t e
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
        F.t[k] = s[k].a1 <= 0.0 ? 1.0 : -1.0;
        F.flip[k] = s[k].a1 <= 0.0 ? 0 : INT_MIN;
        F.k[k] = -(F.t[k] + s[k].a1);
        F.d[k] = (1.0 + F.t[k] * s[k].a1) + s[k].a2;
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
