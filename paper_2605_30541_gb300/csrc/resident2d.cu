// Resident FP32 2D steps: a run of time steps of one or more shots in a single
// cooperative launch whose CTAs keep the wavefield on chip. Three modes: the
// forward solve, the forward recompute that records the imaging terms, and the
// adjoint sweep that consumes them.
//
// The per-step kernel (fwd2d_f32.cu) pays, every step, a launch, a grid-wide
// dependency and a reload of p^n, p^{n-1} and c from L2: 6 to 15 us on grids
// whose arithmetic takes one. On a slice of a few hundred thousand to about a
// million cells (all shots of an FWI survey on a small model, or one shot of a
// field-scale slice) the whole state fits in the SMs' shared memory, so here
// each CTA owns one subdomain of 128 columns and at most WZ = 16 RZ rows for
// the entire run. Subdomain heights vary (RTile descriptors from the host):
// subdomains with absorbing work get fewer rows, so every CTA takes about as
// long per step; warps take ceil(rows / 16) consecutive rows each.
//   - p^n with an 8-cell halo lives in shared memory in two buffers; the
//     other buffer's own cells still hold p^{n-1}, which each thread reads
//     and overwrites with p^{n+1} in place;
//   - the CPML memory variables live in shared memory, on the strips only
//     (RSpan): psi on the absorbing strips (and the 4-cell band beyond the
//     subdomain that a derivative of psi reaches, recomputed redundantly as in
//     the per-step kernel), zeta and the update addend D1 psi + zeta on the
//     strips widened by 4 cells. Outside the strips both recursion
//     coefficients are zero, so everything skipped is exactly zero. x-strip
//     work is spread over all threads (a strip is narrower than a row of
//     warps); z-strip work follows the rows of warps, and zeta_z is fused into
//     the update, which already holds D2z p. The adjoint's multipliers nu and
//     mu (cpml_adj.cu states their recursions) take the same places, with one
//     phase more;
//   - sponge subdomains of a forward solve precompute per cell the update
//     weights 2/(1+a), (1-a)/(1+a) and c/(1+a) (a = c eta dt / 2 is fixed in
//     time), so the step has no division; the gradient's modes round as the
//     per-step kernels' division does (quot2, from 1/(1+a) kept per cell), so
//     that FP16 checkpoints round the same states (with the division itself a
//     gradient of 4 shots of 231 x 381 cells took 8.8 ms instead of 6.3);
//   - a CTA writes the 8 (4 without CPML) border rows and columns of p^{n+1} to
//     its outbox in global memory as 8-byte words (value, step tag), as they
//     are computed; a CTA starts step n by reading its neighbours' words, each
//     until it carries the step's tag, and keeping the values as its halo. The
//     word is one 64-bit access, so a value is never seen without its tag and
//     no fence, counter or second fetch lies on the way: the chain per step is
//     one store, one read and a block barrier. (With a counter per subdomain -
//     store, barrier, release, poll, barrier, fetch, barrier - the exchange
//     alone took 2.55 us: 1000 steps of 241 x 241 cells 3.87 ms, of 669 x 1100
//     with 100 snapshots 6.35 ms; 2.86 and 4.25 ms with the words.) The
//     stencil is a cross, so it needs no corner neighbours; receivers may.
//     Two outbox halves alternate by step parity: a CTA that writes p^{n+1}
//     over p^{n-1} has read p^n from every neighbour that reads it, and each of
//     them sent p^n only after a barrier behind all its reads of p^{n-1}. Tags
//     never repeat between launches, so a word of an earlier run is never taken.
// The launch is cooperative, so all CTAs are co-resident and the waits
// always end; each wait is still bounded (spin_limit polls), after which the
// kernel raises kFlagTimeout and every CTA returns.
//
// Measured (gradients, per-step kernels and this): 16 shots of 241 x 241 cells,
// 1000 steps, CPML, FP16 checkpoints 58.2 and 21.5 ms; 4 shots of 231 x 381,
// 600 steps, sponge, with the forward of the loss 13.0 and 6.1 ms.
//
// The scheme is the leapfrog update with the centred sponge term or the CPML
// memory terms (Sec. 2, App. E.3-E.4), free surface as an odd mirror with
// row 0 held at zero; the per-cell arithmetic is that of the per-step kernel
// (in FP32 pairs; the same roundings but for the sponge weights above).
// Snapshots in FP32 only: an FP16 snapshot's scale needs the grid-wide maximum
// of the previous step, which a schedule without a grid barrier lacks.
#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "f32_tile.cuh"
#include "sim_internal.h"

namespace gsim {
namespace {

using namespace f32;

constexpr int TX = kTileXF, HM = 8, SW = TX + 2 * HM;
constexpr int NWR = kResidentWarps, NTR = NWR * 32;

// Receivers of a subdomain whose entries are kept in shared memory (more
// are read from global memory every step).
constexpr int kRecCache = 128;

__device__ __forceinline__ float4 neg4(const float4 &v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }

// Outbox of a subdomain, one half (words): the top border rows, the bottom
// ones, the left and the right border columns.
constexpr int XN = 0, XS = HM * TX, XWST = 2 * HM * TX, XEST = XWST + 64 * HM, XHALF = kResidentOutbox / 2;
static_assert(XEST + 64 * HM == XHALF, "outbox size");

// four words (value, tag) = 32 bytes
__device__ __forceinline__ void put4(unsigned long long *d, const float4 v, int tag) {
    const unsigned long long t = (unsigned long long)(unsigned)tag << 32;
    const unsigned long long a = t | __float_as_uint(v.x), b = t | __float_as_uint(v.y), c = t | __float_as_uint(v.z),
                             e = t | __float_as_uint(v.w);
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};\nst.relaxed.gpu.global.v2.b64 [%0+16], {%3, %4};\n" ::"l"(d),
                 "l"(a), "l"(b), "l"(c), "l"(e)
                 : "memory");
}
// reads them; true when all four carry the tag
__device__ __forceinline__ bool get4(const unsigned long long *d, int tag, float4 &v) {
    unsigned long long a, b, c, e;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%4];\nld.relaxed.gpu.global.v2.b64 {%2, %3}, [%4+16];\n"
                 : "=l"(a), "=l"(b), "=l"(c), "=l"(e)
                 : "l"(d)
                 : "memory");
    v = make_float4(__uint_as_float((unsigned)a), __uint_as_float((unsigned)b), __uint_as_float((unsigned)c),
                    __uint_as_float((unsigned)e));
    const unsigned t = (unsigned)tag;
    return (unsigned)(a >> 32) == t && (unsigned)(b >> 32) == t && (unsigned)(c >> 32) == t && (unsigned)(e >> 32) == t;
}


// The roundings of the per-step kernel's absorbing cells (fwd2d_f32.cu), which
// the gradient's checkpoints and imaging terms depend on: the first difference
// starts with fma(d_1, p_1 - m_1, d_2 (p_2 - m_2)); psi and zeta_z are
// fma(a, d, b m) (rec2), zeta_x is fma(b, m, a d).
__device__ __forceinline__ float2 d1s2(float2 m1, float2 p1, float2 m2, float2 p2, float2 m3, float2 p3, float2 m4,
                                       float2 p4) {
    float2 r = mul2(splat2(float(kD2)), add2(p2, neg2(m2)));
    r = fma2(splat2(float(kD1)), add2(p1, neg2(m1)), r);
    r = fma2(splat2(float(kD3)), add2(p3, neg2(m3)), r);
    return fma2(splat2(float(kD4)), add2(p4, neg2(m4)), r);
}
__device__ __forceinline__ float2 rec2b(float2 a, float2 d, float2 b, float2 m) { return fma2(b, m, mul2(a, d)); }
// first difference along x of the four cells C from the row's float4s L, C, R
__device__ __forceinline__ void d1x4(const float4 &L, const float4 &C, const float4 &R, float2 &da, float2 &db) {
    const float2 v34 = make_float2(L.w, C.x), v56 = make_float2(C.y, C.z), v12 = make_float2(L.y, L.z),
                 v78 = make_float2(C.w, R.x), v910 = make_float2(R.y, R.z);
    da = d1s2(v34, v56, hi2(L), hi2(C), v12, v78, lo2(L), lo2(R));
    db = d1s2(v56, v78, lo2(C), lo2(R), v34, v910, hi2(L), hi2(R));
}
// and along z at p, rows of pitch ST
template <int ST>
__device__ __forceinline__ void d1z4(const float *p, float2 &da, float2 &db) {
    const float4 m4 = ld4(p - 4 * ST), m3 = ld4(p - 3 * ST), m2 = ld4(p - 2 * ST), m1 = ld4(p - ST), p1 = ld4(p + ST),
                 p2 = ld4(p + 2 * ST), p3 = ld4(p + 3 * ST), p4 = ld4(p + 4 * ST);
    da = d1s2(lo2(m1), lo2(p1), lo2(m2), lo2(p2), lo2(m3), lo2(p3), lo2(m4), lo2(p4));
    db = d1s2(hi2(m1), hi2(p1), hi2(m2), hi2(p2), hi2(m3), hi2(p3), hi2(m4), hi2(p4));
}
// second differences along x of the four cells C from the row's float4s L, C, R
__device__ __forceinline__ void d2x_pairs(const float4 &L, const float4 &C, const float4 &R, float2 &da, float2 &db) {
    const float2 v34 = make_float2(L.w, C.x), v56 = make_float2(C.y, C.z), v12 = make_float2(L.y, L.z),
                 v78 = make_float2(C.w, R.x), v910 = make_float2(R.y, R.z);
    da = d2c2(lo2(C), v34, v56, hi2(L), hi2(C), v12, v78, lo2(L), lo2(R));
    db = d2c2(hi2(C), v56, v78, lo2(C), lo2(R), v34, v910, hi2(L), hi2(R));
}

// OPT: record and adjoint, FP16 imaging terms; forward, the corners are
// exchanged (an instance of its own: one for both took 2.79 ms instead of 2.74
// for 1000 steps of 241 x 241 cells).
template <int RZ, int MODE, bool OPT>
__global__ void __launch_bounds__(NTR, 1) k_resident2d(const __grid_constant__ StepArgs<float> A,
                                                       const __grid_constant__ ResidentArgs R) {
    constexpr int WZ = NWR * RZ;
    constexpr bool ADJ = MODE == kResAdjoint, QH = OPT && MODE != kResForward, CORNERS = OPT && MODE == kResForward;
    extern __shared__ float4 smem4[];
    __shared__ unsigned s_mask[2];  // rows with injected cells
    const RLayout &Y = R.lay;
    float *const S0 = reinterpret_cast<float *>(smem4);
    float *const S1 = S0 + (WZ + 2 * HM) * SW;
    float *const CC = S0 + Y.c;     // WZ x TX: c
    float *const F1 = S0 + Y.f1;    // x strips: psi / nu, chunks [p0, p1)
    float *const F2 = S0 + Y.f2;    // x strips: zeta (own chunks) / mu, chunks [q0, q1)
    float *const AX = S0 + Y.ax;    // x strips: the term, own chunks [a0, a1)
    float *const Z1 = S0 + Y.z1;    // z strips: psi / nu, rows [zp0, zp1)
    float *const Z2 = S0 + Y.z2;    // z strips: zeta (own rows) / mu, rows [zq0, zq1)
    float *const GG = S0 + Y.G;     // adjoint: WZ x TX gradient sums
    float *const KA = S0 + Y.K, *const KB = KA + WZ * TX, *const KC = KB + WZ * TX;  // sponge update weights (exact: KA = 1/(1+a))
    float *const INJ = S0 + Y.inj;  // injected weights (adjoint: values, two halves) of the flagged rows
    // CPML recursion coefficients: x cells [-8, TX + 8), rows [-8, WZ + 8)
    float *const CAX = S0 + Y.coef, *const CBX = CAX + TX + 16, *const CAZ = CBX + TX + 16, *const CBZ = CAZ + WZ + 16;
    int *const RIDX = reinterpret_cast<int *>(S0 + Y.rec);  // receiver cache
    int *const ROFF = RIDX + kRecCache;
    float *const RW = reinterpret_cast<float *>(ROFF + kRecCache);

    const Geom &g = A.g;
    const bool cpml = R.m2[0] || R.m2[1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
    const int ntiles = R.ntiles, lshot = blockIdx.x / ntiles, tile = blockIdx.x - lshot * ntiles, shot = R.shot0 + lshot;
    const RTile *const D = R.tiles + tile;
    const int bx = D->bx, x0 = bx * TX, z0 = D->z0, rows = D->rows, rpw = D->rpw, P = g.P;
    const long long sh = (long long)shot * g.fstride;
    const long long org = cell_off(g, z0, 0, x0);
    float *const gb0 = A.pbuf[0] + sh + org;
    float *const gb1 = A.pbuf[1] + sh + org;
    unsigned long long *const outbox = R.outbox + (long long)blockIdx.x * kResidentOutbox;

    const RSpan sp = resident_span(g, cpml ? (int)SIM_BC_CPML : (int)SIM_BC_NONE, bx, z0, rows, ADJ);
    const int ncx = sp.c1 - sp.c0, nax = sp.a1 - sp.a0;
    const bool hasx = ncx > 0 && A.ca[2], hasz = sp.zc1 > sp.zc0 && A.ca[0];
    const bool spg = A.bc == SIM_BC_SPONGE &&
                     ((g.nbx0 > 0 && x0 < g.nbx0) || (g.nbx1 > 0 && x0 + TX > g.NX - g.nbx1) ||
                      (g.nbz0 > 0 && z0 < g.nbz0) || (g.nbz1 > 0 && z0 + rows > g.NZ - g.nbz1));
    const bool xedge = x0 + TX > g.NX;
    const bool top = g.fs && z0 == 0;
    const int H = cpml ? 8 : 4;                   // exchanged border depth
    const bool hasN = z0 > 0, hasS = z0 + rows < g.NZ, hasW = bx > 0, hasE = x0 + TX < g.NX;
    const int c0 = HM + 4 * lane, gx0 = x0 + 4 * lane, rb = HM + w * rpw;
    const int lo = w * rpw * P + 4 * lane;

    // Shared memory starts at zero: the halo of an absent neighbour, the rows
    // and columns beyond the grid and every CPML value outside the strips.
    for (int i = tid; i < Y.total / 4; i += NTR) smem4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (tid < 2) s_mask[tid] = 0u;
    __syncthreads();

    // run constants
#pragma unroll
    for (int j = 0; j < RZ; j++) {
        const int lz = w * rpw + j;
        if (j < rpw && lz < rows) {
            cp_async16(CC + lz * TX + 4 * lane, A.ch + org + lo + j * P);
            if (ADJ) cp_async16(GG + lz * TX + 4 * lane, A.G + sh + org + lo + j * P);
        }
    }
    if (spg && R.exact_sponge)
        for (int i = tid; i < rows; i += NTR) CAZ[i + 8] = A.E[0][z0 + i];
    if (cpml) {
        for (int i = tid; i < TX + 16; i += NTR) {
            CAX[i] = A.ca[2] ? A.ca[2][x0 - 8 + i] : 0.f;
            CBX[i] = A.cb[2] ? A.cb[2][x0 - 8 + i] : 0.f;
        }
        for (int i = tid; i < WZ + 16; i += NTR) {
            const int gz = z0 - 8 + i;
            const bool in = A.ca[0] && gz >= 0 && gz < g.NZ;
            CAZ[i] = in ? A.ca[0][gz] : 0.f;
            CBZ[i] = in ? A.cb[0][gz] : 0.f;
        }
    }
    if (R.load) {  // p^n0 with its halo, p^{n0-1}, the memory fields
        const float *pc = (R.n0 & 1) ? gb1 : gb0, *pm = (R.n0 & 1) ? gb0 : gb1;
        for (int r = w - HM; r < rows + HM; r += NWR) {
            cp_async16(S0 + (HM + r) * SW + 4 * lane, pc + (long long)r * P - HM + 4 * lane);
            if (lane < 4) cp_async16(S0 + (HM + r) * SW + 128 + 4 * lane, pc + (long long)r * P - HM + 128 + 4 * lane);
            if (r >= 0 && r < rows) cp_async16(S1 + (HM + r) * SW + c0, pm + (long long)r * P + 4 * lane);
        }
        if (hasx) {
            const float *m1 = R.m1i[0] + sh + org, *m2 = R.m2[0] + sh + org;
            for (int i = tid; i < rows * ncx; i += NTR) {
                const int lz = i / ncx, c = sp.c0 + i - lz * ncx;
                cp_async16(F1 + lz * Y.w1 + 4 * (c - sp.p0), m1 + (long long)lz * P + 4 * c - 8);
            }
            const int b0 = ADJ ? sp.m0 : sp.a0, nb = (ADJ ? sp.m1 : sp.a1) - b0, off = ADJ ? sp.q0 : sp.a0;
            for (int i = tid; i < rows * nb; i += NTR) {
                const int lz = i / nb, c = b0 + i - lz * nb;
                cp_async16(F2 + lz * Y.w2 + 4 * (c - off), m2 + (long long)lz * P + 4 * c - 8);
            }
        }
        if (hasz) {
            const float *m1 = R.m1i[1] + sh + org, *m2 = R.m2[1] + sh + org;
            for (int r = sp.zc0 + w; r < sp.zc1; r += NWR)
                cp_async16(Z1 + (r - sp.zp0) * TX + 4 * lane, m1 + (long long)r * P + 4 * lane);
            const int b0 = ADJ ? sp.zm0 : sp.za0, b1 = ADJ ? sp.zm1 : sp.za1, off = ADJ ? sp.zq0 : sp.za0;
            for (int r = b0 + w; r < b1; r += NWR)
                cp_async16(Z2 + (r - off) * TX + 4 * lane, m2 + (long long)r * P + 4 * lane);
        }
    }
    cp_async_wait_all();
    __syncthreads();
    float4 E4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (spg) {
        E4 = __ldg(reinterpret_cast<const float4 *>(A.E[2] + gx0));
        // out = KA p - KB p^{n-1} + KC rhs, a = c (eta_z + eta_x); exact: KA = 1/(1+a)
#pragma unroll
        for (int j = 0; j < RZ; j++) {
            const int lz = w * rpw + j, gz = z0 + lz;
            if (j >= rpw || lz >= rows) continue;
            const float ez = A.E[0][gz];
            const float4 c4 = ld4(CC + lz * TX + 4 * lane);
            float ka[4], kb[4], kc[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const float chv = lane_of(c4, k), es = ez + lane_of(E4, k), a = chv * es, inv = 1.f / (1.f + a);
                ka[k] = R.exact_sponge ? 1.f / __fmaf_rn(chv, es, 1.f) : 2.f * inv;
                kb[k] = (1.f - a) * inv;
                kc[k] = chv * inv;
            }
            st4(KA + lz * TX + 4 * lane, make_float4(ka[0], ka[1], ka[2], ka[3]));
            if (R.exact_sponge) continue;
            st4(KB + lz * TX + 4 * lane, make_float4(kb[0], kb[1], kb[2], kb[3]));
            st4(KC + lz * TX + 4 * lane, make_float4(kc[0], kc[1], kc[2], kc[3]));
        }
    }
    // Injection: the target cells are fixed, so their rows are found once. A
    // point source's value is its weight times w(n); the adjoint's values are
    // sums of residuals, formed a step ahead into the other half of INJ.
    const SimIO *io = A.io;
    const int itile = A.inj_per_shot ? shot * ntiles + tile : tile;
    const int g0 = A.inj_start[itile], g1 = A.inj_start[itile + 1];
    const bool has_inj = g1 > g0;
    for (int gi = g0 + tid; gi < g1; gi += NTR) {
        const int lz = A.inj_grp[gi].cell >> 7;
        atomicOr(&s_mask[lz >> 5], 1u << (lz & 31));
    }
    __syncthreads();
    const unsigned mask0 = s_mask[0], mask1 = s_mask[1];
    auto inj_row = [&](int lz) {  // place of a flagged row
        return lz < 32 ? __popc(mask0 & ((1u << lz) - 1u)) : __popc(mask0) + __popc(mask1 & ((1u << (lz - 32)) - 1u));
    };
    auto inj_flag = [&](int lz) { return ((lz < 32 ? mask0 >> lz : mask1 >> (lz - 32)) & 1u) != 0u; };
    // adjoint: the values of sweep step n (gather row nt - n). A thread's first
    // cell, of one or two entries, has them in registers, and the residuals of
    // the next step are fetched while this one waits for its borders.
    int gplace = -1, gpt0 = 0, gpt1 = 0;
    float gw0 = 0.f, gw1 = 0.f, gr0 = 0.f, gr1 = 0.f;
    if (ADJ && g0 + tid < g1) {
        const InjGroup G = A.inj_grp[g0 + tid];
        if (G.e1 - G.e0 <= 2) {
            gplace = inj_row(G.cell >> 7) * TX + (G.cell & 127);
            gpt0 = gpt1 = A.inj_ent[G.e0].pt;
            gw0 = A.inj_ent[G.e0].w;
            if (G.e1 - G.e0 == 2) gpt1 = A.inj_ent[G.e0 + 1].pt, gw1 = A.inj_ent[G.e0 + 1].w;
        }
    }
    auto resid_row = [&](int n) {
        return static_cast<const float *>(io->resid) + ((long long)shot * A.nt + A.nt - n) * io->nrec;
    };
    auto fetch_residuals = [&](int n) {
        gr0 = gr1 = 0.f;
        if (gplace < 0 || n < 1) return;
        gr0 = resid_row(n)[gpt0];
        if (gw1 != 0.f) gr1 = resid_row(n)[gpt1];
    };
    auto residuals = [&](int n) {
        float *const half = INJ + (n & 1) * Y.injr * TX;
        if (gplace >= 0) half[gplace] = __fmaf_rn(gw1, gr1, gw0 * gr0);
        for (int gi = g0 + tid + (gplace >= 0 ? NTR : 0); gi < g1; gi += NTR) {
            const InjGroup G = A.inj_grp[gi];
            float sum = 0.f;
            if (n >= 1)
                for (int e = G.e0; e < G.e1; e++) sum += A.inj_ent[e].w * resid_row(n)[A.inj_ent[e].pt];
            half[inj_row(G.cell >> 7) * TX + (G.cell & 127)] = sum;
        }
    };
    if (ADJ) {
        fetch_residuals(R.n0);
        residuals(R.n0);
    } else {
        for (int gi = g0 + tid; gi < g1; gi += NTR) {
            const InjGroup G = A.inj_grp[gi];
            float wsum = 0.f;
            for (int e = G.e0; e < G.e1; e++) wsum += A.inj_ent[e].w;
            INJ[inj_row(G.cell >> 7) * TX + (G.cell & 127)] = wsum;
        }
    }
    const bool sample = MODE == kResForward && A.sample;
    const int r0 = sample ? A.rec_start[tile] : 0, r1 = sample ? A.rec_start[tile + 1] : 0;
    const bool rec_cached = r1 - r0 <= kRecCache;
    if (rec_cached)
        for (int e = r0 + tid; e < r1; e += NTR) {
            const RecEntryT<float> Rc = A.rec[e];
            RIDX[e - r0] = Rc.rec;
            ROFF[e - r0] = (HM + Rc.lz) * SW + HM + Rc.lx;
            for (int q = 0; q < 4; q++) RW[4 * (e - r0) + q] = Rc.w[q];
        }
    // The thread's halo float4s (at most two): the words of a neighbour's outbox
    // and the place in the pressure buffer. Rows -H .. -1 come from the bottom
    // rows of the subdomain above, rows >= rows from the top rows of the one
    // below (a last one of fewer than H rows has no more: zeros), columns left
    // and right from the subdomains of the adjacent columns that hold the row.
    // The stencil needs no corner; a receiver between the last row and column
    // and the next ones reads the south-east one (CORNERS). Its subdomain may
    // share no row or column with this one, so it waits in turn for this one's
    // corner: neither then overwrites a word that the other has yet to read.
    int xsrc[2] = {-1, -1}, xdst[2] = {0, 0}, xmir[2] = {-1, -1};  // xmir: the float4's place above the free surface
    {
        const int hq = H / 4, nN = hasN ? 32 * H : 0;
        int up = -1, down = -1;
        for (int k = 0; k < D->nnbr; k++) {
            const RTile &u = R.tiles[D->nbr[k]];
            if (u.bx == bx && u.z0 < z0) up = D->nbr[k];
            if (u.bx == bx && u.z0 > z0) down = D->nbr[k];
        }
        const int nS = hasS ? 32 * min(H, R.tiles[down].rows) : 0, nW = hasW ? rows * hq : 0, nE = hasE ? rows * hq : 0;
        auto side = [&](int dx, int gz) {  // word offset of the neighbour column's subdomain that holds row gz, and its row
            for (int k = 0; k < D->nnbr; k++) {
                const RTile &u = R.tiles[D->nbr[k]];
                if (u.bx == bx + dx && gz >= u.z0 && gz < u.z0 + u.rows)
                    return (lshot * ntiles + D->nbr[k]) * kResidentOutbox + (gz - u.z0) * HM;
            }
            return -1;
        };
        for (int v = 0; v < 2; v++) {
            int i = tid + v * NTR;
            if (i < nN) {
                xsrc[v] = (lshot * ntiles + up) * kResidentOutbox + XS + i * 4;
                xdst[v] = (HM - H + (i >> 5)) * SW + HM + 4 * (i & 31);
                continue;
            }
            i -= nN;
            if (i < nS) {
                xsrc[v] = (lshot * ntiles + down) * kResidentOutbox + XN + i * 4;
                xdst[v] = (HM + rows + (i >> 5)) * SW + HM + 4 * (i & 31);
                continue;
            }
            i -= nS;
            if (i < nW) {
                const int r = i / hq, q = i - r * hq, o = side(-1, z0 + r);
                xsrc[v] = o < 0 ? -1 : o + XEST + 4 * q;
                xdst[v] = (HM + r) * SW + HM - H + 4 * q;
                if (top && r >= 1 && r <= H) xmir[v] = xdst[v] - 2 * r * SW;
                continue;
            }
            i -= nW;
            if (i < nE) {
                const int r = i / hq, q = i - r * hq, o = side(1, z0 + r);
                xsrc[v] = o < 0 ? -1 : o + XWST + 4 * q;
                xdst[v] = (HM + r) * SW + HM + TX + 4 * q;
                if (top && r >= 1 && r <= H) xmir[v] = xdst[v] - 2 * r * SW;
            }
        }
        // the corners, by threads whose second float4 is free: the subdomain that
        // holds one is a neighbour of the one below (south-east) or above (north-west)
        if (CORNERS && tid >= NTR - 2) {
            const bool se = tid == NTR - 1;
            const int via = se ? down : up, z = se ? z0 + rows : z0 - 1;
            for (int k = 0; via >= 0 && k < R.tiles[via].nnbr; k++) {
                const int j = R.tiles[via].nbr[k];
                const RTile &u = R.tiles[j];
                if (u.bx != (se ? bx + 1 : bx - 1) || z < u.z0 || z >= u.z0 + u.rows) continue;
                xsrc[1] = (lshot * ntiles + j) * kResidentOutbox + (se ? XWST : XEST + H - 4) + (z - u.z0) * HM;
                xdst[1] = se ? (HM + rows) * SW + HM + TX : (HM - 1) * SW + HM - 4;
            }
        }
    }
    static_assert(2 * HM * 32 + 2 * 64 * (HM / 4) + 2 <= 2 * NTR, "two halo float4s per thread at most");
    const float *const wav = static_cast<const float *>(io->wavelet);
    float *const gout = static_cast<float *>(io->gather);
    float *const snaps = MODE == kResForward ? static_cast<float *>(io->snaps) : nullptr;
    const int nrec = io->nrec;
    if (top && R.load)  // odd mirror above the free surface: p(-k) = -p(k); later steps write it with p(k)
        for (int k = 1 + w; k <= H; k += NWR)
            for (int c = HM - H + 4 * lane; c < HM + TX + H; c += 128)
                st4(S0 + (HM - k) * SW + c, neg4(ld4(S0 + (HM + k) * SW + c)));
    float wnext = (!ADJ && has_inj && R.n0 < R.n1) ? wav[R.n0] : 0.f;
    __syncthreads();

    for (int n = R.n0; n < R.n1; n++) {
        const int par = (n - R.n0) & 1;
        const unsigned tag = R.tag0 + (unsigned)(n - R.n0);
        float *const cur = par ? S1 : S0;
        float *const nxt = par ? S0 : S1;

        // this step's wavelet sample (fetched one step ahead)
        const float wn = wnext;
        if (!ADJ && has_inj && n + 1 < R.n1) wnext = wav[n + 1];
        // this step's imaging terms, in flight during the wait (FP16: as they lie, two words)
        const long long slot = MODE == kResRecord ? n - R.n0 : R.n1 - 1 - n;
        char *const qs = R.q + slot * R.qstride;
        // FP16 slots: a warp's scale lies in the shot's top ghost rows, which hold nothing else
        float *const qsc = reinterpret_cast<float *>(reinterpret_cast<__half *>(qs) + sh) + tile * NWR + w;
        std::conditional_t<ADJ && QH, uint2, float4> qv[RZ];
        float qs1 = 1.f;
        if (MODE == kResAdjoint) {
            if constexpr (QH) qs1 = *qsc;
#pragma unroll
            for (int j = 0; j < RZ; j++) {
                qv[j] = {};
                if (j >= rpw || w * rpw + j >= rows) continue;
                const long long o = sh + org + lo + j * P;
                if constexpr (ADJ && QH)
                    qv[j] = *reinterpret_cast<const uint2 *>(reinterpret_cast<const __half *>(qs) + o);
                else
                    qv[j] = ld4(reinterpret_cast<const float *>(qs) + o);
            }
        }

        if (ADJ && has_inj && n + 1 < R.n1) fetch_residuals(n + 1);

        bool quit = false;
        if (n > R.n0) {  // the neighbours' borders of p^n become this step's halo
            const unsigned long long *const in = R.outbox + par * XHALF;
            bool need0 = xsrc[0] >= 0, need1 = xsrc[1] >= 0;
            for (long long spins = 0; need0 || need1;) {
                float4 v0, v1;
                const bool ok0 = need0 && get4(in + xsrc[0], tag, v0), ok1 = need1 && get4(in + xsrc[1], tag, v1);
                if (ok0) {
                    st4(cur + xdst[0], v0);
                    if (xmir[0] >= 0) st4(cur + xmir[0], neg4(v0));
                    need0 = false;
                }
                if (ok1) {
                    st4(cur + xdst[1], v1);
                    if (xmir[1] >= 0) st4(cur + xmir[1], neg4(v1));
                    need1 = false;
                }
                if (!(need0 || need1)) break;
                if (++spins > R.spin_limit) {
                    quit = true;
                    atomicOr(A.flags, kFlagTimeout);
                    break;
                }
                if ((spins & 1023) == 0 && (*reinterpret_cast<volatile unsigned *>(A.flags) & kFlagTimeout)) {
                    quit = true;
                    break;
                }
            }
        }
        if (__syncthreads_or(quit)) return;
        if (!ADJ) {
            // CPML psi^n = b psi^{n-1} + a D1 p^n (scaled by h) on the strips
            if (hasx)
                for (int i = tid; i < rows * ncx; i += NTR) {
                    const int lz = i / ncx, c = sp.c0 + (i - lz * ncx);
                    const float *row = cur + (HM + lz) * SW + 4 * c;
                    const float4 a4 = ld4(CAX + 4 * c), b4 = ld4(CBX + 4 * c);
                    float *px = F1 + lz * Y.w1 + 4 * (c - sp.p0);
                    const float4 old = ld4(px);
                    float2 da, db;
                    d1x4(ld4(row - 4), ld4(row), ld4(row + 4), da, db);
                    const float2 pa = rec2(lo2(a4), da, lo2(b4), lo2(old)), pb = rec2(hi2(a4), db, hi2(b4), hi2(old));
                    st4(px, make_float4(pa.x, pa.y, pb.x, pb.y));
                }
            if (hasz)
                for (int r = sp.zc0 + w; r < sp.zc1; r += NWR) {
                    const float *col = cur + (HM + r) * SW + c0;
                    float2 da, db;
                    d1z4<SW>(col, da, db);
                    const float2 a2 = splat2(CAZ[r + 8]), b2 = splat2(CBZ[r + 8]);
                    float *pz = Z1 + (r - sp.zp0) * TX + 4 * lane;
                    const float4 old = ld4(pz);
                    const float2 pa = rec2(a2, da, b2, lo2(old)), pb = rec2(a2, db, b2, hi2(old));
                    st4(pz, make_float4(pa.x, pa.y, pb.x, pb.y));
                }
            if (hasx || hasz) __syncthreads();
            // zeta_x^n = b zeta_x^{n-1} + a (D2x p^n + D1x psi_x^n) and the addend
            // D1x psi_x^n + zeta_x^n on the widened x-strips
            if (hasx && nax > 0) {
                for (int i = tid; i < rows * nax; i += NTR) {
                    const int lz = i / nax, c = sp.a0 + (i - lz * nax);
                    const float *row = cur + (HM + lz) * SW + 4 * c, *px = F1 + lz * Y.w1 + 4 * (c - sp.p0);
                    const float4 a4 = ld4(CAX + 4 * c), b4 = ld4(CBX + 4 * c);
                    float *zp = F2 + lz * Y.w2 + 4 * (c - sp.a0);
                    const float4 z4 = ld4(zp);
                    float2 xa, xb, da, db;
                    d2x_pairs(ld4(row - 4), ld4(row), ld4(row + 4), xa, xb);
                    d1x4(ld4(px - 4), ld4(px), ld4(px + 4), da, db);
                    const float2 za = rec2b(lo2(a4), add2(xa, da), lo2(b4), lo2(z4));
                    const float2 zb = rec2b(hi2(a4), add2(xb, db), hi2(b4), hi2(z4));
                    st4(zp, make_float4(za.x, za.y, zb.x, zb.y));
                    const float2 ea = add2(da, za), eb = add2(db, zb);
                    st4(AX + lz * Y.wa + 4 * (c - sp.a0), make_float4(ea.x, ea.y, eb.x, eb.y));
                }
                __syncthreads();
            }
        } else if (hasx || hasz) {
            // nu^k = b nu^{k+1} + u^{k+1}
            if (hasx)
                for (int i = tid; i < rows * ncx; i += NTR) {
                    const int lz = i / ncx, c = sp.c0 + (i - lz * ncx);
                    const float4 u = ld4(cur + (HM + lz) * SW + 4 * c), b4 = ld4(CBX + 4 * c);
                    float *px = F1 + lz * Y.w1 + 4 * (c - sp.p0);
                    const float4 old = ld4(px);
                    const float2 na = fma2(lo2(b4), lo2(old), lo2(u)), nb = fma2(hi2(b4), hi2(old), hi2(u));
                    st4(px, make_float4(na.x, na.y, nb.x, nb.y));
                }
            if (hasz)
                for (int r = sp.zc0 + w; r < sp.zc1; r += NWR) {
                    const float4 u = ld4(cur + (HM + r) * SW + c0);
                    const float2 b2 = splat2(CBZ[r + 8]);
                    float *pz = Z1 + (r - sp.zp0) * TX + 4 * lane;
                    const float4 old = ld4(pz);
                    const float2 na = fma2(b2, lo2(old), lo2(u)), nb = fma2(b2, hi2(old), hi2(u));
                    st4(pz, make_float4(na.x, na.y, nb.x, nb.y));
                }
            __syncthreads();
            // mu^k = b mu^{k+1} - D1 (u^{k+1} + a nu^k)
            if (hasx && sp.m1 > sp.m0) {
                const int nm = sp.m1 - sp.m0;
                auto wx = [&](const float *row, const float *px, int c) {  // u + a nu of chunk c
                    const float4 u = ld4(row), nu = ld4(px), a4 = ld4(CAX + 4 * c);
                    const float2 wa = fma2(lo2(a4), lo2(nu), lo2(u)), wb = fma2(hi2(a4), hi2(nu), hi2(u));
                    return make_float4(wa.x, wa.y, wb.x, wb.y);
                };
                for (int i = tid; i < rows * nm; i += NTR) {
                    const int lz = i / nm, c = sp.m0 + (i - lz * nm);
                    const float *row = cur + (HM + lz) * SW + 4 * c, *px = F1 + lz * Y.w1 + 4 * (c - sp.p0);
                    const float4 b4 = ld4(CBX + 4 * c);
                    float *mp = F2 + lz * Y.w2 + 4 * (c - sp.q0);
                    const float4 old = ld4(mp);
                    float2 da, db;
                    d1x_pairs(wx(row - 4, px - 4, c - 1), wx(row, px, c), wx(row + 4, px + 4, c + 1), da, db);
                    const float2 ma = fma2(lo2(b4), lo2(old), neg2(da)), mb = fma2(hi2(b4), hi2(old), neg2(db));
                    st4(mp, make_float4(ma.x, ma.y, mb.x, mb.y));
                }
            }
            if (hasz && sp.zm1 > sp.zm0) {
                auto wz = [&](int r) {
                    const float4 u = ld4(cur + (HM + r) * SW + c0), nu = ld4(Z1 + (r - sp.zp0) * TX + 4 * lane);
                    const float2 a2 = splat2(CAZ[r + 8]);
                    const float2 wa = fma2(a2, lo2(nu), lo2(u)), wb = fma2(a2, hi2(nu), hi2(u));
                    return make_float4(wa.x, wa.y, wb.x, wb.y);
                };
                for (int r = sp.zm0 + w; r < sp.zm1; r += NWR) {
                    float2 da, db;
                    d1_pairs(wz(r - 4), wz(r - 3), wz(r - 2), wz(r - 1), wz(r + 1), wz(r + 2), wz(r + 3), wz(r + 4), da, db);
                    const float2 b2 = splat2(CBZ[r + 8]);
                    float *mp = Z2 + (r - sp.zq0) * TX + 4 * lane;
                    const float4 old = ld4(mp);
                    const float2 ma = fma2(b2, lo2(old), neg2(da)), mb = fma2(b2, hi2(old), neg2(db));
                    st4(mp, make_float4(ma.x, ma.y, mb.x, mb.y));
                }
            }
            __syncthreads();
            // the bracket of the x axis: D2 (a nu) - D1 (a mu)
            if (hasx && nax > 0) {
                auto am = [&](const float *p, int c) {
                    const float4 v = ld4(p), a4 = ld4(CAX + 4 * c);
                    return make_float4(a4.x * v.x, a4.y * v.y, a4.z * v.z, a4.w * v.w);
                };
                for (int i = tid; i < rows * nax; i += NTR) {
                    const int lz = i / nax, c = sp.a0 + (i - lz * nax);
                    const float *np = F1 + lz * Y.w1 + 4 * (c - sp.p0), *mp = F2 + lz * Y.w2 + 4 * (c - sp.q0);
                    float2 xa, xb, da, db;
                    d2x_pairs(am(np - 4, c - 1), am(np, c), am(np + 4, c + 1), xa, xb);
                    d1x_pairs(am(mp - 4, c - 1), am(mp, c), am(mp + 4, c + 1), da, db);
                    st4(AX + lz * Y.wa + 4 * (c - sp.a0),
                        make_float4(xa.x - da.x, xa.y - da.y, xb.x - db.x, xb.y - db.y));
                }
                __syncthreads();
            }
        }

        // update: p^{n+1} into the other buffer, borders to the outbox
        float4 zw[RZ + 8];
#pragma unroll
        for (int j = 0; j < RZ + 8; j++) zw[j] = ld4(cur + (rb - 4 + j) * SW + c0);
        float tmax = 0.f;
        const bool inx = hasx && lane + 2 >= sp.a0 && lane + 2 < sp.a1;
        unsigned long long *const ob = outbox + (par ^ 1) * XHALF;
#pragma unroll
        for (int j = 0; j < RZ; j++) {
            const int lz = w * rpw + j;
            if (j >= rpw || lz >= rows) continue;
            const float4 C = zw[j + 4];
            const Pairs4 d = d2_pairs(ld4(cur + (rb + j) * SW + c0 - 4), C, ld4(cur + (rb + j) * SW + c0 + 4), zw + j);
            float2 ra = add2(d.za, d.xa), rbb = add2(d.zb, d.xb);
            const float4 pp4 = ld4(nxt + (rb + j) * SW + c0);  // p^{n-1}
            const float4 c4 = ld4(CC + lz * TX + 4 * lane);
            // CPML terms: x from the phase above; z in place on the widened z-strips
            const bool zrow = hasz && lz >= sp.za0 && lz < sp.za1;
            if (inx || zrow) {
                float2 ea = make_float2(0.f, 0.f), eb = ea;
                if (inx) {
                    const float4 ax4 = ld4(AX + lz * Y.wa + 4 * (lane + 2 - sp.a0));
                    ea = lo2(ax4), eb = hi2(ax4);
                }
                if (zrow) {
                    const float *z1 = Z1 + (lz - sp.zp0) * TX + 4 * lane;
                    if (!ADJ) {  // zeta_z^n = b zeta_z^{n-1} + a (D2z p^n + D1z psi_z^n)
                        float2 da, db;
                        d1z4<TX>(z1, da, db);
                        float *zp = Z2 + (lz - sp.za0) * TX + 4 * lane;
                        const float4 z4 = ld4(zp);
                        const float2 a2 = splat2(CAZ[lz + 8]), b2 = splat2(CBZ[lz + 8]);
                        const float2 za = rec2(a2, add2(d.za, da), b2, lo2(z4)), zb = rec2(a2, add2(d.zb, db), b2, hi2(z4));
                        st4(zp, make_float4(za.x, za.y, zb.x, zb.y));
                        ea = add2(ea, add2(da, za));
                        eb = add2(eb, add2(db, zb));
                    } else {  // D2 (a nu) - D1 (a mu)
                        const float *z2 = Z2 + (lz - sp.zq0) * TX + 4 * lane;
                        float4 an[9], m[9];
#pragma unroll
                        for (int k = 0; k < 9; k++) {
                            const float a = CAZ[lz + 4 + k];
                            const float4 v = ld4(z1 + (k - 4) * TX), u = ld4(z2 + (k - 4) * TX);
                            an[k] = make_float4(a * v.x, a * v.y, a * v.z, a * v.w);
                            m[k] = make_float4(a * u.x, a * u.y, a * u.z, a * u.w);
                        }
                        const float2 d2a = d2c2(lo2(an[4]), lo2(an[3]), lo2(an[5]), lo2(an[2]), lo2(an[6]), lo2(an[1]),
                                                lo2(an[7]), lo2(an[0]), lo2(an[8]));
                        const float2 d2b = d2c2(hi2(an[4]), hi2(an[3]), hi2(an[5]), hi2(an[2]), hi2(an[6]), hi2(an[1]),
                                                hi2(an[7]), hi2(an[0]), hi2(an[8]));
                        float2 da, db;
                        d1_pairs(m[0], m[1], m[2], m[3], m[5], m[6], m[7], m[8], da, db);
                        ea = add2(ea, add2(d2a, neg2(da)));
                        eb = add2(eb, add2(d2b, neg2(db)));
                    }
                }
                ra = add2(ra, ea);
                rbb = add2(rbb, eb);
            }
            if (has_inj && inj_flag(lz)) {
                const float4 v = ld4(INJ + ((ADJ ? (n & 1) * Y.injr : 0) + inj_row(lz)) * TX + 4 * lane);
                const float f = ADJ ? 1.f : wn;
                ra.x = __fmaf_rn(A.src_scale, v.x * f, ra.x);
                ra.y = __fmaf_rn(A.src_scale, v.y * f, ra.y);
                rbb.x = __fmaf_rn(A.src_scale, v.z * f, rbb.x);
                rbb.y = __fmaf_rn(A.src_scale, v.w * f, rbb.y);
            }
            float res[4], qk[4];
            const float rhs[4] = {ra.x, ra.y, rbb.x, rbb.y};
            if (!spg) {
                const float4 o = plain4(C, pp4, c4, ra, rbb);
                res[0] = o.x, res[1] = o.y, res[2] = o.z, res[3] = o.w;
#pragma unroll
                for (int k = 0; k < 4; k++) qk[k] = 0.f * (res[k] - lane_of(pp4, k)) - rhs[k];
            } else if (R.exact_sponge) {
                const float ez = CAZ[lz + 8];
                const float4 y4 = ld4(KA + lz * TX + 4 * lane);
                const float2 one = splat2(1.f), two = splat2(2.f), ea = add2(splat2(ez), lo2(E4)), eb = add2(splat2(ez), hi2(E4));
                const float2 ta = fma2(lo2(c4), ra, fma2(neg2(fma2(neg2(lo2(c4)), ea, one)), lo2(pp4), mul2(two, lo2(C))));
                const float2 tb = fma2(hi2(c4), rbb, fma2(neg2(fma2(neg2(hi2(c4)), eb, one)), hi2(pp4), mul2(two, hi2(C))));
                const float2 oa = quot2(ta, fma2(lo2(c4), ea, one), lo2(y4)), ob2 = quot2(tb, fma2(hi2(c4), eb, one), hi2(y4));
                res[0] = oa.x, res[1] = oa.y, res[2] = ob2.x, res[3] = ob2.y;
                qk[0] = __fmaf_rn(ea.x, oa.x - pp4.x, -ra.x), qk[1] = __fmaf_rn(ea.y, oa.y - pp4.y, -ra.y);
                qk[2] = __fmaf_rn(eb.x, ob2.x - pp4.z, -rbb.x), qk[3] = __fmaf_rn(eb.y, ob2.y - pp4.w, -rbb.y);
            } else {
                const float4 ka = ld4(KA + lz * TX + 4 * lane), kb = ld4(KB + lz * TX + 4 * lane),
                             kc = ld4(KC + lz * TX + 4 * lane);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    res[k] = lane_of(ka, k) * lane_of(C, k) - lane_of(kb, k) * lane_of(pp4, k) + lane_of(kc, k) * rhs[k];
                    qk[k] = 0.f;
                }
            }
            if (xedge) {
#pragma unroll
                for (int k = 0; k < 4; k++)
                    if (gx0 + k >= g.NX) res[k] = 0.f;
            }
            if (top && lz == 0) res[0] = res[1] = res[2] = res[3] = 0.f;
            const float4 r4 = make_float4(res[0], res[1], res[2], res[3]);
            if (top && lz >= 1 && lz <= H) st4(nxt + (HM - lz) * SW + c0, neg4(r4));  // odd mirror above the free surface
            st4(nxt + (rb + j) * SW + c0, r4);
            if (RZ < 3 && n + 1 < R.n1) {
                if (hasN && lz < H) put4(ob + XN + lz * TX + 4 * lane, r4, tag + 1);
                if (hasS && lz >= rows - H) put4(ob + XS + (lz - rows + H) * TX + 4 * lane, r4, tag + 1);
                if (hasW && 4 * lane < H) put4(ob + XWST + lz * HM + 4 * lane, r4, tag + 1);
                if (hasE && 4 * lane >= TX - H) put4(ob + XEST + lz * HM + 4 * lane - (TX - H), r4, tag + 1);
            }
            if constexpr (MODE == kResRecord) {
                qv[j] = make_float4(qk[0], qk[1], qk[2], qk[3]);
                if (QH)
                    tmax = fmaxf(tmax, fmaxf(fmaxf(fabsf(qk[0]), fabsf(qk[1])), fmaxf(fabsf(qk[2]), fabsf(qk[3]))));
                else
                    st4(reinterpret_cast<float *>(qs) + sh + org + lo + j * P, qv[j]);
            }
            if constexpr (ADJ) {
                float *gp = GG + lz * TX + 4 * lane;
                float4 gv = ld4(gp), q;
                if constexpr (QH) {
                    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&qv[j].x)),
                                 b = __half22float2(*reinterpret_cast<const __half2 *>(&qv[j].y));
                    q = make_float4(a.x * qs1, a.y * qs1, b.x * qs1, b.y * qs1);
                } else {
                    q = qv[j];
                }
                gv.x += res[0] * q.x;
                gv.y += res[1] * q.y;
                gv.z += res[2] * q.z;
                gv.w += res[3] * q.w;
                st4(gp, gv);
            }
        }
        // Borders of tall subdomains, from the rows just written: few instances of
        // the sending code for the instruction cache, and the side columns of all
        // rows at once (with 4 rows per warp a gradient of 16 shots 22.32 -> 21.49
        // ms, with 3 a slice 4.03 -> 4.01; with 1 or 2 rows, where a send per row
        // in place starts earlier, 2.84 -> 2.90 and 6.13 -> 6.17)
        if (RZ >= 3 && n + 1 < R.n1) {
            __syncwarp();
            const int w0 = w * rpw, w1 = min(w0 + rpw, rows);
            if (hasN)
#pragma unroll 1
                for (int lz = w0; lz < min(w1, H); lz++)
                    put4(ob + XN + lz * TX + 4 * lane, ld4(nxt + (HM + lz) * SW + c0), tag + 1);
            if (hasS)
#pragma unroll 1
                for (int lz = max(w0, rows - H); lz < w1; lz++)
                    put4(ob + XS + (lz - rows + H) * TX + 4 * lane, ld4(nxt + (HM + lz) * SW + c0), tag + 1);
            // lane: (row, side, float4)
            const int b = cpml ? 2 : 1, lz = w0 + (lane >> b), east = (lane >> (b - 1)) & 1, q = cpml ? lane & 1 : 0;
            if (lz < w1 && (east ? hasE : hasW))
                put4(ob + (east ? XEST : XWST) + lz * HM + 4 * q, ld4(nxt + (HM + lz) * SW + HM + (east ? TX - H : 0) + 4 * q),
                     tag + 1);
        }
        if constexpr (MODE == kResRecord && QH) {  // one power-of-two scale per warp and step
            const float s = pow2_scale(warp_max(tmax)), inv = 1.f / s;
            if (lane == 0) *qsc = s;
#pragma unroll
            for (int j = 0; j < RZ; j++) {
                if (j >= rpw || w * rpw + j >= rows) continue;
                const __half2 a = __floats2half2_rn(qv[j].x * inv, qv[j].y * inv),
                              b = __floats2half2_rn(qv[j].z * inv, qv[j].w * inv);
                uint2 u;
                u.x = *reinterpret_cast<const unsigned *>(&a);
                u.y = *reinterpret_cast<const unsigned *>(&b);
                *reinterpret_cast<uint2 *>(reinterpret_cast<__half *>(qs) + sh + org + lo + j * P) = u;
            }
        }
        if (ADJ && has_inj && n + 1 < R.n1) residuals(n + 1);

        // Off the critical path, while the words travel: receivers and the
        // snapshot sample p^n, still held in this buffer until the next step's
        // update (behind the next barrier) overwrites it.
        if (r1 > r0 && gout) {
            const long long rowo = ((long long)shot * A.nt + n) * nrec;
            for (int e = tid; e < r1 - r0; e += NTR) {
                int ri, off;
                float w4[4];
                if (rec_cached) {
                    ri = RIDX[e];
                    off = ROFF[e];
                    for (int q = 0; q < 4; q++) w4[q] = RW[4 * e + q];
                } else {
                    const RecEntryT<float> Rc = A.rec[r0 + e];
                    ri = Rc.rec;
                    off = (HM + Rc.lz) * SW + HM + Rc.lx;
                    for (int q = 0; q < 4; q++) w4[q] = Rc.w[q];
                }
                const float *b = cur + off;
                const float val = w4[0] * b[0] + w4[1] * b[1] + w4[2] * b[SW] + w4[3] * b[SW + 1];
                gout[rowo + ri] = val;
                if (!isfinite(val)) atomicOr(A.flags, kFlagUnstable);
            }
        }
        if (snaps && A.nsnap > 0 && n >= A.snap_begin && n < A.snap_end && (n - A.snap_begin) % A.snap_every == 0) {
            const int snap_k = (n - A.snap_begin) / A.snap_every;
            const long long sbase = ((long long)shot * A.nsnap + snap_k) * g.nz * g.nx;
#pragma unroll
            for (int j = 0; j < RZ; j++) {
                const int gz = z0 + w * rpw + j;
                if (j >= rpw || w * rpw + j >= rows || gz < g.oz || gz >= g.oz + g.nz) continue;
                const float4 p4 = ld4(cur + (rb + j) * SW + c0);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const int gx = gx0 + k;
                    if (gx < g.ox || gx >= g.ox + g.nx) continue;
                    snaps[sbase + (long long)(gz - g.oz) * g.nx + (gx - g.ox)] = lane_of(p4, k);
                }
            }
        }
    }

    // final state: p^{n1} and p^{n1-1} into the global buffers of the per-step
    // layout, own cells only, each thread copying the cells it wrote; the
    // memory fields' own cells on the strips, and the gradient sums
    if (R.n1 > R.n0) {
        const bool odd = (R.n1 - R.n0) & 1;
        const float *fin = odd ? S1 : S0, *prv = odd ? S0 : S1;
        float *gl = (R.n1 & 1) ? gb1 : gb0, *gp = (R.n1 & 1) ? gb0 : gb1;
#pragma unroll
        for (int j = 0; j < RZ; j++) {
            const int lz = w * rpw + j;
            if (j >= rpw || lz >= rows) continue;
            st4(gl + lo + j * P, ld4(fin + (rb + j) * SW + c0));
            st4(gp + lo + j * P, ld4(prv + (rb + j) * SW + c0));
            if (ADJ) st4(A.G + sh + org + lo + j * P, ld4(GG + lz * TX + 4 * lane));
        }
        if (R.store_mem && (hasx || hasz)) {
            __syncthreads();
            if (hasx) {
                float *m1 = R.m1o[0] + sh + org, *m2 = R.m2[0] + sh + org;
                const int k0 = max(sp.c0, 2), nk = min(sp.c1, 2 + TX / 4) - k0;
                for (int i = tid; i < rows * max(nk, 0); i += NTR) {
                    const int lz = i / nk, c = k0 + i - lz * nk;
                    st4(m1 + (long long)lz * P + 4 * c - 8, ld4(F1 + lz * Y.w1 + 4 * (c - sp.p0)));
                }
                const int b0 = ADJ ? max(sp.m0, 2) : sp.a0, nb = (ADJ ? min(sp.m1, 2 + TX / 4) : sp.a1) - b0,
                          off = ADJ ? sp.q0 : sp.a0;
                for (int i = tid; i < rows * max(nb, 0); i += NTR) {
                    const int lz = i / nb, c = b0 + i - lz * nb;
                    st4(m2 + (long long)lz * P + 4 * c - 8, ld4(F2 + lz * Y.w2 + 4 * (c - off)));
                }
            }
            if (hasz) {
                float *m1 = R.m1o[1] + sh + org, *m2 = R.m2[1] + sh + org;
                for (int r = max(sp.zc0, 0) + w; r < min(sp.zc1, rows); r += NWR)
                    st4(m1 + (long long)r * P + 4 * lane, ld4(Z1 + (r - sp.zp0) * TX + 4 * lane));
                const int b0 = ADJ ? max(sp.zm0, 0) : sp.za0, b1 = ADJ ? min(sp.zm1, rows) : sp.za1,
                          off = ADJ ? sp.zq0 : sp.za0;
                for (int r = b0 + w; r < b1; r += NWR)
                    st4(m2 + (long long)r * P + 4 * lane, ld4(Z2 + (r - off) * TX + 4 * lane));
            }
        }
    }
}

template <int RZ, int MODE, bool OPT>
cudaError_t launch_rz(const StepArgs<float> &a, const ResidentArgs &r, int nshots, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r.ntiles * nshots);
    cfg.blockDim = dim3(NTR);
    cfg.dynamicSmemBytes = (size_t)r.lay.total * sizeof(float);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_resident2d<RZ, MODE, OPT>, a, r);
}

template <int RZ>
cudaError_t launch_mode(const StepArgs<float> &a, const ResidentArgs &r, int mode, int nshots, cudaStream_t st) {
    const bool qh = a.q_fp16 != 0;
    if (mode == kResForward)
        return r.corners ? launch_rz<RZ, kResForward, true>(a, r, nshots, st) : launch_rz<RZ, kResForward, false>(a, r, nshots, st);
    if (mode == kResRecord)
        return qh ? launch_rz<RZ, kResRecord, true>(a, r, nshots, st) : launch_rz<RZ, kResRecord, false>(a, r, nshots, st);
    return qh ? launch_rz<RZ, kResAdjoint, true>(a, r, nshots, st) : launch_rz<RZ, kResAdjoint, false>(a, r, nshots, st);
}

template <int RZ>
cudaError_t configure_rz() {
    cudaError_t e = cudaSuccess;
    for (auto k : {k_resident2d<RZ, kResForward, false>, k_resident2d<RZ, kResForward, true>, k_resident2d<RZ, kResRecord, false>,
                   k_resident2d<RZ, kResRecord, true>, k_resident2d<RZ, kResAdjoint, false>, k_resident2d<RZ, kResAdjoint, true>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentMaxSmem - 64);
    return e;
}

}  // namespace

// Shared-memory layout of a launch over the given subdomains; false when it
// does not fit. injr: rows with injected cells a subdomain has at most.
bool resident2d_layout(const Geom &g, int bc, int rz, int mode, bool exact_sponge, const std::vector<RTile> &tiles, int injr,
                       RLayout &Y) {
    const int WZ = kResidentWarps * rz;
    const bool adj = mode == kResAdjoint, cpml = bc == SIM_BC_CPML;
    int w1 = 0, w2 = 0, wa = 0, z1 = 0, z2 = 0;
    if (cpml)
        for (const RTile &t : tiles) {
            const RSpan s = resident_span(g, bc, t.bx, t.z0, t.rows, adj);
            w1 = std::max(w1, 4 * (s.p1 - s.p0));
            wa = std::max(wa, 4 * (s.a1 - s.a0));
            w2 = std::max(w2, adj ? 4 * (s.q1 - s.q0) : 4 * (s.a1 - s.a0));
            z1 = std::max(z1, s.zp1 - s.zp0);
            z2 = std::max(z2, adj ? s.zq1 - s.zq0 : s.za1 - s.za0);
        }
    Y = RLayout{};
    Y.w1 = w1;
    Y.w2 = w2;
    Y.wa = wa;
    Y.injr = injr;
    long long o = 2LL * (WZ + 2 * HM) * SW;
    auto take = [&](long long n) {
        const long long at = o;
        o += (n + 3) / 4 * 4;
        return (int)at;
    };
    Y.c = take((long long)WZ * TX);
    Y.coef = take(bc != SIM_BC_NONE ? 2 * (TX + 16) + 2 * (WZ + 16) : 0);
    Y.f1 = take((long long)WZ * w1);
    Y.f2 = take((long long)WZ * w2);
    Y.ax = take((long long)WZ * wa);
    Y.z1 = take((long long)z1 * TX);
    Y.z2 = take((long long)z2 * TX);
    Y.G = take(adj ? (long long)WZ * TX : 0);
    Y.K = take(bc == SIM_BC_SPONGE ? (exact_sponge ? 1LL : 3LL) * WZ * TX : 0);
    Y.inj = take((long long)(adj ? 2 : 1) * injr * TX);
    Y.rec = take(mode == kResForward ? 6 * kRecCache : 0);
    Y.total = (int)std::min<long long>(o, 1 << 28);
    return o * (long long)sizeof(float) + 64 <= (long long)kResidentMaxSmem;
}

cudaError_t configure_resident2d() {
    cudaError_t e = configure_rz<1>();
    if (e == cudaSuccess) e = configure_rz<2>();
    if (e == cudaSuccess) e = configure_rz<3>();
    if (e == cudaSuccess) e = configure_rz<4>();
    return e;
}

cudaError_t launch_resident2d(const StepArgs<float> &a, const ResidentArgs &r, int rz, int mode, int nshots,
                              cudaStream_t st) {
    switch (rz) {
        case 1: return launch_mode<1>(a, r, mode, nshots, st);
        case 2: return launch_mode<2>(a, r, mode, nshots, st);
        case 3: return launch_mode<3>(a, r, mode, nshots, st);
        case 4: return launch_mode<4>(a, r, mode, nshots, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gsim
