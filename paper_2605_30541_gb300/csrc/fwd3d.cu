// 3D time step of the acoustic scheme (FP32).
//
// Main kernel: a z-march over (x, y) tiles (2.5D blocking). A CTA of 8 warps
// owns a column of 1024 cells of the grid, 64 x 16 or 32 x 32 where the planes
// are staged by tensor-memory-accelerator copies that one thread issues
// (k_step3d_tma, the only form that runs unasked) and 128 x 8 where every
// thread copies its share by cp.async (k_step3d, which GSIM_ZMARCH=async selects:
// the form the tests compare the other with). Each thread owns 4 consecutive x
// cells of a row and keeps the 9 planes z-4 .. z+4 of those cells in a register
// queue, so p^n is read from memory once per cell for the z-derivative. The
// planes with their radius-4 x/y halo are staged into a shared-memory ring
// ahead of use. The update is the leapfrog step with the
// centred sponge term (Eq. cerjan_pde), the free-surface plane z = 0 held at
// zero with an odd mirror above it (Eq. free_surface), and no boundary
// arithmetic outside absorbing tiles.
//
// The CPML addends of each axis and the receiver samples come from one launch
// before the march (cpml3d.cu), the march injects the point sources; snapshot
// output and the adjoint sweep's injection are side kernels.
#include <cfloat>
#include <climits>

#include <cudaTypedefs.h>

#include "sim_internal.h"
#include "stencil.cuh"

namespace gsim {
namespace {

constexpr int TX = kTileXF, NW = 8, NTH = NW * 32, SW3 = TX + 8;

__device__ __forceinline__ float lane4(const float4 &v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}
__device__ __forceinline__ float4 ld4g(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// The four cells of one thread at one plane: x window L, C, R (C the cells),
// the nine y rows yv (yv[4] = C) and the nine z planes z0..z8 (z4 = C) of
// p^n. The second differences run in cell pairs (0, 1) and (2, 3) with the
// pair arithmetic, in d2c's order of roundings; rhs = D2x + D2y + D2z. The
// plain update p^{n+1} = 2 p - p^{n-1} + c rhs is fma(c, rhs, fma(2, p,
// -p^{n-1})), also in pairs; the sponge update (Eq. cerjan_pde) runs per
// cell. Both z-marches call this, so they give the same bits.
struct Cells4 {
    float res[4], rhs[4];
};
__device__ __forceinline__ Cells4 cells4(const float4 &L, const float4 &C, const float4 &R, const float4 (&yv)[9],
                                         const float4 &z0, const float4 &z1, const float4 &z2, const float4 &z3,
                                         const float4 &z5, const float4 &z6, const float4 &z7, const float4 &z8,
                                         const float4 &pp4, const float4 &ch4, bool spg, float es0,
                                         const float4 &Ex4) {
    // x: pairs of the 12-float window; (v3, v4), (v5, v6), (v1, v2), (v7, v8), (v9, v10) straddle float4s
    const float2 v34 = make_float2(L.w, C.x), v56 = make_float2(C.y, C.z), v12 = make_float2(L.y, L.z),
                 v78 = make_float2(C.w, R.x), v910 = make_float2(R.y, R.z);
    const float2 xa = d2c2(lo2(C), v34, v56, hi2(L), hi2(C), v12, v78, lo2(L), lo2(R));
    const float2 xb = d2c2(hi2(C), v56, v78, lo2(C), lo2(R), v34, v910, hi2(L), hi2(R));
    const float2 ya = d2c2(lo2(C), lo2(yv[3]), lo2(yv[5]), lo2(yv[2]), lo2(yv[6]), lo2(yv[1]), lo2(yv[7]),
                           lo2(yv[0]), lo2(yv[8]));
    const float2 yb = d2c2(hi2(C), hi2(yv[3]), hi2(yv[5]), hi2(yv[2]), hi2(yv[6]), hi2(yv[1]), hi2(yv[7]),
                           hi2(yv[0]), hi2(yv[8]));
    const float2 za = d2c2(lo2(C), lo2(z3), lo2(z5), lo2(z2), lo2(z6), lo2(z1), lo2(z7), lo2(z0), lo2(z8));
    const float2 zb = d2c2(hi2(C), hi2(z3), hi2(z5), hi2(z2), hi2(z6), hi2(z1), hi2(z7), hi2(z0), hi2(z8));
    const float2 ra = add2(add2(xa, ya), za), rb = add2(add2(xb, yb), zb);
    Cells4 o;
    o.rhs[0] = ra.x, o.rhs[1] = ra.y, o.rhs[2] = rb.x, o.rhs[3] = rb.y;
    if (!spg) {
        const float2 two = splat2(2.f);
        const float2 oa = fma2(lo2(ch4), ra, fma2(two, lo2(C), neg2(lo2(pp4))));
        const float2 ob = fma2(hi2(ch4), rb, fma2(two, hi2(C), neg2(hi2(pp4))));
        o.res[0] = oa.x, o.res[1] = oa.y, o.res[2] = ob.x, o.res[3] = ob.y;
    } else {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const float p = lane4(C, k), chv = lane4(ch4, k), pp = lane4(pp4, k);
            const float a = chv * (es0 + lane4(Ex4, k));
            o.res[k] = quot1(2.f * p - (1.f - a) * pp + chv * o.rhs[k], 1.f + a);
        }
    }
    return o;
}
__device__ __forceinline__ void cp16(void *smem, const void *gmem) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
// The CPML addends (cpml3d.cu) of one thread's row of four cells (gy, gx0 ..)
// in a tile at (x0, y0): p^{n+1} += c (addend) axis by axis, in the order x,
// z, y; the addend is part of the Laplacian in the record mode's imaging
// term. Tiles and planes away from the strips test block-uniform flags.
struct AddRows {
    const float *x, *y, *z;  // the row's addends at plane 0 (z: at slot 0); NULL: none
    long long px, py, pz;    // plane strides
    int zl, zh;              // planes < zl and >= zh take z addends (none: every plane lies between)
    bool xy;                 // the tile meets an x or y strip
    __device__ __forceinline__ AddRows(const Add3 &D, const Geom &g, int shot, int gy, int gx0, int x0, int tx, int y0, int ty)
        : x(nullptr), y(nullptr), z(nullptr) {
        const bool row = gy < g.NY && gx0 < g.NX;
        px = (long long)g.NY * D.nxw;
        py = (long long)D.nyw * g.P;
        pz = (long long)g.NY * g.P;
        if (D.a[2] && row && (gx0 < D.xl || gx0 >= D.xs))
            x = D.a[2] + shot * D.st[2] + (long long)gy * D.nxw + (gx0 < D.xl ? gx0 : D.xl + gx0 - D.xs);
        if (D.a[1] && row && (gy < D.yl || gy >= D.yh))
            y = D.a[1] + shot * D.st[1] + (long long)(gy < D.yl ? gy : D.yl + gy - D.yh) * g.P + gx0;
        if (D.a[0] && row) z = D.a[0] + shot * D.st[0] + (long long)gy * g.P + gx0;
        zl = D.a[0] ? D.zl : 0;
        zh = D.a[0] ? D.zh : INT_MAX;
        xy = (D.a[2] && (x0 < D.xl || x0 + tx > D.xs)) || (D.a[1] && (y0 < D.yl || y0 + ty > D.yh));
    }
    __device__ __forceinline__ bool zin(int pl) const { return pl < zl || pl >= zh; }
    __device__ __forceinline__ const float *zrow(int pl) const { return z + (pl < zl ? pl : zl + pl - zh) * pz; }
    __device__ __forceinline__ static void add(const float4 v, const float4 &c, float *res, float *qk) {
        res[0] = __fmaf_rn(c.x, v.x, res[0]), qk[0] -= v.x;
        res[1] = __fmaf_rn(c.y, v.y, res[1]), qk[1] -= v.y;
        res[2] = __fmaf_rn(c.z, v.z, res[2]), qk[2] -= v.z;
        res[3] = __fmaf_rn(c.w, v.w, res[3]), qk[3] -= v.w;
    }
    // straight from memory
    __device__ __forceinline__ void apply(int pl, const float4 &c, float *res, float *qk) const {
        if (x) add(ld4g(x + pl * px), c, res, qk);
        if (z && zin(pl)) add(ld4g(zrow(pl)), c, res, qk);
        if (y) add(ld4g(y + pl * py), c, res, qk);
    }
};
// One corner c of a shot's point source into p^{n+1} (already updated); with
// qs (record mode), its share E d - h^2 s of the imaging term.
__device__ __noinline__ void inject3(const StepArgs<float> &A, const Pt3 &P, int c, int shot, int n, int row, float *qs) {
    const Geom &g = A.g;
    const long long o = P.cell[c], so = (long long)shot * g.fstride + o;
    float es = 0.f;
    if (A.bc == SIM_BC_SPONGE) {
        const long long r = o - g.org, PP = (long long)g.PY * g.P;
        const int z = (int)(r / PP), y = (int)((r % PP) / g.P), x = (int)(r % g.P);
        es = A.E[0][z] + A.E[1][y] + A.E[2][x];
    }
    const float sum = P.w[c] * static_cast<const float *>(A.io->wavelet)[row], chv = A.ch[o];
    const float d = chv * A.src_scale * sum / (1.f + chv * es);
    A.pbuf[(n + 1) & 1][so] += d;
    if (qs) qs[so] += es * d - A.src_scale * sum;
}

// Staged planes in flight: while plane z is computed, planes z+1 .. z+4 are
// ready or arriving and plane z+5 is being requested. A ring slot holds the
// plane's p^n with its x/y halo, and p^{n-1} and c of the CTA's own cells;
// the register queue takes plane z+4's own cells from its slot, so after the
// prologue every global read of the march is a cp.async issued five planes
// ahead of its use.
constexpr int NS3 = 6;
template <int RY>
constexpr int slot3d() {
    return (NW * RY + 8) * SW3 + 2 * NW * RY * TX;
}

// MODE (kModeForward / kModeRecord / kModeAdjoint) as in the 2D kernel: the
// record sweep also writes the imaging term Q'^n = E (p^{n+1} - p^{n-1}) -
// h^2 L p^n of each cell to qs (the source's share is added by the injection
// kernel), the adjoint sweep adds u^{n+1} Q'^n, read from qs, to Gs.
template <int RY, int MODE>
__global__ void __launch_bounds__(NTH, 2) k_step3d(const StepArgs<float> A, const int n, const int zchunk,
                                                   const Add3 D, float *qs, float *Gs) {
    constexpr int TY = NW * RY, NR = TY + 8;  // staged rows per plane
    constexpr int SLOT = slot3d<RY>();
    extern __shared__ float4 sm3[];
    float *const ring = reinterpret_cast<float *>(sm3);

    const Geom &g = A.g;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int nchunk = (g.NZ + zchunk - 1) / zchunk;
    const int shot = blockIdx.z / nchunk, zb = (blockIdx.z % nchunk) * zchunk;
    const int ze = min(zb + zchunk, g.NZ);
    const long long PP = (long long)g.PY * g.P;  // plane pitch
    const long long sh = (long long)shot * g.fstride;
    const float *pc = A.pbuf[n & 1] + sh;
    float *pn = A.pbuf[(n + 1) & 1] + sh;
    const int gx0 = x0 + 4 * lane;
    const bool xedge = x0 + TX > g.NX;
    const bool spg = A.bc == SIM_BC_SPONGE &&
                     ((g.nbx0 > 0 && x0 < g.nbx0) || (g.nbx1 > 0 && x0 + TX > g.NX - g.nbx1) ||
                      (g.nby0 > 0 && y0 < g.nby0) || (g.nby1 > 0 && y0 + TY > g.NY - g.nby1) || g.nbz0 > 0 ||
                      g.nbz1 > 0);
    float4 Ex4 = make_float4(0, 0, 0, 0);
    float Ey[RY];
#pragma unroll
    for (int r = 0; r < RY; r++) Ey[r] = 0.f;
    if (spg) {
        Ex4 = __ldg(reinterpret_cast<const float4 *>(A.E[2] + gx0));
#pragma unroll
        for (int r = 0; r < RY; r++) Ey[r] = __ldg(A.E[1] + y0 + w * RY + r);
    }
    // offsets of (z = 0, y0 + w RY, gx0), of the staged plane's corner and of the tile's corner
    const long long own0 = cell_off(g, 0, y0 + w * RY, gx0);
    const long long halo0 = cell_off(g, 0, y0 - 4, x0 - 4);
    const long long tile0 = cell_off(g, 0, y0, x0);

    cudaGridDependencySynchronize();

    // register queue: planes z-4 .. z+4 of this thread's cells
    float4 q[9][RY];
    auto load_plane = [&](int z, int r) -> float4 {
        if (z < 0) {
            if (!g.fs) return make_float4(0, 0, 0, 0);
            const float4 v = *reinterpret_cast<const float4 *>(pc + own0 + (long long)(-z) * PP + r * g.P);
            return make_float4(-v.x, -v.y, -v.z, -v.w);
        }
        return *reinterpret_cast<const float4 *>(pc + own0 + (long long)z * PP + r * g.P);
    };
#pragma unroll
    for (int k = 0; k < 8; k++)
#pragma unroll
        for (int r = 0; r < RY; r++) q[k + 1][r] = load_plane(zb - 4 + k, r);

    // plane z into its slot: p^n with halo, and (for planes this CTA
    // updates) p^{n-1} and c of the own cells
    auto stage = [&](int z) {
        float *dst = ring + (z % NS3) * SLOT;
        const float *src = pc + halo0 + (long long)z * PP;
        for (int rr = w; rr < NR; rr += NW) {
            cp16(dst + rr * SW3 + 4 * lane, src + rr * g.P + 4 * lane);
            if (lane < 2) cp16(dst + rr * SW3 + 128 + 4 * lane, src + rr * g.P + 128 + 4 * lane);
        }
        if (z < ze) {
            float *dpp = dst + NR * SW3, *dch = dpp + TY * TX;
            const long long o = tile0 + (long long)z * PP;
            for (int rr = w; rr < TY; rr += NW) {
                cp16(dpp + rr * TX + 4 * lane, pn + o + rr * g.P + 4 * lane);
                cp16(dch + rr * TX + 4 * lane, A.ch + o + rr * g.P + 4 * lane);
            }
        }
        cp_commit();
    };
#pragma unroll
    for (int k = 0; k < NS3 - 1; k++) stage(zb + k);

    for (int z = zb; z < ze; z++) {
        stage(z + NS3 - 1);
        cp_wait<1>();
        __syncthreads();
        const float *cur = ring + (z % NS3) * SLOT;
        const float *ahead = ring + ((z + 4) % NS3) * SLOT;
#pragma unroll
        for (int k = 0; k < 8; k++)
#pragma unroll
            for (int r = 0; r < RY; r++) q[k][r] = q[k + 1][r];
#pragma unroll
        for (int r = 0; r < RY; r++)
            q[8][r] = *reinterpret_cast<const float4 *>(ahead + (w * RY + r + 4) * SW3 + 4 + 4 * lane);
        const float ez = spg ? __ldg(A.E[0] + z) : 0.f;
#pragma unroll
        for (int r = 0; r < RY; r++) {
            const int ly = w * RY + r, gy = y0 + ly;
            const float *row = cur + (ly + 4) * SW3 + 4 + 4 * lane;  // this thread's float4 in the staged plane
            const float4 L = *reinterpret_cast<const float4 *>(row - 4), C = *reinterpret_cast<const float4 *>(row),
                         R = *reinterpret_cast<const float4 *>(row + 4);
            float4 yv[9];
#pragma unroll
            for (int m = 0; m < 9; m++) yv[m] = *reinterpret_cast<const float4 *>(row + (m - 4) * SW3);
            const float4 pp4 = *reinterpret_cast<const float4 *>(cur + NR * SW3 + ly * TX + 4 * lane);
            const float4 ch4 = *reinterpret_cast<const float4 *>(cur + NR * SW3 + TY * TX + ly * TX + 4 * lane);
            const Cells4 cu = cells4(L, C, R, yv, q[0][r], q[1][r], q[2][r], q[3][r], q[5][r], q[6][r], q[7][r],
                                     q[8][r], pp4, ch4, spg, ez + Ey[r], Ex4);
            float res[4], qk[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                res[k] = cu.res[k];
                const float es = spg ? ez + Ey[r] + lane4(Ex4, k) : 0.f;
                qk[k] = es * (res[k] - lane4(pp4, k)) - cu.rhs[k];
            }
            AddRows(D, g, shot, gy, gx0, x0, TX, y0, TY).apply(z, ch4, res, qk);
            if (xedge) {
#pragma unroll
                for (int k = 0; k < 4; k++)
                    if (gx0 + k >= g.NX) res[k] = 0.f;
            }
            if (g.fs && z == 0) res[0] = res[1] = res[2] = res[3] = 0.f;
            if (gy < g.NY) {
                const long long o = own0 + (long long)z * PP + r * g.P;
                *reinterpret_cast<float4 *>(pn + o) = make_float4(res[0], res[1], res[2], res[3]);
                if (MODE == kModeRecord)
                    *reinterpret_cast<float4 *>(qs + sh + o) = make_float4(qk[0], qk[1], qk[2], qk[3]);
                if (MODE == kModeAdjoint) {
                    const float4 q4 = *reinterpret_cast<const float4 *>(qs + sh + o);
                    float4 g4 = *reinterpret_cast<const float4 *>(Gs + sh + o);
                    g4.x += res[0] * q4.x;
                    g4.y += res[1] * q4.y;
                    g4.z += res[2] * q4.z;
                    g4.w += res[3] * q4.w;
                    *reinterpret_cast<float4 *>(Gs + sh + o) = g4;
                }
            }
        }
        __syncthreads();  // this slot is restaged at the next plane
    }
    cp_wait<0>();  // no copy into shared memory outlives the block
}

// ---------------------------------------------------------------- z-march with TMA
//
// The same update as k_step3d, with the planes staged by the tensor memory
// accelerator: one thread issues, per plane z, three bulk tensor copies (p^n
// of plane z + 4 with its radius-4 x/y halo into the halo ring, for the
// register queue now and as the plane's own stencil rows four planes later;
// p^{n-1} and c of plane z's own cells into the own ring) and arms one
// mbarrier with their byte count; every thread waits on it once per plane.
// Groups are staged AHEAD planes before their use.
//
// A plane is 96 pair-arithmetic instructions per float4, and the march used to
// spend 250 more on three waits with 64-bit counters, generic addresses, votes
// and the ring bookkeeping (352 warp instructions per 128 cells, 112 us at
// 170 x 227 x 273 x 2 shots). One group per plane, rings of 8 and 4 slots with
// the loop unrolled by 4 (slot addresses are constants but for the halves of
// the halo ring, which swap), offsets instead of pointers and no vote leave 264
// and 88 us, the CPML addends' read included.
//
// A wait that gives up (bounded) marks its thread, which waits no more and
// goes on with whatever its slots hold; the leader then stages no more, waits
// (bounded) for the copies in flight, and the kernel sets kFlagTimeout.
//
// Tiles of TW x TY cells, TW = 64 or 32 and TW TY = 1024: a warp takes 128 / TW
// rows. They stage 1.7 and 1.6 cells per cell (a 128 x 8 tile: 2.1; it was
// slower by 3% at 172 x 152 rows, 5% at 1060 x 1060 and 12% at 273 x 227) and
// waste few lanes past a ragged edge. The autotuner times both.
constexpr int AHEAD = 3, NSH = AHEAD + 5, NSO = AHEAD + 1;  // planes z .. z + 4 + AHEAD; z .. z + AHEAD
static_assert(NSH == 8 && NSO == 4, "the plane loop is unrolled by 4");
template <int TW>
struct Tile3 {
    static constexpr int RPW = TX / TW, TY = NW * RPW, SW = TW + 8;
    static constexpr int HALO = (TY + 8) * SW * 4, OWN = TY * TW * 4, OSLOT = 2 * OWN;
    static constexpr int ADD = 2 * 3 * NTH * 16;            // CPML addends of two planes, a slot per thread and axis
    static constexpr int OWN0 = NSH * HALO, ADD0 = OWN0 + NSO * OSLOT, BAR0 = ADD0 + ADD;
    static constexpr size_t SMEM = (size_t)BAR0 + (NSO + 1) * sizeof(unsigned long long);
    static_assert(HALO % 128 == 0 && OWN % 128 == 0, "TMA destinations are 128-byte aligned");
    static_assert(SMEM <= 113 * 1024, "two CTAs per SM");
};

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned b, unsigned cnt) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(b), "r"(cnt) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(b), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned b, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(b), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(unsigned b, unsigned parity, int limit) {
    if (mbar_try(b, parity)) return true;
    for (int i = 1; i < limit; i++)
        if (mbar_try(b, parity)) return true;
    return false;
}
__device__ __forceinline__ void tma_load4(unsigned dst, const CUtensorMap *m, int x, int y, int z, int w, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(m)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load3(unsigned dst, const CUtensorMap *m, int x, int y, int z, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(m)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// src, row: the shots' point sources and the wavelet row injected (src NULL: none)
template <int MODE, int TW>
__global__ void __launch_bounds__(NTH, 2) k_step3d_tma(const StepArgs<float> A, const __grid_constant__ Tma3 M,
                                                       const int n, const int zchunk, const int ms, const Add3 D,
                                                       const Pt3 *src, const int row, float *qs, float *Gs,
                                                       const int spin) {
    using T3 = Tile3<TW>;
    constexpr int TY = T3::TY, SW = T3::SW, HALO = T3::HALO, OSLOT = T3::OSLOT, OWN = T3::OWN;
    extern __shared__ __align__(128) unsigned char sm_t[];
    const unsigned s0 = smem_u32(sm_t), bar0 = s0 + T3::BAR0;  // barriers: one per own slot, then the first planes'

    const Geom &g = A.g;
    const int tid = threadIdx.x, lx = 4 * (tid % (TW / 4)), w = tid / (TW / 4);  // cell and row in the tile
    const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TY;
    const int nchunk = (g.NZ + zchunk - 1) / zchunk;
    const int shot = blockIdx.z / nchunk, zb = (blockIdx.z % nchunk) * zchunk;
    const int ze = min(zb + zchunk, g.NZ);
    const long long PP = (long long)g.PY * g.P;
    const long long sh = (long long)shot * g.fstride;
    const int gx0 = x0 + lx, gy = y0 + w;
    const bool xedge = x0 + TW > g.NX, live = gy < g.NY && gx0 < g.NX;  // cells past the grid stay zero: no store
    const bool spg = A.bc == SIM_BC_SPONGE &&
                     ((g.nbx0 > 0 && x0 < g.nbx0) || (g.nbx1 > 0 && x0 + TW > g.NX - g.nbx1) ||
                      (g.nby0 > 0 && y0 < g.nby0) || (g.nby1 > 0 && y0 + TY > g.NY - g.nby1) || g.nbz0 > 0 ||
                      g.nbz1 > 0);
    float4 Ex4 = make_float4(0, 0, 0, 0);
    float Ey = 0.f;
    if (spg) {
        Ex4 = __ldg(reinterpret_cast<const float4 *>(A.E[2] + gx0));
        Ey = __ldg(A.E[1] + gy);
    }
    const long long own0 = cell_off(g, 0, gy, gx0);
    const AddRows add(D, g, shot, gy, gx0, x0, TW, y0, TY);
    float4 *const aslot = reinterpret_cast<float4 *>(sm_t + T3::ADD0) + tid;
    // tensor coordinates of the padded layout: (x, y, z) + kGhost; w = buffer parity * ms + shot
    const int tx = x0 + kGhost, ty = y0 + kGhost;
    const int wcur = (n & 1) * ms + shot, wprev = ((n + 1) & 1) * ms + shot;
    if (tid == 0) {
        for (int k = 0; k <= NSO; k++) mbar_init(bar0 + 8 * k, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();

    cudaGridDependencySynchronize();

    // thread 0: the group of plane z into halo slot kh (plane z + 4) and own slot ks
    auto stage = [&](int z, int kh, int ks) {
        const unsigned bar = bar0 + 8 * ks, dst = s0 + T3::OWN0 + ks * OSLOT;
        mbar_expect(bar, HALO + OSLOT);
        tma_load4(s0 + kh * HALO, &M.ph, tx - 4, ty - 4, z + 4 + kGhost, wcur, bar);
        tma_load4(dst, &M.po, tx, ty, z + kGhost, wprev, bar);
        tma_load3(dst + OWN, &M.c, tx, ty, z + kGhost, bar);
    };
    if (tid == 0) {
        mbar_expect(bar0 + 8 * NSO, 4 * HALO);
        for (int k = 0; k < 4; k++)
            tma_load4(s0 + k * HALO, &M.ph, tx - 4, ty - 4, zb + k + kGhost, wcur, bar0 + 8 * NSO);
        for (int k = 0; k < AHEAD; k++)
            if (zb + k < ze) stage(zb + k, k + 4, k);
    }
    // CPML addends of the coming plane into the thread's slots (x, y, z of two
    // planes); slots of an axis the thread has no addend of stay zero
    const float *ax = add.x + zb * add.px, *ay = add.y + zb * add.py;
    bool zn = false;  // the coming plane takes z addends
    auto fetch = [&](int z, int half) {
        float4 *const v = aslot + half * 3 * NTH;
        if (add.xy) {
            if (add.x) cp16(v, ax);
            if (add.y) cp16(v + NTH, ay);
            ax += add.px;
            ay += add.py;
        }
        zn = add.zin(z);
        if (zn && add.z) cp16(v + 2 * NTH, add.zrow(z));
        cp_commit();
    };
    for (int k = 0; k < 6; k++)
        if (!(k % 3 == 0 ? add.x : k % 3 == 1 ? add.y : add.z)) aslot[k * NTH] = make_float4(0.f, 0.f, 0.f, 0.f);
    fetch(zb, 0);

    // register queue of this thread's cells: plane z + m lives in q[(j + m + 4) % 9]
    // at step j of a block of 4 planes
    const unsigned rowo = ((w + 4) * SW + 4 + lx) * 4;  // the thread's float4 in a halo slot
    float4 q[9];
    {
        const float *pc = A.pbuf[n & 1] + sh + own0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int z = zb - 4 + k;
            float4 v = make_float4(0, 0, 0, 0);
            if (z >= 0) {
                v = ld4g(pc + (long long)z * PP);
            } else if (g.fs) {
                const float4 u = ld4g(pc + (long long)(-z) * PP);
                v = make_float4(-u.x, -u.y, -u.z, -u.w);
            }
            q[k] = v;
        }
    }
    int zbad = mbar_wait(bar0 + 8 * NSO, 0, spin) ? ze : zb - 1;  // plane at which this thread gave up waiting (ze: none)
#pragma unroll
    for (int k = 0; k < 4; k++) q[4 + k] = *reinterpret_cast<const float4 *>(sm_t + k * HALO + rowo);

    unsigned ha = 0, hb = 4;  // first halo slots of planes zz .. zz + 3 and zz + 4 .. zz + 7
    unsigned par = 0;         // phase of the own slots
    float *out = A.pbuf[(n + 1) & 1] + sh + own0 + (long long)zb * PP;
    long long orow = sh + own0 + (long long)zb * PP;  // record / adjoint: this thread's float4 of plane z
    for (int zz = zb; zz < ze; zz += 4) {
        const unsigned char *const ra = sm_t + ha * HALO + rowo, *const rb = sm_t + hb * HALO + rowo;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int z = zz + j;
            if (z >= ze) break;
            // into the slots plane z - 1 used
            if (tid == 0 && z + AHEAD < ze && zbad == ze) stage(z + AHEAD, j == 0 ? hb + 3 : ha + j - 1, (j + 3) % NSO);
            // the next plane's addends, a plane ahead of their use (the tiles at the
            // strips would wait on their latency every plane)
            const bool zadd = zn;
            if (z + 1 < ze) fetch(z + 1, (j + 1) & 1);
            else cp_commit();
            float4 qa = make_float4(0, 0, 0, 0), ga = qa;
            if (MODE == kModeAdjoint && live) {
                qa = ld4g(qs + orow);
                ga = ld4g(Gs + orow);
            }
            if (zbad == ze && !mbar_wait(bar0 + 8 * j, par, spin)) zbad = z;
            const unsigned char *const cur = ra + j * HALO, *const own = sm_t + T3::OWN0 + j * OSLOT + 16 * tid;
            q[(j + 8) % 9] = *reinterpret_cast<const float4 *>(rb + j * HALO);
            const float ez = spg ? __ldg(A.E[0] + z) : 0.f;
            const float *pr = reinterpret_cast<const float *>(cur);
            const float4 L = ld4g(pr - 4), C = ld4g(pr), R = ld4g(pr + 4);
            float4 yv[9];
#pragma unroll
            for (int m = 0; m < 9; m++) yv[m] = m == 4 ? C : ld4g(pr + (m - 4) * SW);
            const float4 pp4 = *reinterpret_cast<const float4 *>(own), ch4 = *reinterpret_cast<const float4 *>(own + OWN);
            const Cells4 cu = cells4(L, C, R, yv, q[j % 9], q[(j + 1) % 9], q[(j + 2) % 9], q[(j + 3) % 9], q[(j + 5) % 9],
                                     q[(j + 6) % 9], q[(j + 7) % 9], q[(j + 8) % 9], pp4, ch4, spg, ez + Ey, Ex4);
            float res[4], qk[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                res[k] = cu.res[k];
                const float es = spg ? ez + Ey + lane4(Ex4, k) : 0.f;
                qk[k] = es * (res[k] - lane4(pp4, k)) - cu.rhs[k];
            }
            if (add.xy | zadd) {
                cp_wait<1>();
                const float4 *const v = aslot + (j & 1) * 3 * NTH;
                if (add.xy) AddRows::add(v[0], ch4, res, qk);
                if (zadd) AddRows::add(v[2 * NTH], ch4, res, qk);
                if (add.xy) AddRows::add(v[NTH], ch4, res, qk);
            }
            if (xedge) {
#pragma unroll
                for (int k = 0; k < 4; k++)
                    if (gx0 + k >= g.NX) res[k] = 0.f;
            }
            if (g.fs && z == 0) res[0] = res[1] = res[2] = res[3] = 0.f;
            if (live) {
                *reinterpret_cast<float4 *>(out) = make_float4(res[0], res[1], res[2], res[3]);
                if (MODE == kModeRecord) *reinterpret_cast<float4 *>(qs + orow) = make_float4(qk[0], qk[1], qk[2], qk[3]);
                if (MODE == kModeAdjoint) {
                    ga.x += res[0] * qa.x;
                    ga.y += res[1] * qa.y;
                    ga.z += res[2] * qa.z;
                    ga.w += res[3] * qa.w;
                    *reinterpret_cast<float4 *>(Gs + orow) = ga;
                }
            }
            out += PP;
            if (MODE != kModeForward) orow += PP;
            __syncthreads();  // every thread is done with plane z's slots before they are restaged
        }
        // plane zz + 4 + m back to q[(m + 4) % 9] for the next block
        const float4 t0 = q[0], t1 = q[1], t2 = q[2];
#pragma unroll
        for (int k = 0; k < 5; k++) q[k] = q[k + 4];
        q[5] = t0;
        q[6] = t1;
        q[7] = t2;
        const unsigned t = ha;
        ha = hb;
        hb = t;
        par ^= 1;
    }
    cp_wait<0>();  // no copy outlives the thread
    // a leader that waited for every group knows that its copies have landed;
    // one that gave up waits (bounded) for those still in flight: the group it
    // gave up on and the AHEAD it had staged beyond (or the first planes')
    if (zbad < ze) {
        atomicOr(A.flags, kFlagTimeout);
        if (tid == 0) {
            if (zbad < zb) mbar_wait(bar0 + 8 * NSO, 0, spin);
            for (int z = max(zbad, zb); z < min(ze, max(zbad, zb) + AHEAD + 1); z++)
                mbar_wait(bar0 + 8 * ((z - zb) % NSO), ((z - zb) / NSO) & 1, spin);
        }
    }
    __syncthreads();
    // the source corners among the cells this CTA has written
    if (MODE != kModeAdjoint && src && tid < 8 && src[shot].cell[tid] >= 0) {
        const long long o = src[shot].cell[tid], r = o - g.org;
        const int z = (int)(r / PP), y = (int)(r % PP / g.P), x = (int)(r % g.P);
        if (x >= x0 && x < x0 + TW && y >= y0 && y < y0 + TY && z >= zb && z < ze)
            inject3(A, src[shot], tid, shot, n, row, MODE == kModeRecord ? qs : nullptr);
    }
}

// ---------------------------------------------------------------- points (3D)

// point sources into p^{n+1} (one thread per shot and corner). The TMA march
// injects on its own.
__global__ void k_inject3d(const StepArgs<float> A, const int n, const int row, const Pt3 *src, int nshots, float *qs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 8 * nshots && src[i >> 3].cell[i & 7] >= 0) inject3(A, src[i >> 3], i & 7, i >> 3, n, row, qs);
}

// The adjoint sweep's injection: residuals into u^{n+1} by target cell
// (deterministic order of the entries of a cell), the cell's G gaining the
// injected part.
__global__ void k_inj3d(const StepArgs<float> A, const int n, const int row, const Inj3 *grp, const int ngrp,
                        const InjE3 *ent, const float *qs, float *Gs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ngrp || row < 0 || row >= A.nt) return;
    const Inj3 G = grp[i];
    const int shot = blockIdx.y;
    const Geom &g = A.g;
    const SimIO *io = A.io;
    const float *r = static_cast<const float *>(io->resid) + ((long long)shot * A.nt + row) * io->nrec;
    float sum = 0.f;
    for (int e = G.e0; e < G.e1; e++) sum += ent[e].w * r[ent[e].pt];
    const long long o = G.cell, so = (long long)shot * g.fstride + o;
    float es = 0.f;
    if (A.bc == SIM_BC_SPONGE) {
        const long long r = o - g.org, PP = (long long)g.PY * g.P;
        const int z = (int)(r / PP), y = (int)((r % PP) / g.P), x = (int)(r % g.P);
        es = A.E[0][z] + A.E[1][y] + A.E[2][x];
    }
    const float chv = A.ch[o];
    const float d = chv * A.src_scale * sum / (1.f + chv * es);
    A.pbuf[(n + 1) & 1][so] += d;
    Gs[so] += d * qs[so];
}

// interior of p^n into the snapshot stack (FP32), or its max |p| (FP16 pass 1)
__global__ void k_snap3d(const StepArgs<float> A, const StepTime t, int pass) {
    const Geom &g = A.g;
    const int shot = blockIdx.y;
    const float *p = A.pbuf[t.n & 1] + (long long)shot * g.fstride;
    const long long nint = (long long)g.nz * g.ny * g.nx;
    const SimIO *io = A.io;
    const long long base = ((long long)shot * A.nsnap + t.snap_k) * nint;
    const float s = (pass == 2) ? pow2_scale(__uint_as_float(io->snap_max[shot * A.nsnap + t.snap_k])) : 1.f;
    float m = 0.f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nint; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % g.nx);
        const long long zy = i / g.nx;
        const int y = (int)(zy % g.ny), z = (int)(zy / g.ny);
        const float v = p[cell_off(g, z + g.oz, y + g.oy, x + g.ox)];
        if (pass == 0) static_cast<float *>(io->snaps)[base + i] = v;
        else if (pass == 1) m = fmaxf(m, fabsf(v));
        else static_cast<__half *>(io->snaps)[base + i] = __float2half_rn(v / s);
    }
    if (pass == 1) {
        m = warp_max(m);
        if ((threadIdx.x & 31) == 0) {
            if (!(m <= FLT_MAX)) atomicOr(A.flags, kFlagUnstable);
            else atomicMax(&io->snap_max[shot * A.nsnap + t.snap_k], __float_as_uint(m));
        }
    }
    if (pass == 2 && blockIdx.x == 0 && threadIdx.x == 0) io->snap_scale[shot * A.nsnap + t.snap_k] = s;
}

template <int RY>
size_t smem3d() {
    return (size_t)NS3 * slot3d<RY>() * sizeof(float);
}

}  // namespace


// Tensor maps of one launch (host): the pressure buffers pbuf[0] (both
// parities of max_shots shots, fstride apart) and c, in the padded layout.
cudaError_t make_maps(const StepArgs<float> &a, int tw, Tma3 &m) {
    static PFN_cuTensorMapEncodeTiled_v12000 enc = nullptr;
    if (!enc) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return cudaErrorNotSupported;
        enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const Geom &g = a.g;
    const long long ms = (a.pbuf[1] - a.pbuf[0]) / g.fstride;
    const long long planes = g.fstride / ((long long)g.PY * g.P);
    // x extent: the ghost columns left of the grid, the grid and the 4 columns
    // of the last cells' halo; columns past it (the padding of the last x tile,
    // all zeros) come as the copy's zero fill instead of DRAM reads
    const cuuint64_t nxt = std::min<cuuint64_t>((cuuint64_t)g.P, (cuuint64_t)(kGhost + g.NX + 4));
    const cuuint64_t dims[4] = {nxt, (cuuint64_t)g.PY, (cuuint64_t)planes, (cuuint64_t)(2 * ms)};
    const cuuint64_t strides[3] = {(cuuint64_t)g.P * 4, (cuuint64_t)g.PY * g.P * 4, (cuuint64_t)g.fstride * 4};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    const cuuint32_t w = (cuuint32_t)tw, r = NW * TX / w, bh[4] = {w + 8, r + 8, 1, 1}, bo[4] = {w, r, 1, 1};
    CUresult q = enc(&m.ph, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.pbuf[0], dims, strides, bh, one,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (q == CUDA_SUCCESS)
        q = enc(&m.po, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.pbuf[0], dims, strides, bo, one,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (q == CUDA_SUCCESS)
        q = enc(&m.c, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(a.ch), dims, strides, bo, one,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return q == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int TW>
cudaError_t configure_tma() {
    cudaError_t e = cudaSuccess;
    for (auto k : {k_step3d_tma<kModeForward, TW>, k_step3d_tma<kModeRecord, TW>, k_step3d_tma<kModeAdjoint, TW>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile3<TW>::SMEM);
    return e;
}

cudaError_t configure_step3d() {
    cudaError_t e = configure_tma<64>();
    if (e == cudaSuccess) e = configure_tma<32>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step3d<1, kModeForward>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem3d<1>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step3d<1, kModeRecord>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem3d<1>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step3d<1, kModeAdjoint>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem3d<1>());
    return e;
}

template <int RY, int MODE>
cudaError_t launch_step3d_mode(cudaLaunchConfig_t &cfg, const StepArgs<float> &a, int n, int zchunk, const Add3 &D,
                               float *qs, float *Gs) {
    cfg.dynamicSmemBytes = smem3d<RY>();
    return cudaLaunchKernelEx(&cfg, k_step3d<RY, MODE>, a, n, zchunk, D, qs, Gs);
}

template <int TW>
cudaError_t launch_tma(cudaLaunchConfig_t &cfg, const StepArgs<float> &a, int n, int zchunk, int mode, const Add3 &D,
                       const Pt3 *src, int row, float *qs, float *Gs) {
    Tma3 m;
    if (cudaError_t e = make_maps(a, TW, m)) return e;
    cfg.gridDim.x = (a.g.NX + TW - 1) / TW;
    cfg.gridDim.y = (a.g.NY + Tile3<TW>::TY - 1) / Tile3<TW>::TY;
    cfg.dynamicSmemBytes = Tile3<TW>::SMEM;
    const int ms = (int)((a.pbuf[1] - a.pbuf[0]) / a.g.fstride);
    const int spin = 1 << 22;
    if (mode == kModeRecord)
        return cudaLaunchKernelEx(&cfg, k_step3d_tma<kModeRecord, TW>, a, m, n, zchunk, ms, D, src, row, qs, Gs, spin);
    if (mode == kModeAdjoint)
        return cudaLaunchKernelEx(&cfg, k_step3d_tma<kModeAdjoint, TW>, a, m, n, zchunk, ms, D, src, row, qs, Gs, spin);
    return cudaLaunchKernelEx(&cfg, k_step3d_tma<kModeForward, TW>, a, m, n, zchunk, ms, D, src, row, qs, Gs, spin);
}

cudaError_t launch_step3d(const StepArgs<float> &a, int n, const ZShape &zs, int nshots, cudaStream_t st, bool pdl, int mode,
                          const Add3 &D, const Pt3 *src, int row, float *qs, float *Gs) {
    const int zchunk = zs.chunk, nchunk = (a.g.NZ + zchunk - 1) / zchunk;
    if (row < 0 || row >= a.nt) src = nullptr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.ntx, (a.g.NY + NW - 1) / NW, nchunk * nshots);
    cfg.blockDim = dim3(NTH);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    if (zs.variant != kZMarchAsync)
        return zs.tile == 32 ? launch_tma<32>(cfg, a, n, zchunk, mode, D, src, row, qs, Gs)
                             : launch_tma<64>(cfg, a, n, zchunk, mode, D, src, row, qs, Gs);
    cudaError_t e = mode == kModeRecord    ? launch_step3d_mode<1, kModeRecord>(cfg, a, n, zchunk, D, qs, Gs)
                    : mode == kModeAdjoint ? launch_step3d_mode<1, kModeAdjoint>(cfg, a, n, zchunk, D, qs, Gs)
                                           : launch_step3d_mode<1, kModeForward>(cfg, a, n, zchunk, D, qs, Gs);
    if (e != cudaSuccess || !src) return e;
    k_inject3d<<<(8 * nshots + 63) / 64, 64, 0, st>>>(a, n, row, src, nshots, mode == kModeRecord ? qs : nullptr);
    return cudaGetLastError();
}

cudaError_t launch_inj3d(const StepArgs<float> &a, int n, int row, const Inj3 *grp, int ngrp, const InjE3 *ent,
                         int nshots, const float *qs, float *Gs, cudaStream_t st) {
    if (ngrp <= 0) return cudaSuccess;
    k_inj3d<<<dim3((ngrp + 127) / 128, nshots), 128, 0, st>>>(a, n, row, grp, ngrp, ent, qs, Gs);
    return cudaGetLastError();
}

cudaError_t launch_snap3d(const StepArgs<float> &a, const StepTime &t, int fp16, int nshots, cudaStream_t st) {
    if (fp16) {
        k_snap3d<<<dim3(608, nshots), 256, 0, st>>>(a, t, 1);
        k_snap3d<<<dim3(608, nshots), 256, 0, st>>>(a, t, 2);
    } else {
        k_snap3d<<<dim3(608, nshots), 256, 0, st>>>(a, t, 0);
    }
    return cudaGetLastError();
}

}  // namespace gsim
