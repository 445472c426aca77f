// CPML memory terms of the 3D step, every axis in one launch before the
// z-march (fwd3d.cu): psi^n and zeta^n on the strips, and the addend
// D1 psi^n + zeta^n of each axis on its strip widened by 4 cells, written to
// a compact array that the march adds (Add3):
//   psi^n  = b psi^{n-1}  + a D1 p^n
//   zeta^n = b zeta^{n-1} + a (D2 p^n + D1 psi^n)
//   p^{n+1} = (plain update) + c (addend of x) + c (addend of z) + c (addend of y)
// and, for the adjoint sweep, the multipliers nu and mu and the bracket
// -D1 (a mu) + D2 (a nu) (cpml_adj.cu states the recursions).
//
// Bound by HBM on volumes larger than L2 and by latency below that. One pass
// per axis after the march (a thread walking one column of a strip, reading
// c and reading and writing p^{n+1} once more per axis) cost 0.88 ms of a
// 3.17 ms step of 649 x 1060 x 1060 cells and, three short launches of 150 to
// 370 CTAs each, 104 of 225 us at 170 x 227 x 273 x 2 shots. This launch takes
// 62 us there, and the march pays the addends' read.
// Here a block owns all rows of one strip range for 128 columns at one
// position of the third axis (z and y axes: k_cpml3d's column blocks), so
// psi can be updated in place; its warps take runs of rows, with register
// windows along the axis; x strips go by blocks of row ends. Strips these do not take (columns of more than kColRows rows, a z
// range within reach of a free surface, x strips over 44 cells or close
// together) go through k_psi3d + k_add3d, one thread per four cells.
#include <algorithm>

#include "f32_tile.cuh"
#include "sim_internal.h"
#include "stencil.cuh"

namespace gsim {
namespace {

using f32::ld4;
using f32::st4;

constexpr int kColRows = 72;   // longest widened range of a column block
constexpr int NT = 128;        // threads per block
constexpr int CW = 128;        // cells across a column block
constexpr int kRowEnds = 64;   // row ends per block
constexpr int kMaxQ = 12;      // float4s of a widened x strip end

__device__ __forceinline__ float lane4(const float4 &v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}
// 16-byte copy that writes zeros (reads nothing) when v is false
__device__ __forceinline__ void cp16z(float *dst, const float *gmem, bool v) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(gmem), "r"(v ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ long long axis_stride(const Geom &g, int ax) {
    return ax == 0 ? (long long)g.PY * g.P : (ax == 1 ? (long long)g.P : 1LL);
}
// the float4 starting at cell x holds x-strip cells
__device__ __forceinline__ bool xstrip4(const Geom &g, int x) {
    return x + 3 >= 0 && x < g.NX && ((g.nbx0 > 0 && x < g.nbx0) || (g.nbx1 > 0 && x + 3 >= g.NX - g.nbx1));
}

// second differences along x of the four cells C from the row's float4s L, C, R
__device__ __forceinline__ void d2x_pairs(const float4 &L, const float4 &C, const float4 &R, float2 &da, float2 &db) {
    const float2 v34 = make_float2(L.w, C.x), v56 = make_float2(C.y, C.z), v12 = make_float2(L.y, L.z),
                 v78 = make_float2(C.w, R.x), v910 = make_float2(R.y, R.z);
    da = d2c2(lo2(C), v34, v56, hi2(L), hi2(C), v12, v78, lo2(L), lo2(R));
    db = d2c2(hi2(C), v56, v78, lo2(C), lo2(R), v34, v910, hi2(L), hi2(R));
}

// ---------------------------------------------------------------- plan of one launch

struct ColRanges {
    int n;            // ranges (0 to 2)
    int s0[2], s1[2]; // [s0, s1) along the axis: the strips widened by 4
};
struct XEnds {
    int ne;            // strip ends (0 to 2)
    int xa[2], nq[2];  // 8 cells before the widened strip (a multiple of 4), its float4s
};
struct Plan3 {
    Add3 D;
    ColRanges c[2];           // z, y
    XEnds E;                  // x
    int nbr[2];               // column blocks per range of z and y
    int nb[3];                // column blocks of z and y, blocks of x row ends
    int nbx;                  // blocks per strip end of x
    long long xrows;          // rows (z, y) of the x axis
    const Pt3 *rec;           // receivers sampled by the launch's last blocks (p^n into the gather)
    int nrec, nbs;
};

// ---------------------------------------------------------------- columns (z and y axes)

// Rows [i0, i1) of the block's L that warp w takes.
__device__ __forceinline__ void warp_rows(int L, int w, int &i0, int &i1) {
    i0 = L * w / (NT / 32);
    i1 = L * (w + 1) / (NT / 32);
}

// A column block: rows s0 .. s1 - 1 of axis ax (0: z, 1: y) of 32 consecutive
// float4 columns, counted along x and then along the third axis (no lane is
// lost to a ragged x extent). Forward: f = p^n, m0 = psi, m1 = zeta; adjoint:
// f = u^{k+1}, m0 = nu, m1 = mu. Both memory fields are updated in place.
template <bool ADJ>
__device__ __forceinline__ void col_block(const StepArgs<float> &A, const Plan3 &Q, int ax, int k, int blk,
                                          const float *f, float *m0, float *m1, float *add, float *sm) {
    const Geom &g = A.g;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nx4 = (g.NX + 3) >> 2, nu = ax == 0 ? g.NY : g.NZ;
    const int col = min(32 * blk + lane, nx4 * nu - 1), u = col / nx4, x = 4 * (col - u * nx4);
    const bool act = 32 * blk + lane < nx4 * nu && !(g.fs && ax == 1 && u == 0);  // the free-surface row stays zero
    const int N = ax == 0 ? g.NZ : g.NY, lo = ax == 0 ? g.nbz0 : g.nby0, hi = ax == 0 ? g.nbz1 : g.nby1;
    const long long s = axis_stride(g, ax);
    const int s0 = Q.c[ax].s0[k], s1 = Q.c[ax].s1[k], L = s1 - s0;
    const long long o0 = ax == 0 ? cell_off(g, 0, u, x) : cell_off(g, u, 0, x);  // row 0 of the column
    f += o0, m0 += o0, m1 += o0;
    const float *ca = A.ca[ax], *cb = A.cb[ax];
    auto strip = [&](int r) { return (lo > 0 && r >= 0 && r < lo) || (hi > 0 && r >= N - hi && r < N); };
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    constexpr int FH = ADJ ? 4 : 8;       // rows of f beyond the range
    float *F = sm + 4 * lane;             // L + 2 FH rows of f from s0 - FH
    float *S = F + (L + 2 * FH) * CW;     // L + 8 rows of m0 from s0 - 4, zero off the strip
    float *Z = S + (L + 8) * CW;          // forward: L rows of m1 from s0; adjoint: L + 8 from s0 - 4
    constexpr int ZH = ADJ ? 4 : 0, NWB = NT / 32;
    {   // rows w, w + NWB, ...: pointers advance by a stride
        const float *p = f + (s0 - FH + w) * s;
        for (int i = w; i < L + 2 * FH; i += NWB, p += NWB * s) cp16z(F + i * CW, p, act);
        const long long o = (s0 - 4 + w) * s;
        const float *p0 = m0 + o, *p1 = m1 + o;
        for (int i = w; i < L + 8; i += NWB, p0 += NWB * s, p1 += NWB * s) {
            const bool in = i >= 4 && i < L + 4;
            float *const z = Z + (i - 4 + ZH) * CW;
            if (in && strip(s0 - 4 + i)) {
                cp16z(S + i * CW, p0, act);
                cp16z(z, p1, act);
            } else {
                st4(S + i * CW, zero);
                if (ADJ || in) st4(z, zero);
            }
        }
    }
    f32::cp_async_wait_all();
    __syncthreads();
    int i0, i1;
    warp_rows(L, w, i0, i1);
    // the thread's rows of the memory fields and of the addend (a range's slots are consecutive)
    float *q0 = m0 + (s0 + i0) * s, *q1 = m1 + (s0 + i0) * s;
    const int l1 = ax == 0 ? Q.D.zl : Q.D.yl, h0 = ax == 0 ? Q.D.zh : Q.D.yh, r0 = s0 + i0;
    const int slot = r0 < l1 ? r0 : l1 + r0 - h0;
    const long long as = ax == 0 ? (long long)g.NY * g.P : g.P;
    float *out = add + (ax == 0 ? (long long)slot * g.NY + u : (long long)u * Q.D.nyw + slot) * g.P + x;

    // Rows i0 .. i1 - 1, blocks of 9 unrolled: the 9-row register windows W (rows
    // i .. i + 8 of the array at w0) and V (v0; NULL: none) rotate by renaming.
    // fn(i, place of row i's window) reads W[(k + m) % 9].
    float4 W[9], V[9];
    auto windows = [&](const float *w0, const float *v0, auto fn) {
#pragma unroll
        for (int m = 0; m < 8; m++) {
            W[m] = ld4(w0 + (i0 + m) * CW);
            if (v0) V[m] = ld4(v0 + (i0 + m) * CW);
        }
        for (int ib = i0; ib < i1; ib += 9) {
#pragma unroll
            for (int k = 0; k < 9; k++) {
                const int i = ib + k;
                if (i >= i1) break;
                W[(k + 8) % 9] = ld4(w0 + (i + 8) * CW);
                if (v0) V[(k + 8) % 9] = ld4(v0 + (i + 8) * CW);
                fn(i, k);
            }
        }
    };
    auto d1 = [](const float4 *X, int k, float2 &da, float2 &db) {
        f32::d1_pairs(X[k % 9], X[(k + 1) % 9], X[(k + 2) % 9], X[(k + 3) % 9], X[(k + 5) % 9], X[(k + 6) % 9],
                      X[(k + 7) % 9], X[(k + 8) % 9], da, db);
    };
    auto d2 = [](const float4 *X, int k, float2 &da, float2 &db) {
        const float4 &c = X[(k + 4) % 9], &m1 = X[(k + 3) % 9], &p1 = X[(k + 5) % 9], &m2 = X[(k + 2) % 9],
                     &p2 = X[(k + 6) % 9], &m3 = X[(k + 1) % 9], &p3 = X[(k + 7) % 9], &m4 = X[k % 9], &p4 = X[(k + 8) % 9];
        da = d2c2(lo2(c), lo2(m1), lo2(p1), lo2(m2), lo2(p2), lo2(m3), lo2(p3), lo2(m4), lo2(p4));
        db = d2c2(hi2(c), hi2(m1), hi2(p1), hi2(m2), hi2(p2), hi2(m3), hi2(p3), hi2(m4), hi2(p4));
    };
    if (!ADJ) {
        windows(F + 4 * CW, nullptr, [&](int i, int k) {  // psi^n of row r
            const int r = s0 + i;
            if (strip(r)) {
                const float a = __ldg(ca + r), b = __ldg(cb + r);
                float2 da, db;
                d1(W, k, da, db);
                const float4 old = ld4(S + (i + 4) * CW);
                const float2 pa = f32::rec2(splat2(a), da, splat2(b), lo2(old));
                const float2 pb = f32::rec2(splat2(a), db, splat2(b), hi2(old));
                const float4 ps = make_float4(pa.x, pa.y, pb.x, pb.y);
                st4(S + (i + 4) * CW, ps);
                if (act) st4(q0, ps);
            }
            q0 += s;
        });
        __syncthreads();
        windows(F + 4 * CW, S, [&](int i, int k) {  // zeta^n and the addend of row r
            const int r = s0 + i;
            float a = 0.f, b = 0.f;
            const bool in = strip(r);
            if (in) {
                a = __ldg(ca + r);
                b = __ldg(cb + r);
            }
            const float4 zo = ld4(Z + i * CW);
            float2 d2a, d2b, dsa, dsb;
            d2(W, k, d2a, d2b);
            d1(V, k, dsa, dsb);
            const float2 za = f32::rec2(splat2(a), add2(d2a, dsa), splat2(b), lo2(zo));
            const float2 zb = f32::rec2(splat2(a), add2(d2b, dsb), splat2(b), hi2(zo));
            if (act) {
                if (in) st4(q1, make_float4(za.x, za.y, zb.x, zb.y));
                const float2 aa = add2(dsa, za), ab = add2(dsb, zb);
                st4(out, make_float4(aa.x, aa.y, ab.x, ab.y));
            }
            q1 += s;
            out += as;
        });
    } else {
        // nu^k = b nu + u of the strip rows (S then holds a nu^k), w = u + a nu^k (F)
        for (int i = i0; i < i1; i++, q0 += s) {
            const int r = s0 + i;
            if (!strip(r)) continue;
            const float a = __ldg(ca + r), b = __ldg(cb + r);
            const float4 uo = ld4(F + (i + 4) * CW), no = ld4(S + (i + 4) * CW);
            const float2 na = fma2(splat2(b), lo2(no), lo2(uo)), nb = fma2(splat2(b), hi2(no), hi2(uo));
            if (act) st4(q0, make_float4(na.x, na.y, nb.x, nb.y));
            const float2 pa = mul2(splat2(a), na), pb = mul2(splat2(a), nb);
            st4(S + (i + 4) * CW, make_float4(pa.x, pa.y, pb.x, pb.y));
            const float2 wa = add2(lo2(uo), pa), wb = add2(hi2(uo), pb);
            st4(F + (i + 4) * CW, make_float4(wa.x, wa.y, wb.x, wb.y));
        }
        __syncthreads();
        windows(F, nullptr, [&](int i, int k) {  // mu^k = b mu - D1 w of the strip rows (Z then holds a mu^k)
            const int r = s0 + i;
            if (strip(r)) {
                const float a = __ldg(ca + r), b = __ldg(cb + r);
                float2 da, db;
                d1(W, k, da, db);
                const float4 mo = ld4(Z + (i + 4) * CW);
                const float2 ma = fma2(splat2(b), lo2(mo), neg2(da)), mb = fma2(splat2(b), hi2(mo), neg2(db));
                if (act) st4(q1, make_float4(ma.x, ma.y, mb.x, mb.y));
                const float2 pa = mul2(splat2(a), ma), pb = mul2(splat2(a), mb);
                st4(Z + (i + 4) * CW, make_float4(pa.x, pa.y, pb.x, pb.y));
            }
            q1 += s;
        });
        __syncthreads();
        windows(S, Z, [&](int, int k) {  // the bracket D2 (a nu) - D1 (a mu)
            float2 d2a, d2b, dsa, dsb;
            d2(W, k, d2a, d2b);
            d1(V, k, dsa, dsb);
            const float2 ea = add2(d2a, neg2(dsa)), eb = add2(d2b, neg2(dsb));
            if (act) st4(out, make_float4(ea.x, ea.y, eb.x, eb.y));
            out += as;
        });
    }
}

// ---------------------------------------------------------------- row ends (x axis)
//
// A block takes kRowEnds consecutive (z, y) rows at one strip end. All their
// f, m0 and m1 (the memory fields on strip cells, zeros elsewhere) are staged
// by cp.async first; then each phase deals the rows' float4s out to all
// threads (a half-warp per row end kept 6 to 9 of 16 lanes busy and formed
// each row's addresses in every lane: 530 instructions per pair of ends).
// Lane index j of a row end: cells xa + 4 j, j in [0, nq + 4); the strip's
// float4s update the memory fields, j in [2, nq + 2) write the addend.
template <bool ADJ>
__device__ __forceinline__ void row_ends(const StepArgs<float> &A, const Plan3 &Q, int blk, const float *f, float *m0,
                                         float *m1, float *add, float *sm) {
    const Geom &g = A.g;
    const int e = blk >= Q.nbx, xa = e ? Q.E.xa[1] : Q.E.xa[0], nq = e ? Q.E.nq[1] : Q.E.nq[0], J = nq + 4;
    const long long r0 = (long long)(blk - e * Q.nbx) * kRowEnds;
    const int rows = (int)min((long long)kRowEnds, Q.xrows - r0);
    long long *const base = reinterpret_cast<long long *>(sm);        // field offset of the row's cell xa; -1: held row
    float *const F = sm + 2 * kRowEnds, *const S = F + kRowEnds * J * 4, *const Z = S + kRowEnds * J * 4;
    const int tid = threadIdx.x;
    if (tid < rows) {
        const unsigned row = (unsigned)(r0 + tid), z = row / (unsigned)g.NY, y = row - z * (unsigned)g.NY;
        base[tid] = g.fs && z == 0 ? -1 : cell_off(g, (int)z, (int)y, xa);  // the free-surface row stays zero
    }
    __syncthreads();
    // the strip's float4s: j in [j0, j1)
    int j0 = J, j1 = 0;
    for (int j = 1; j < nq + 3; j++)
        if (xstrip4(g, xa + 4 * j)) j0 = min(j0, j), j1 = j + 1;
    const int ns = max(0, j1 - j0);
    // fn(row, float4 m of its n) over the block's rows, dealt out to the threads
    auto deal = [&](int n, auto fn) {
        if (n <= 0) return;
        const int dr = NT / n, dm = NT - dr * n;
        int r = tid / n, m = tid - r * n;
        while (r < rows) {
            fn(r, m);
            r += dr;
            m += dm;
            if (m >= n) m -= n, r++;
        }
    };
    deal(J, [&](int r, int j) {
        const int i = 4 * (r * J + j);
        const long long o = base[r];
        const bool in = o >= 0, st = in && j >= j0 && j < j1;
        const long long p = (in ? o : 0) + 4 * j;
        cp16z(F + i, f + p, in);
        cp16z(S + i, m0 + p, st);
        cp16z(Z + i, m1 + p, st);
    });
    f32::cp_async_wait_all();
    __syncthreads();
    const float *const ca = A.ca[2] + xa, *const cb = A.cb[2] + xa;
    float *const ad = add + r0 * Q.D.nxw + (xa + 8 < Q.D.xl ? xa + 8 : Q.D.xl + xa + 8 - Q.D.xs);  // the first row's float4 2
    if (!ADJ) {
        deal(ns, [&](int r, int m) {  // psi^n
            const int j = j0 + m;
            const long long o = base[r];
            if (o < 0) return;
            const float *p = F + 4 * (r * J + j);
            float *s = S + 4 * (r * J + j);
            const float4 a4 = ld4(ca + 4 * j), b4 = ld4(cb + 4 * j), old = ld4(s);
            float2 da, db;
            f32::d1x_pairs(ld4(p - 4), ld4(p), ld4(p + 4), da, db);
            const float2 pa = f32::rec2(lo2(a4), da, lo2(b4), lo2(old)), pb = f32::rec2(hi2(a4), db, hi2(b4), hi2(old));
            const float4 ps = make_float4(pa.x, pa.y, pb.x, pb.y);
            st4(s, ps);
            st4(m0 + o + 4 * j, ps);
        });
        __syncthreads();
        deal(nq, [&](int r, int m) {  // zeta^n and the addend
            const int j = 2 + m;
            const long long o = base[r];
            if (o < 0) return;
            const float *p = F + 4 * (r * J + j), *s = S + 4 * (r * J + j);
            const bool in = j >= j0 && j < j1;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 a4 = in ? ld4(ca + 4 * j) : zero, b4 = in ? ld4(cb + 4 * j) : zero, zo = ld4(Z + 4 * (r * J + j));
            float2 xd, yd, da, db;
            d2x_pairs(ld4(p - 4), ld4(p), ld4(p + 4), xd, yd);
            f32::d1x_pairs(ld4(s - 4), ld4(s), ld4(s + 4), da, db);
            const float2 za = f32::rec2(lo2(a4), add2(xd, da), lo2(b4), lo2(zo));
            const float2 zb = f32::rec2(hi2(a4), add2(yd, db), hi2(b4), hi2(zo));
            if (in) st4(m1 + o + 4 * j, make_float4(za.x, za.y, zb.x, zb.y));
            const float2 aa = add2(da, za), ab = add2(db, zb);
            st4(ad + r * Q.D.nxw + 4 * m, make_float4(aa.x, aa.y, ab.x, ab.y));
        });
    } else {
        deal(ns, [&](int r, int m) {  // nu^k (S then holds a nu^k) and w = u + a nu^k (F)
            const int j = j0 + m;
            const long long o = base[r];
            if (o < 0) return;
            float *p = F + 4 * (r * J + j), *s = S + 4 * (r * J + j);
            const float4 a4 = ld4(ca + 4 * j), b4 = ld4(cb + 4 * j), u = ld4(p), old = ld4(s);
            const float2 na = fma2(lo2(b4), lo2(old), lo2(u)), nb = fma2(hi2(b4), hi2(old), hi2(u));
            st4(m0 + o + 4 * j, make_float4(na.x, na.y, nb.x, nb.y));
            const float2 pa = mul2(lo2(a4), na), pb = mul2(hi2(a4), nb);
            st4(s, make_float4(pa.x, pa.y, pb.x, pb.y));
            const float2 wa = add2(lo2(u), pa), wb = add2(hi2(u), pb);
            st4(p, make_float4(wa.x, wa.y, wb.x, wb.y));
        });
        __syncthreads();
        deal(ns, [&](int r, int m) {  // mu^k (Z then holds a mu^k)
            const int j = j0 + m;
            const long long o = base[r];
            if (o < 0) return;
            const float *p = F + 4 * (r * J + j);
            float *t = Z + 4 * (r * J + j);
            const float4 a4 = ld4(ca + 4 * j), b4 = ld4(cb + 4 * j), mo = ld4(t);
            float2 da, db;
            f32::d1x_pairs(ld4(p - 4), ld4(p), ld4(p + 4), da, db);
            const float2 ma = fma2(lo2(b4), lo2(mo), neg2(da)), mb = fma2(hi2(b4), hi2(mo), neg2(db));
            st4(m1 + o + 4 * j, make_float4(ma.x, ma.y, mb.x, mb.y));
            const float2 pa = mul2(lo2(a4), ma), pb = mul2(hi2(a4), mb);
            st4(t, make_float4(pa.x, pa.y, pb.x, pb.y));
        });
        __syncthreads();
        deal(nq, [&](int r, int m) {  // the bracket
            const int j = 2 + m;
            if (base[r] < 0) return;
            const float *s = S + 4 * (r * J + j), *t = Z + 4 * (r * J + j);
            float2 xd, yd, da, db;
            d2x_pairs(ld4(s - 4), ld4(s), ld4(s + 4), xd, yd);
            f32::d1x_pairs(ld4(t - 4), ld4(t), ld4(t + 4), da, db);
            const float2 ea = add2(xd, neg2(da)), eb = add2(yd, neg2(db));
            st4(ad + r * Q.D.nxw + 4 * m, make_float4(ea.x, ea.y, eb.x, eb.y));
        });
    }
}

// receivers: p^n into row n of the gather
__device__ __forceinline__ void sample3(const StepArgs<float> &A, const Plan3 &Q, int n, int r, int shot, const float *p) {
    if (r >= Q.nrec) return;
    const Pt3 P = Q.rec[r];
    float v = 0.f;
#pragma unroll
    for (int c = 0; c < 8; c++)
        if (P.cell[c] >= 0) v += P.w[c] * p[P.cell[c]];
    static_cast<float *>(A.io->gather)[((long long)shot * A.nt + n) * Q.nrec + r] = v;
    if (!isfinite(v)) atomicOr(A.flags, kFlagUnstable);
}

// Memory fields of the axes: forward psi, zeta; adjoint nu, mu.
struct Mem3 {
    const float *f;  // p^n, or u^{k+1}
    float *m0[3], *m1[3];
};

template <bool ADJ>
__global__ void __launch_bounds__(NT, 4) k_cpml3d(const StepArgs<float> A, const Plan3 Q, const Mem3 M, const int n) {
    extern __shared__ float4 sm4[];
    const int shot = blockIdx.y;
    const long long sh = (long long)shot * A.g.fstride;
    int b = blockIdx.x;
    cudaGridDependencySynchronize();
#pragma unroll
    for (int ax = 0; ax < 2; ax++) {
        if (b < Q.nb[ax]) {
            const int k = b >= Q.nbr[ax];
            col_block<ADJ>(A, Q, ax, k, b - k * Q.nbr[ax], M.f + sh, M.m0[ax] + sh, M.m1[ax] + sh,
                           Q.D.a[ax] + shot * Q.D.st[ax], reinterpret_cast<float *>(sm4));
            return;
        }
        b -= Q.nb[ax];
    }
    if (b < Q.nb[2]) {
        row_ends<ADJ>(A, Q, b, M.f + sh, M.m0[2] + sh, M.m1[2] + sh, Q.D.a[2] + shot * Q.D.st[2],
                      reinterpret_cast<float *>(sm4));
        return;
    }
    if (!ADJ) sample3(A, Q, n, (b - Q.nb[2]) * NT + threadIdx.x, shot, M.f + sh);
}

// ---------------------------------------------------------------- other strip layouts (forward)
//
// One thread per float4 column: psi on the strips first (k_psi3d), then zeta
// and the addend on the widened strips (k_add3d). A box's x-range is rounded
// out to multiples of 4 (cells so added lie outside the strips, where both
// recursion coefficients are zero, or beyond the grid, where c is zero, so
// they stay zero and add nothing). Item i of a box is float4 column i mod C
// of row i / C, rows ordered (z, y).
struct Box {
    int z0, z1, y0, y1, x0, x1;
};
__device__ __forceinline__ bool box_item(const Box &b, long long i, int &z, int &y, int &x) {
    const int nc = (b.x1 - b.x0) >> 2, ny = b.y1 - b.y0;
    if (nc <= 0 || ny <= 0) return false;
    const long long row = i / nc;
    x = b.x0 + 4 * (int)(i - row * nc);
    y = b.y0 + (int)(row % ny);
    z = b.z0 + (int)(row / ny);
    return z < b.z1;
}
__device__ __forceinline__ long long box_items(const Box &b) {
    return (long long)(b.z1 - b.z0) * (b.y1 - b.y0) * ((b.x1 - b.x0) >> 2);
}

// D1 of the float4 at o along axis stride s (s > 1), or along x from a
// 12-float window (s == 1)
__device__ __forceinline__ float4 d1_4(const float *f, long long o, long long s) {
    float r[4];
    if (s == 1) {
        const float4 L = ld4(f + o - 4), C = ld4(f + o), R = ld4(f + o + 4);
        const float v[12] = {L.x, L.y, L.z, L.w, C.x, C.y, C.z, C.w, R.x, R.y, R.z, R.w};
#pragma unroll
        for (int k = 0; k < 4; k++)
            r[k] = float(kD1) * (v[5 + k] - v[3 + k]) + float(kD2) * (v[6 + k] - v[2 + k]) +
                   float(kD3) * (v[7 + k] - v[1 + k]) + float(kD4) * (v[8 + k] - v[k]);
    } else {
        float4 a = ld4(f + o + s), b = ld4(f + o - s);
        r[0] = float(kD1) * (a.x - b.x); r[1] = float(kD1) * (a.y - b.y);
        r[2] = float(kD1) * (a.z - b.z); r[3] = float(kD1) * (a.w - b.w);
        a = ld4(f + o + 2 * s), b = ld4(f + o - 2 * s);
        r[0] += float(kD2) * (a.x - b.x); r[1] += float(kD2) * (a.y - b.y);
        r[2] += float(kD2) * (a.z - b.z); r[3] += float(kD2) * (a.w - b.w);
        a = ld4(f + o + 3 * s), b = ld4(f + o - 3 * s);
        r[0] += float(kD3) * (a.x - b.x); r[1] += float(kD3) * (a.y - b.y);
        r[2] += float(kD3) * (a.z - b.z); r[3] += float(kD3) * (a.w - b.w);
        a = ld4(f + o + 4 * s), b = ld4(f + o - 4 * s);
        r[0] += float(kD4) * (a.x - b.x); r[1] += float(kD4) * (a.y - b.y);
        r[2] += float(kD4) * (a.z - b.z); r[3] += float(kD4) * (a.w - b.w);
    }
    return make_float4(r[0], r[1], r[2], r[3]);
}
// D2 of the float4 at o along axis stride s (same conventions)
__device__ __forceinline__ float4 d2_4(const float *f, long long o, long long s) {
    float r[4];
    if (s == 1) {
        const float4 L = ld4(f + o - 4), C = ld4(f + o), R = ld4(f + o + 4);
        const float v[12] = {L.x, L.y, L.z, L.w, C.x, C.y, C.z, C.w, R.x, R.y, R.z, R.w};
#pragma unroll
        for (int k = 0; k < 4; k++)
            r[k] = d2c<float>(v[4 + k], v[3 + k], v[5 + k], v[2 + k], v[6 + k], v[1 + k], v[7 + k], v[k], v[8 + k]);
    } else {
        const float4 c = ld4(f + o);
        const float4 m1 = ld4(f + o - s), p1 = ld4(f + o + s), m2 = ld4(f + o - 2 * s), p2 = ld4(f + o + 2 * s);
        const float4 m3 = ld4(f + o - 3 * s), p3 = ld4(f + o + 3 * s), m4 = ld4(f + o - 4 * s),
                     p4 = ld4(f + o + 4 * s);
#pragma unroll
        for (int k = 0; k < 4; k++)
            r[k] = d2c<float>(lane4(c, k), lane4(m1, k), lane4(p1, k), lane4(m2, k), lane4(p2, k), lane4(m3, k),
                              lane4(p3, k), lane4(m4, k), lane4(p4, k));
    }
    return make_float4(r[0], r[1], r[2], r[3]);
}
__device__ __forceinline__ void coef4(const StepArgs<float> &A, int ax, int z, int y, int x, float4 &a4, float4 &b4) {
    if (ax == 2) {
        a4 = ld4(A.ca[2] + x);
        b4 = ld4(A.cb[2] + x);
    } else {
        const int k = ax == 0 ? z : y;
        const float a = A.ca[ax][k], b = A.cb[ax][k];
        a4 = make_float4(a, a, a, a);
        b4 = make_float4(b, b, b, b);
    }
}

__global__ void k_psi3d(const StepArgs<float> A, const int n, const int ax, const Box b0, const Box b1) {
    cudaGridDependencySynchronize();
    const Geom &g = A.g;
    const long long s = axis_stride(g, ax);
    const long long n0 = box_items(b0), n1 = box_items(b1);
    const int shot = blockIdx.y;
    const long long sh = (long long)shot * g.fstride;
    const float *p = A.pbuf[n & 1] + sh;
    float *psi = A.psi[ax][0] + sh;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n0 + n1;
         i += (long long)gridDim.x * blockDim.x) {
        int z, y, x;
        if (!(i < n0 ? box_item(b0, i, z, y, x) : box_item(b1, i - n0, z, y, x))) continue;
        const long long o = cell_off(g, z, y, x);
        float4 a4, b4;
        coef4(A, ax, z, y, x, a4, b4);
        const float4 d = d1_4(p, o, s), old = ld4(psi + o);
        *reinterpret_cast<float4 *>(psi + o) = make_float4(b4.x * old.x + a4.x * d.x, b4.y * old.y + a4.y * d.y,
                                                           b4.z * old.z + a4.z * d.z, b4.w * old.w + a4.w * d.w);
    }
}

// zeta^n = b zeta^{n-1} + a (D2 p^n + D1 psi^n) and the addend D1 psi^n + zeta^n
// on the strips of one axis widened by 4 cells (where D1 psi is non-zero).
__global__ void k_add3d(const StepArgs<float> A, const Add3 D, const int n, const int ax, const Box b0, const Box b1) {
    cudaGridDependencySynchronize();
    const Geom &g = A.g;
    const long long s = axis_stride(g, ax);
    const long long n0 = box_items(b0), n1 = box_items(b1);
    const int shot = blockIdx.y;
    const long long sh = (long long)shot * g.fstride;
    const float *p = A.pbuf[n & 1] + sh;
    float *add = D.a[ax] + shot * D.st[ax];
    const float *psi = A.psi[ax][0] + sh;
    float *zeta = A.zeta[ax] + sh;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n0 + n1;
         i += (long long)gridDim.x * blockDim.x) {
        int z, y, x;
        if (!(i < n0 ? box_item(b0, i, z, y, x) : box_item(b1, i - n0, z, y, x))) continue;
        if (g.fs && z == 0) continue;
        const long long o = cell_off(g, z, y, x);
        float4 d2;
        if (ax == 0 && g.fs && z < 4) {  // z-derivative across the free surface: odd mirror
            float r[4];
            for (int k = 0; k < 4; k++) {
                float c[9];
                for (int m = -4; m <= 4; m++) {
                    const int zz = z + m;
                    c[m + 4] = zz < 0 ? -p[cell_off(g, -zz, y, x + k)] : p[cell_off(g, zz, y, x + k)];
                }
                r[k] = d2c<float>(c[4], c[3], c[5], c[2], c[6], c[1], c[7], c[0], c[8]);
            }
            d2 = make_float4(r[0], r[1], r[2], r[3]);
        } else {
            d2 = d2_4(p, o, s);
        }
        float4 a4, b4;
        coef4(A, ax, z, y, x, a4, b4);
        const float4 dps = d1_4(psi, o, s), zo = ld4(zeta + o);
        const float4 zt = make_float4(b4.x * zo.x + a4.x * (d2.x + dps.x), b4.y * zo.y + a4.y * (d2.y + dps.y),
                                      b4.z * zo.z + a4.z * (d2.z + dps.z), b4.w * zo.w + a4.w * (d2.w + dps.w));
        st4(zeta + o, zt);
        const long long oa = ax == 0   ? ((long long)(z < D.zl ? z : D.zl + z - D.zh) * g.NY + y) * g.P + x
                             : ax == 1 ? ((long long)z * D.nyw + (y < D.yl ? y : D.yl + y - D.yh)) * g.P + x
                                       : ((long long)z * g.NY + y) * D.nxw + (x < D.xl ? x : D.xl + x - D.xs);
        st4(add + oa, make_float4(dps.x + zt.x, dps.y + zt.y, dps.z + zt.z, dps.w + zt.w));
    }
}

size_t col_smem(int L, bool adj) {
    return (size_t)CW * sizeof(float) * (adj ? 3 * (L + 8) : (L + 16) + (L + 8) + L);
}

size_t row_smem(int nq) { return sizeof(float) * kRowEnds * (2 + 3 * 4 * (size_t)(nq + 4)); }

// Strip ranges of an axis widened by 4 cells; strips that meet are one range.
ColRanges col_ranges(int N, int lo, int hi) {
    ColRanges R{};
    const int l1 = lo > 0 ? std::min(N, lo + 4) : 0, h0 = hi > 0 ? std::max(0, N - hi - 4) : N;
    if (l1 > 0 && h0 < N && l1 >= h0) {
        R.n = 1;
        R.s1[0] = N;
        return R;
    }
    if (l1 > 0) R.s1[R.n++] = l1;
    if (h0 < N) R.s0[R.n] = h0, R.s1[R.n++] = N;
    return R;
}

// The row-end blocks take widened strips of at most kMaxQ float4s whose ends are
// apart (no cell's psi formed twice).
bool x_ends(const Geom &g, XEnds &E) {
    const int NX = g.NX;
    int qa[2], qb[2], m = 0;
    if (g.nbx0 > 0) qa[m] = 0, qb[m++] = std::min(NX, g.nbx0 + 4);
    if (g.nbx1 > 0) qa[m] = std::max(0, NX - g.nbx1 - 4), qb[m++] = NX;
    bool ok = m > 0 && (m < 2 || qa[1] - qb[0] >= 16);
    E = XEnds{};
    for (int k = 0; k < m && ok; k++) {
        const int q4 = qa[k] & ~3, nq = (qb[k] - q4 + 3) >> 2;
        E.xa[k] = q4 - 8;
        E.nq[k] = nq;
        ok = nq <= kMaxQ;
    }
    E.ne = m;
    return ok;
}

// The axes k_cpml3d takes (bit per axis) and its plan; smem: bytes a block needs.
int plan3(const StepArgs<float> &a, const Add3 &D, bool adj, Plan3 &Q, size_t &smem) {
    const Geom &g = a.g;
    Q = Plan3{};
    Q.D = D;
    smem = 0;
    int took = 0;
    for (int ax = 0; ax < 2; ax++) {
        if (!a.ca[ax]) continue;
        const ColRanges R = ax == 0 ? col_ranges(g.NZ, g.nbz0, g.nbz1) : col_ranges(g.NY, g.nby0, g.nby1);
        int most = 0;
        for (int k = 0; k < R.n; k++) most = std::max(most, R.s1[k] - R.s0[k]);
        const bool mirror = ax == 0 && g.fs && R.n > 0 && R.s0[0] < 4;  // D2 across the free surface
        if (most > kColRows || mirror) continue;
        took |= 1 << ax;
        Q.c[ax] = R;
        Q.nbr[ax] = (int)(((long long)(ax == 0 ? g.NY : g.NZ) * ((g.NX + 3) >> 2) + 31) / 32);
        Q.nb[ax] = R.n * Q.nbr[ax];
        if (R.n) smem = std::max(smem, col_smem(most, adj));
    }
    if (a.ca[2] && x_ends(g, Q.E)) {
        took |= 4;
        Q.xrows = (long long)g.NZ * g.NY;
        Q.nbx = (int)((Q.xrows + kRowEnds - 1) / kRowEnds);
        Q.nb[2] = Q.E.ne * Q.nbx;
        smem = std::max(smem, row_smem(std::max(Q.E.nq[0], Q.E.nq[1])));
    }
    return took;
}

template <typename K, typename... Args>
cudaError_t launch(K k, dim3 grid, int threads, size_t smem, cudaStream_t st, bool pdl, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace

Add3 add3_layout(const Geom &g, const bool on[3], long long elems[3]) {
    Add3 D{};
    const ColRanges rz = col_ranges(g.NZ, on[0] ? g.nbz0 : 0, on[0] ? g.nbz1 : 0);
    const ColRanges ry = col_ranges(g.NY, on[1] ? g.nby0 : 0, on[1] ? g.nby1 : 0);
    auto ends = [](const ColRanges &R, int N, int &l, int &h) {
        l = 0, h = N;
        for (int k = 0; k < R.n; k++) {
            if (R.s0[k] == 0) l = R.s1[k];
            else h = R.s0[k];
        }
        return l + N - h;
    };
    D.nzw = ends(rz, g.NZ, D.zl, D.zh);
    D.nyw = ends(ry, g.NY, D.yl, D.yh);
    D.xe = (g.NX + 3) & ~3;
    D.xl = on[2] && g.nbx0 > 0 ? std::min(D.xe, (g.nbx0 + 4 + 3) & ~3) : 0;
    D.xs = on[2] && g.nbx1 > 0 ? std::max(0, g.NX - g.nbx1 - 4) & ~3 : D.xe;
    if (D.xl >= D.xs && D.xl > 0) D.xl = D.xs = D.xe;  // ends that meet: one range
    D.nxw = D.xl + D.xe - D.xs;
    elems[0] = (long long)D.nzw * g.NY * g.P;
    elems[1] = (long long)g.NZ * D.nyw * g.P;
    elems[2] = (long long)g.NZ * g.NY * D.nxw;
    for (int ax = 0; ax < 3; ax++) D.st[ax] = elems[ax];
    return D;
}

cudaError_t configure_cpml3d() {
    static_assert(kRowEnds * (2 + 12 * (kMaxQ + 4)) <= CW * (3 * kColRows + 24), "the row ends' staging fits the opt-in");
    cudaError_t e = cudaFuncSetAttribute(k_cpml3d<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)col_smem(kColRows, false));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cpml3d<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)col_smem(kColRows, true));
    return e;
}

cudaError_t launch_cpml3d(const StepArgs<float> &a, const Add3 &D, int n, const Pt3 *rec, int nrec, int nshots,
                          cudaStream_t st, bool pdl) {
    const Geom &g = a.g;
    Plan3 Q;
    size_t smem;
    const int took = plan3(a, D, false, Q, smem);
    const int N[3] = {g.NZ, g.NY, g.NX};
    const int lo[3] = {g.nbz0, g.nby0, g.nbx0}, hi[3] = {g.nbz1, g.nby1, g.nbx1};
    for (int ax = 0; ax < 3; ax++) {
        if (!a.ca[ax] || (took >> ax & 1)) continue;
        for (int phase = 0; phase < 2; phase++) {
            const int widen = phase == 0 ? 0 : 4;
            int a0 = 0, a1 = lo[ax] > 0 ? std::min(N[ax], lo[ax] + widen) : 0;
            int b0 = hi[ax] > 0 ? std::max(0, N[ax] - hi[ax] - widen) : N[ax], b1 = N[ax];
            if (a1 > b0) {  // strips meet: one box
                a1 = b1;
                b0 = b1;
            }
            Box B0{0, g.NZ, 0, g.NY, 0, g.NX}, B1 = B0;
            auto set = [&](Box &b, int s0, int s1) {
                if (ax == 0) { b.z0 = s0; b.z1 = s1; }
                else if (ax == 1) { b.y0 = s0; b.y1 = s1; }
                else { b.x0 = s0; b.x1 = s1; }
            };
            set(B0, a0, a1);
            set(B1, b0, b1);
            // float4 columns: x-ranges rounded out to multiples of 4; boxes that then
            // touch or overlap become one box (so no cell is updated twice)
            auto round4 = [](Box &b) {
                if (b.x1 <= b.x0) return;
                b.x0 = b.x0 & ~3;
                b.x1 = (b.x1 + 3) & ~3;
            };
            round4(B0);
            round4(B1);
            const bool empty0 = B0.z1 <= B0.z0 || B0.y1 <= B0.y0 || B0.x1 <= B0.x0;
            const bool empty1 = B1.z1 <= B1.z0 || B1.y1 <= B1.y0 || B1.x1 <= B1.x0;
            if (ax == 2 && !empty0 && !empty1 && B0.x1 >= B1.x0) {
                B0.x1 = B1.x1;
                B1 = Box{0, 0, 0, 0, 0, 0};
            }
            const long long items = (long long)(B0.z1 - B0.z0) * (B0.y1 - B0.y0) * ((B0.x1 - B0.x0) >> 2) +
                                    (long long)(B1.z1 - B1.z0) * (B1.y1 - B1.y0) * ((B1.x1 - B1.x0) >> 2);
            if (items <= 0) continue;
            const dim3 grid((int)std::min<long long>((items + 255) / 256, 152 * 16), nshots);
            const cudaError_t e = phase == 0 ? launch(k_psi3d, grid, 256, 0, st, pdl, a, n, ax, B0, B1)
                                             : launch(k_add3d, grid, 256, 0, st, pdl, a, D, n, ax, B0, B1);
            if (e != cudaSuccess) return e;
        }
    }
    Q.rec = rec;
    Q.nrec = rec ? nrec : 0;
    Q.nbs = (Q.nrec + NT - 1) / NT;
    const int blocks = Q.nb[0] + Q.nb[1] + Q.nb[2] + Q.nbs;
    if (blocks == 0) return cudaSuccess;
    Mem3 M{};
    M.f = a.pbuf[n & 1];
    for (int ax = 0; ax < 3; ax++) {
        M.m0[ax] = a.psi[ax][0];
        M.m1[ax] = a.zeta[ax];
    }
    return launch(k_cpml3d<false>, dim3(blocks, nshots), NT, smem, st, pdl, a, Q, M, n);
}

bool cpml3d_adjoint_fits(const StepArgs<float> &a) {
    Plan3 Q;
    size_t smem;
    const int took = plan3(a, Add3{}, true, Q, smem);
    for (int ax = 0; ax < 3; ax++)
        if (a.ca[ax] && !(took >> ax & 1)) return false;
    return true;
}

cudaError_t launch_cpml3d_adjoint(const StepArgs<float> &a, const Add3 &D, const CpmlAdjArgs<float> &c, int nshots,
                                  cudaStream_t st, bool pdl) {
    Plan3 Q;
    size_t smem;
    plan3(a, D, true, Q, smem);
    Mem3 M{};
    M.f = c.u;
    for (int ax = 0; ax < 3; ax++) {
        M.m0[ax] = c.nu[ax][0];
        M.m1[ax] = c.mu[ax];
    }
    const int blocks = Q.nb[0] + Q.nb[1] + Q.nb[2];
    if (blocks == 0) return cudaSuccess;
    return launch(k_cpml3d<true>, dim3(blocks, nshots), NT, smem, st, pdl, a, Q, M, 0);
}

}  // namespace gsim
