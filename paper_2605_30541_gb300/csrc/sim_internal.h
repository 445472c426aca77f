// Internal declarations of libsim: field layout, kernel argument blocks and
// the launch entry points each translation unit provides. Host code is C++17.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/sim.h"

namespace gsim {

// ---------------------------------------------------------------- layout
//
// Every field (pressure ping-pong buffers, c = (v dt / h)^2, velocity, CPML
// memory) uses one padded layout per shot: the computational grid (interior +
// absorbing cells, NZ x NY x NX) surrounded by kGhost cells of zeros on every
// side, rows padded to a multiple of 32 elements. The ghost cells are never
// written, so a stencil that reads them sees p = 0 (Dirichlet) without a
// bounds check. Cell (z, y, x) of the computational grid sits at
//     org + (z * PY + y) * P + x
// where PY is the number of rows per z-plane (1 in 2D).
constexpr int kGhost = 8;      // >= the widest halo any kernel reads (CPML recompute)
constexpr int kTileX2 = 32;    // 2D tile (x) of the generic (any precision) stencil kernel
constexpr int kTileZ2 = 16;    // 2D tile (z) of the generic kernel
constexpr int kTileXF = 128;   // 2D tile (x) of the FP32 kernel; its z extent is tuned (8, 16, 32)
constexpr int kProfAlign = 128; // per-axis profile segments: aligned starts, room for a whole last tile
constexpr int kRoundX = 128;   // padded extents round up to these, so any tile
constexpr int kRoundZ = 32;    //   of the tuned set stays inside the allocation
constexpr int kRoundY = 32;
constexpr int kMinmaxBlocks = 512;  // partial (min, max, bad) triples written by launch_minmax

struct Geom {
    int ndim;
    int NZ, NY, NX;        // computational grid
    int nz, ny, nx;        // interior
    int oz, oy, ox;        // interior origin in the computational grid
    int nbz0, nbz1, nby0, nby1, nbx0, nbx1;
    int P;                 // row pitch (elements)
    int PY;                // rows per z-plane (1 in 2D)
    long long fstride;     // elements per field
    long long org;         // offset of cell (0,0,0)
    int fs;                // free surface on top
};

__host__ __device__ inline long long cell_off(const Geom &g, int z, int y, int x) {
    return g.org + ((long long)z * g.PY + y) * g.P + x;
}

// Receiver: base cell of its linear-interpolation stencil (local to the tile
// that samples it) and the 4 (2D) or 8 (3D) corner weights, corner order
// (dz, dy, dx) with dx fastest.
template <typename W>
struct RecEntryT {
    int rec;
    int lz, ly, lx;
    W w[8];
};

// Injection: one group per target cell of a tile, summing its entries in a
// fixed order (so the result is deterministic), value = weight * input[pt].
struct InjGroup {
    int cell;   // local linear index lz * TX + lx (2D) / (lz*TY + ly)*TX + lx (3D)
    int e0, e1; // entry range
    int pad;
};
template <typename W>
struct InjEntryT {
    int pt;     // index of the input value (shot for a source, receiver for a residual)
    W w;
};

// Per-call I/O block, resident on the device and refreshed before each run,
// so captured graphs stay valid across calls.
struct SimIO {
    const void *wavelet;     // [nt] (shared by the shots)
    void *gather;            // [nshots][nt][nrec]
    void *snaps;             // [nshots][nsnap][interior]
    float *snap_scale;       // [nshots][nsnap]
    unsigned *snap_max;      // [nshots][nsnap] float bits of max |p|
    const void *resid;       // [nshots][nt][nrec] adjoint residual
    int nrec;
    int nshots;
    int snap_fp16;
    int pad;
};

enum : unsigned { kFlagUnstable = 1u, kFlagTimeout = 2u };

template <typename T>
struct StepArgs {
    Geom g;
    T *pbuf[2];              // ping-pong bases (per shot: + shot * fstride)
    const T *ch;             // (v dt / h)^2, field layout, shared by the shots
    const T *E[3];           // sponge profile per axis: eta h^2 / (2 dt); NULL = none
    const T *ca[3], *cb[3];  // CPML recursion coefficients per axis; NULL = axis absent
    T *psi[3][2];            // CPML psi ping-pong (scaled by h), per shot stride fstride
    T *zeta[3];              // CPML zeta (scaled by h^2)
    int bc;
    T src_scale;             // h^(2-d)
    int ntx, nty, ntz;       // tiles per shot
    int nt;
    int nsnap, snap_every, snap_begin, snap_end;
    // receivers (tile-local lists, shared by the shots)
    const int *rec_start;
    const RecEntryT<T> *rec;
    // injection (sources: per shot and tile; residuals: per tile)
    const int *inj_start;
    const InjGroup *inj_grp;
    const InjEntryT<T> *inj_ent;
    int inj_per_shot;        // 1: inj lists are indexed by shot * ntiles + tile
    int inj_kind;            // 0: value = wavelet[n]; 1: value = resid[shot][n][pt]
    const SimIO *io;
    unsigned *flags;
    int sample;              // 1: receivers sample p^n into io->gather
    int inj_reverse;         // 1: injection row = nt - n (adjoint sweep), rows >= nt inject 0
    // adjoint-state imaging term Q'^n = E (p^{n+1} - p^{n-1}) - h^2 (L p^n + s^n), per cell
    void *qslot;             // this launch's slot, field layout per shot (T, or half when q_fp16)
    float *qscale;           // FP16 slots: power-of-two scale per [shot][tile]
    int q_fp16;
    T *G;                    // adjoint sweep: G += u^{n+1} Q'^n, field layout per shot
    const T *cext;           // adjoint sweep of a CPML problem: per-cell term added to the Laplacian
};

// Per-launch facts of one step, resolved on the host (so the kernel does no
// integer division on them): buffer parity / gather row, snapshot index to
// write (-1: none), snapshot index whose FP16 scale this step's output feeds
// (-1: none), injection row (-1: none), and the imaging-term slot.
struct StepTime {
    int n;
    int snap_k;
    int max_k;
    int inj_row;
    void *qslot;
    float *qscale;
};

// CPML terms of the adjoint sweep (cpml_adj.cu): the multipliers nu (of
// zeta) and mu (of psi) of each absorbing axis, nu ping-ponged by step
// parity; in 2D the term `ext` the step kernel adds to the Laplacian of u
// (A.cext), in 3D c times that term added to u^k after the update.
template <typename T>
struct CpmlAdjArgs {
    const T *u;   // u^{k+1}, field layout per shot
    T *nu[3][2];  // [axis][parity] (absent axes unused)
    T *mu[3];     // [axis]
    T *ext;       // 2D: the bracket, added to the Laplacian by the step kernel
    T *uo;        // 3D: u^k, receives c times the bracket (NULL in 2D)
    const T *q;   // 3D: the recorded imaging term of the step
    T *G;         // 3D: gradient accumulator
};
template <typename T>
cudaError_t launch_cpml_adjoint(const StepArgs<T> &a, const CpmlAdjArgs<T> &c, int parity, int nshots,
                                cudaStream_t st);

// Step kernel modes: plain forward; forward that records Q'^n; adjoint sweep
// that accumulates G from the recorded Q'.
enum StepMode { kModeForward = 0, kModeRecord = 1, kModeAdjoint = 2 };

// A point of the 3D path: field offsets of its 8 trilinear corners (-1 where
// the weight is zero or the corner is a held free-surface cell) and weights.
struct Pt3 {
    long long cell[8];
    float w[8];
};

// Batch (persistent) execution: see k_batch2d in fwd2d_f32.cu.
struct BatchMember {
    int slice;       // index into BatchArgs::slices
    int shot;
    int tile0;       // first of this member's tiles within one step of its group
    int done0;       // offset of this member's per-tile step counters
};
struct BatchGroup {
    long long base;  // first item of the group
    int T;           // tiles per step over the group's members
    int m0, m1;      // member range
};
struct BatchArgs {
    const StepArgs<float> *slices;
    const BatchGroup *groups;
    int ngroups;
    int nmembers;
    const BatchMember *members;
    int *done;                 // per (slice, shot, tile): steps completed
    unsigned long long *head;  // work counter
    long long total;           // items
    long long spin_limit;      // polls before a wait gives up
    unsigned *flags;           // kFlagTimeout on a wait that gave up
};
cudaError_t launch_batch2d(const BatchArgs &b, int tz, bool cpml, int grid, cudaStream_t st);
// Stepped batch (k_multi2d): step n of every member in one launch of
// nblocks = all members' tiles; members' tile0 is global (prefix over members).
cudaError_t launch_multi2d(const BatchArgs &b, int tz, bool cpml, int nblocks, int n, cudaStream_t st, bool pdl);
int batch_blocks_per_sm(int tz, bool cpml);

// Row march (march2d.cu): the 2D FP32 forward step as warps that each walk
// down the rows [z0, z1) of one 128-column strip (bx) of one member (slice,
// shot). The warps take the nitems segments in order from the step's
// counter ctr[n & 1] (ctr[0] zeroed before the first step; each step zeroes
// the next step's). tz is the tile height of the slices' receiver and
// injection lists.
constexpr int kMarchW = 128;
struct MarchSeg {
    int slice, shot, bx, z0, z1;
    int pad[3];
};
struct MarchArgs {
    const StepArgs<float> *slices;
    const MarchSeg *segs;
    unsigned *ctr;
    int nwarps;
    int nitems;
    int tz;
    int pad;
};
cudaError_t configure_march2d();
int march2d_warps_per_sm(bool cpml);
cudaError_t launch_march2d(const MarchArgs &m, bool cpml, const StepTime &t, cudaStream_t st, bool pdl);

// Temporal blocking of the row march (march2x.cu): two steps per pass for
// members without CPML. A member (slice, shot) has two more pressure fields
// (p3 and p3 + pstride: the four fields alternate as two pairs over the
// passes) and up to four source corners; items are MarchSeg over 120-column
// strips (slice = member index). Receivers are TBSample entries sampled
// after each pass.
constexpr int kTBW = 120;
struct TBMember {
    int slice, shot;
    float *p3;             // third and fourth pressure fields of the slice (per shot: + shot * fstride)
    long long pstride;     // from the third field to the fourth
    int nsrc, pad;
    int sz[4], sx[4];      // source corners: computational-grid row and column
    float sw[4];           // bilinear weights
};
struct TBSample {
    int member, rec;
    int z, x;              // base cell (computational grid) of the 2 x 2 corners
    float w[4];            // corner weights (z, x), (z, x+1), (z+1, x), (z+1, x+1)
};
struct TBArgs {
    const StepArgs<float> *slices;
    const TBMember *members;
    const MarchSeg *segs;
    const TBSample *samples;
    unsigned *ctr;         // two per-pass item counters
    int nitems;
    int pad;
    long long nsamples;
};
struct TBPass {
    int k;                 // pass index: even passes read fields 0, 1, odd passes fields 2, 3
    int n;                 // first step of the pass
    int two;               // 1: steps n and n + 1; 0: step n only
    int inj0, inj1;        // wavelet rows injected at the two steps (-1: none)
    int pad;
};
cudaError_t configure_march2x();
int march2x_warps_per_sm();
cudaError_t launch_march2x(const TBArgs &b, const TBPass &t, int nwarps, cudaStream_t st);

// 3D step (fwd3d.cu, cpml3d.cu). Per step: snapshot, CPML addends and
// receiver samples, z-march update with the addends and the sources.
// z-march variants: kZMarchAsync stages each plane by per-thread 16-byte
// cp.async copies; kZMarchTma by bulk tensor copies (TMA) issued by one
// thread, completion on mbarriers.
enum { kZMarchAsync = 1, kZMarchTma = 6 };
// CPML addends of the 3D step: per axis a compact array over the cells of its
// strips widened by 4 (z: slots of whole (y, x) planes; y: slots of x rows in
// every plane; x: the float4s from the strip ends of every row), one after
// another for the shots.
struct Add3 {
    float *a[3];        // z, y, x; NULL: axis absent
    long long st[3];    // elements per shot
    int zl, zh, nzw;    // planes z < zl (slot z) and z >= zh (slot zl + z - zh)
    int yl, yh, nyw;    // rows y alike
    int xl, xs, xe, nxw; // float4s starting in [0, xl) and [xs, xe); nxw floats per row
};
Add3 add3_layout(const Geom &g, const bool on[3], long long elems[3]);
struct Pt3;
cudaError_t configure_cpml3d();
// psi^n, zeta^n and the addends of every absorbing axis, and (rec) the
// receivers' samples of p^n into the gather
cudaError_t launch_cpml3d(const StepArgs<float> &a, const Add3 &D, int n, const Pt3 *rec, int nrec, int nshots,
                          cudaStream_t st, bool pdl);
// the adjoint sweep's multipliers (in place: parity 0 of nu) and brackets, for
// strip layouts that fit; the z-march of the sweep adds the brackets
bool cpml3d_adjoint_fits(const StepArgs<float> &a);
cudaError_t launch_cpml3d_adjoint(const StepArgs<float> &a, const Add3 &D, const CpmlAdjArgs<float> &c, int nshots,
                                  cudaStream_t st, bool pdl);
struct Tma3 {
    CUtensorMap ph;  // p (both parities, all shots): one plane of a tile with its 4-cell x / y halo
    CUtensorMap po;  // the same buffers: one plane of a tile's own cells
    CUtensorMap c;   // c = (v dt / h)^2: likewise
};
cudaError_t configure_step3d();
struct ZShape {
    int variant = kZMarchTma;
    int tile = 64;   // columns of a CTA's tile (TMA: 64 or 32 of 1024 cells; cp.async: 128 x 8)
    int chunk = 0;   // planes per CTA
};
// src, row: the shots' point sources and the wavelet row they inject (NULL, or
// a row outside the record: none)
cudaError_t launch_step3d(const StepArgs<float> &a, int n, const ZShape &zs, int nshots, cudaStream_t st, bool pdl, int mode,
                          const Add3 &D, const Pt3 *src, int row, float *qs = nullptr, float *Gs = nullptr);
// 3D residual injection grouped by target cell (the adjoint sweep): group =
// cell offset within a field and entry range, the same for every shot.
struct Inj3 {
    long long cell;
    int e0, e1;
};
struct InjE3 {
    int pt;
    float w;
};
cudaError_t launch_inj3d(const StepArgs<float> &a, int n, int row, const Inj3 *grp, int ngrp, const InjE3 *ent,
                         int nshots, const float *qs, float *Gs, cudaStream_t st);
cudaError_t launch_snap3d(const StepArgs<float> &a, const StepTime &t, int fp16, int nshots, cudaStream_t st);

// Resident execution (resident2d.cu): one cooperative launch runs steps [n0, n1)
// of 2D FP32 shots whose state fits on chip; each CTA of kResidentWarps warps
// owns one subdomain: columns [128 bx, 128 bx + 128), rows [z0, z0 + rows) with
// rows <= 16 RZ, warps taking rpw rows each. nbr lists the subdomains whose
// borders form its halo (same shot).
constexpr int kResidentWarps = 16;
constexpr size_t kResidentMaxSmem = 227 * 1024;
constexpr int kResidentMaxNbr = 11;
constexpr int kResidentOutbox = 2 * (2 * 8 * 128 + 2 * 64 * 8);  // words: two halves of border rows and columns
struct RTile {
    int bx, z0, rows, rpw;
    int nnbr;
    int nbr[kResidentMaxNbr];
};

// CPML work of one subdomain. Columns in float4 chunks (chunk c: the cells
// 4c - 8 .. 4c - 5 of the subdomain, c in [0, 36)), rows subdomain-local; the
// memory fields are non-zero on the strips only, the terms that use them on
// the strips widened by 4. Forward: first field psi, second zeta; adjoint: nu
// and mu (kept on the ring of 8 and 4 cells round the subdomain that the
// transposed derivatives reach, recomputed redundantly as psi is on 4).
struct RSpan {
    int c0, c1;   // chunks of the first field that are updated
    int m0, m1;   // adjoint: chunks of the second
    int a0, a1;   // own chunks that take the term
    int p0, p1;   // chunks of the first field kept (zeros round [c0, c1) for the derivative windows)
    int q0, q1;   // adjoint: of the second
    int zc0, zc1, zm0, zm1, za0, za1, zp0, zp1, zq0, zq1;  // the same along z, in rows
};
__host__ __device__ inline void strip_hull(int o, int N, int nb0, int nb1, int c0, int c1, int &lo, int &hi) {
    lo = 1 << 30;
    hi = -(1 << 30);
    if (nb0 > 0) {
        const int a = -o > c0 ? -o : c0, b = nb0 - o < c1 ? nb0 - o : c1;
        if (a < b) lo = a < lo ? a : lo, hi = b > hi ? b : hi;
    }
    if (nb1 > 0) {
        const int a = N - nb1 - o > c0 ? N - nb1 - o : c0, b = N - o < c1 ? N - o : c1;
        if (a < b) lo = a < lo ? a : lo, hi = b > hi ? b : hi;
    }
}
__host__ __device__ inline RSpan resident_span(const Geom &g, int bc, int bx, int z0, int rows, bool adj) {
    RSpan s{};
    if (bc != SIM_BC_CPML) return s;
    const int x0 = bx * kTileXF, ring = adj ? 8 : 4;
    auto mn = [](int a, int b) { return a < b ? a : b; };
    auto mx = [](int a, int b) { return a > b ? a : b; };
    int lo, hi;
    strip_hull(x0, g.NX, g.nbx0, g.nbx1, -ring, kTileXF + ring, lo, hi);
    if (lo < hi) {
        s.c0 = (lo + 8) >> 2, s.c1 = (hi + 11) >> 2;
        s.p0 = s.c0, s.p1 = s.c1;
        const int al = mx(0, lo - 4), ah = mn(kTileXF, hi + 4);
        if (al < ah) s.a0 = (al + 8) >> 2, s.a1 = (ah + 11) >> 2;
        if (adj) {
            strip_hull(x0, g.NX, g.nbx0, g.nbx1, -4, kTileXF + 4, lo, hi);
            if (lo < hi) {
                s.m0 = (lo + 8) >> 2, s.m1 = (hi + 11) >> 2;
                s.p0 = mn(s.p0, s.m0 - 1), s.p1 = mx(s.p1, s.m1 + 1);
            }
            s.q0 = s.m0, s.q1 = s.m1;
            if (s.a0 < s.a1) {
                if (s.q0 >= s.q1) s.q0 = s.a0, s.q1 = s.a1;
                s.q0 = mn(s.q0, s.a0 - 1), s.q1 = mx(s.q1, s.a1 + 1);
            }
        }
        if (s.a0 < s.a1) s.p0 = mn(s.p0, s.a0 - 1), s.p1 = mx(s.p1, s.a1 + 1);
    }
    strip_hull(z0, g.NZ, g.nbz0, g.nbz1, -ring, rows + ring, lo, hi);
    if (lo < hi) {
        s.zc0 = lo, s.zc1 = hi;
        s.zp0 = lo, s.zp1 = hi;
        s.za0 = mx(0, lo - 4), s.za1 = mn(rows, hi + 4);
        if (s.za0 >= s.za1) s.za0 = s.za1 = 0;
        if (adj) {
            strip_hull(z0, g.NZ, g.nbz0, g.nbz1, -4, rows + 4, lo, hi);
            if (lo < hi) {
                s.zm0 = lo, s.zm1 = hi;
                s.zp0 = mn(s.zp0, lo - 4), s.zp1 = mx(s.zp1, hi + 4);
            }
            s.zq0 = s.zm0, s.zq1 = s.zm1;
            if (s.za0 < s.za1) {
                if (s.zq0 >= s.zq1) s.zq0 = s.za0, s.zq1 = s.za1;
                s.zq0 = mn(s.zq0, s.za0 - 4), s.zq1 = mx(s.zq1, s.za1 + 4);
            }
        }
        if (s.za0 < s.za1) s.zp0 = mn(s.zp0, s.za0 - 4), s.zp1 = mx(s.zp1, s.za1 + 4);
    }
    return s;
}

// Shared memory of a launch (floats; the same for every CTA): offsets and the
// widths of the compact CPML arrays (the largest over the subdomains).
struct RLayout {
    int c, coef, f1, f2, ax, z1, z2, G, K, inj, rec;  // offsets
    int w1, w2, wa;                                   // floats per row of f1, f2, ax
    int injr;                                         // rows with injected cells a subdomain may have
    int total;
};
enum { kResForward = 0, kResRecord = 1, kResAdjoint = 2 };
struct ResidentArgs {
    unsigned long long *outbox;  // kResidentOutbox words per CTA
    long long spin_limit;
    const RTile *tiles;  // device array, per shot
    int ntiles;
    int shot0;           // first shot of the launch
    int n0, n1;          // steps (adjoint: sweep index n = nt - k)
    unsigned tag0;       // words of step n carry tag0 + n - n0; no earlier launch has used tags from tag0 on
    int load;            // start from the state in the global fields (else from rest)
    int store_mem;       // leave the CPML memory in the global fields too
    int exact_sponge;    // the sponge update with its division, as the per-step kernels have it
    RLayout lay;
    // CPML memory, field layout (x, z): forward psi in, psi out, zeta; adjoint nu, mu
    float *m1i[2], *m1o[2], *m2[2];
    // imaging-term slots of the launch's steps (record: slot n - n0; adjoint: slot n1 - 1 - n); FP16
    // slots keep a scale per (subdomain, warp) in the top ghost rows of each shot's field
    char *q;
    long long qstride;
    int corners;  // a receiver reads the cell past a subdomain's last row and column: exchange it
};
cudaError_t configure_resident2d();
bool resident2d_layout(const Geom &g, int bc, int rz, int mode, bool exact_sponge, const std::vector<RTile> &tiles, int injr,
                       RLayout &lay);
cudaError_t launch_resident2d(const StepArgs<float> &a, const ResidentArgs &r, int rz, int mode, int nshots,
                              cudaStream_t st);

// Message returned by sim_last_error(NULL) for failures of this thread.
void set_thread_error(const char *msg);

// Launchers (one translation unit each).
template <typename T>
cudaError_t launch_step2d(const StepArgs<T> &a, int n, int nshots, int mode, cudaStream_t st);

// FP32 kernel with a 128 x tz tile (tz in {8, 16, 32}).
// pdl: let step n+1 launch while step n drains (programmatic dependent launch);
// the kernel waits for its predecessor before reading any field.
cudaError_t launch_step2d_f32(const StepArgs<float> &a, const StepTime &t, int tz, int nshots, int mode,
                              cudaStream_t st, bool pdl);
cudaError_t configure_step2d_f32();

// Checkpoint of the CPML memory of one axis: only the boxes of its strips
// (the memory is zero elsewhere), compact [shot][rows][x] with, in FP16, a
// power-of-two scale per (shot, box row). row0 / elem0 are prefix sums over
// the boxes (row0[n] rows and elem0[n] elements per shot).
struct CkBox {
    int z0, z1, y0, y1, x0, x1;
};
constexpr int kMaxCkBoxes = 2;
struct CkBoxes {
    int n;
    CkBox b[kMaxCkBoxes];
    long long row0[kMaxCkBoxes + 1];
    long long elem0[kMaxCkBoxes + 1];
};
// One checkpoint: the two pressure fields (compact [shot][NZ NY NX] copies, in
// FP16 with a power-of-two scale per 2D tile, ntx x ntz of them) and the CPML
// memory, two fields per absorbing axis.
template <typename T>
struct CkArgs {
    int fp16, nshots, ntx, ntz, nmem;
    T *state[2];
    void *state_copy[2];
    float *state_scale[2];
    T *mem[6];
    void *mem_copy[6];
    float *mem_scale[6];
    CkBoxes box[3];
    unsigned block0[6];  // set by the launch
};
template <typename T>
cudaError_t launch_checkpoint(const Geom &g, CkArgs<T> c, bool store, cudaStream_t st);
// res = g - d (all shots), per-block partial sums of res^2 / 2 into part.
template <typename T>
cudaError_t launch_residual(const T *g, const T *d, T *res, long long n, double *part, int nblocks, cudaStream_t st);
// acc[interior] += sum over shots and replicated padding cells of -2 G / (v h^2).
template <typename T>
cudaError_t launch_fold_gradient(const Geom &g, const T *G, long long gshot, int nshots, const T *vpad,
                                 double inv_h2, double *acc, cudaStream_t st);
template <typename T>
cudaError_t launch_add_gradient(const double *acc, T *grad, long long n, cudaStream_t st);

template <typename T>
cudaError_t launch_setup_model(const Geom &g, const T *vel, T *ch, T *vpad, double dt_over_h,
                               cudaStream_t st);
template <typename T>
cudaError_t launch_minmax(const Geom &g, const T *vel, double *out2, cudaStream_t st);
template <typename T>
cudaError_t launch_check_finite(const Geom &g, const T *f, int nshots, unsigned *flags,
                                cudaStream_t st);

}  // namespace gsim
