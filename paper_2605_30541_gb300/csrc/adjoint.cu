// Support kernels of the adjoint-state gradient: checkpoint store/restore
// (FP32/FP64 copy or FP16 with a power-of-two scale per tile; the CPML
// memory of an axis only on the boxes of its strips, where it can be
// non-zero, with a scale per row), the data
// residual with its misfit, and the final FP64 fold of the per-shot imaging
// sums onto the interior velocity cells (absorbing cells replicate the
// nearest interior cell, so their contributions land on the edge cells).
#include <cfloat>

#include "sim_internal.h"
#include "stencil.cuh"

namespace gsim {
namespace {

constexpr int TX = kTileX2, TZ = kTileZ2, BX = 32, BY = 8, RZ = TZ / BY, NTH = BX * BY;

__device__ __forceinline__ float tile_max(float v, float *red) {
    const int tid = threadIdx.x;
    v = warp_max(v);
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    float m = tid < NTH / 32 ? red[tid & 31] : 0.f;
    if (tid < 32) m = warp_max(m);
    __syncthreads();
    if (tid == 0) red[0] = m;
    __syncthreads();
    return red[0];
}

// Rows of the computational grid: r = z NY + y (r = z in 2D), NZ NY rows of NX cells.
__device__ __forceinline__ long long row_off(const Geom &g, int r, int x) {
    return cell_off(g, r / g.NY, r % g.NY, x);
}

// A checkpoint is stored or restored by one launch: its first CTAs take the two
// pressure fields, a CTA per (tile of rows x columns, shot, field), the others
// the CPML memory, a warp per (box row, shot) of each field. (With a launch per
// field, twelve per segment of a 2D CPML gradient, 16 shots of 241 x 241 cells
// in 32 segments took 24.2 ms instead of 23.1, one shot of 132 x 152 x 172 in
// 11 segments 14.4 instead of 13.8.)
//
// The compact copy of a pressure field is [shot][NZ NY NX], in FP16 with a
// scale per tile.
template <typename T, bool STORE>
__device__ __forceinline__ void state_tile(const Geom &g, const CkArgs<T> &C, int w, int bx, int bz, int shot, float *red) {
    const int x0 = bx * TX, z0 = bz * TZ, nrow = g.NZ * g.NY;
    const int tx = threadIdx.x & (BX - 1), ty = threadIdx.x / BX;
    T *f = C.state[w] + (long long)shot * g.fstride;
    float *scale = C.state_scale[w] + (long long)shot * C.ntx * C.ntz + bz * C.ntx + bx;
    void *cmp = C.state_copy[w];
    T v[RZ];
    float sc = 1.f;
    if (STORE) {
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < RZ; k++) {
            const int gz = z0 + ty + k * BY, gx = x0 + tx;
            v[k] = (gz < nrow && gx < g.NX) ? f[row_off(g, gz, gx)] : T(0);
            m = fmaxf(m, fabsf((float)v[k]));
        }
        if (C.fp16) {
            const float s = pow2_scale(tile_max(m, red));
            sc = 1.f / s;
            if (threadIdx.x == 0) *scale = s;
        }
    } else if (C.fp16) {
        sc = *scale;
    }
#pragma unroll
    for (int k = 0; k < RZ; k++) {
        const int gz = z0 + ty + k * BY, gx = x0 + tx;
        if (gz >= nrow || gx >= g.NX) continue;
        const long long ci = ((long long)shot * nrow + gz) * g.NX + gx;
        if (STORE) {
            if (C.fp16) static_cast<__half *>(cmp)[ci] = __float2half_rn((float)v[k] * sc);
            else static_cast<T *>(cmp)[ci] = v[k];
        } else {
            f[row_off(g, gz, gx)] =
                C.fp16 ? T(__half2float(static_cast<const __half *>(cmp)[ci]) * sc) : static_cast<const T *>(cmp)[ci];
        }
    }
}

// Boxes of the computational grid (the CPML strips of one axis): one warp per
// (row of a box, shot). A box row is the x run [x0, x1) at one (z, y); the
// compact copy is [shot][rows of box 0, box 1, ...][x] and, in FP16, carries
// one power-of-two scale per (shot, row).
__device__ __forceinline__ int box_of(const CkBoxes &B, long long r) {
    int k = 0;
    while (k + 1 < B.n && B.row0[k + 1] <= r) k++;
    return k;
}

template <typename T, bool STORE>
__device__ __forceinline__ void box_row(const Geom &g, const CkArgs<T> &C, int j, long long w) {
    const int lane = threadIdx.x & 31;
    const CkBoxes &B = C.box[j / 2];
    const long long rows = B.row0[B.n];
    if (w >= rows * C.nshots) return;
    const int shot = (int)(w / rows);
    const long long r = w - (long long)shot * rows;
    const int k = box_of(B, r);
    const CkBox &b = B.b[k];
    const long long lr = r - B.row0[k];
    const int ny = b.y1 - b.y0, len = b.x1 - b.x0;
    const int z = b.z0 + (int)(lr / ny), y = b.y0 + (int)(lr % ny);
    T *f = C.mem[j] + (long long)shot * g.fstride + cell_off(g, z, y, b.x0);
    void *cmp = C.mem_copy[j];
    const long long e0 = (long long)shot * B.elem0[B.n] + B.elem0[k] + lr * len;
    const long long si = (long long)shot * rows + r;
    if (STORE) {
        float inv = 1.f;
        if (C.fp16) {
            float m = 0.f;
            for (int i = lane; i < len; i += 32) m = fmaxf(m, fabsf((float)f[i]));
            const float sc = pow2_scale(warp_max(m));
            inv = 1.f / sc;
            if (lane == 0) C.mem_scale[j][si] = sc;
        }
        for (int i = lane; i < len; i += 32) {
            if (C.fp16) static_cast<__half *>(cmp)[e0 + i] = __float2half_rn((float)f[i] * inv);
            else static_cast<T *>(cmp)[e0 + i] = f[i];
        }
    } else {
        const float sc = C.fp16 ? C.mem_scale[j][si] : 1.f;
        for (int i = lane; i < len; i += 32)
            f[i] = C.fp16 ? T(__half2float(static_cast<const __half *>(cmp)[e0 + i]) * sc)
                          : static_cast<const T *>(cmp)[e0 + i];
    }
}

template <typename T, bool STORE>
__global__ void __launch_bounds__(NTH) k_checkpoint(const Geom g, const __grid_constant__ CkArgs<T> C) {
    __shared__ float red[NTH / 32];
    unsigned b = blockIdx.x;
    const unsigned tiles = (unsigned)C.ntx * C.ntz, states = 2u * tiles * C.nshots;
    if (b < states) {
        const unsigned t = b % tiles, q = b / tiles;
        state_tile<T, STORE>(g, C, q & 1, t % C.ntx, t / C.ntx, q >> 1, red);
        return;
    }
    b -= states;
    int j = 0;
    while (j + 1 < C.nmem && b >= C.block0[j + 1]) j++;
    box_row<T, STORE>(g, C, j, (long long)(b - C.block0[j]) * (NTH / 32) + (threadIdx.x >> 5));
}

template <typename T>
__global__ void k_residual(const T *__restrict__ gath, const T *__restrict__ d, T *res, long long n, double *part) {
    __shared__ double sm[256];
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const T r = gath[i] - d[i];
        res[i] = r;
        acc += 0.5 * (double)r * (double)r;
    }
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

// Interior cell i gathers every computational cell whose velocity copies it:
// itself, plus the absorbing cells beyond it when it sits on an edge (a line
// of them on a face, a block on an edge or corner: (nb + 1)^3 cells on a 3D
// corner). Per cell the shots' imaging terms are summed in FP64 and scaled by
// -2 / (h^2 v) once; the cells of a block share v. A thread walking a corner
// block serially held the whole fold up (201 x 201 + 20 cells, 16 shots: 0.72
// ms; 100 x 120 x 140 + 16 cells: 3.1 ms), so the cells that gather nothing
// else go one per thread (k_fold) and the others one per warp, blocks of over
// kFoldWide cells by the whole CTA (k_fold_edge): 0.036 and 0.17 ms with them.
struct Faces {       // which ends of each axis gather absorbing cells
    int n[3];        // interior extents (z, y, x)
    int lo[3], hi[3];
    long long cells; // interior cells on one of them
};

template <typename T>
__device__ __forceinline__ double shots_sum(const T *G, long long gshot, int nshots, long long o) {
    double gs = 0.0;
    for (int s = 0; s < nshots; s++) gs += (double)G[s * gshot + o];
    return gs;
}

template <typename T>
__global__ void k_fold(const Geom g, const Faces F, const T *__restrict__ G, long long gshot, int nshots,
                       const T *__restrict__ vpad, double inv_h2, double *acc) {
    const long long nint = (long long)g.nz * g.ny * g.nx;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nint; i += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(i % g.nx);
        const long long zy = i / g.nx;
        const int iy = (int)(zy % g.ny), iz = (int)(zy / g.ny);
        if ((F.lo[0] && iz == 0) || (F.hi[0] && iz == g.nz - 1) || (F.lo[1] && iy == 0) || (F.hi[1] && iy == g.ny - 1) ||
            (F.lo[2] && ix == 0) || (F.hi[2] && ix == g.nx - 1))
            continue;
        const long long o = cell_off(g, iz + g.oz, iy + g.oy, ix + g.ox);
        acc[i] += -2.0 * inv_h2 / (double)vpad[o] * shots_sum(G, gshot, nshots, o);
    }
}

constexpr int kFoldWarps = 4;
constexpr long long kFoldWide = 512;

// Cell b of the interior cells on a gathering face: the z faces over all
// (y, x), then the y faces over the other z, then the x faces over the rest.
__device__ __forceinline__ void face_cell(const Faces &F, long long b, int *q) {
    const long long n0 = F.n[0], n1 = F.n[1], n2 = F.n[2];
    const int f0 = F.lo[0] + F.hi[0], f1 = F.lo[1] + F.hi[1], f2 = F.lo[2] + F.hi[2];
    auto end = [&](int ax, int k) { return k == 0 && F.lo[ax] ? 0 : F.n[ax] - 1; };  // the k-th face's index
    if (b < f0 * n1 * n2) {
        q[0] = end(0, (int)(b / (n1 * n2)));
        q[1] = (int)(b / n2 % n1);
        q[2] = (int)(b % n2);
        return;
    }
    b -= f0 * n1 * n2;
    const long long m0 = n0 - f0, m1 = n1 - f1;
    if (b < m0 * f1 * n2) {
        q[0] = (int)(b / (f1 * n2)) + F.lo[0];
        q[1] = end(1, (int)(b / n2 % f1));
        q[2] = (int)(b % n2);
        return;
    }
    b -= m0 * f1 * n2;
    q[0] = (int)(b / (m1 * f2)) + F.lo[0];
    q[1] = (int)(b / f2 % m1) + F.lo[1];
    q[2] = end(2, (int)(b % f2));
}

template <typename T>
__global__ void __launch_bounds__(kFoldWarps * 32) k_fold_edge(const Geom g, const Faces F, const T *__restrict__ G,
                                                               long long gshot, int nshots, const T *__restrict__ vpad,
                                                               double inv_h2, double *acc) {
    __shared__ double part[kFoldWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto block = [&](long long b, int *a, int *n, long long *i) {  // the computational cells cell b gathers
        int q[3];
        face_cell(F, b, q);
        const int o[3] = {g.oz, g.oy, g.ox}, N[3] = {g.NZ, g.NY, g.NX};
#pragma unroll
        for (int k = 0; k < 3; k++) {
            a[k] = q[k] == 0 ? 0 : q[k] + o[k];
            n[k] = (q[k] == F.n[k] - 1 ? N[k] : q[k] + o[k] + 1) - a[k];
        }
        *i = ((long long)q[0] * g.ny + q[1]) * g.nx + q[2];
        return (long long)n[0] * n[1] * n[2];
    };
    auto strided = [&](const int *a, const int *n, auto c0, auto cells, int step) {
        using I = decltype(cells);
        const I nx = (I)n[2], ny = (I)n[1];
        double s = 0.0;
#pragma unroll 4
        for (I c = c0; c < cells; c += (I)step) {
            const I r = c / nx;
            s += shots_sum(G, gshot, nshots, cell_off(g, a[0] + (int)(r / ny), a[1] + (int)(r % ny), a[2] + (int)(c % nx)));
        }
        return s;
    };
    auto sum = [&](const int *a, const int *n, int c0, long long cells, int step) {
        double s = cells >> 31 ? strided(a, n, (long long)c0, cells, step)
                               : strided(a, n, (unsigned)c0, (unsigned)cells, step);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    auto add = [&](const int *a, long long i, double s) {
        acc[i] += -2.0 * inv_h2 / (double)vpad[cell_off(g, a[0], a[1], a[2])] * s;
    };
    const long long b0 = blockIdx.x * (long long)kFoldWarps;
    int a[3], n[3];
    long long i;
    if (b0 + w < F.cells) {
        const long long cells = block(b0 + w, a, n, &i);
        if (cells <= kFoldWide) {
            const double s = sum(a, n, lane, cells, 32);
            if (lane == 0) add(a, i, s);
        }
    }
    for (int k = 0; k < kFoldWarps && b0 + k < F.cells; k++) {
        const long long cells = block(b0 + k, a, n, &i);
        if (cells <= kFoldWide) continue;
        const double s = sum(a, n, threadIdx.x, cells, kFoldWarps * 32);
        if (lane == 0) part[w] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int j = 0; j < kFoldWarps; j++) t += part[j];
            add(a, i, t);
        }
        __syncthreads();
    }
}

template <typename T>
__global__ void k_add(const double *__restrict__ acc, T *grad, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        grad[i] += (T)acc[i];
}

}  // namespace

template <typename T>
cudaError_t launch_checkpoint(const Geom &g, CkArgs<T> c, bool store, cudaStream_t st) {
    long long blocks = 0;
    for (int j = 0; j < c.nmem; j++) {
        const CkBoxes &B = c.box[j / 2];
        c.block0[j] = (unsigned)blocks;
        blocks += (B.row0[B.n] * c.nshots + NTH / 32 - 1) / (NTH / 32);
    }
    blocks += 2LL * c.ntx * c.ntz * c.nshots;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (store) k_checkpoint<T, true><<<(unsigned)blocks, NTH, 0, st>>>(g, c);
    else k_checkpoint<T, false><<<(unsigned)blocks, NTH, 0, st>>>(g, c);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_residual(const T *g, const T *d, T *res, long long n, double *part, int nblocks, cudaStream_t st) {
    k_residual<T><<<nblocks, 256, 0, st>>>(g, d, res, n, part);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fold_gradient(const Geom &g, const T *G, long long gshot, int nshots, const T *vpad,
                                 double inv_h2, double *acc, cudaStream_t st) {
    Faces F{};
    const int n[3] = {g.nz, g.ny, g.nx}, o[3] = {g.oz, g.oy, g.ox}, N[3] = {g.NZ, g.NY, g.NX};
    long long plain = 1;  // interior cells on no gathering face
    for (int k = 0; k < 3; k++) {
        F.n[k] = n[k];
        F.lo[k] = o[k] > 0;
        F.hi[k] = N[k] > o[k] + n[k] && !(F.lo[k] && n[k] == 1);  // one cell gathers both ends: one face
        plain *= n[k] - F.lo[k] - F.hi[k];
    }
    F.cells = (long long)g.nz * g.ny * g.nx - plain;
    if (plain > 0) k_fold<T><<<1216, 256, 0, st>>>(g, F, G, gshot, nshots, vpad, inv_h2, acc);
    if (F.cells > 0)
        k_fold_edge<T><<<(unsigned)((F.cells + kFoldWarps - 1) / kFoldWarps), kFoldWarps * 32, 0, st>>>(
            g, F, G, gshot, nshots, vpad, inv_h2, acc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_add_gradient(const double *acc, T *grad, long long n, cudaStream_t st) {
    k_add<T><<<1216, 256, 0, st>>>(acc, grad, n);
    return cudaGetLastError();
}

#define INST(T)                                                                                               \
    template cudaError_t launch_checkpoint<T>(const Geom &, CkArgs<T>, bool, cudaStream_t);                   \
    template cudaError_t launch_residual<T>(const T *, const T *, T *, long long, double *, int, cudaStream_t); \
    template cudaError_t launch_fold_gradient<T>(const Geom &, const T *, long long, int, const T *,      \
                                                 double, double *, cudaStream_t);                             \
    template cudaError_t launch_add_gradient<T>(const double *, T *, long long, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace gsim
