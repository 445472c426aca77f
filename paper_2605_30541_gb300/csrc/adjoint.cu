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
    const int tid = threadIdx.y * BX + threadIdx.x;
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

// One CTA per (tile of rows x columns, shot); the compact copy of a state is
// [shot][NZ NY NX].
template <typename T>
__global__ void __launch_bounds__(NTH) k_store(const Geom g, const T *__restrict__ field, void *dst, float *scale,
                                               int fp16, long long sstride, int ntx) {
    __shared__ float red[NTH / 32];
    const int x0 = blockIdx.x * TX, z0 = blockIdx.y * TZ, shot = blockIdx.z, nrow = g.NZ * g.NY;
    const int tile = blockIdx.y * ntx + blockIdx.x, ntiles = ntx * gridDim.y;
    const T *f = field + (long long)shot * g.fstride;
    T v[RZ];
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < RZ; k++) {
        const int gz = z0 + threadIdx.y + k * BY, gx = x0 + threadIdx.x;
        v[k] = (gz < nrow && gx < g.NX) ? f[row_off(g, gz, gx)] : T(0);
        m = fmaxf(m, fabsf((float)v[k]));
    }
    float inv = 1.f;
    if (fp16) {
        const float s = pow2_scale(tile_max(m, red));
        inv = 1.f / s;
        if (threadIdx.x == 0 && threadIdx.y == 0) scale[(long long)shot * ntiles + tile] = s;
    }
#pragma unroll
    for (int k = 0; k < RZ; k++) {
        const int gz = z0 + threadIdx.y + k * BY, gx = x0 + threadIdx.x;
        if (gz >= nrow || gx >= g.NX) continue;
        const long long ci = shot * sstride + (long long)gz * g.NX + gx;
        if (fp16) static_cast<__half *>(dst)[ci] = __float2half_rn((float)v[k] * inv);
        else static_cast<T *>(dst)[ci] = v[k];
    }
}

template <typename T>
__global__ void __launch_bounds__(NTH) k_load(const Geom g, T *field, const void *src, const float *scale, int fp16,
                                              long long sstride, int ntx) {
    const int x0 = blockIdx.x * TX, z0 = blockIdx.y * TZ, shot = blockIdx.z, nrow = g.NZ * g.NY;
    const int tile = blockIdx.y * ntx + blockIdx.x, ntiles = ntx * gridDim.y;
    T *f = field + (long long)shot * g.fstride;
    const float s = fp16 ? scale[(long long)shot * ntiles + tile] : 1.f;
#pragma unroll
    for (int k = 0; k < RZ; k++) {
        const int gz = z0 + threadIdx.y + k * BY, gx = x0 + threadIdx.x;
        if (gz >= nrow || gx >= g.NX) continue;
        const long long ci = shot * sstride + (long long)gz * g.NX + gx;
        f[row_off(g, gz, gx)] =
            fp16 ? T(__half2float(static_cast<const __half *>(src)[ci]) * s) : static_cast<const T *>(src)[ci];
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
__global__ void __launch_bounds__(256) k_boxes(const Geom g, const CkBoxes B, T *field, void *cmp, float *scale,
                                               int fp16, int nshots) {
    const int lane = threadIdx.x & 31;
    const long long rows = B.row0[B.n];
    const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    if (w >= rows * nshots) return;
    const int shot = (int)(w / rows);
    const long long r = w - (long long)shot * rows;
    const int k = box_of(B, r);
    const CkBox &b = B.b[k];
    const long long lr = r - B.row0[k];
    const int ny = b.y1 - b.y0, len = b.x1 - b.x0;
    const int z = b.z0 + (int)(lr / ny), y = b.y0 + (int)(lr % ny);
    T *f = field + (long long)shot * g.fstride + cell_off(g, z, y, b.x0);
    const long long e0 = (long long)shot * B.elem0[B.n] + B.elem0[k] + lr * len;
    const long long si = (long long)shot * rows + r;
    if (STORE) {
        float inv = 1.f;
        if (fp16) {
            float m = 0.f;
            for (int i = lane; i < len; i += 32) m = fmaxf(m, fabsf((float)f[i]));
            const float sc = pow2_scale(warp_max(m));
            inv = 1.f / sc;
            if (lane == 0) scale[si] = sc;
        }
        for (int i = lane; i < len; i += 32) {
            if (fp16) static_cast<__half *>(cmp)[e0 + i] = __float2half_rn((float)f[i] * inv);
            else static_cast<T *>(cmp)[e0 + i] = f[i];
        }
    } else {
        const float sc = fp16 ? scale[si] : 1.f;
        for (int i = lane; i < len; i += 32)
            f[i] = fp16 ? T(__half2float(static_cast<const __half *>(cmp)[e0 + i]) * sc) : static_cast<const T *>(cmp)[e0 + i];
    }
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
cudaError_t launch_store_state(const Geom &g, const T *field, void *dst, float *scale, int fp16, int nshots,
                               long long shot_stride, int ntx, int ntz, cudaStream_t st) {
    k_store<T><<<dim3(ntx, ntz, nshots), dim3(BX, BY), 0, st>>>(g, field, dst, scale, fp16, shot_stride, ntx);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_load_state(const Geom &g, T *field, const void *src, const float *scale, int fp16, int nshots,
                              long long shot_stride, int ntx, int ntz, cudaStream_t st) {
    k_load<T><<<dim3(ntx, ntz, nshots), dim3(BX, BY), 0, st>>>(g, field, src, scale, fp16, shot_stride, ntx);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_store_boxes(const Geom &g, const CkBoxes &b, const T *field, void *dst, float *scale, int fp16,
                               int nshots, cudaStream_t st) {
    const long long warps = b.row0[b.n] * nshots;
    if (warps == 0) return cudaSuccess;
    k_boxes<T, true><<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(g, b, const_cast<T *>(field), dst, scale, fp16,
                                                                  nshots);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_load_boxes(const Geom &g, const CkBoxes &b, T *field, const void *src, const float *scale,
                              int fp16, int nshots, cudaStream_t st) {
    const long long warps = b.row0[b.n] * nshots;
    if (warps == 0) return cudaSuccess;
    k_boxes<T, false><<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(g, b, field, const_cast<void *>(src),
                                                                   const_cast<float *>(scale), fp16, nshots);
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
    template cudaError_t launch_store_state<T>(const Geom &, const T *, void *, float *, int, int, long long,  \
                                               int, int, cudaStream_t);                                       \
    template cudaError_t launch_load_state<T>(const Geom &, T *, const void *, const float *, int, int,        \
                                              long long, int, int, cudaStream_t);                             \
    template cudaError_t launch_store_boxes<T>(const Geom &, const CkBoxes &, const T *, void *, float *, int, int, \
                                               cudaStream_t);                                                \
    template cudaError_t launch_load_boxes<T>(const Geom &, const CkBoxes &, T *, const void *, const float *, int, \
                                              int, cudaStream_t);                                            \
    template cudaError_t launch_residual<T>(const T *, const T *, T *, long long, double *, int, cudaStream_t); \
    template cudaError_t launch_fold_gradient<T>(const Geom &, const T *, long long, int, const T *,      \
                                                 double, double *, cudaStream_t);                             \
    template cudaError_t launch_add_gradient<T>(const double *, T *, long long, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace gsim
