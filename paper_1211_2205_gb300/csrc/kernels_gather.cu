// Gather kernel of the half-step pass and small helper kernels.
//
// k_gather_pass updates every output component of one grid at one point per
// thread: W = sum_k cx_k (u_k(right) - u_k(left)) + sum_k cy_k (u_k(up) -
// u_k(down)) with cx = -Mx[j][k]/dx, cy = -My[j][k]/dy (the weighted sparse
// sum of section 5.5 over eq. central_differences), then the exact sub-step
// u <- a u + b (W + q) (eq. sub_step_solution with a = exp(-c tau),
// b = tau E(-c tau), tau = dt/2 for a half-step, dt for the fused even pair
// or a merged odd pair).  It serves FP64 runs, the slab system and any N.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "pdl.h"

namespace starmap {

namespace {

// Write u at point (x, y) of a component and its boundary copies.
template <class T>
__device__ __forceinline__ void store_point(T* comp, long pitch, int x, int y, int nx, int ny,
                                            bool xnode, bool ynode, int px, int py, T v) {
    comp[(long)(y + 1) * pitch + x] = v;
    int gxa = -2, gxb = -2;
    if (px) { if (x == nx - 1) gxa = -1; if (x == 0) gxb = nx; }
    else if (!xnode) { if (x == 0) gxa = -1; if (x == nx - 1) gxb = nx; }
    if (gxa != -2) comp[(long)(y + 1) * pitch + gxa] = v;
    if (gxb != -2) comp[(long)(y + 1) * pitch + gxb] = v;
    int gya = -2, gyb = -2;
    if (py) { if (y == ny - 1) gya = -1; if (y == 0) gyb = ny; }
    else if (!ynode) { if (y == 0) gya = -1; if (y == ny - 1) gyb = ny; }
    if (gya != -2) comp[(long)(gya + 1) * pitch + x] = v;
    if (gyb != -2) comp[(long)(gyb + 1) * pitch + x] = v;
}

// Corner boundary copy t (0: (-1,-1), 1: (nx,-1), 2: (-1,ny), 3: (nx,ny)):
// where both axes keep a copy on that side, the x rule applied to the y
// copy.  The passes never read corners; the fused step's even update does
// at the points it adds beyond a periodic edge next to a corner.
template <class T>
__device__ __forceinline__ void corner_ghost(T* comp, long pitch, int nx, int ny, bool xnode, bool ynode,
                                             int px, int py, int t) {
    const bool hx = px || !xnode, hy = py || !ynode;
    if (!hx || !hy) return;
    const bool right = t & 1, top = t & 2;
    const int gx = right ? nx : -1, gy = top ? ny : -1;
    const int sx = right ? (px ? 0 : nx - 1) : (px ? nx - 1 : 0);
    const int sy = top ? (py ? 0 : ny - 1) : (py ? ny - 1 : 0);
    comp[(long)(gy + 1) * pitch + gx] = comp[(long)(sy + 1) * pitch + sx];
}

// Boundary copies of one component as independent items.  A column copy
// lands in a 32-byte sector that holds nothing else of use, so the item
// that writes it stores the sector whole (fewer partial stores, which make
// DRAM read the sector first):
//   items [0, ny)                row y's gap [nx, pitch): the sector holding
//                                nx (the interior values in it kept, row y's
//                                right copy at nx, zero padding) and the row's
//                                last sector (row y + 1's left copy at
//                                pitch - 1, zero padding)
//   items [.., + 2 nx)           rows -1 and ny (where the y axis keeps copies)
//   4 items                      single stores: row 0's left copy and the
//                                corners (-1,-1), (nx,-1), (nx,ny); the corner
//                                (-1,ny) is row ny - 1's gap
// Only padding lies between nx and pitch - 1 (pitch >= nx + 6); the copies
// follow the rules of store_point, corners those of corner_ghost.
// (Reading the boundary values costs a 128-byte line each from DRAM: one
// line per row and side is what bounds this kernel.)
__device__ __forceinline__ void store_sector(float* dst, const float (&v)[8]) {
    reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

__host__ __device__ __forceinline__ int ghost_items(int nx, int ny, bool hx, bool hy) {
    return (hx ? ny : 0) + (hy ? 2 * nx : 0) + 4;
}

__device__ __forceinline__ void ghost_item(float* comp, long pitch, int nx, int ny, bool xnode, bool ynode,
                                           int px, int py, int i) {
    constexpr int EPS = 32 / (int)sizeof(float);     // elements per 32-byte sector
    const bool hx = px || !xnode, hy = py || !ynode;
    const int xl = px ? nx - 1 : 0, xr = px ? 0 : nx - 1;          // sources of the left / right copies
    const int ylo = py ? ny - 1 : 0, yhi = py ? 0 : ny - 1;        // sources of rows -1 and ny
    auto at = [&](int x, int y) -> float& { return comp[(long)(y + 1) * pitch + x]; };
    if (hx) {
        if (i < ny) {
            const int y = i;
            float* row = &at(0, y);
            const int a0 = nx & ~(EPS - 1), b0 = (int)pitch - EPS;
            float sa[EPS];
#pragma unroll
            for (int e = 0; e < EPS; ++e) {
                const int x = a0 + e;
                sa[e] = x < nx ? row[x] : (x == nx ? row[xr] : 0.f);
            }
            // left copy of row y + 1 (for the last row: the corner (-1, ny))
            const float left = y + 1 < ny ? at(xl, y + 1) : (hy ? at(xl, yhi) : 0.f);
            if (a0 == b0) {
                sa[EPS - 1] = left;
            } else {
                float sb[EPS];
#pragma unroll
                for (int e = 0; e < EPS; ++e) sb[e] = 0.f;
                sb[EPS - 1] = left;
                store_sector(row + b0, sb);
            }
            store_sector(row + a0, sa);
            return;
        }
        i -= ny;
    }
    if (hy) {
        if (i < nx) { at(i, -1) = at(i, ylo); return; }
        if (i < 2 * nx) { at(i - nx, ny) = at(i - nx, yhi); return; }
        i -= 2 * nx;
    }
    if (i == 0) { if (hx) at(-1, 0) = at(xl, 0); return; }
    if (!hx || !hy) return;
    if (i == 1) at(-1, -1) = at(xl, ylo);
    else if (i == 2) at(nx, -1) = at(xr, ylo);
    else if (i == 3) at(nx, ny) = at(xr, yhi);
}

// w + sum_k c[k] (p[k] - m[k]) over the first n of up to four terms, in
// order, as straight lines: an FP64 operation predicated off takes its 64
// clocks of the unit all the same.
template <class T>
__device__ __forceinline__ T add_terms(T w, int n, const T (&c)[MAXC], const T (&p)[MAXC], const T (&m)[MAXC]) {
    static_assert(MAXC == 4, "up to four couplings per direction");
    switch (n) {
        case 4:
            return w + c[0] * (p[0] - m[0]) + c[1] * (p[1] - m[1]) + c[2] * (p[2] - m[2]) + c[3] * (p[3] - m[3]);
        case 3: return w + c[0] * (p[0] - m[0]) + c[1] * (p[1] - m[1]) + c[2] * (p[2] - m[2]);
        case 2: return w + c[0] * (p[0] - m[0]) + c[1] * (p[1] - m[1]);
        case 1: return w + c[0] * (p[0] - m[0]);
        default: return w;
    }
}

// Both output grids of a pass in one launch: blockIdx.z = slice, the first
// A.slices[0] of them on output grid 0, the others on grid 1; output t of a
// grid goes to slice (t - begin) mod slices.  On small grids, where a thread
// has one output, the launch, a table load and a chain of loads and FP64
// operations (64 clocks each, one at a time per warp) are the pass: the
// tables and decay coefficients, host-written, are loaded before the
// previous pass is waited for (pdl.h).
// ROWS: a row of blocks per row of points (blockIdx.y), for long rows: no
// division, and with more warps in flight (72 registers instead of 88) and
// all loads of an output together.  us per pass, without / with: FP32 P_1
// 1500^2 50 / 39, P_3 142 / 106, P_39 256^2 352 / 241; slab of 60000 cells
// FP64 P_63 38 / 31.
template <class T, bool ROWS>
__device__ __forceinline__ void gather_pass(const GatherArgs<T>& A) {
    pdl_trigger();
    if (ROWS) pdl_wait();
    const int K = (int)blockIdx.z < A.slices[0] ? 0 : 1;
    const int slice = (int)blockIdx.z - (K ? A.slices[0] : 0);
    const GridDev<T>& G = A.out[K];
    const int nx = G.nx, ny = G.ny;
    int ix, iy;
    bool inside;
    if (ROWS) {
        ix = blockIdx.x * blockDim.x + threadIdx.x;
        iy = blockIdx.y;
        inside = ix < nx && iy < ny;
    } else {
        // points in rows one after the other: no lanes idle at a row's end (an FP64 operation costs a warp of
        // four lanes what it costs a whole one)
        const unsigned long long point = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
        inside = point < (unsigned long long)nx * ny;
        iy = point >> 32 ? (int)(point / nx) : (int)((unsigned)point / (unsigned)nx);
        ix = (int)(point - (unsigned long long)iy * nx);
    }
    const bool xnode = (A.grid[K] & 1) != 0, ynode = (A.grid[K] & 2) != 0;
    const long pitch = A.pitch;
    // right / upper neighbour in the partner grid (eq. central_differences)
    const T* Xb = A.xin[K].base + (long)(iy + 1) * pitch + ix + (xnode ? A.p[0] : 1 - A.p[0]);
    const T* Yb = A.yin[K].base + (long)(iy + 1 + (ynode ? A.p[1] : 1 - A.p[1])) * pitch + ix;
    const long cxs = A.xin[K].cstride, cys = A.yin[K].cstride;
    T* self = G.base + (long)(iy + 1) * pitch + ix;
    const long cidx = inside ? (long)iy * G.cp + ix : 0;
    const long plane = (long)G.cp * ny;
    bool waited = ROWS;
    for (int t = A.begin[K] + slice; t < A.end[K]; t += A.slices[K]) {
        const GatherOut o = A.outs[t];
        const GatherCoef<T> c = A.coefs[t];
        const T* cf = G.coef + ((long)o.cls * 4 + 2 * A.which) * plane + cidx;
        const T a = cf[0];
        const T bb = cf[plane];
        const T q = o.src >= 0 ? A.src[o.src][cidx] : T(0);
        if (!waited) {
            pdl_wait();
            waited = true;
        }
        if (!inside) continue;
        T r[MAXC], l[MAXC], u[MAXC], d[MAXC];
#pragma unroll
        for (int k = 0; k < MAXC; ++k) {
            const T* x = Xb + (long)o.xin[k] * cxs;
            const T* y = Yb + (long)o.yin[k] * cys;
            r[k] = k < o.nxt ? x[0] : T(0);
            l[k] = k < o.nxt ? x[-1] : T(0);
            u[k] = k < o.nyt ? y[0] : T(0);
            d[k] = k < o.nyt ? y[-pitch] : T(0);
        }
        T* comp = G.base + (long)o.local * G.cstride;
        const T old = self[(long)o.local * G.cstride];
        T w = add_terms<T>(T(0), o.nxt, c.cx, r, l);
        w = add_terms<T>(w, o.nyt, c.cy, u, d);
        if (o.src >= 0) w += q;
        const T v = a * old + bb * w;
        store_point(comp, pitch, ix, iy, nx, ny, xnode, ynode, A.p[0], A.p[1], v);
    }
    if (!waited) pdl_wait();
}
template <class T>
__global__ void __launch_bounds__(128) k_gather_pass(const __grid_constant__ GatherArgs<T> A) {
    gather_pass<T, false>(A);
}
template <class T>
__global__ void __launch_bounds__(128, 7) k_gather_rows(const __grid_constant__ GatherArgs<T> A) {
    gather_pass<T, true>(A);
}

// Refresh the boundary copies of components [kbegin, kend) of one grid.
template <class T>
__global__ void k_fill_ghosts(const GhostArgs<T> A) {
    const GridDev<T>& G = A.g;
    const long per = 2L * G.nx + 2L * G.ny;
    const long total = per * (A.kend - A.kbegin);
    const bool xnode = (A.grid & 1) != 0, ynode = (A.grid & 2) != 0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const int k = A.kbegin + (int)(t / per);
        long r = t % per;
        int x, y;
        if (r < G.nx) { x = (int)r; y = 0; }
        else if (r < 2L * G.nx) { x = (int)(r - G.nx); y = G.ny - 1; }
        else if (r < 2L * G.nx + G.ny) { x = 0; y = (int)(r - 2L * G.nx); }
        else { x = G.nx - 1; y = (int)(r - 2L * G.nx - G.ny); }
        T* comp = G.base + (long)k * G.cstride;
        const T v = comp[(long)(y + 1) * A.pitch + x];
        store_point(comp, A.pitch, x, y, G.nx, G.ny, xnode, ynode, A.p[0], A.p[1], v);
    }
    const long corners = 4L * (A.kend - A.kbegin);
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < corners; t += (long)gridDim.x * blockDim.x)
        corner_ghost(G.base + (long)(A.kbegin + t / 4) * G.cstride, A.pitch, G.nx, G.ny, xnode, ynode, A.p[0], A.p[1],
                     (int)(t % 4));
}

// Boundary copies of the odd grids after a fused step, whose kernel leaves
// them out: blockIdx.y runs over the components of both grids, threads over
// the items of a component (ghost_item).
__global__ void k_fill_ghosts_pass(const GhostPassArgs A) {
    const int c = blockIdx.y;
    const int which = c < A.g[0].K ? 0 : 1;
    const GridDev<float>& G = A.g[which];
    const int k = which ? c - A.g[0].K : c;
    const bool xnode = (A.grid[which] & 1) != 0, ynode = (A.grid[which] & 2) != 0;
    float* comp = G.base + (long)k * G.cstride;
    const int nx = G.nx, ny = G.ny;
    const int items = ghost_items(nx, ny, A.p[0] || !xnode, A.p[1] || !ynode);
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < items; r += gridDim.x * blockDim.x)
        ghost_item(comp, A.pitch, nx, ny, xnode, ynode, A.p[0], A.p[1], r);
}

// Deterministic FP64 reduction: per-block partials (mass, sum of squares,
// non-finite count) over all rows of all grids, then one block sums them in
// a fixed order.
template <class T>
__global__ void k_reduce_partials(const ReduceArgs<T> A, double* partials) {
    __shared__ double sh[3][256];
    double mass = 0.0, sq = 0.0, bad = 0.0;
    long rows_total = 0;
    for (int g = 0; g < 4; ++g) rows_total += (long)A.g[g].K * A.g[g].ny;
    for (long r = blockIdx.x; r < rows_total; r += gridDim.x) {
        long rr = r;
        int g = 0;
        while (rr >= (long)A.g[g].K * A.g[g].ny) { rr -= (long)A.g[g].K * A.g[g].ny; ++g; }
        const GridDev<T>& G = A.g[g];
        const int k = (int)(rr / G.ny), y = (int)(rr % G.ny);
        const T* row = G.base + (long)k * G.cstride + (long)(y + A.row0) * A.pitch;
        for (int x = threadIdx.x; x < G.nx; x += blockDim.x) {
            const double v = (double)row[x];
            if (!isfinite(v)) { bad += 1.0; continue; }
            sq += v * v;
            if (g == 0 && k == 0) mass += v;
        }
    }
    sh[0][threadIdx.x] = mass;
    sh[1][threadIdx.x] = sq;
    sh[2][threadIdx.x] = bad;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < 3; ++q) partials[blockIdx.x * 3 + q] = sh[q][0];
}

__global__ void k_reduce_final(const double* partials, int nblocks, double cell, double* out) {
    __shared__ double sh[3][256];
    double acc[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
        for (int q = 0; q < 3; ++q) acc[q] += partials[b * 3 + q];
    for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] = acc[q];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sh[0][0] * cell;
        out[1] = sqrt(sh[1][0] * cell);
        out[2] = sh[2][0];
    }
}

template <class T>
__global__ void k_axpby(T* out, const T* x, const T* y, double alpha, double beta, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = (T)(alpha * (double)x[i] + beta * (double)y[i]);
}

int status_of(cudaError_t e) { return e == cudaSuccess ? 0 : -4; }

}  // namespace

static int sm_count_gather() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
    }
    return n;
}

template <class T>
int launch_gather_pass(GatherArgs<T> a, void* stream) {
    long points = 0;
    int outs = 0;
    for (int K = 0; K < 2; ++K) {
        if (a.end[K] <= a.begin[K]) continue;
        points = std::max(points, (long)a.out[K].nx * a.out[K].ny);
        outs += a.end[K] - a.begin[K];
    }
    if (outs == 0 || points == 0) return 0;
    // one thread per point walks a slice of a grid's outputs; on a small grid
    // the outputs are dealt over more slices, so that about two waves of
    // threads fill the GPU
    const int width = 128;
    const long threads = (points + width - 1) / width * width;
    const long want = 2L * 2048 * sm_count_gather();
    for (int K = 0; K < 2; ++K) {
        const int n = a.end[K] - a.begin[K];
        const long z = threads >= want ? 1 : (want * std::max(n, 0) / outs + threads - 1) / threads;
        a.slices[K] = n <= 0 ? 0 : (int)std::min<long>(std::min<long>(std::max<long>(z, 1), n), 64);
    }
    // By rows where a sixteenth of the lanes at most is idle for it, from the size on where the loads' latency
    // and not the launch's counts.  us per pass, without / with: FP32 256^2 P_1 (98 k values) 2.3 / 3.2, P_7 12.9 /
    // 12.1, 512^2 P_1 (393 k) 5.5 / 5.6, P_2 9.3 / 8.8; slabs of 10000 cells, FP64 P_15 (80 k) 2.9 / 4.2, P_31 5.2 /
    // 4.9, FP32 P_63 (320 k) 5.0 / 5.1; 120 x 90 (a fifteenth idle) P_60 99 / 102
    const int nxmax = std::max(a.out[0].nx, a.out[1].nx), nymax = std::max(a.out[0].ny, a.out[1].ny);
    const int per_row = (nxmax + width - 1) / width;
    const bool rows = points * outs >= (sizeof(T) == 8 ? 150000 : 500000) && 16L * per_row * width <= 17L * nxmax &&
                      nymax <= 65535;
    const dim3 grid = rows ? dim3(per_row, nymax, a.slices[0] + a.slices[1])
                           : dim3((unsigned)(threads / width), 1, a.slices[0] + a.slices[1]);
    const cudaError_t e = launch_pdl(rows ? k_gather_rows<T> : k_gather_pass<T>, grid, dim3(width), 0,
                                     (cudaStream_t)stream, threads < want, a);
    return status_of(e != cudaSuccess ? e : cudaGetLastError());
}

template <class T>
int launch_fill_ghosts(const GhostArgs<T>& a, void* stream) {
    if (a.kend <= a.kbegin || a.g.nx == 0) return 0;
    long total = (2L * a.g.nx + 2L * a.g.ny) * (a.kend - a.kbegin);
    int blocks = (int)((total + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    k_fill_ghosts<T><<<blocks, 256, 0, (cudaStream_t)stream>>>(a);
    return status_of(cudaGetLastError());
}

int launch_fill_ghosts_pass(const GhostPassArgs& a, void* stream) {
    const int K = a.g[0].K + a.g[1].K;
    if (K <= 0) return 0;
    const int len = std::max(ghost_items(a.g[0].nx, a.g[0].ny, true, true), ghost_items(a.g[1].nx, a.g[1].ny, true, true));
    const dim3 grid((len + 255) / 256, K);
    k_fill_ghosts_pass<<<grid, 256, 0, (cudaStream_t)stream>>>(a);
    return status_of(cudaGetLastError());
}

template <class T>
int launch_reduce(const ReduceArgs<T>& a, double* partials, int nblocks, double* result, void* stream) {
    k_reduce_partials<T><<<nblocks, 256, 0, (cudaStream_t)stream>>>(a, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return status_of(e);
    k_reduce_final<<<1, 256, 0, (cudaStream_t)stream>>>(partials, nblocks, a.cell, result);
    return status_of(cudaGetLastError());
}

template <class T>
int launch_axpby(T* out, const T* x, const T* y, double alpha, double beta, size_t n, void* stream) {
    if (n == 0) return 0;
    size_t blocks = (n + 255) / 256;
    if (blocks > 65536) blocks = 65536;
    k_axpby<T><<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(out, x, y, alpha, beta, n);
    return status_of(cudaGetLastError());
}

template int launch_gather_pass<float>(GatherArgs<float>, void*);
template int launch_gather_pass<double>(GatherArgs<double>, void*);
template int launch_fill_ghosts<float>(const GhostArgs<float>&, void*);
template int launch_fill_ghosts<double>(const GhostArgs<double>&, void*);
template int launch_reduce<float>(const ReduceArgs<float>&, double*, int, double*, void*);
template int launch_reduce<double>(const ReduceArgs<double>&, double*, int, double*, void*);
template int launch_axpby<float>(float*, const float*, const float*, double, double, size_t, void*);
template int launch_axpby<double>(double*, const double*, const double*, double, double, size_t, void*);

}  // namespace starmap
