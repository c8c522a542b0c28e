// FP64 half-step pass of the 2D real P_N system, moments streamed by order.
//
// A thread owns a point of one output kind (R: G21 / G11, I: G12 / G22) and
// walks the inputs (l', q') of the pass in order, like the tiled FP32 kernel
// (tiled_kernel.cuh, which explains the reach of an input, the partial sums
// and the stages): each input's two half-grid differences (eq.
// central_differences) are formed once per point and kind, where the gather
// kernel forms them for every target that uses them.
//
// The couplings of a target to the R and the I input of one (l', q') have the
// same size (both are parts of one complex coefficient of eq. Pncomplex):
// My = r Mx, r = -1 (R targets) or 1 (I targets) for the targets of m = m' + 1
// (Pm, N0) and the opposite for those of m = m' - 1 (P0, Np); stream_build
// checks every entry.  So with s = d_x + r (dx/dy) d_y and t = d_x - r (dx/dy)
// d_y each target takes one weighted term per input, not two.
//
// What bounds it: the FP64 units.  One operation of a warp takes 64 clocks of
// its scheduler's unit, predicated off or not (P_39 on 256^2: 14 828 of them
// per scheduler keep it busy 82 % of 1 140 895 clocks).  Per value a pass spends 8 to
// 9.7 of them (N = 5 to 39: two differences, s and t, four weighted terms,
// the decayed update) where the gather kernel spends 11.5 to 17; loads,
// tables and addresses issue in their shadow.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "pdl.h"
#include "stream.h"

namespace starmap {

// The records of one pass and kind, with the component each of them completes
// (-1: none).
struct Records {
    std::vector<StreamRec> rec;
    std::vector<PairRec> pair;
    std::vector<int> rec_comp, pair_comp;
    size_t rec_at = 0, pair_at = 0;                                    // bytes into the device buffer
};

struct StreamTables {
    Records r[2][2];                                                   // [P][K]
    std::vector<unsigned char> image;                                  // of the device buffer
    DevTable dev;
    int N = 1;
    int slots = 0;                                                     // partial sums per thread
    double rho = 1.0;                                                  // dx / dy
    int sms = 1;
    int resident[2] = {1, 1};                                          // streaming blocks on an SM, pass P
};

namespace {

struct KernelArgs {
    GridDev<double> own[2], other[2], out[2];   // per kind: its input grid, the other kind's, its output grid
    const StreamRec* rec[2];
    const PairRec* pair[2];
    int outs[2], slices[2];     // k_pair_pass: outputs of a kind, blockIdx.y's slices of them
    int out_grid[2];
    // slots is not read by the kernels: with these two others alone the compiler gives k_stream_pass 64 registers
    // instead of 70, and P_63 takes 2 % longer, P_13 2 % at 256^2 (and 1 % less at 512^2)
    int count, slots, which;
    long pitch;
    int p[2];
    double rho, minus_rho;      // (a negation on the device is an FP64 operation)
    double* const* src;
};

// A thread's point of the output grid of kind K (points in rows one after
// the other: no lanes idle at a row's end).
struct Point {
    const double *bx, *by;      // right / upper neighbours in the input grids, component 0
    double* bo;                 // the point, component 0
    long cidx;                  // its coefficients and sources
    // boundary copies (section 4.2): along x at +xo (and +xo2), along y at +yo (and +yo2), 0 for none
    long xo, xo2, yo, yo2;
    bool inside;
};

__device__ __forceinline__ Point point_of(const KernelArgs& A, int K) {
    Point p;
    const GridDev<double>& G = A.out[K];
    const int nx = G.nx, ny = G.ny;
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    p.inside = i < (unsigned long long)nx * ny;
    const int y = i >> 32 ? (int)(i / nx) : (int)((unsigned)i / (unsigned)nx);
    const int x = (int)(i - (unsigned long long)y * nx);
    const long pitch = A.pitch;
    const bool xnode = A.out_grid[K] & 1, ynode = A.out_grid[K] & 2;
    p.bx = A.own[K].base + (long)(y + 1) * pitch + x + (xnode ? A.p[0] : 1 - A.p[0]);
    p.by = A.other[K].base + (long)(y + 1 + (ynode ? A.p[1] : 1 - A.p[1])) * pitch + x;
    p.bo = G.base + (long)(y + 1) * pitch + x;
    p.cidx = p.inside ? (long)y * G.cp + x : 0;
    p.xo = p.xo2 = p.yo = p.yo2 = 0;
    if (A.p[0] || !xnode) {
        if (x == (A.p[0] ? nx - 1 : 0)) p.xo = -1 - x;
        if (x == (A.p[0] ? 0 : nx - 1)) (p.xo ? p.xo2 : p.xo) = nx - x;
    }
    if (A.p[1] || !ynode) {
        if (y == (A.p[1] ? ny - 1 : 0)) p.yo = (long)(-1 - y) * pitch;
        if (y == (A.p[1] ? 0 : ny - 1)) (p.yo ? p.yo2 : p.yo) = (long)(ny - y) * pitch;
    }
    return p;
}

__device__ __forceinline__ void store(double* d, const Point& p, double u) {
    d[0] = u;
    if (p.xo || p.yo) {
        if (p.xo) d[p.xo] = u;
        if (p.xo2) d[p.xo2] = u;
        if (p.yo) {
            d[p.yo] = u;
            if (p.xo) d[p.yo + p.xo] = u;
            if (p.xo2) d[p.yo + p.xo2] = u;
        }
        if (p.yo2) {
            d[p.yo2] = u;
            if (p.xo) d[p.yo2 + p.xo] = u;
            if (p.xo2) d[p.yo2 + p.xo2] = u;
        }
    }
}

// The first C pairs, in order, as one straight line (see the kernel below on
// predicated FP64 operations).
template <int C>
__device__ __forceinline__ double pair_sum(const PairRec& r, const double (&v)[4][4], double rho, double minus_rho) {
    double W = 0.0;
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const double s = fma(r.t >> k & 1 ? minus_rho : rho, v[k][2] - v[k][3], v[k][0] - v[k][1]);
        W = k ? fma(r.w[k], s, W) : r.w[k] * s;
    }
    return W;
}

// Small grids: one output per thread (blockIdx.y: slices of the outputs of
// both kinds), the same operations on it in the same order as the stages
// above, so both kernels give the same values bit for bit.  A pass is then
// the launch, one chain of loads and one of 10 to 18 FP64 operations; records
// and coefficients, host-written, are loaded before the previous pass is
// waited for.  100^2 P_5: 13 us per pass with a launch per grid, tables in
// local memory and no overlap, 5.5 so.
// Wide: the same on large grids of N <= 2, where the streamed chain is too
// short to be worth its stages and the warps in flight are what counts: 64
// registers instead of 94.
__device__ __forceinline__ void pair_pass(const KernelArgs& A) {
    pdl_trigger();
    const int K = (int)blockIdx.y < A.slices[0] ? 0 : 1;
    const int slice = (int)blockIdx.y - (K ? A.slices[0] : 0);
    const GridDev<double>& G = A.out[K];
    const Point pt = point_of(A, K);
    const long cx = A.own[K].cstride, cy = A.other[K].cstride, pitch = A.pitch;
    const long plane = (long)G.cp * G.ny;
    const double rho = K == 0 ? A.minus_rho : A.rho, minus_rho = K == 0 ? A.rho : A.minus_rho;
    bool waited = false;
    for (int i = slice; i < A.outs[K]; i += A.slices[K]) {
        const PairRec r = A.pair[K][i];
        const double* cf = G.coef + ((long)r.cls * 4 + 2 * A.which) * plane + pt.cidx;
        const double a = cf[0], b = cf[plane];
        const double q = r.src >= 0 ? A.src[r.src][pt.cidx] : 0.0;
        if (!waited) {
            pdl_wait();
            waited = true;
        }
        if (!pt.inside) continue;
        double v[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double *px = pt.bx + r.own[k] * cx, *py = pt.by + r.other[k] * cy;
            v[k][0] = r.own[k] >= 0 ? px[0] : 0.0;
            v[k][1] = r.own[k] >= 0 ? px[-1] : 0.0;
            v[k][2] = r.other[k] >= 0 ? py[0] : 0.0;
            v[k][3] = r.other[k] >= 0 ? py[-pitch] : 0.0;
        }
        double* d = pt.bo + r.out * G.cstride;
        const double old = d[0];
        double W = 0.0;
        switch (r.count) {
            case 4: W = pair_sum<4>(r, v, rho, minus_rho); break;
            case 3: W = pair_sum<3>(r, v, rho, minus_rho); break;
            case 2: W = pair_sum<2>(r, v, rho, minus_rho); break;
            case 1: W = pair_sum<1>(r, v, rho, minus_rho); break;
            default: break;
        }
        if (r.src >= 0) W += q;
        store(d, pt, fma(a, old, b * W));
    }
    if (!waited) pdl_wait();
}

constexpr int THREADS = 128;
__global__ void __launch_bounds__(THREADS) k_pair_pass(const __grid_constant__ KernelArgs A) { pair_pass(A); }
__global__ void __launch_bounds__(THREADS, 8) k_pair_pass_wide(const __grid_constant__ KernelArgs A) { pair_pass(A); }

// Seven blocks of 128 on an SM (up to N = 39 or so): a pass over 256^2 points
// is one wave of blocks.  256^2 P_13: 114 us per pass with the gather kernel,
// 75 so.  (-rho is an operand modifier of the multiply-add here; with a second
// register for it the compiler schedules the loop worse, 85.)
__global__ void __launch_bounds__(THREADS, 7) k_stream_pass(const __grid_constant__ KernelArgs A) {
    extern __shared__ __align__(16) unsigned char raw[];
    StreamRec* rec = reinterpret_cast<StreamRec*>(raw);
    const int K = blockIdx.y;
    {
        const int4* s = reinterpret_cast<const int4*>(A.rec[K]);
        int4* d = reinterpret_cast<int4*>(rec);
        for (int i = threadIdx.x; i < A.count * (int)(sizeof(StreamRec) / 16); i += blockDim.x) d[i] = __ldg(s + i);
    }
    __syncthreads();
    // host-written data above, the state below
    pdl_trigger();
    pdl_wait();
    const GridDev<double>& G = A.out[K];
    const Point pt = point_of(A, K);
    if (!pt.inside) return;
    double* part = reinterpret_cast<double*>(rec + A.count) + threadIdx.x;      // slot s at part[s blockDim.x]
    const int T = blockDim.x;
    const long pitch = A.pitch;
    const double *bx = pt.bx, *by = pt.by;
    double* const bo = pt.bo;
    const long cx = A.own[K].cstride, cy = A.other[K].cstride, co = G.cstride;
    const long cidx = pt.cidx, plane = (long)G.cp * G.ny;
    const double rho = K == 0 ? -A.rho : A.rho;
    double W = 0.0, t = 0.0, a = 0.0, b = 0.0;
    int cls = -1;
    // the values of a stage: right, left, upper, lower, old
    auto load = [&](const StreamRec& r, double (&v)[5]) {
        const double* px = bx + r.own * cx;
        const double* py = by + r.other * cy;
        v[0] = r.own >= 0 ? px[0] : 0.0;
        v[1] = r.own >= 0 ? px[-1] : 0.0;
        v[2] = r.other >= 0 ? py[0] : 0.0;
        v[3] = r.other >= 0 ? py[-pitch] : 0.0;
        v[4] = r.out >= 0 ? bo[r.out * co] : 0.0;
    };
    auto stage = [&](int k, const double (&v)[5], double (&next)[5]) {
        const StreamRec& r = rec[k];
        if (k + 1 < A.count) load(rec[k + 1], next);
        if (r.out >= 0 && r.cls != cls) {
            cls = r.cls;
            const double* cf = G.coef + ((long)cls * 4 + 2 * A.which) * plane + cidx;
            a = cf[0];
            b = cf[plane];
        }
        if (r.pre >= 0) W = part[r.pre * T];
        double n = 0.0;
        // an FP64 operation takes its 64 clocks of the unit also where it is predicated off or its result
        // is dropped: each kind of stage has its own straight line of those it needs
        auto sums = [&](bool p0, bool np, bool pm, bool n0, bool need_t) {
            if (p0) W = fma(r.p0, t, W);
            if (np) n = r.np * t;
            const double dx = v[0] - v[1], dy = v[2] - v[3];
            if (need_t) t = fma(-rho, dy, dx);
            if (pm || n0) {
                const double s = fma(rho, dy, dx);
                if (pm) W = fma(r.pm, s, W);
                if (n0) n = fma(r.n0, s, n);
            }
        };
        // m' = 0: one input, no targets of m' - 1
        auto single = [&](bool p0, bool np, bool pm, bool n0, bool own) {
            if (p0) W = fma(r.p0, t, W);
            if (np) n = r.np * t;
            const double s = own ? v[0] - v[1] : rho * (v[2] - v[3]);
            if (pm) W = fma(r.pm, s, W);
            if (n0) n = fma(r.n0, s, n);
        };
        switch (r.op) {
            case OP_FULL: sums(true, true, true, true, true); break;
            case OP_HEAD: sums(false, false, false, true, true); break;
            case OP_FULL_TOP: sums(true, false, true, false, true); break;
            case OP_HEAD_TOP: sums(false, false, false, false, true); break;
            case OP_TAIL: W = fma(r.p0, t, W); n = r.np * t; break;
            case OP_TAIL_TOP: W = fma(r.p0, t, W); break;
            case OP_OWN: single(true, true, true, true, true); break;
            case OP_OTHER: single(true, true, true, true, false); break;
            case OP_OWN_TOP: single(true, false, true, false, true); break;
            case OP_OTHER_TOP: single(true, false, true, false, false); break;
            case OP_OWN_HEAD: single(false, false, false, true, true); break;
            case OP_OTHER_HEAD: single(false, false, false, true, false); break;
            default: break;
        }
        if (r.out >= 0) {
            if (r.src >= 0) W += A.src[r.src][cidx];
            const double u = fma(a, v[4], b * W);
            store(bo + r.out * co, pt, u);
        }
        W = r.post >= 0 ? part[r.post * T] : 0.0;
        if (r.store >= 0) part[r.store * T] = n;
    };
    double v0[5], v1[5];
    load(rec[0], v0);
    for (int k = 0; k < A.count; k += 2) {
        stage(k, v0, v1);
        if (k + 1 < A.count) stage(k + 1, v1, v0);
    }
}

// index of (l, m, imag) in the real ordering of eq. transformation
int comp_index(int l, int m, int imag) { return l * (l + 1) / 2 + (m > 0 ? 2 * ((l - m) / 2) + imag : l); }
int nq(int l) { return l < 0 ? 0 : l / 2 + 1; }

// Records of pass P and kind K; false where the system lacks the structure.
bool build_records(const SystemMatrices& sys, const std::vector<char>& frozen, int P, int K, double dx, double dy,
                   Records& R) {
    const int n = sys.ncomp;
    const int N = sys.moms[n - 1].l;
    const int gin[2] = {P == 1 ? 0 : 1, P == 1 ? 3 : 2}, gout[2] = {P == 1 ? 1 : 0, P == 1 ? 2 : 3};
    bool ok = true;
    long covered = 0;
    // component (L, q) of kind k, or -1
    auto comp = [&](int L, int q, int k) -> int {
        if (L < 0 || L > N || q < 0 || q >= nq(L) || (k && L - 2 * q < 1)) return -1;
        const int j = comp_index(L, L - 2 * q, k);
        const Moment& m = sys.moms[j];
        if (m.l != L || m.m != L - 2 * q || (int)m.imag != k || m.grid != (L % 2 == P ? gout[k] : gin[k])) ok = false;
        return j;
    };
    // weight of the target (L, q) for the inputs (lp, ql), sign r of its My
    auto weight = [&](int L, int q, int lp, int ql, double r) -> double {
        const int t = comp(L, q, K), own = comp(lp, ql, K), other = comp(lp, ql, 1 - K);
        if (t < 0) return 0.0;
        const double mx = own >= 0 ? sys.Mx[(size_t)t * n + own] : 0.0;
        const double my = other >= 0 ? sys.My[(size_t)t * n + other] : 0.0;
        covered += (mx != 0.0) + (my != 0.0);
        if (own >= 0 && other >= 0 && std::fabs(my - r * mx) > 1e-14) ok = false;
        return -(own >= 0 ? mx : r * my) / dx;
    };
    const double r = K == 0 ? -1.0 : 1.0;       // Pm and N0; the opposite for P0 and Np
    const int first = 1 - P;
    auto finish = [&](StreamRec& e, int L, int q) -> int {
        const int j = comp(L, q, K);
        if (j < 0 || frozen[j]) return -1;
        e.out = (int16_t)sys.moms[j].local;
        return j;
    };
    auto add = [&](const StreamRec& e, int j) {
        R.rec.push_back(e);
        R.rec_comp.push_back(j);
    };
    const StreamRec none = {0.0, 0.0, 0.0, 0.0, -1, -1, -1, -1, 0, -1, -1, -1, OP_NONE, {0, 0, 0}};
    int last = first;
    for (int lp = first; lp <= N; lp += 2) {
        last = lp;
        const int nin = nq(lp), nqp = lp > first ? nq(lp - 1) : 0;
        for (int q = 0; q < nin + (lp & 1); ++q) {
            StreamRec e = none;
            int target = -1;
            if (q > 0) {
                e.p0 = weight(lp - 1, q - 1, lp, q - 1, -r);
                e.np = weight(lp + 1, q, lp, q - 1, -r);
                target = finish(e, lp - 1, q - 1);
            }
            if (q < nin) {
                const int own = comp(lp, q, K), other = comp(lp, q, 1 - K);
                e.own = (int16_t)(own >= 0 ? sys.moms[own].local : -1);
                e.other = (int16_t)(other >= 0 ? sys.moms[other].local : -1);
                if (q > 0) e.pm = weight(lp - 1, q - 1, lp, q, r);
                e.n0 = weight(lp + 1, q, lp, q, r);
                if (q < nqp) e.post = (int8_t)q;
            }
            // the operations the stage has (a target that does not exist has zero weight and no slot)
            const bool both = e.own >= 0 && e.other >= 0, none_in = e.own < 0 && e.other < 0;
            const bool done = q > 0 && comp(lp - 1, q - 1, K) >= 0, next = comp(lp + 1, q, K) >= 0;
            const bool later = comp(lp - 1, q, K) >= 0 || comp(lp + 1, q + 1, K) >= 0;
            if (both) e.op = q == 0 ? (next ? OP_HEAD : OP_HEAD_TOP) : next ? OP_FULL : OP_FULL_TOP;
            else if (none_in) e.op = next ? OP_TAIL : done ? OP_TAIL_TOP : OP_NONE;
            else if (q == 0) e.op = e.own >= 0 ? OP_OWN_HEAD : OP_OTHER_HEAD;
            else if (e.own >= 0) e.op = next ? OP_OWN : OP_OWN_TOP;
            else e.op = next ? OP_OTHER : OP_OTHER_TOP;
            if (q < nin && none_in) ok = false;
            if (q < nin && later && !both) ok = false;
            if (lp + 1 <= N && q < nq(lp + 1)) e.store = (int8_t)q;
            add(e, target);
        }
    }
    if (last + 1 <= N)
        for (int q = 0; q < nq(last + 1); ++q) {
            StreamRec e = none;
            e.pre = (int8_t)q;
            const int target = finish(e, last + 1, q);
            add(e, target);
        }
    // the same sums output by output
    for (int j = 0; j < n; ++j) {
        const Moment& m = sys.moms[j];
        if (m.grid != gout[K] || frozen[j]) continue;
        PairRec p = {};
        const int q = (m.l - m.m) / 2;
        const int il[4] = {m.l - 1, m.l - 1, m.l + 1, m.l + 1}, iq[4] = {q - 1, q, q, q + 1};
        for (int k = 0; k < 4; ++k) p.own[k] = p.other[k] = -1;
        for (int k = 0; k < 4; ++k) {
            const int own = comp(il[k], iq[k], K), other = comp(il[k], iq[k], 1 - K);
            if (own < 0 && other < 0) continue;
            const int c = p.count++;
            if (own >= 0) p.own[c] = (int16_t)sys.moms[own].local;
            if (other >= 0) p.other[c] = (int16_t)sys.moms[other].local;
            if (!(k & 1)) p.t |= (int8_t)(1 << c);
            const long had = covered;
            p.w[c] = weight(m.l, q, il[k], iq[k], k & 1 ? r : -r);
            covered = had;
        }
        p.out = (int16_t)m.local;
        R.pair.push_back(p);
        R.pair_comp.push_back(j);
    }
    // every target of the kind once, every coupling once
    long targets = 0, total = 0;
    for (int j = 0; j < n; ++j) {
        if (sys.moms[j].grid != gout[K]) continue;
        targets += !frozen[j];
        for (int k = 0; k < n; ++k)
            total += (sys.Mx[(size_t)j * n + k] != 0.0) + (sys.My[(size_t)j * n + k] != 0.0);
    }
    for (const StreamRec& e : R.rec) targets -= e.out >= 0;
    return ok && targets == 0 && covered == total;
}

size_t stream_smem(const StreamTables& t, int P) {
    return t.r[P][0].rec.size() * sizeof(StreamRec) + (size_t)t.slots * THREADS * sizeof(double);
}

}  // namespace

int stream_build(const SystemMatrices& sys, const std::vector<char>& frozen, double dx, double dy, StreamTables** out) {
    *out = nullptr;
    StreamTables* t = new StreamTables();
    for (int P = 0; P < 2; ++P)
        for (int K = 0; K < 2; ++K)
            if (!build_records(sys, frozen, P, K, dx, dy, t->r[P][K])) {
                delete t;
                return 0;
            }
    t->N = sys.moms[sys.ncomp - 1].l;
    t->slots = nq(t->N);
    t->rho = dx / dy;
    size_t bytes = 0;
    auto place = [&](size_t n) {
        const size_t at = bytes;
        bytes = (bytes + n + 255) / 256 * 256;
        return at;
    };
    for (int P = 0; P < 2; ++P)
        for (int K = 0; K < 2; ++K) {
            Records& R = t->r[P][K];
            R.rec_at = place(R.rec.size() * sizeof(StreamRec));
            R.pair_at = place(R.pair.size() * sizeof(PairRec));
        }
    t->image.assign(bytes, 0);
    int dev = 0, most = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&t->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncSetAttribute(k_stream_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess) {
        delete t;
        return -4;
    }
    for (int P = 0; P < 2; ++P)
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t->resident[P], k_stream_pass, THREADS, stream_smem(*t, P)) !=
            cudaSuccess) {
            delete t;
            return -4;
        }
    *out = t;
    return 0;
}

int stream_update(StreamTables* t, const std::vector<int>& comp_class, const std::vector<int>& src_slot) {
    for (int P = 0; P < 2; ++P)
        for (int K = 0; K < 2; ++K) {
            Records& R = t->r[P][K];
            auto set = [&](auto& e, int j) {
                if (j < 0) return;
                e.cls = (int8_t)comp_class[j];
                e.src = (int16_t)src_slot[j];
            };
            for (size_t i = 0; i < R.rec.size(); ++i) set(R.rec[i], R.rec_comp[i]);
            for (size_t i = 0; i < R.pair.size(); ++i) set(R.pair[i], R.pair_comp[i]);
            std::memcpy(t->image.data() + R.rec_at, R.rec.data(), R.rec.size() * sizeof(StreamRec));
            if (!R.pair.empty())
                std::memcpy(t->image.data() + R.pair_at, R.pair.data(), R.pair.size() * sizeof(PairRec));
        }
    return table_upload(t->dev, t->image.data(), t->image.size()) == cudaSuccess ? 0 : -4;
}

void stream_destroy(StreamTables* t) {
    if (!t) return;
    table_free(t->dev);
    delete t;
}

int stream_pass(const StreamTables* t, const StreamArgs& a, void* stream) {
    KernelArgs k;
    const int P = a.P;
    const int gin[2] = {P == 1 ? 0 : 1, P == 1 ? 3 : 2}, gout[2] = {P == 1 ? 1 : 0, P == 1 ? 2 : 3};
    long points = 0;
    for (int K = 0; K < 2; ++K) {
        k.own[K] = a.g[gin[K]];
        k.other[K] = a.g[gin[1 - K]];
        k.out[K] = a.g[gout[K]];
        k.out_grid[K] = gout[K];
        const Records& R = t->r[P][K];
        const unsigned char* dev = static_cast<const unsigned char*>(t->dev.p);
        k.rec[K] = reinterpret_cast<const StreamRec*>(dev + R.rec_at);
        k.pair[K] = reinterpret_cast<const PairRec*>(dev + R.pair_at);
        k.outs[K] = (int)R.pair.size();
        k.slices[K] = 0;
        points = std::max(points, (long)k.out[K].nx * k.out[K].ny);
    }
    k.count = (int)t->r[P][0].rec.size();
    k.slots = t->slots;
    k.which = a.which;
    k.pitch = a.pitch;
    k.p[0] = a.p[0];
    k.p[1] = a.p[1];
    k.rho = t->rho;
    k.minus_rho = -t->rho;
    k.src = a.src;
    const long blocks = (points + THREADS - 1) / THREADS;
    cudaError_t e;
    // Streamed: two threads per point, whose chains of stages need about two
    // warps per scheduler of the GPU to hide one another (the fewer stages, the
    // more).  us per pass, output by output / streamed: P_3 200^2 7.8 / 8.3,
    // 220^2 8.8 / 8.4, 512^2 33 / 28; P_5 175^2 11.7 / 12.3, 190^2 13.3 / 12.3,
    // 256^2 21 / 16; P_7 175^2 19.1 / 18.4, P_13 54 / 45, P_39 429 / 336; 256^2
    // P_13 112 / 74, P_39 905 / 585.  At N <= 2 an input has too few targets:
    // P_2 512^2 16.6 (wide) / 18.7, P_1 7.8 / 12.3.
    const long from = t->N >= 7 ? 200 : t->N >= 5 ? 230 : 300;
    if (t->N > 2 && points >= from * t->sms) {
        // A pass overlaps the previous one's tail only where that one's blocks
        // fill the SMs evenly: early blocks take whatever slots it leaves, and
        // an SM then runs its full number of them while another has a few.
        // 220^2 P_13 (five blocks per SM of seven) 75 us with, 55 without; 175^2
        // P_39 496 and 336; 256^2 P_5 (6.7 of seven) 16.3 and 18.1.
        const bool overlap = blocks <= 1024 && 2 * blocks > (long)t->sms * (t->resident[P] - 1);
        e = launch_pdl(k_stream_pass, dim3((unsigned)blocks, 2), dim3(THREADS), stream_smem(*t, P), (cudaStream_t)stream,
                       overlap, k);
    } else {
        // one output per thread (up to 64 slices per kind).  Wide, us per pass,
        // without / with: P_1 256^2 3.6 / 4.0, 350^2 5.6 / 4.9, 512^2 9.1 / 7.8,
        // 1500 x 1300 57 / 47; P_2 256^2 6.7 / 6.1, 512^2 18.5 / 16.6, 1500 x 1300 137 / 115
        for (int K = 0; K < 2; ++K) k.slices[K] = std::min(k.outs[K], 64);
        const bool wide = t->N <= 2 && points >= (t->N == 1 ? 500 : 400) * (long)t->sms;
        e = launch_pdl(wide ? k_pair_pass_wide : k_pair_pass, dim3((unsigned)blocks, k.slices[0] + k.slices[1]),
                       dim3(THREADS), 0, (cudaStream_t)stream, true, k);
    }
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : -4;
}

}  // namespace starmap
