// C ABI of the StaRMAP stepper: handle lifetime, problem data, schedules,
// read-out and checkpoints.  See include/starmap.h for the contract.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include <sys/stat.h>

#include "host_math.h"
#include "internal.h"
#include "mlp.h"
#include "stream.h"
#include "tiled.h"
#include "../../include/starmap.h"

namespace starmap {
std::atomic<int>& alloc_fail_countdown() {
    static std::atomic<int> countdown{0};
    return countdown;
}
}  // namespace starmap

using namespace starmap;

namespace {
thread_local std::string g_create_error;
// Tile grid of a batch instance and the cost of one of its tiles (pipeline
// stages of its longer pass).
struct BatchShape { int tx, ty, cost; };
}

struct starmap_s {
    starmap_config cfg{};
    SystemMatrices sys;
    int ncomp = 0;
    double dx = 0, dy = 0, dt = 0, t = 0;
    long steps = 0;
    int p[2] = {1, 1};
    int nxg[4] = {0, 0, 0, 0}, nyg[4] = {0, 0, 0, 0}, Kg[4] = {0, 0, 0, 0};
    int cpg[4] = {0, 0, 0, 0};            // row pitch of a grid's coefficients and sources on the device
    long pitch = 0, rows = 0;
    std::vector<int> members[4];          // component ids per grid, by local index
    size_t esize = 8;
    bool fp32 = false;
    void* alloc[4] = {nullptr, nullptr, nullptr, nullptr};
    void* base[4] = {nullptr, nullptr, nullptr, nullptr};
    void* alloc1[4] = {nullptr, nullptr, nullptr, nullptr};   // second state set (fused schedule)
    void* base1[4] = {nullptr, nullptr, nullptr, nullptr};
    long cstride[4] = {0, 0, 0, 0};
    size_t grid_bytes[4] = {0, 0, 0, 0};
    void* coef[4] = {nullptr, nullptr, nullptr, nullptr};
    int ncls_alloc = 0;
    int nclasses = 2;
    std::vector<int> comp_class;
    std::vector<double> sl_factor;        // empty = isotropic
    std::vector<double> sig_a[4], sig_s[4];
    std::vector<int> src_slot;            // per component, -1 if none
    std::vector<void*> src_dev;           // by slot
    DevTable src_ptrs_dev;
    std::vector<GatherOut> outs;          // the gather kernel's outputs (empty where another kernel runs)
    std::vector<int> outs_comp;           // and their components
    DevTable outs_dev, coefs_dev;
    int tbeg[4] = {0, 0, 0, 0}, tend[4] = {0, 0, 0, 0};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    double* partials = nullptr;
    double* result = nullptr;
    int red_blocks = 608;
    void* prev[4] = {nullptr, nullptr, nullptr, nullptr};
    bool have_output = false;
    double out_lambda = 1.0;
    bool ghosts_dirty = true;
    int kernel_used = STARMAP_KERNEL_GATHER;
    TiledPlan* tiled = nullptr;
    StreamTables* stream64 = nullptr;     // FP64 2D passes (null: the gather kernel)
    bool stream_tried = false;
    // learned closure (STARMAP_CLOSURE_MLP8)
    int closure = STARMAP_CLOSURE_NONE;
    int nsys = 0;                          // order of the assembled system
    std::vector<char> frozen;              // per component: left alone by the even passes
    float* net_params = nullptr;           // FP32 parameters (device)
    mlp::Packed* net = nullptr;            // BF16 packed network (device)
    bool net_ready = false;
    float* ctr = nullptr;                  // closure scratch (input fragments, scales, I_8 centre values)
    float* lsig = nullptr;                 // log(1 + sigma_a), log(1 + sigma_s0) at the cell centres
    bool lsig_dirty = true;
    int engine = mlp::ENGINE_TCGEN05;      // tensor-core path of the closure network
    int* closure_err = nullptr;            // bounded-wait flag of the tcgen05 network
    unsigned long version = 0;             // bumped whenever the tiled pass parameters change
    // periodic health check (starmap_set_health_check)
    long health_every = 0;                 // steps per span, 0 = off
    double health_growth = 1.05;
    void* snap[4] = {nullptr, nullptr, nullptr, nullptr};   // state at the end of the last span that passed
    double snap_t = 0.0;
    long snap_steps = 0;
    long health_good_steps = 0;
    double health_l2_good = 0.0, health_l2_failed = std::nan("");
    std::vector<double> src_sq;            // per component: sum of the squared source values at its grid points
    // time-dependent material and sources (starmap_set_time_dependence)
    starmap_field_fn td_fn = nullptr;
    void* td_user = nullptr;
    std::vector<int> td_src;               // components with a source
    std::vector<double> gx[4], gy[4];      // point coordinates of each grid, [y][x]
    std::string err;
};

struct starmap_batch_s {
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int schedule = STARMAP_SCHEDULE_MERGED;
    int variant = 1;                       // tile height of every instance (see starmap_batch_create)
    int shape = 0;                         // the batch kernel (tiled_batch_shape)
    double tuned_ms[2] = {-1.0, -1.0};     // autotuner: ms per step with 10-row / 5-row tiles (-1: not timed)
    int strip = 192;                       // stages per strip of short tiles (batch_plan)
    bool from_cache = false;               // the tuning came from the cache file
    std::vector<BatchShape> shapes;        // per instance: tiles and stages (for re-planning)
    int slots = 0;                         // resident CTA slots of the persistent grid
    std::vector<starmap_t*> inst;
    std::vector<unsigned long> uploaded;   // parameter version of each instance on the device
    std::vector<char> staging;             // host copy of the parameter blocks
    void* dev_params = nullptr;
    void* dev_items = nullptr;             // per CTA: strided runs (instance, first tile, count, stride)
    int* dev_off = nullptr;                // CTA b's runs: items[off[b]] .. items[off[b + 1] - 1]
    int smem = 0;
    int grid = 0;
    std::vector<std::pair<long, cudaGraphExec_t>> graphs;   // captured step sequences by step count
    std::string err;
};

namespace {

int fail(starmap_t* h, int code, const std::string& msg) {
    if (h) h->err = msg; else g_create_error = msg;
    return code;
}

int cuda_fail(starmap_t* h, cudaError_t e, const char* what) {
    return fail(h, STARMAP_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define CK(call, what) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return cuda_fail(h, e_, what); } while (0)

// Surface a bounded-wait failure of the tiled kernel or of the tcgen05
// closure network (synchronises the stream).
int poll_kernel(starmap_t* h) {
    if (h->closure_err) {
        int flag = 0;
        if (cudaMemcpyAsync(&flag, h->closure_err, sizeof(int), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
            cudaStreamSynchronize(h->stream) != cudaSuccess)
            return fail(h, STARMAP_E_CUDA, "reading the closure error flag failed");
        if (flag) {
            cudaMemsetAsync(h->closure_err, 0, sizeof(int), h->stream);
            return fail(h, STARMAP_E_TIMEOUT, "a bounded wait in the closure network gave up");
        }
    }
    if (!h->tiled) return STARMAP_OK;
    int rc = tiled_poll(h->tiled, h->stream);
    if (rc == -6) return fail(h, STARMAP_E_TIMEOUT, tiled_error(h->tiled));
    if (rc) return fail(h, STARMAP_E_CUDA, tiled_error(h->tiled));
    return STARMAP_OK;
}

template <class T>
GridDev<T> grid_dev(const starmap_t* h, int g) {
    GridDev<T> d;
    d.base = (T*)h->base[g];
    d.cstride = h->cstride[g];
    d.nx = h->nxg[g];
    d.ny = h->nyg[g];
    d.K = h->Kg[g];
    d.coef = (T*)h->coef[g];
    d.cp = h->cpg[g];
    return d;
}

int class_of(const starmap_t* h, int l) {
    if (h->sl_factor.empty()) return l == 0 ? 0 : 1;
    return l;
}

// The gather kernel's tables (couplings once; classes, source slots).
template <class T>
int build_gather(starmap_t* h) {
    const int n = h->ncomp;
    if (h->outs.empty()) {
        std::vector<GatherOut> outs;
        std::vector<int> comps;
        std::vector<GatherCoef<T>> coefs;
        for (int g = 0; g < 4; ++g) {
            h->tbeg[g] = (int)outs.size();
            for (int j : h->members[g]) {
                if (h->frozen[j]) continue;
                GatherOut o{};
                GatherCoef<T> c{};
                o.local = h->sys.moms[j].local;
                for (int k = 0; k < n; ++k) {
                    double mx = h->sys.Mx[(size_t)j * n + k];
                    double my = h->sys.My[(size_t)j * n + k];
                    if (mx != 0.0) {
                        if (h->sys.moms[k].grid != (g ^ 1) || o.nxt >= MAXC)
                            return fail(h, STARMAP_E_UNSUPPORTED, "x-coupling outside the staggered pattern");
                        o.xin[o.nxt] = h->sys.moms[k].local;
                        c.cx[o.nxt] = (T)(-mx / h->dx);
                        ++o.nxt;
                    }
                    if (my != 0.0) {
                        if (h->sys.moms[k].grid != (g ^ 2) || o.nyt >= MAXC)
                            return fail(h, STARMAP_E_UNSUPPORTED, "y-coupling outside the staggered pattern");
                        o.yin[o.nyt] = h->sys.moms[k].local;
                        c.cy[o.nyt] = (T)(-my / h->dy);
                        ++o.nyt;
                    }
                }
                outs.push_back(o);
                comps.push_back(j);
                coefs.push_back(c);
            }
            h->tend[g] = (int)outs.size();
        }
        CK(table_upload(h->coefs_dev, coefs.data(), coefs.size() * sizeof(GatherCoef<T>)), "cudaMalloc tables");
        h->outs = outs;
        h->outs_comp = comps;
    }
    for (size_t i = 0; i < h->outs.size(); ++i) {
        h->outs[i].cls = h->comp_class[h->outs_comp[i]];
        h->outs[i].src = h->src_slot[h->outs_comp[i]];
    }
    CK(table_upload(h->outs_dev, h->outs.data(), h->outs.size() * sizeof(GatherOut)), "cudaMalloc tables");
    return STARMAP_OK;
}

// The pass tables of the handle's kernel.  What follows from the system alone
// is assembled once; a source or a new set of decay classes changes the
// entries' classes and source slots and uploads them into the same buffers.
template <class T>
int build_tables(starmap_t* h) {
    if (h->tiled) {
        int rc = tiled_update(h->tiled, h->sys, h->comp_class, h->src_slot, h->src_dev, h->frozen, h->dx, h->dy);
        if (rc) return fail(h, rc, tiled_error(h->tiled));
        ++h->version;
        return STARMAP_OK;
    }
    // source pointers by slot, at most one per component
    std::vector<void*> ptrs(h->src_dev.begin(), h->src_dev.end());
    ptrs.resize(h->ncomp, nullptr);
    CK(table_upload(h->src_ptrs_dev, ptrs.data(), ptrs.size() * sizeof(void*)), "cudaMalloc sources");
    if (!h->fp32 && h->cfg.system == STARMAP_PN2D && !h->stream64 && !h->stream_tried) {
        if (stream_build(h->sys, h->frozen, h->dx, h->dy, &h->stream64))
            return fail(h, STARMAP_E_CUDA, "streamed tables");
        h->stream_tried = true;
    }
    if (h->stream64) {
        if (stream_update(h->stream64, h->comp_class, h->src_slot)) return fail(h, STARMAP_E_CUDA, "cudaMalloc tables");
    } else {
        int rc = build_gather<T>(h);
        if (rc) return rc;
    }
    ++h->version;
    return STARMAP_OK;
}

int rebuild_tables(starmap_t* h) {
    return h->fp32 ? build_tables<float>(h) : build_tables<double>(h);
}

// Rows of nx values to device rows of cp.  A 2D copy of pageable memory takes
// 5 to 7 us longer than a plain one (replacing a source, before the wait of
// about 4 us below, FP64 and FP32 64^2: 18.8 and 11.5 us, FP32 150^2: 38 and
// 33), so the copy is plain where it
// needs no further pass over the values: rows without padding, and FP32, whose
// conversion writes padded rows as well.  (FP64 padded on the host: 100^2 24 ->
// 27 us, 1023 x 700 514 -> 863; a narrow FP32 grid would mostly send padding.)
template <class T>
cudaError_t upload_rows(void* d, const double* q, int nx, int ny, int cp, cudaStream_t stream) {
    const size_t row = (size_t)nx * sizeof(T), pitch = (size_t)cp * sizeof(T);
    const bool convert = sizeof(T) != sizeof(double);
    std::unique_ptr<T[]> rows;
    const void* from = q;
    int w = nx;                                         // of a row at `from`
    if (convert) {
        if (cp <= 2 * nx) w = cp;
        rows.reset(new T[(size_t)w * ny]);
        if (w == nx) std::copy(q, q + (size_t)nx * ny, rows.get());
        else
            for (int y = 0; y < ny; ++y) {
                T* r = std::copy(q + (size_t)y * nx, q + (size_t)(y + 1) * nx, rows.get() + (size_t)y * w);
                std::fill(r, rows.get() + (size_t)(y + 1) * w, T(0));
            }
        from = rows.get();
    }
    // on the handle's stream, and waited for: a blocking copy of pageable memory may return before its last part has
    // landed, and the passes' stream does not wait for the default one
    const cudaError_t e = w == cp ? cudaMemcpyAsync(d, from, pitch * ny, cudaMemcpyHostToDevice, stream)
                                  : cudaMemcpy2DAsync(d, pitch, from, row, row, ny, cudaMemcpyHostToDevice, stream);
    return e == cudaSuccess ? cudaStreamSynchronize(stream) : e;
}

// Decay coefficients of grid g from the stored material (section 5.5/5.7):
// class 0: c = Sigma_a; class l >= 1: c = Sigma_a + Sigma_s0 - Sigma_sl.
// Stored as a = exp(-c dt/2), b = dt/2 E(-c dt/2), A = exp(-c dt), B = dt E(-c dt).
template <class T>
int upload_coefficients(starmap_t* h, int g) {
    const long plane = (long)h->cpg[g] * h->nyg[g];     // rows padded to cpg (the padding is never used)
    if (plane == 0) return STARMAP_OK;
    std::vector<T> buf((size_t)h->nclasses * 4 * plane);
    const std::vector<double>& sa = h->sig_a[g];
    const std::vector<double>& ss = h->sig_s[g];
    const double dt = h->dt;
    const int nx = h->nxg[g], ny = h->nyg[g];
    for (int cls = 0; cls < h->nclasses; ++cls) {
        for (int y = 0; y < ny; ++y) {
            T* dst = buf.data() + (size_t)cls * 4 * plane + (size_t)y * h->cpg[g];
            for (int x = 0; x < nx; ++x, ++dst) {
                const size_t i = (size_t)y * nx + x;
                double c;
                if (cls == 0) c = sa[i];
                else if (h->sl_factor.empty()) c = sa[i] + ss[i];
                else c = sa[i] + ss[i] - ss[i] * h->sl_factor[cls];
                dst[0] = (T)std::exp(-c * dt / 2);
                dst[plane] = (T)(dt / 2 * expm1div(-c * dt / 2));
                dst[2 * plane] = (T)std::exp(-c * dt);
                dst[3 * plane] = (T)(dt * expm1div(-c * dt));
            }
        }
    }
    CK(cudaMemcpyAsync(h->coef[g], buf.data(), buf.size() * sizeof(T), cudaMemcpyHostToDevice, h->stream), "upload coefficients");
    CK(cudaStreamSynchronize(h->stream), "upload coefficients");
    return STARMAP_OK;
}

int ensure_coef_alloc(starmap_t* h) {
    if (h->ncls_alloc >= h->nclasses) return STARMAP_OK;
    for (int g = 0; g < 4; ++g) {
        if (h->coef[g]) { cudaFree(h->coef[g]); h->coef[g] = nullptr; }
        size_t bytes = std::max<size_t>(1, (size_t)h->nclasses * 4 * h->cpg[g] * h->nyg[g]) * h->esize;
        CK(dev_alloc(&h->coef[g], bytes), "cudaMalloc coefficients");
    }
    h->ncls_alloc = h->nclasses;
    return STARMAP_OK;
}

int upload_all_coefficients(starmap_t* h) {
    int rc = ensure_coef_alloc(h);
    if (rc) return rc;
    for (int g = 0; g < 4; ++g) {
        rc = h->fp32 ? upload_coefficients<float>(h, g) : upload_coefficients<double>(h, g);
        if (rc) return rc;
    }
    return STARMAP_OK;
}

template <class T>
int fill_ghosts_all(starmap_t* h) {
    for (int g = 0; g < 4; ++g) {
        GhostArgs<T> a;
        a.g = grid_dev<T>(h, g);
        a.pitch = h->pitch;
        a.grid = g;
        a.p[0] = h->p[0];
        a.p[1] = h->p[1];
        a.kbegin = 0;
        a.kend = h->Kg[g];
        if (launch_fill_ghosts<T>(a, h->stream)) return cuda_fail(h, cudaGetLastError(), "ghost fill");
    }
    h->ghosts_dirty = false;
    return STARMAP_OK;
}

// One pass over the output grids of a parity.  odd: grids G21, G12;
// even: G11, G22.  which: 0 half-step coefficients, 1 full-step.
template <class T>
int run_pass(starmap_t* h, bool odd, int which) {
    if (h->kernel_used != STARMAP_KERNEL_GATHER) {
        int rc = tiled_pass(h->tiled, odd, which, h->stream);
        if (rc) return fail(h, rc, tiled_error(h->tiled));
        return STARMAP_OK;
    }
    if (h->stream64) {
        StreamArgs a;
        for (int g = 0; g < 4; ++g) a.g[g] = grid_dev<double>(h, g);
        a.pitch = h->pitch;
        a.p[0] = h->p[0];
        a.p[1] = h->p[1];
        a.P = odd ? 1 : 0;
        a.which = which;
        a.src = (double* const*)h->src_ptrs_dev.p;
        if (stream_pass(h->stream64, a, h->stream)) return cuda_fail(h, cudaGetLastError(), "FP64 pass");
        return STARMAP_OK;
    }
    GatherArgs<T> a;
    for (int q = 0; q < 2; ++q) {
        const int g = q == 0 ? (odd ? 1 : 0) : (odd ? 2 : 3);
        a.out[q] = grid_dev<T>(h, g);
        a.xin[q] = grid_dev<T>(h, g ^ 1);
        a.yin[q] = grid_dev<T>(h, g ^ 2);
        a.grid[q] = g;
        a.begin[q] = h->tbeg[g];
        a.end[q] = h->tend[g];
        a.slices[q] = 0;
    }
    a.pitch = h->pitch;
    a.p[0] = h->p[0];
    a.p[1] = h->p[1];
    a.which = which;
    a.outs = (const GatherOut*)h->outs_dev.p;
    a.coefs = (const GatherCoef<T>*)h->coefs_dev.p;
    a.src = (T* const*)h->src_ptrs_dev.p;
    if (launch_gather_pass<T>(a, h->stream)) return cuda_fail(h, cudaGetLastError(), "gather pass");
    return STARMAP_OK;
}

// The closure kernels are unrolled over the grid placement of components
// 0..44 (mlp::GRID45); check it against the handle's own placement.
bool closure_layout_ok(const starmap_t* h) {
    const int n = std::min(h->ncomp, mlp::NMOM + mlp::NOUT);
    for (int j = 0; j < n; ++j)
        if (h->sys.moms[j].grid != mlp::GRID45[j]) return false;
    return true;
}

// log(1 + sigma) of grid G11's material, FP32 on the device (network inputs).
int ensure_lsig(starmap_t* h) {
    const size_t M = (size_t)h->nxg[0] * h->nyg[0];
    if (!h->lsig) CK(dev_alloc(&h->lsig, std::max<size_t>(1, 2 * M) * sizeof(float)), "cudaMalloc closure inputs");
    if (!h->lsig_dirty) return STARMAP_OK;
    std::vector<float> buf(2 * M);
    for (size_t i = 0; i < M; ++i) {
        buf[i] = (float)std::log1p(h->sig_a[0][i]);
        buf[M + i] = (float)std::log1p(h->sig_s[0][i]);
    }
    CK(cudaMemcpyAsync(h->lsig, buf.data(), buf.size() * sizeof(float), cudaMemcpyHostToDevice, h->stream),
       "upload closure inputs");
    CK(cudaStreamSynchronize(h->stream), "upload closure inputs");
    h->lsig_dirty = false;
    return STARMAP_OK;
}

template <class T>
mlp::ClosureArgs<T> closure_args(const starmap_t* h) {
    mlp::ClosureArgs<T> a;
    for (int g = 0; g < 4; ++g) a.g[g] = grid_dev<T>(h, g);
    a.pitch = h->pitch;
    a.p[0] = h->p[0];
    a.p[1] = h->p[1];
    a.nx = h->nxg[0];
    a.ny = h->nyg[0];
    for (int j = 0; j < mlp::NMOM + mlp::NOUT; ++j) {
        a.slot[j] = j < h->ncomp ? make_int2(h->sys.moms[j].grid, h->sys.moms[j].local) : make_int2(0, 0);
        a.col[j] = a.g[a.slot[j].x].base + (long)a.slot[j].y * a.g[a.slot[j].x].cstride;
    }
    const size_t M = (size_t)a.nx * a.ny;
    a.lsa = h->lsig;
    a.lss = h->lsig + M;
    return a;
}

// Network prediction of the order-8 moments from the current state.
template <class T>
int run_closure(starmap_t* h) {
    if (!h->net_ready) return fail(h, STARMAP_E_STATE, "closure handle stepped before starmap_set_closure");
    int rc = ensure_lsig(h);
    if (rc) return rc;
    const size_t M = (size_t)h->nxg[0] * h->nyg[0];
    if (!h->ctr) CK(dev_alloc(&h->ctr, std::max<size_t>(1, (size_t)mlp::closure_scratch_floats((long)M)) * sizeof(float)),
                    "cudaMalloc closure scratch");
    if (!h->closure_err) {
        CK(dev_alloc(&h->closure_err, sizeof(int)), "cudaMalloc closure flag");
        CK(cudaMemsetAsync(h->closure_err, 0, sizeof(int), h->stream), "closure flag");
    }
    if (mlp::closure<T>(closure_args<T>(h), h->net, h->ctr, h->engine, h->closure_err, h->stream))
        return cuda_fail(h, cudaGetLastError(), "closure");
    return STARMAP_OK;
}

// Odd pass, preceded by the closure where there is one.
template <class T>
int odd_pass(starmap_t* h, int which) {
    if (h->closure) { int rc = run_closure<T>(h); if (rc) return rc; }
    return run_pass<T>(h, true, which);
}

// Boundary copies of the odd grids of state set `set` (0: base, 1: base1).
int refresh_odd(starmap_t* h, int set) {
    GhostPassArgs ga;
    const int go[2] = {1, 2};
    for (int q = 0; q < 2; ++q) {
        ga.g[q] = grid_dev<float>(h, go[q]);
        if (set) ga.g[q].base = (float*)h->base1[go[q]];
        ga.grid[q] = go[q];
    }
    ga.pitch = h->pitch;
    ga.p[0] = h->p[0];
    ga.p[1] = h->p[1];
    if (launch_fill_ghosts_pass(ga, h->stream)) return cuda_fail(h, cudaGetLastError(), "ghost refresh");
    return STARMAP_OK;
}

// The inner steps of the merged schedule, E_dt O_dt each, as fused launches
// two at a time (set 0 -> set 1 -> set 0); an odd count runs one unfused.
// (FP32: the schedule needs the tiled kernel.)
int fused_inner_steps(starmap_t* h, long m) {
    int rc;
    if (m % 2) {
        if ((rc = run_pass<float>(h, false, 1)) || (rc = odd_pass<float>(h, 1))) return rc;
        --m;
    }
    for (long i = 0; i < m; ++i) {
        const int dir = (int)(i & 1);
        rc = tiled_fused_step(h->tiled, dir, h->stream);
        if (rc) return fail(h, rc, tiled_error(h->tiled));
        if ((rc = refresh_odd(h, 1 - dir))) return rc;
    }
    return STARMAP_OK;
}

template <class T>
int do_steps(starmap_t* h, long n) {
    if (n <= 0) return STARMAP_OK;
    if (h->closure && !h->net_ready) return fail(h, STARMAP_E_STATE, "closure handle stepped before starmap_set_closure");
    if (h->ghosts_dirty) { int rc = fill_ghosts_all<T>(h); if (rc) return rc; }
    int rc;
    if (h->cfg.schedule == STARMAP_SCHEDULE_FUSED) {
        if ((rc = odd_pass<T>(h, 0))) return rc;
        if ((rc = fused_inner_steps(h, n - 1))) return rc;
        if ((rc = run_pass<T>(h, false, 1))) return rc;
        if ((rc = odd_pass<T>(h, 0))) return rc;
    } else if (h->cfg.schedule == STARMAP_SCHEDULE_MERGED) {
        if ((rc = odd_pass<T>(h, 0))) return rc;
        for (long i = 0; i < n; ++i) {
            if ((rc = run_pass<T>(h, false, 1))) return rc;
            if ((rc = odd_pass<T>(h, i == n - 1 ? 0 : 1))) return rc;
        }
    } else {
        for (long i = 0; i < n; ++i) {
            if ((rc = odd_pass<T>(h, 0))) return rc;
            if ((rc = run_pass<T>(h, false, 1))) return rc;
            if ((rc = odd_pass<T>(h, 0))) return rc;
        }
    }
    h->t += n * h->dt;
    h->steps += n;
    return STARMAP_OK;
}

int check_j(starmap_t* h, int j) {
    if (!h) return STARMAP_E_ARG;
    if (j < 0 || j >= h->ncomp) return fail(h, STARMAP_E_ARG, "component index out of range");
    return STARMAP_OK;
}

size_t comp_points(const starmap_t* h, int j) {
    int g = h->sys.moms[j].grid;
    return (size_t)h->nxg[g] * h->nyg[g];
}

char* comp_ptr(const starmap_t* h, int j, void* const* bases) {
    const Moment& m = h->sys.moms[j];
    return (char*)bases[m.grid] + ((size_t)m.local * h->cstride[m.grid] + h->pitch) * h->esize;
}

// copy component j from a device layout (bases) to a host array in the run's precision
int download_raw(starmap_t* h, int j, void* const* bases, void* dst) {
    int g = h->sys.moms[j].grid;
    CK(cudaMemcpy2DAsync(dst, h->nxg[g] * h->esize, comp_ptr(h, j, bases), h->pitch * h->esize,
                         h->nxg[g] * h->esize, h->nyg[g], cudaMemcpyDeviceToHost, h->stream), "download");
    return STARMAP_OK;
}

int upload_raw(starmap_t* h, int j, const void* src) {
    int g = h->sys.moms[j].grid;
    CK(cudaMemcpy2DAsync(comp_ptr(h, j, h->base), h->pitch * h->esize, src, h->nxg[g] * h->esize,
                         h->nxg[g] * h->esize, h->nyg[g], cudaMemcpyHostToDevice, h->stream), "upload");
    h->ghosts_dirty = true;
    return STARMAP_OK;
}

int download_double(starmap_t* h, int j, void* const* bases, double* out) {
    size_t np = comp_points(h, j);
    if (int rc = poll_kernel(h)) return rc;
    if (h->fp32) {
        std::vector<float> tmp(np);
        int rc = download_raw(h, j, bases, tmp.data());
        if (rc) return rc;
        CK(cudaStreamSynchronize(h->stream), "download");
        for (size_t i = 0; i < np; ++i) out[i] = tmp[i];
    } else {
        int rc = download_raw(h, j, bases, out);
        if (rc) return rc;
        CK(cudaStreamSynchronize(h->stream), "download");
    }
    return STARMAP_OK;
}

void release(starmap_t* h) {
    for (int g = 0; g < 4; ++g) {
        if (h->alloc[g]) cudaFree(h->alloc[g]);
        if (h->coef[g]) cudaFree(h->coef[g]);
        if (h->prev[g]) cudaFree(h->prev[g]);
    }
    for (void* p : h->src_dev) if (p) cudaFree(p);
    table_free(h->src_ptrs_dev);
    table_free(h->outs_dev);
    table_free(h->coefs_dev);
    if (h->partials) cudaFree(h->partials);
    if (h->result) cudaFree(h->result);
    if (h->net_params) cudaFree(h->net_params);
    if (h->net) cudaFree(h->net);
    if (h->ctr) cudaFree(h->ctr);
    if (h->lsig) cudaFree(h->lsig);
    if (h->closure_err) cudaFree(h->closure_err);
    for (int g = 0; g < 4; ++g) if (h->snap[g]) cudaFree(h->snap[g]);
    for (int g = 0; g < 4; ++g) if (h->alloc1[g]) cudaFree(h->alloc1[g]);
    if (h->tiled) tiled_destroy(h->tiled);
    stream_destroy(h->stream64);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
}


}  // namespace

extern "C" {

namespace {
// The work-unit plan of a batch (below).
int batch_plan(const std::vector<BatchShape>& shapes, int slots, std::vector<int4>& items, std::vector<int>& off,
               int strip_stages = 192);
}  // namespace

void starmap_config_default(starmap_config* c) {
    if (!c) return;
    std::memset(c, 0, sizeof(*c));
    c->system = STARMAP_PN2D;
    c->N = 1;
    c->ax[0] = 0; c->ax[1] = 1; c->ax[2] = 0; c->ax[3] = 1;
    c->n[0] = 16; c->n[1] = 16;
    c->bc[0] = STARMAP_PERIODIC; c->bc[1] = STARMAP_PERIODIC;
    c->cn = 0.5;
    c->dt = 0;
    c->precision = STARMAP_FP64;
    c->schedule = STARMAP_SCHEDULE_LITERAL;
    c->kernel = STARMAP_KERNEL_AUTO;
    c->cuda_stream = nullptr;
    c->closure = STARMAP_CLOSURE_NONE;
}

int starmap_host_matrices(int system, int N, int cap, double* Mx, double* My, int* grid, int* order,
                          double* lambda_max) {
    SystemMatrices s;
    std::string err;
    if (!build_system(system, N, s, err)) return fail(nullptr, STARMAP_E_ARG, err);
    if (cap < s.ncomp) return fail(nullptr, STARMAP_E_ARG, "capacity below the number of components");
    int n = s.ncomp;
    for (int i = 0; i < n; ++i) {
        for (int j = 0; j < n; ++j) {
            if (Mx) Mx[(size_t)i * n + j] = s.Mx[(size_t)i * n + j];
            if (My) My[(size_t)i * n + j] = s.My[(size_t)i * n + j];
        }
        if (grid) grid[i] = s.moms[i].grid;
        if (order) order[i] = s.moms[i].l;
    }
    if (lambda_max) *lambda_max = s.lambda_max;
    return STARMAP_OK;
}

int starmap_direction_moments(int system, int N, double mu, double phi, double* out, size_t count) {
    std::vector<double> v;
    std::string err;
    if (!direction_moments(system, N, mu, phi, v, err)) return fail(nullptr, STARMAP_E_ARG, err);
    if (!out || count < v.size()) return fail(nullptr, STARMAP_E_ARG, "out needs ncomp doubles");
    std::copy(v.begin(), v.end(), out);
    return STARMAP_OK;
}

int starmap_tiled_schedule(int N, int parity, int frozen_top, double dx, double dy,
                           int* stages, size_t stage_capacity, float* coef, size_t coef_capacity,
                           int* fin, size_t fin_capacity, long* counts) {
    std::vector<int> st, fi;
    std::vector<float> co;
    std::string err;
    const int rc = tiled_schedule(N, parity, frozen_top != 0, dx, dy, st, co, fi, err);
    if (rc) return fail(nullptr, rc == -8 ? STARMAP_E_UNSUPPORTED : STARMAP_E_ARG, err);
    if (stages) std::copy(st.begin(), st.begin() + std::min(st.size(), stage_capacity * 4), stages);
    if (coef) std::copy(co.begin(), co.begin() + std::min(co.size(), coef_capacity * 16), coef);
    if (fin) std::copy(fi.begin(), fi.begin() + std::min(fi.size(), fin_capacity), fin);
    if (counts) {
        counts[0] = (long)(st.size() / 4);
        counts[1] = (long)(co.size() / 16);
        counts[2] = (long)fi.size();
    }
    return STARMAP_OK;
}

int starmap_batch_plan(const int* tiles_x, const int* tiles_y, const int* cost, int count, int slots,
                       int* items, size_t item_capacity, int* off, size_t off_capacity, long* counts) {
    if (count < 1 || slots < 1 || !tiles_x || !tiles_y || !cost)
        return fail(nullptr, STARMAP_E_ARG, "batch_plan needs count >= 1, slots >= 1 and the shape arrays");
    std::vector<BatchShape> shapes(count);
    for (int i = 0; i < count; ++i) {
        if (tiles_x[i] < 1 || tiles_y[i] < 1 || cost[i] < 0 || (long long)tiles_x[i] * tiles_y[i] > 0x7fffffffll)
            return fail(nullptr, STARMAP_E_ARG, "batch_plan: bad shape of instance " + std::to_string(i));
        shapes[i] = {tiles_x[i], tiles_y[i], cost[i]};
    }
    std::vector<int4> it;
    std::vector<int> of;
    const int grid = batch_plan(shapes, slots, it, of);
    if (grid < 1) return fail(nullptr, STARMAP_E_ARG, "too many tiles in one batch");
    if (items)
        for (size_t e = 0; e < std::min(it.size(), item_capacity); ++e) {
            items[4 * e] = it[e].x; items[4 * e + 1] = it[e].y; items[4 * e + 2] = it[e].z; items[4 * e + 3] = it[e].w;
        }
    if (off) std::copy(of.begin(), of.begin() + std::min(of.size(), off_capacity), off);
    if (counts) { counts[0] = grid; counts[1] = (long)it.size(); }
    return STARMAP_OK;
}

int starmap_host_expm1div(double* c, size_t count) {
    if (!c && count) return STARMAP_E_ARG;
    for (size_t i = 0; i < count; ++i) c[i] = expm1div(c[i]);
    return STARMAP_OK;
}

// starmap_create; shape: see TiledGeometry.
static int create_handle(const starmap_config* cfg, int shape, starmap_t** out) {
    if (!out) return fail(nullptr, STARMAP_E_ARG, "out is NULL");
    *out = nullptr;
    if (!cfg) return fail(nullptr, STARMAP_E_ARG, "cfg is NULL");
    const starmap_config& c = *cfg;
    if (c.system != STARMAP_PN2D && c.system != STARMAP_SLAB) return fail(nullptr, STARMAP_E_ARG, "unknown system");
    if (c.N < 1 || c.N > 63) return fail(nullptr, STARMAP_E_ARG, "N must be in [1, 63]");
    if (c.n[0] < 1 || c.n[1] < 1 || c.n[0] > (1 << 16) || c.n[1] > (1 << 16))
        return fail(nullptr, STARMAP_E_ARG, "grid size out of range");
    if (!(c.ax[1] > c.ax[0]) || !(c.ax[3] > c.ax[2])) return fail(nullptr, STARMAP_E_ARG, "empty domain");
    for (int d = 0; d < 2; ++d)
        if (c.bc[d] != STARMAP_PERIODIC && c.bc[d] != STARMAP_EXTRAPOLATION)
            return fail(nullptr, STARMAP_E_ARG, "unknown boundary condition");
    if (c.precision != STARMAP_FP64 && c.precision != STARMAP_FP32) return fail(nullptr, STARMAP_E_ARG, "unknown precision");
    if (c.schedule != STARMAP_SCHEDULE_LITERAL && c.schedule != STARMAP_SCHEDULE_MERGED &&
        c.schedule != STARMAP_SCHEDULE_FUSED)
        return fail(nullptr, STARMAP_E_ARG, "unknown schedule");
    if (c.schedule == STARMAP_SCHEDULE_FUSED &&
        (c.closure != STARMAP_CLOSURE_NONE || c.system != STARMAP_PN2D || c.precision != STARMAP_FP32 ||
         c.kernel == STARMAP_KERNEL_GATHER))
        return fail(nullptr, STARMAP_E_UNSUPPORTED, "the fused schedule needs the tiled kernel: FP32, 2D, no closure");
    if (c.kernel < STARMAP_KERNEL_AUTO || c.kernel > STARMAP_KERNEL_TILED_SHORT) return fail(nullptr, STARMAP_E_ARG, "unknown kernel");
    if (c.closure != STARMAP_CLOSURE_NONE && c.closure != STARMAP_CLOSURE_MLP8)
        return fail(nullptr, STARMAP_E_ARG, "unknown closure");
    if (c.closure == STARMAP_CLOSURE_MLP8) {
        if (c.system != STARMAP_PN2D || c.N != 7)
            return fail(nullptr, STARMAP_E_UNSUPPORTED, "the learned closure is defined for the 2D system with N = 7");
    }

    starmap_t* h = new (std::nothrow) starmap_t();
    if (!h) return fail(nullptr, STARMAP_E_NOMEM, "host allocation failed");
    h->cfg = c;
    h->closure = c.closure;
    h->nsys = c.closure == STARMAP_CLOSURE_MLP8 ? 8 : c.N;
    std::string err;
    if (!build_system(c.system, h->nsys, h->sys, err)) { delete h; return fail(nullptr, STARMAP_E_ARG, err); }
    h->ncomp = h->sys.ncomp;
    h->frozen.assign(h->ncomp, 0);
    if (h->closure) {
        for (int j = 0; j < h->ncomp; ++j) h->frozen[j] = h->sys.moms[j].l == h->nsys;
        if (!closure_layout_ok(h)) { delete h; return fail(nullptr, STARMAP_E_UNSUPPORTED, "moment placement differs from the closure kernels'"); }
    }
    h->dx = (c.ax[1] - c.ax[0]) / c.n[0];
    h->dy = (c.ax[3] - c.ax[2]) / c.n[1];
    for (int d = 0; d < 2; ++d) h->p[d] = c.bc[d] == STARMAP_PERIODIC ? 1 : 0;
    const double hmin = c.system == STARMAP_SLAB ? h->dx : std::min(h->dx, h->dy);
    const double bound = c.system == STARMAP_SLAB ? 1.0 : 1.0 / std::sqrt(2.0);
    if (c.dt > 0) {
        h->dt = c.dt;
    } else {
        if (!(c.cn > 0)) { delete h; return fail(nullptr, STARMAP_E_ARG, "cn must be positive"); }
        h->dt = c.cn * hmin / h->sys.lambda_max;
    }
    if (h->dt * h->sys.lambda_max / hmin > bound * (1 + 1e-12)) {
        delete h;
        return fail(nullptr, STARMAP_E_CFL, "time step beyond the CFL bound (cn <= 1/sqrt(2) in 2D, 1 in slab)");
    }
    // grids (section 5.2)
    for (int g = 0; g < 4; ++g) {
        bool xnode = g & 1, ynode = g & 2;
        h->nxg[g] = xnode ? c.n[0] + 1 - h->p[0] : c.n[0];
        h->nyg[g] = ynode ? c.n[1] + 1 - h->p[1] : c.n[1];
        h->Kg[g] = h->sys.grid_count[g];
        h->cpg[g] = (h->nxg[g] + 31) / 32 * 32;
    }
    for (int j = 0; j < h->ncomp; ++j) h->members[h->sys.moms[j].grid].push_back(j);
    for (int g = 0; g < 4; ++g)
        std::sort(h->members[g].begin(), h->members[g].end(),
                  [&](int a, int b) { return h->sys.moms[a].local < h->sys.moms[b].local; });
    h->fp32 = c.precision == STARMAP_FP32;
    h->esize = h->fp32 ? 4 : 8;
    int nxmax = 0, nymax = 0;
    for (int g = 0; g < 4; ++g) { nxmax = std::max(nxmax, h->nxg[g]); nymax = std::max(nymax, h->nyg[g]); }
    h->pitch = ((nxmax + 6 + 31) / 32) * 32;
    h->rows = nymax + 2;
    h->comp_class.resize(h->ncomp);
    h->nclasses = 2;
    for (int j = 0; j < h->ncomp; ++j) h->comp_class[j] = class_of(h, h->sys.moms[j].l);
    h->src_slot.assign(h->ncomp, -1);
    for (int g = 0; g < 4; ++g) {
        size_t plane = (size_t)h->nxg[g] * h->nyg[g];
        h->sig_a[g].assign(plane, 0.0);
        h->sig_s[g].assign(plane, 0.0);
    }
    // kernel choice
    bool tiled_ok = tiled_supported(c.system, h->nsys, c.precision);
    const bool want_tiled = c.kernel >= STARMAP_KERNEL_TILED;
    if (want_tiled && !tiled_ok) {
        delete h;
        return fail(nullptr, STARMAP_E_UNSUPPORTED, "tiled kernel needs FP32, the 2D P_N system, N <= 63 and TMA support");
    }
    int variant = tiled_default_variant(h->nsys, nxmax, nymax);
    if (c.kernel == STARMAP_KERNEL_TILED_TALL) variant = 0;
    if (c.kernel == STARMAP_KERNEL_TILED_SHORT) variant = 1;
    h->kernel_used = (want_tiled || (c.kernel == STARMAP_KERNEL_AUTO && tiled_ok))
                         ? (variant ? STARMAP_KERNEL_TILED_SHORT : STARMAP_KERNEL_TILED_TALL) : STARMAP_KERNEL_GATHER;

    // device resources
    cudaError_t e;
    if (c.cuda_stream) { h->stream = (cudaStream_t)c.cuda_stream; h->own_stream = false; }
    else {
        e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) { int rc = cuda_fail(nullptr, e, "cudaStreamCreate"); delete h; return rc; }
        h->own_stream = true;
    }
    auto bail = [&](int rc) { if (rc != STARMAP_OK) { std::string m = h->err; release(h); delete h; g_create_error = m; } return rc; };
    for (int g = 0; g < 4; ++g) {
        h->cstride[g] = h->rows * h->pitch;
        size_t elems = LEAD + (size_t)std::max(1, h->Kg[g]) * h->cstride[g] + h->pitch;
        h->grid_bytes[g] = elems * h->esize;
        e = dev_alloc(&h->alloc[g], h->grid_bytes[g]);
        if (e != cudaSuccess) return bail(fail(h, e == cudaErrorMemoryAllocation ? STARMAP_E_NOMEM : STARMAP_E_CUDA,
                                                std::string("cudaMalloc state: ") + cudaGetErrorString(e)));
        e = cudaMemsetAsync(h->alloc[g], 0, h->grid_bytes[g], h->stream);
        if (e != cudaSuccess) return bail(cuda_fail(h, e, "cudaMemset state"));
        h->base[g] = (char*)h->alloc[g] + LEAD * h->esize;
    }
    e = dev_alloc(&h->partials, (size_t)h->red_blocks * 3 * sizeof(double));
    if (e != cudaSuccess) return bail(cuda_fail(h, e, "cudaMalloc reduction"));
    e = dev_alloc(&h->result, 4 * sizeof(double));
    if (e != cudaSuccess) return bail(cuda_fail(h, e, "cudaMalloc reduction"));
    if (h->kernel_used != STARMAP_KERNEL_GATHER) {
        TiledGeometry geo;
        for (int g = 0; g < 4; ++g) {
            geo.base[g] = h->base[g]; geo.cstride[g] = h->cstride[g];
            geo.nx[g] = h->nxg[g]; geo.ny[g] = h->nyg[g]; geo.K[g] = h->Kg[g]; geo.cp[g] = h->cpg[g];
        }
        geo.pitch = h->pitch; geo.rows = h->rows; geo.p[0] = h->p[0]; geo.p[1] = h->p[1]; geo.N = h->nsys; geo.shape = shape;
        geo.variant = h->kernel_used == STARMAP_KERNEL_TILED_SHORT ? 1 : 0;
        int rc = tiled_create(geo, &h->tiled);
        if (rc) { std::string m = h->tiled ? tiled_error(h->tiled) : "tiled kernel setup failed"; return bail(fail(h, rc, m)); }
    }
    int rc = upload_all_coefficients(h);
    if (rc) return bail(rc);
    if (h->tiled) { for (int g = 0; g < 4; ++g) tiled_set_coef(h->tiled, g, h->coef[g], h->nclasses); }
    rc = rebuild_tables(h);
    if (rc == STARMAP_E_UNSUPPORTED && h->tiled && h->kernel_used == STARMAP_KERNEL_TILED_TALL &&
        (c.kernel == STARMAP_KERNEL_AUTO || c.kernel == STARMAP_KERNEL_TILED)) {
        // at the highest orders the partial sums and tables of the 10-row
        // tiles leave no room for a ring: the 5-row tiles (half the partial
        // sums, one CTA per SM where needed)
        tiled_destroy(h->tiled);
        h->tiled = nullptr;
        h->err.clear();
        TiledGeometry geo;
        for (int g = 0; g < 4; ++g) {
            geo.base[g] = h->base[g]; geo.cstride[g] = h->cstride[g];
            geo.nx[g] = h->nxg[g]; geo.ny[g] = h->nyg[g]; geo.K[g] = h->Kg[g]; geo.cp[g] = h->cpg[g];
        }
        geo.pitch = h->pitch; geo.rows = h->rows; geo.p[0] = h->p[0]; geo.p[1] = h->p[1]; geo.N = h->nsys; geo.shape = shape;
        geo.variant = 1;
        rc = tiled_create(geo, &h->tiled);
        if (rc) return bail(fail(h, rc, h->tiled ? tiled_error(h->tiled) : "tiled kernel setup failed"));
        h->kernel_used = STARMAP_KERNEL_TILED_SHORT;
        for (int g = 0; g < 4; ++g) tiled_set_coef(h->tiled, g, h->coef[g], h->nclasses);
        rc = rebuild_tables(h);
    }
    if (rc == STARMAP_E_UNSUPPORTED && h->tiled && c.kernel == STARMAP_KERNEL_AUTO) {
        // beyond that the gather kernel
        tiled_destroy(h->tiled);
        h->tiled = nullptr;
        h->kernel_used = STARMAP_KERNEL_GATHER;
        h->err.clear();
        rc = rebuild_tables(h);
    }
    if (rc) return bail(rc);
    if (c.schedule == STARMAP_SCHEDULE_FUSED) {
        // the second state set the fused steps alternate with
        if (!h->tiled) return bail(fail(h, STARMAP_E_UNSUPPORTED, "the fused schedule needs the tiled kernel"));
        for (int g = 0; g < 4; ++g) {
            e = dev_alloc(&h->alloc1[g], h->grid_bytes[g]);
            if (e != cudaSuccess) return bail(fail(h, e == cudaErrorMemoryAllocation ? STARMAP_E_NOMEM : STARMAP_E_CUDA,
                                                    std::string("cudaMalloc second state: ") + cudaGetErrorString(e)));
            e = cudaMemsetAsync(h->alloc1[g], 0, h->grid_bytes[g], h->stream);
            if (e != cudaSuccess) return bail(cuda_fail(h, e, "cudaMemset second state"));
            h->base1[g] = (char*)h->alloc1[g] + LEAD * h->esize;
        }
        rc = tiled_fused_setup(h->tiled, h->base1);
        if (rc) return bail(fail(h, rc, tiled_error(h->tiled)));
    }
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return bail(cuda_fail(h, e, "create"));
    *out = h;
    return STARMAP_OK;
}

int starmap_create(const starmap_config* cfg, starmap_t** out) { return create_handle(cfg, -1, out); }

void starmap_destroy(starmap_t* h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    release(h);
    delete h;
}

const char* starmap_last_error(const starmap_t* h) {
    return h ? h->err.c_str() : g_create_error.c_str();
}

int starmap_num_moments(const starmap_t* h) { return h ? h->ncomp : 0; }
double starmap_dt(const starmap_t* h) { return h ? h->dt : 0.0; }
double starmap_time(const starmap_t* h) { return h ? h->t : 0.0; }
long starmap_steps_done(const starmap_t* h) { return h ? h->steps : 0; }
int starmap_kernel(const starmap_t* h) { return h ? h->kernel_used : 0; }

int starmap_moment_info(const starmap_t* hc, int j, int* l, int* m, int* is_imag, int* grid, int* nx, int* ny) {
    starmap_t* h = const_cast<starmap_t*>(hc);
    int rc = check_j(h, j);
    if (rc) return rc;
    const Moment& mo = h->sys.moms[j];
    if (l) *l = mo.l;
    if (m) *m = mo.m;
    if (is_imag) *is_imag = mo.imag ? 1 : 0;
    if (grid) *grid = mo.grid;
    if (nx) *nx = h->nxg[mo.grid];
    if (ny) *ny = h->nyg[mo.grid];
    return STARMAP_OK;
}

int starmap_grid_info(const starmap_t* hc, int g, int* nx, int* ny, double* x0, double* y0, double* dx, double* dy) {
    starmap_t* h = const_cast<starmap_t*>(hc);
    if (!h) return STARMAP_E_ARG;
    if (g < 0 || g > 3) return fail(h, STARMAP_E_ARG, "grid index out of range");
    bool xnode = g & 1, ynode = g & 2;
    if (nx) *nx = h->nxg[g];
    if (ny) *ny = h->nyg[g];
    // eq. grid11 / staggered_grids: cells at (i - 1/2) h, nodes at i h, i from p
    if (x0) *x0 = h->cfg.ax[0] + (xnode ? h->p[0] * h->dx : 0.5 * h->dx);
    if (y0) *y0 = h->cfg.ax[2] + (ynode ? h->p[1] * h->dy : 0.5 * h->dy);
    if (dx) *dx = h->dx;
    if (dy) *dy = h->dy;
    return STARMAP_OK;
}

int starmap_set_material(starmap_t* h, int g, const double* sigma_a, const double* sigma_s0, size_t count) {
    if (!h) return STARMAP_E_ARG;
    if (g < 0 || g > 3) return fail(h, STARMAP_E_ARG, "grid index out of range");
    size_t plane = (size_t)h->nxg[g] * h->nyg[g];
    if (count != plane) return fail(h, STARMAP_E_ARG, "material size does not match the grid");
    if (!sigma_a || !sigma_s0) return fail(h, STARMAP_E_ARG, "material array is NULL");
    for (size_t i = 0; i < plane; ++i) {
        if (!std::isfinite(sigma_a[i]) || !std::isfinite(sigma_s0[i]))
            return fail(h, STARMAP_E_NONFINITE, "material contains NaN or Inf");
    }
    CK(cudaStreamSynchronize(h->stream), "set_material");
    h->sig_a[g].assign(sigma_a, sigma_a + plane);
    h->sig_s[g].assign(sigma_s0, sigma_s0 + plane);
    if (g == 0) h->lsig_dirty = true;
    int rc = ensure_coef_alloc(h);
    if (rc) return rc;
    rc = h->fp32 ? upload_coefficients<float>(h, g) : upload_coefficients<double>(h, g);
    if (rc) return rc;
    if (h->tiled) tiled_set_coef(h->tiled, g, h->coef[g], h->nclasses);
    ++h->version;
    return STARMAP_OK;
}

int starmap_set_scattering_factors(starmap_t* h, const double* factor, int count) {
    if (!h) return STARMAP_E_ARG;
    CK(cudaStreamSynchronize(h->stream), "set_scattering_factors");
    if (!factor) {
        h->sl_factor.clear();
        h->nclasses = 2;
    } else {
        if (count != h->nsys + 1)
            return fail(h, STARMAP_E_ARG, "factor must have one entry per order of the system (N+1; 9 with the closure)");
        h->sl_factor.assign(factor, factor + count);
        h->nclasses = h->nsys + 1;
    }
    for (int j = 0; j < h->ncomp; ++j) h->comp_class[j] = class_of(h, h->sys.moms[j].l);
    int rc = upload_all_coefficients(h);
    if (rc) return rc;
    if (h->tiled) for (int g = 0; g < 4; ++g) tiled_set_coef(h->tiled, g, h->coef[g], h->nclasses);
    return rebuild_tables(h);
}

int starmap_set_source(starmap_t* h, int j, const double* q, size_t count) {
    int rc = check_j(h, j);
    if (rc) return rc;
    if (h->frozen[j] && q) return fail(h, STARMAP_E_ARG, "the order-8 components of the closure take no source");
    CK(cudaStreamSynchronize(h->stream), "set_source");
    size_t np = comp_points(h, j);
    const int g = h->sys.moms[j].grid;
    if (!q) {
        if (j < (int)h->src_sq.size()) h->src_sq[j] = 0.0;
        if (h->src_slot[j] >= 0) {
            int s = h->src_slot[j];
            cudaFree(h->src_dev[s]);
            h->src_dev[s] = nullptr;
            h->src_slot[j] = -1;
            // compact slots
            std::vector<void*> keep;
            std::vector<int> remap(h->src_dev.size(), -1);
            for (size_t i = 0; i < h->src_dev.size(); ++i)
                if (h->src_dev[i]) { remap[i] = (int)keep.size(); keep.push_back(h->src_dev[i]); }
            for (int k = 0; k < h->ncomp; ++k) if (h->src_slot[k] >= 0) h->src_slot[k] = remap[h->src_slot[k]];
            h->src_dev = keep;
        }
        return rebuild_tables(h);
    }
    if (count != np) return fail(h, STARMAP_E_ARG, "source size does not match the grid of the component");
    const bool new_slot = h->src_slot[j] < 0;
    if (new_slot) {
        void* d = nullptr;
        CK(dev_alloc(&d, (size_t)h->cpg[g] * h->nyg[g] * h->esize), "cudaMalloc source");
        h->src_slot[j] = (int)h->src_dev.size();
        h->src_dev.push_back(d);
    }
    void* d = h->src_dev[h->src_slot[j]];
    if (h->src_sq.size() != (size_t)h->ncomp) h->src_sq.assign(h->ncomp, 0.0);
    double sq = 0.0;
    for (size_t i = 0; i < np; ++i) sq += q[i] * q[i];
    h->src_sq[j] = sq;
    const int nx = h->nxg[g], ny = h->nyg[g], cp = h->cpg[g];
    CK(h->fp32 ? upload_rows<float>(d, q, nx, ny, cp, h->stream) : upload_rows<double>(d, q, nx, ny, cp, h->stream),
       "upload source");
    // the pass tables only change when a component gains a source
    return new_slot ? rebuild_tables(h) : STARMAP_OK;
}

int starmap_set_moment(starmap_t* h, int j, const double* u, size_t count) {
    int rc = check_j(h, j);
    if (rc) return rc;
    size_t np = comp_points(h, j);
    if (!u || count != np) return fail(h, STARMAP_E_ARG, "moment size does not match the grid of the component");
    if (h->fp32) {
        std::vector<float> tmp(u, u + np);
        rc = upload_raw(h, j, tmp.data());
        if (rc) return rc;
        CK(cudaStreamSynchronize(h->stream), "set_moment");
    } else {
        rc = upload_raw(h, j, u);
        if (rc) return rc;
        CK(cudaStreamSynchronize(h->stream), "set_moment");
    }
    h->have_output = false;
    return STARMAP_OK;
}

}  // extern "C"

namespace {

// Rows [y0, y0 + rows) of every component of grid g <-> a packed buffer
// [component][row][x] (one 3D copy; buf host or device memory).
int copy_rows(starmap_t* h, int g, int y0, int rows, void* buf, size_t bytes, bool pack) {
    if (!h) return STARMAP_E_ARG;
    if (g < 0 || g > 3) return fail(h, STARMAP_E_ARG, "grid index out of range");
    if (y0 < 0 || rows < 0 || y0 + rows > h->nyg[g]) return fail(h, STARMAP_E_ARG, "rows leave the grid");
    const size_t need = (size_t)h->Kg[g] * rows * h->nxg[g] * h->esize;
    if (bytes != need) return fail(h, STARMAP_E_ARG, "buffer size does not match components x rows x nx of the grid");
    if (need == 0) return STARMAP_OK;
    if (!buf) return fail(h, STARMAP_E_ARG, "null buffer");
    if (int rc = poll_kernel(h)) return rc;
    char* dev = (char*)h->base[g] + (size_t)(y0 + 1) * h->pitch * h->esize;
    cudaPitchedPtr state = make_cudaPitchedPtr(dev, h->pitch * h->esize, h->nxg[g] * h->esize, h->rows);
    cudaPitchedPtr packed = make_cudaPitchedPtr(buf, h->nxg[g] * h->esize, h->nxg[g] * h->esize, rows);
    cudaMemcpy3DParms p = {};
    p.srcPtr = pack ? state : packed;
    p.dstPtr = pack ? packed : state;
    p.extent = make_cudaExtent(h->nxg[g] * h->esize, rows, h->Kg[g]);
    p.kind = cudaMemcpyDefault;
    CK(cudaMemcpy3DAsync(&p, h->stream), pack ? "pack rows" : "unpack rows");
    if (!pack) { h->ghosts_dirty = true; h->have_output = false; }
    return STARMAP_OK;
}

}  // namespace

extern "C" {

int starmap_pack_rows(starmap_t* h, int g, int y0, int rows, void* buf, size_t bytes) {
    return copy_rows(h, g, y0, rows, buf, bytes, true);
}

int starmap_unpack_rows(starmap_t* h, int g, int y0, int rows, const void* buf, size_t bytes) {
    return copy_rows(h, g, y0, rows, const_cast<void*>(buf), bytes, false);
}

int starmap_clear(starmap_t* h) {
    if (!h) return STARMAP_E_ARG;
    for (int g = 0; g < 4; ++g)
        CK(cudaMemsetAsync(h->alloc[g], 0, h->grid_bytes[g], h->stream), "clear");
    h->t = 0.0;
    h->steps = 0;
    h->have_output = false;
    h->ghosts_dirty = false;      // all ghosts are zero, consistent with the zero state
    return STARMAP_OK;
}

int starmap_set_time(starmap_t* h, double t) {
    if (!h) return STARMAP_E_ARG;
    h->t = t;
    return STARMAP_OK;
}

}  // extern "C"

namespace {

// FP64 reduction of the whole state, res = {mass, l2, nonfinite}
// (synchronises the stream).
int reduce_state(starmap_t* h, double* res) {
    int rc;
    if (h->fp32) {
        ReduceArgs<float> a;
        for (int g = 0; g < 4; ++g) a.g[g] = grid_dev<float>(h, g);
        a.pitch = h->pitch; a.cell = h->dx * h->dy;
        rc = launch_reduce<float>(a, h->partials, h->red_blocks, h->result, h->stream);
    } else {
        ReduceArgs<double> a;
        for (int g = 0; g < 4; ++g) a.g[g] = grid_dev<double>(h, g);
        a.pitch = h->pitch; a.cell = h->dx * h->dy;
        rc = launch_reduce<double>(a, h->partials, h->red_blocks, h->result, h->stream);
    }
    if (rc) return cuda_fail(h, cudaGetLastError(), "reduction");
    if ((rc = poll_kernel(h))) return rc;
    CK(cudaMemcpyAsync(res, h->result, 3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "reduction read-back");
    CK(cudaStreamSynchronize(h->stream), "reduction");
    return STARMAP_OK;
}

double source_l2(const starmap_t* h) {
    double s = 0.0;
    for (double v : h->src_sq) s += v;
    return std::sqrt(s * h->dx * h->dy);
}

int health_copy(starmap_t* h, bool save) {
    for (int g = 0; g < 4; ++g) {
        if (save) CK(cudaMemcpyAsync(h->snap[g], h->alloc[g], h->grid_bytes[g], cudaMemcpyDeviceToDevice, h->stream), "health copy");
        else CK(cudaMemcpyAsync(h->alloc[g], h->snap[g], h->grid_bytes[g], cudaMemcpyDeviceToDevice, h->stream), "health restore");
    }
    if (save) { h->snap_t = h->t; h->snap_steps = h->steps; }
    else { h->t = h->snap_t; h->steps = h->snap_steps; h->ghosts_dirty = true; }
    return STARMAP_OK;
}

// Steps in spans of health_every with the FP64 check after each span; on
// failure the state of the last span that passed comes back.
template <class T>
int do_steps_checked(starmap_t* h, long n) {
    if (n <= 0) return STARMAP_OK;
    for (int g = 0; g < 4; ++g)
        if (!h->snap[g]) CK(dev_alloc(&h->snap[g], h->grid_bytes[g]), "cudaMalloc health copy");
    double res[3];
    int rc = reduce_state(h, res);
    if (rc) return rc;
    h->health_good_steps = h->steps;
    h->health_l2_good = res[1];
    h->health_l2_failed = std::nan("");
    if (starmap_health_verdict(res[1], res[1], 0.0, 0.0, 1.0, (long)res[2]) != STARMAP_OK) {
        h->health_l2_failed = res[1];
        return fail(h, STARMAP_E_NONFINITE, "health check: the state holds NaN or Inf before stepping");
    }
    if ((rc = health_copy(h, true))) return rc;
    for (long done = 0; done < n;) {
        const long k = std::min(h->health_every, n - done);
        if ((rc = do_steps<T>(h, k))) return rc;
        if ((rc = reduce_state(h, res))) return rc;
        const int v = starmap_health_verdict(h->health_l2_good, res[1], k * h->dt, source_l2(h), h->health_growth,
                                             (long)res[2]);
        if (v != STARMAP_OK) {
            h->health_l2_failed = res[1];
            if ((rc = health_copy(h, false))) return rc;
            return fail(h, v, v == STARMAP_E_NONFINITE
                                  ? "health check: NaN or Inf after a span; state reset to the last span that passed"
                                  : "health check: L2 norm grew past its bound; state reset to the last span that passed");
        }
        h->health_good_steps = h->steps;
        h->health_l2_good = res[1];
        done += k;
        if (done < n && (rc = health_copy(h, true))) return rc;
    }
    return STARMAP_OK;
}

}  // namespace

extern "C" {

int starmap_health_verdict(double l2_start, double l2_end, double t_span, double q_l2, double growth,
                           long nonfinite) {
    if (nonfinite > 0 || !std::isfinite(l2_start) || !std::isfinite(l2_end)) return STARMAP_E_NONFINITE;
    if (l2_end > growth * (l2_start + t_span * q_l2)) return STARMAP_E_GROWTH;
    return STARMAP_OK;
}

int starmap_set_health_check(starmap_t* h, long every, double growth) {
    if (!h) return STARMAP_E_ARG;
    if (every < 0 || !(growth >= 1.0) || !std::isfinite(growth))
        return fail(h, STARMAP_E_ARG, "health check: every must be >= 0 and growth >= 1");
    h->health_every = every;
    h->health_growth = growth;
    if (every == 0) {
        CK(cudaStreamSynchronize(h->stream), "health check off");
        for (int g = 0; g < 4; ++g) if (h->snap[g]) { cudaFree(h->snap[g]); h->snap[g] = nullptr; }
    }
    return STARMAP_OK;
}

int starmap_health(const starmap_t* h, long* good_steps, double* l2_good, double* l2_failed) {
    if (!h) return STARMAP_E_ARG;
    if (good_steps) *good_steps = h->health_good_steps;
    if (l2_good) *l2_good = h->health_l2_good;
    if (l2_failed) *l2_failed = h->health_l2_failed;
    return STARMAP_OK;
}

int starmap_set_time_dependence(starmap_t* h, starmap_field_fn fn, void* user, const int* source_comps,
                                int n_sources) {
    if (!h) return STARMAP_E_ARG;
    if (!fn) {
        h->td_fn = nullptr;
        h->td_user = nullptr;
        h->td_src.clear();
        return STARMAP_OK;
    }
    if (n_sources < 0 || (n_sources > 0 && !source_comps)) return fail(h, STARMAP_E_ARG, "bad source list");
    std::vector<char> seen(h->ncomp, 0);
    for (int i = 0; i < n_sources; ++i) {
        const int j = source_comps[i];
        if (j < 0 || j >= h->ncomp) return fail(h, STARMAP_E_ARG, "source component out of range");
        if (h->frozen[j]) return fail(h, STARMAP_E_ARG, "the order-8 components of the closure take no source");
        if (seen[j]++) return fail(h, STARMAP_E_ARG, "source component listed twice");
    }
    for (int g = 0; g < 4; ++g) {
        double x0, y0, dx, dy;
        int nx, ny;
        starmap_grid_info(h, g, &nx, &ny, &x0, &y0, &dx, &dy);
        h->gx[g].resize((size_t)nx * ny);
        h->gy[g].resize((size_t)nx * ny);
        for (int k = 0; k < ny; ++k)
            for (int i = 0; i < nx; ++i) {
                h->gx[g][(size_t)k * nx + i] = x0 + i * dx;
                h->gy[g][(size_t)k * nx + i] = y0 + k * dy;
            }
    }
    // components that had a source and are not listed lose it
    for (int j = 0; j < h->ncomp; ++j)
        if (!seen[j] && h->src_slot[j] >= 0) {
            int rc = starmap_set_source(h, j, nullptr, 0);
            if (rc) return rc;
        }
    h->td_fn = fn;
    h->td_user = user;
    h->td_src.assign(source_comps, source_comps + n_sources);
    return STARMAP_OK;
}

}  // extern "C"

namespace {

// Material and sources of a time-dependent problem at time t, through the
// caller's callback.
int load_fields_at(starmap_t* h, double t) {
    std::vector<double> a, s;
    for (int g = 0; g < 4; ++g) {
        const size_t np = h->gx[g].size();
        if (np == 0) continue;
        a.resize(np);
        s.resize(np);
        if (h->td_fn(h->td_user, STARMAP_FIELD_SIGMA_A, t, g, h->gx[g].data(), h->gy[g].data(), np, a.data()) ||
            h->td_fn(h->td_user, STARMAP_FIELD_SIGMA_S0, t, g, h->gx[g].data(), h->gy[g].data(), np, s.data()))
            return fail(h, STARMAP_E_ARG, "time-dependence callback failed (material)");
        int rc = starmap_set_material(h, g, a.data(), s.data(), np);
        if (rc) return rc;
    }
    for (int j : h->td_src) {
        const int g = h->sys.moms[j].grid;
        const size_t np = h->gx[g].size();
        a.resize(np);
        if (h->td_fn(h->td_user, STARMAP_FIELD_SOURCE + j, t, g, h->gx[g].data(), h->gy[g].data(), np, a.data()))
            return fail(h, STARMAP_E_ARG, "time-dependence callback failed (source)");
        int rc = starmap_set_source(h, j, a.data(), np);
        if (rc) return rc;
    }
    return STARMAP_OK;
}

}  // namespace

extern "C" {

int starmap_step(starmap_t* h, long nsteps) {
    if (!h) return STARMAP_E_ARG;
    if (nsteps < 0) return fail(h, STARMAP_E_ARG, "negative step count");
    h->have_output = false;
    if (h->td_fn) {
        for (long i = 0; i < nsteps; ++i) {
            int rc = load_fields_at(h, h->t + 0.5 * h->dt);
            if (rc) return rc;
            // one step of the merged schedule is O_1/2 E O_1/2 with the fused even pair: the literal step
            if (h->health_every > 0)
                rc = h->fp32 ? do_steps_checked<float>(h, 1) : do_steps_checked<double>(h, 1);
            else
                rc = h->fp32 ? do_steps<float>(h, 1) : do_steps<double>(h, 1);
            if (rc) return rc;
        }
        return STARMAP_OK;
    }
    if (h->health_every > 0)
        return h->fp32 ? do_steps_checked<float>(h, nsteps) : do_steps_checked<double>(h, nsteps);
    return h->fp32 ? do_steps<float>(h, nsteps) : do_steps<double>(h, nsteps);
}

int starmap_pass(starmap_t* h, int parity, int which) {
    if (!h) return STARMAP_E_ARG;
    if (parity == 2) {
        // two fused inner steps (set 0 -> set 1 -> set 0)
        if (h->cfg.schedule != STARMAP_SCHEDULE_FUSED || which != 1)
            return fail(h, STARMAP_E_ARG, "parity 2 (a fused pair) needs the fused schedule and which = 1");
        h->have_output = false;
        if (h->ghosts_dirty) { int rc = fill_ghosts_all<float>(h); if (rc) return rc; }
        return fused_inner_steps(h, 2);
    }
    if ((parity != 0 && parity != 1) || (which != 0 && which != 1)) return fail(h, STARMAP_E_ARG, "parity and which must be 0 or 1");
    h->have_output = false;
    if (h->closure && parity == 1 && !h->net_ready)
        return fail(h, STARMAP_E_STATE, "closure handle stepped before starmap_set_closure");
    if (h->fp32) {
        if (h->ghosts_dirty) { int rc = fill_ghosts_all<float>(h); if (rc) return rc; }
        return parity == 1 ? odd_pass<float>(h, which) : run_pass<float>(h, false, which);
    }
    if (h->ghosts_dirty) { int rc = fill_ghosts_all<double>(h); if (rc) return rc; }
    return parity == 1 ? odd_pass<double>(h, which) : run_pass<double>(h, false, which);
}

int starmap_advance_to(starmap_t* h, double t_out) {
    if (!h) return STARMAP_E_ARG;
    const double eps = 1e-12 * std::max(1.0, std::fabs(t_out));
    if (t_out < h->t - eps) return fail(h, STARMAP_E_ARG, "t_out lies before the current time");
    for (int g = 0; g < 4; ++g) {
        if (!h->prev[g]) CK(dev_alloc(&h->prev[g], h->grid_bytes[g]), "cudaMalloc output level");
    }
    if (t_out <= h->t + eps) {
        for (int g = 0; g < 4; ++g)
            CK(cudaMemcpyAsync(h->prev[g], h->alloc[g], h->grid_bytes[g], cudaMemcpyDeviceToDevice, h->stream), "copy level");
        h->out_lambda = 1.0;
        h->have_output = true;
        return STARMAP_OK;
    }
    long n = (long)std::ceil((t_out - h->t) / h->dt - 1e-9);
    if (n < 1) n = 1;
    int rc = starmap_step(h, n - 1);
    if (rc) return rc;
    if (h->ghosts_dirty) {
        rc = h->fp32 ? fill_ghosts_all<float>(h) : fill_ghosts_all<double>(h);
        if (rc) return rc;
    }
    for (int g = 0; g < 4; ++g)
        CK(cudaMemcpyAsync(h->prev[g], h->alloc[g], h->grid_bytes[g], cudaMemcpyDeviceToDevice, h->stream), "copy level");
    double t0 = h->t;
    rc = starmap_step(h, 1);
    if (rc) return rc;
    h->out_lambda = (t_out - t0) / h->dt;
    h->have_output = true;
    return STARMAP_OK;
}

int starmap_output(starmap_t* h, int j, double* out, size_t count) {
    int rc = check_j(h, j);
    if (rc) return rc;
    if (!h->have_output) return fail(h, STARMAP_E_STATE, "no output level: call starmap_advance_to first");
    size_t np = comp_points(h, j);
    if (!out || count != np) return fail(h, STARMAP_E_ARG, "output size does not match the grid of the component");
    std::vector<double> a(np), b(np);
    void* prevb[4];
    for (int g = 0; g < 4; ++g) prevb[g] = h->prev[g] ? (char*)h->prev[g] + LEAD * h->esize : nullptr;
    if ((rc = download_double(h, j, prevb, a.data()))) return rc;
    if ((rc = download_double(h, j, h->base, b.data()))) return rc;
    const double lam = h->out_lambda;
    for (size_t i = 0; i < np; ++i) out[i] = (1.0 - lam) * a[i] + lam * b[i];
    return STARMAP_OK;
}

int starmap_moments(starmap_t* h, int j, double* out, size_t count) {
    int rc = check_j(h, j);
    if (rc) return rc;
    size_t np = comp_points(h, j);
    if (!out || count != np) return fail(h, STARMAP_E_ARG, "output size does not match the grid of the component");
    return download_double(h, j, h->base, out);
}

int starmap_moments_window(starmap_t* h, int j, int i0, int k0, int nx, int ny, double* out, size_t count) {
    int rc = check_j(h, j);
    if (rc) return rc;
    const int g = h->sys.moms[j].grid;
    if (i0 < 0 || k0 < 0 || nx < 0 || ny < 0 || i0 + nx > h->nxg[g] || k0 + ny > h->nyg[g])
        return fail(h, STARMAP_E_ARG, "window leaves the grid of the component");
    if (!out || count != (size_t)nx * ny) return fail(h, STARMAP_E_ARG, "output size does not match the window");
    if (nx == 0 || ny == 0) return STARMAP_OK;
    if ((rc = poll_kernel(h))) return rc;
    const char* src = comp_ptr(h, j, h->base) + ((size_t)k0 * h->pitch + i0) * h->esize;
    std::vector<char> tmp((size_t)nx * ny * h->esize);
    CK(cudaMemcpy2DAsync(tmp.data(), nx * h->esize, src, h->pitch * h->esize, nx * h->esize, ny,
                         cudaMemcpyDeviceToHost, h->stream), "download window");
    CK(cudaStreamSynchronize(h->stream), "download window");
    for (size_t i = 0; i < (size_t)nx * ny; ++i)
        out[i] = h->fp32 ? (double)((const float*)tmp.data())[i] : ((const double*)tmp.data())[i];
    return STARMAP_OK;
}

int starmap_diagnostics(starmap_t* h, double* mass, double* l2, long* nonfinite) {
    if (!h) return STARMAP_E_ARG;
    double res[3];
    int rc = reduce_state(h, res);
    if (rc) return rc;
    if (mass) *mass = res[0];
    if (l2) *l2 = res[1];
    if (nonfinite) *nonfinite = (long)res[2];
    if (res[2] > 0) return fail(h, STARMAP_E_NONFINITE, "state contains NaN or Inf");
    return STARMAP_OK;
}

int starmap_device_ptr(starmap_t* h, int j, void** ptr, long* pitch, long* offset) {
    int rc = check_j(h, j);
    if (rc) return rc;
    const Moment& m = h->sys.moms[j];
    if (ptr) *ptr = (char*)h->base[m.grid] + (size_t)m.local * h->cstride[m.grid] * h->esize;
    if (pitch) *pitch = h->pitch;
    if (offset) *offset = h->pitch;
    return STARMAP_OK;
}

size_t starmap_state_bytes(const starmap_t* h) {
    if (!h) return 0;
    size_t s = 0;
    for (int j = 0; j < h->ncomp; ++j) s += comp_points(h, j) * h->esize;
    return s + 2 * sizeof(double);
}

int starmap_get_state(starmap_t* h, void* buf, size_t bytes) {
    if (!h) return STARMAP_E_ARG;
    if (!buf || bytes < starmap_state_bytes(h)) return fail(h, STARMAP_E_ARG, "state buffer too small");
    if (int rc = poll_kernel(h)) return rc;
    char* p = (char*)buf;
    for (int j = 0; j < h->ncomp; ++j) {
        int rc = download_raw(h, j, h->base, p);
        if (rc) return rc;
        p += comp_points(h, j) * h->esize;
    }
    CK(cudaStreamSynchronize(h->stream), "get_state");
    double meta[2] = {h->t, (double)h->steps};
    std::memcpy(p, meta, sizeof(meta));
    return STARMAP_OK;
}

int starmap_set_state(starmap_t* h, const void* buf, size_t bytes) {
    if (!h) return STARMAP_E_ARG;
    if (!buf || bytes < starmap_state_bytes(h)) return fail(h, STARMAP_E_ARG, "state buffer too small");
    const char* p = (const char*)buf;
    for (int j = 0; j < h->ncomp; ++j) {
        int rc = upload_raw(h, j, p);
        if (rc) return rc;
        p += comp_points(h, j) * h->esize;
    }
    CK(cudaStreamSynchronize(h->stream), "set_state");
    double meta[2];
    std::memcpy(meta, p, sizeof(meta));
    h->t = meta[0];
    h->steps = (long)meta[1];
    h->have_output = false;
    return STARMAP_OK;
}

int starmap_debug_fail_allocation(int n) {
    if (n < 0) return fail(nullptr, STARMAP_E_ARG, "the allocation to fail is counted from 1 (0 disables)");
    starmap::alloc_fail_countdown().store(n);
    return STARMAP_OK;
}

int starmap_selftest_bounded_wait(void) {
    int gave_up = 0, tc_gave_up = 0;
    if (tiled_wait_selftest(&gave_up) || mlp::tc_wait_selftest(&tc_gave_up))
        return fail(nullptr, STARMAP_E_CUDA, "bounded-wait self-test could not run");
    if (!gave_up) return fail(nullptr, STARMAP_E_STATE, "bounded wait did not give up on a barrier nothing arrives at");
    if (!tc_gave_up)
        return fail(nullptr, STARMAP_E_STATE, "a network kernel's bounded wait did not give up as it must");
    return fail(nullptr, STARMAP_E_TIMEOUT, "bounded waits gave up as expected");
}

int starmap_selftest_abort_drain(int* us) {
    if (!us) return fail(nullptr, STARMAP_E_ARG, "us is NULL");
    if (tiled_drain_selftest(us)) return fail(nullptr, STARMAP_E_CUDA, "drain self-test could not run");
    return STARMAP_OK;
}

int starmap_sync(starmap_t* h) {
    if (!h) return STARMAP_E_ARG;
    CK(cudaStreamSynchronize(h->stream), "sync");
    return poll_kernel(h);
}

int starmap_set_closure(starmap_t* h, const float* params, size_t count) {
    if (!h) return STARMAP_E_ARG;
    if (!h->closure) return fail(h, STARMAP_E_STATE, "handle was created without a closure");
    if (!params || count != (size_t)mlp::NPARAM) return fail(h, STARMAP_E_ARG, "closure needs STARMAP_MLP_PARAMS floats");
    for (size_t i = 0; i < count; ++i)
        if (!std::isfinite(params[i])) return fail(h, STARMAP_E_NONFINITE, "closure parameters contain NaN or Inf");
    if (!h->net_params) CK(dev_alloc(&h->net_params, (size_t)mlp::NPARAM * sizeof(float)), "cudaMalloc closure");
    if (!h->net) CK(dev_alloc(&h->net, sizeof(mlp::Packed)), "cudaMalloc closure");
    CK(cudaMemcpyAsync(h->net_params, params, count * sizeof(float), cudaMemcpyHostToDevice, h->stream), "upload closure");
    if (mlp::pack(h->net_params, h->net, h->stream)) return cuda_fail(h, cudaGetLastError(), "pack closure");
    CK(cudaStreamSynchronize(h->stream), "set_closure");
    h->net_ready = true;
    return STARMAP_OK;
}

int starmap_set_closure_engine(starmap_t* h, int engine) {
    if (!h) return STARMAP_E_ARG;
    if (engine != STARMAP_MLP_ENGINE_MMA_SYNC && engine != STARMAP_MLP_ENGINE_TCGEN05)
        return fail(h, STARMAP_E_ARG, "unknown network engine");
    h->engine = engine == STARMAP_MLP_ENGINE_TCGEN05 ? mlp::ENGINE_TCGEN05 : mlp::ENGINE_MMA_SYNC;
    return STARMAP_OK;
}

int starmap_closure_samples(starmap_t* h, float* X, float* scale, float* targets, size_t count) {
    if (!h) return STARMAP_E_ARG;
    if (h->cfg.system != STARMAP_PN2D || h->nsys < 7)
        return fail(h, STARMAP_E_UNSUPPORTED, "closure samples need the 2D system with N >= 7");
    if (targets && h->nsys < 8) return fail(h, STARMAP_E_UNSUPPORTED, "order-8 targets need N >= 8");
    if (!closure_layout_ok(h)) return fail(h, STARMAP_E_UNSUPPORTED, "moment placement differs from the closure kernels'");
    const size_t M = (size_t)h->nxg[0] * h->nyg[0];
    if (!X || !scale || count != M) return fail(h, STARMAP_E_ARG, "samples need X, scale and count = n_x * n_y");
    if (h->ghosts_dirty) {
        int rc = h->fp32 ? fill_ghosts_all<float>(h) : fill_ghosts_all<double>(h);
        if (rc) return rc;
    }
    int rc = ensure_lsig(h);
    if (rc) return rc;
    rc = h->fp32 ? mlp::samples<float>(closure_args<float>(h), X, scale, targets, h->stream)
                 : mlp::samples<double>(closure_args<double>(h), X, scale, targets, h->stream);
    if (rc) return cuda_fail(h, cudaGetLastError(), "closure samples");
    return STARMAP_OK;
}


// ---------------------------------------------------------------- batches
namespace {
thread_local std::string g_batch_create_error;

int bfail(starmap_batch_t* b, int code, const std::string& msg) {
    if (b) b->err = msg; else g_batch_create_error = msg;
    return code;
}

void batch_release(starmap_batch_t* b) {
    for (auto& gx : b->graphs) cudaGraphExecDestroy(gx.second);
    b->graphs.clear();
    for (starmap_t* h : b->inst) starmap_destroy(h);
    b->inst.clear();
    if (b->dev_params) cudaFree(b->dev_params);
    if (b->dev_items) cudaFree(b->dev_items);
    if (b->dev_off) cudaFree(b->dev_off);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
}

// Upload the pass parameters of instances whose tables changed.
int batch_sync_params(starmap_batch_t* b) {
    const size_t pb = 4 * tiled_params_bytes();
    bool any = false;
    for (size_t i = 0; i < b->inst.size(); ++i) {
        starmap_t* h = b->inst[i];
        if (b->uploaded[i] == h->version) continue;
        if (tiled_export_params(h->tiled, b->staging.data() + i * pb))
            return bfail(b, STARMAP_E_STATE, "instance tables not built");
        // the batch kernel runs with the shared memory sized at creation
        if (std::max(tiled_smem_bytes(h->tiled, 0), tiled_smem_bytes(h->tiled, 1)) > b->smem)
            return bfail(b, STARMAP_E_STATE, "instance " + std::to_string(i) + " outgrew the batch's shared memory");
        b->uploaded[i] = h->version;
        any = true;
    }
    if (!any) return STARMAP_OK;
    cudaError_t e = cudaMemcpyAsync(b->dev_params, b->staging.data(), b->staging.size(), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bfail(b, STARMAP_E_CUDA, std::string("upload batch parameters: ") + cudaGetErrorString(e));
    return STARMAP_OK;
}

// The pass launches of one starmap_batch_step(b, n) (same schedules as do_steps).
int batch_issue(starmap_batch_t* b, long n) {
    auto pass = [&](int P, int w) {
        return tiled_batch_pass(b->dev_params, b->dev_items, b->dev_off, P, w, b->grid, b->smem, b->shape,
                                b->stream);
    };
    if (b->schedule == STARMAP_SCHEDULE_MERGED) {
        if (pass(1, 0)) return STARMAP_E_CUDA;
        for (long i = 0; i < n; ++i) {
            if (pass(0, 1)) return STARMAP_E_CUDA;
            if (pass(1, i == n - 1 ? 0 : 1)) return STARMAP_E_CUDA;
        }
    } else {
        for (long i = 0; i < n; ++i)
            if (pass(1, 0) || pass(0, 1) || pass(1, 0)) return STARMAP_E_CUDA;
    }
    return STARMAP_OK;
}
}  // namespace

namespace {
// Work units of all instances (heaviest instance first) form one list
// dealt to the resident CTAs (below) so that every CTA gets about the same
// work and at any time the CTAs work on one contiguous band of the list
// (x-neighbouring units run side by side and share their halo columns in
// L2).  A unit is
//  * for short tiles (few stages): a strip of consecutive tiles in y,
//    about STRIP_STAGES stages long, streamed through one pipeline (the
//    next tile's halo row is still in L2; setup, fill and drain are paid
//    once per strip);
//  * for long tiles: one tile; a CTA's tiles of one instance are then a
//    single run with stride grid (the band of tiles moves down the grid in
//    lockstep, so vertical neighbours also share halo rows in L2).
// Items are (instance, first tile, tile count, tile stride); CTA c runs
// items[off[c]] .. items[off[c + 1] - 1].  Returns the grid (0 if the
// lists would not fit 32-bit indices).
int batch_plan(const std::vector<BatchShape>& shapes, int slots, std::vector<int4>& items, std::vector<int>& off,
               int strip_stages_max) {
    const int count = (int)shapes.size();
    constexpr int STRIP_MAX_STAGES = 48;     // tiles up to this long go in strips
    // stages per strip: strip_stages_max (192 unless the batch autotuner
    // chose 96 or 384), halved while the list would hold fewer than four
    // units per CTA (a few small instances must still fill the GPU)
    std::vector<int> strip(count, 1);
    long long total_units = 0;
    for (int strip_stages = std::max(1, strip_stages_max);; strip_stages /= 2) {
        total_units = 0;
        for (int i = 0; i < count; ++i) {
            const int tx = shapes[i].tx, ty = shapes[i].ty;
            const int c = std::max(1, shapes[i].cost);
            strip[i] = c <= STRIP_MAX_STAGES ? std::max(1, std::min(ty, (strip_stages + c - 1) / c)) : 1;
            total_units += strip[i] > 1 ? (long long)tx * ((ty + strip[i] - 1) / strip[i]) : (long long)tx * ty;
        }
        if (total_units >= 4LL * slots || strip_stages <= 1) break;
    }
    const int grid = (int)std::max(1LL, std::min<long long>(total_units, std::max(1, slots)));
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        return (double)shapes[a].tx * shapes[a].ty * shapes[a].cost > (double)shapes[c].tx * shapes[c].ty * shapes[c].cost;
    });
    // Instances are dealt in that order, each to the CTAs by current load:
    // the strips of a short-tile instance in chunks of `grid` units, the
    // heaviest units of a chunk to the least-loaded CTAs; the tiles of a
    // long-tile instance as one strided run per CTA (residue k: tiles k,
    // k + grid, ...), the residues with one tile more to the least-loaded
    // CTAs.  Every CTA still works through the instances in the same order,
    // so at any time the CTAs share one band of the list.
    std::vector<std::vector<int4>> per(grid);
    std::vector<long long> load(grid, 0);
    std::vector<int> ctas(grid);
    auto by_load = [&]() {
        for (int c = 0; c < grid; ++c) ctas[c] = c;
        std::stable_sort(ctas.begin(), ctas.end(), [&](int a, int c) { return load[a] < load[c]; });
    };
    std::vector<int4> units;
    for (int i : order) {
        const int tx = shapes[i].tx, ty = shapes[i].ty;
        const long long c = shapes[i].cost;
        if (strip[i] > 1) {
            const int S = strip[i];
            units.clear();
            for (int y0 = 0; y0 < ty; y0 += S)
                for (int x = 0; x < tx; ++x) units.push_back(make_int4(i, y0 * tx + x, std::min(S, ty - y0), tx));
            for (size_t r = 0; r < units.size(); r += (size_t)grid) {
                const size_t end = std::min(units.size(), r + (size_t)grid);
                std::stable_sort(units.begin() + r, units.begin() + end,
                                 [](const int4& a, const int4& b) { return a.z > b.z; });
                by_load();
                for (size_t e = r; e < end; ++e) {
                    const int cta = ctas[e - r];
                    per[cta].push_back(units[e]);
                    load[cta] += (long long)units[e].z * c;
                }
            }
        } else {
            const int tiles = tx * ty, q = tiles / grid, rem = tiles % grid;
            by_load();
            for (int k = 0; k < grid; ++k) {
                const int n = q + (k < rem ? 1 : 0);
                if (n == 0) continue;
                per[ctas[k]].push_back(make_int4(i, k, n, grid));
                load[ctas[k]] += (long long)n * c;
            }
        }
    }
    items.clear();
    off.assign(grid + 1, 0);
    for (int cta = 0; cta < grid; ++cta) {
        off[cta] = (int)items.size();
        items.insert(items.end(), per[cta].begin(), per[cta].end());
        if (items.size() > 0x7fffffffu) return 0;
    }
    off[grid] = (int)items.size();
    return grid;
}

// (Re)plan the work units with strips of about `strip` stages, upload the
// lists and drop the captured step graphs (they hold the old lists).
int batch_replan(starmap_batch_t* b, int strip) {
    std::vector<int4> it;
    std::vector<int> off;
    const int grid = batch_plan(b->shapes, b->slots, it, off, strip);
    if (grid < 1) return bfail(b, STARMAP_E_ARG, "too many tiles in one batch");
    cudaError_t e = cudaStreamSynchronize(b->stream);
    for (auto& gx : b->graphs) cudaGraphExecDestroy(gx.second);
    b->graphs.clear();
    if (b->dev_items) { cudaFree(b->dev_items); b->dev_items = nullptr; }
    if (b->dev_off) { cudaFree(b->dev_off); b->dev_off = nullptr; }
    if (e == cudaSuccess) e = dev_alloc(&b->dev_off, off.size() * sizeof(int));
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->dev_off, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = dev_alloc(&b->dev_items, std::max<size_t>(1, it.size()) * sizeof(int4));
    if (e == cudaSuccess && !it.empty())
        e = cudaMemcpyAsync(b->dev_items, it.data(), it.size() * sizeof(int4), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bfail(b, e == cudaErrorMemoryAllocation ? STARMAP_E_NOMEM : STARMAP_E_CUDA,
                                       std::string("batch plan upload: ") + cudaGetErrorString(e));
    b->grid = grid;
    b->strip = strip;
    return STARMAP_OK;
}

// Build a batch whose instances use tile height `variant` (0: 10 rows, 1: 5 rows).
int batch_build(const starmap_config* cfgs, int count, int variant, starmap_batch_t** out) {
    *out = nullptr;
    if (!cfgs || count < 1) return bfail(nullptr, STARMAP_E_ARG, "a batch needs at least one configuration");
    starmap_batch_t* b = new (std::nothrow) starmap_batch_t();
    if (!b) return bfail(nullptr, STARMAP_E_NOMEM, "host allocation failed");
    auto bail = [&](int rc) {
        std::string m = b->err;
        batch_release(b);
        delete b;
        g_batch_create_error = m;
        return rc;
    };
    b->schedule = cfgs[0].schedule;
    if (b->schedule != STARMAP_SCHEDULE_LITERAL && b->schedule != STARMAP_SCHEDULE_MERGED)
        return bail(bfail(b, STARMAP_E_ARG, "unknown schedule"));
    cudaError_t e;
    if (cfgs[0].cuda_stream) {
        b->stream = (cudaStream_t)cfgs[0].cuda_stream;
    } else {
        e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) return bail(bfail(b, STARMAP_E_CUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e)));
        b->own_stream = true;
    }
    std::vector<BatchShape> shapes;
    b->variant = variant;
    int max_N = 1;                         // one kernel runs every instance
    for (int i = 0; i < count; ++i) max_N = std::max(max_N, cfgs[i].N);
    b->shape = tiled_batch_shape(variant, max_N);
    for (int i = 0; i < count; ++i) {
        starmap_config c = cfgs[i];
        if (c.system != STARMAP_PN2D || c.precision != STARMAP_FP32 || c.closure != STARMAP_CLOSURE_NONE)
            return bail(bfail(b, STARMAP_E_UNSUPPORTED, "batch instance " + std::to_string(i) +
                                                            ": batches hold FP32 2D P_N instances without closure"));
        c.kernel = b->variant ? STARMAP_KERNEL_TILED_SHORT : STARMAP_KERNEL_TILED_TALL;
        c.schedule = b->schedule;
        c.cuda_stream = b->stream;
        starmap_t* h = nullptr;
        int rc = create_handle(&c, b->shape, &h);
        if (rc) return bail(bfail(b, rc, "batch instance " + std::to_string(i) + ": " + g_create_error));
        b->inst.push_back(h);
        int tx = 0, ty = 0;
        tiled_tile_grid(h->tiled, &tx, &ty);
        const int cost = std::max(tiled_stage_count(h->tiled, 0), tiled_stage_count(h->tiled, 1));
        if ((long long)tx * ty * cost > 0x7fffffffll)
            return bail(bfail(b, STARMAP_E_ARG, "batch instance " + std::to_string(i) + ": too many pipeline stages"));
        shapes.push_back({tx, ty, cost});
        b->smem = std::max(b->smem, std::max(tiled_smem_bytes(h->tiled, 0), tiled_smem_bytes(h->tiled, 1)));
    }
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    b->slots = sms * tiled_batch_ctas(b->smem, b->shape);   // resident CTAs of the persistent grid
    b->shapes = shapes;
    int rc = tiled_batch_prepare(b->smem, b->shape);
    if (rc) return bail(bfail(b, rc, "batch kernel needs more shared memory than the device offers"));
    b->staging.assign((size_t)count * 4 * tiled_params_bytes(), 0);
    b->uploaded.assign(count, ~0ul);
    e = dev_alloc(&b->dev_params, b->staging.size());
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bail(bfail(b, e == cudaErrorMemoryAllocation ? STARMAP_E_NOMEM : STARMAP_E_CUDA,
                                            std::string("batch setup: ") + cudaGetErrorString(e)));
    rc = batch_sync_params(b);
    if (rc) return bail(rc);
    rc = batch_replan(b, b->strip);
    if (rc) return bail(rc);
    *out = b;
    return STARMAP_OK;
}

// Device time of `steps` batched steps (CUDA events on the batch stream).
int batch_time(starmap_batch_t* b, long steps, double* ms) {
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return STARMAP_E_CUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return STARMAP_E_CUDA; }
    int rc = starmap_batch_step(b, 1);                     // warm-up: graph capture and first touch
    if (!rc) rc = cudaEventRecord(e0, b->stream) == cudaSuccess ? 0 : STARMAP_E_CUDA;
    if (!rc) rc = starmap_batch_step(b, steps);
    if (!rc) rc = cudaEventRecord(e1, b->stream) == cudaSuccess ? 0 : STARMAP_E_CUDA;
    if (!rc) rc = cudaEventSynchronize(e1) == cudaSuccess ? 0 : STARMAP_E_CUDA;
    float t = 0.f;
    if (!rc) rc = cudaEventElapsedTime(&t, e0, e1) == cudaSuccess ? 0 : STARMAP_E_CUDA;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (!rc) rc = starmap_batch_sync(b);
    *ms = t / (double)steps;
    return rc;
}

// Back to t = 0, step 0 (the tuning steps ran on the zero state).
void batch_reset_clock(starmap_batch_t* b) {
    for (starmap_t* h : b->inst) {
        h->t = 0.0;
        h->steps = 0;
        h->have_output = false;
    }
}
}  // namespace

}  // extern "C"

namespace {

// The autotuner's cache: one line per batch signature, "signature rows
// strip ms" (the last line of a signature wins).
std::string tune_cache_path() {
    const char* env = std::getenv("STARMAP_TUNE_CACHE");
    if (env) return std::string(env) == "off" ? std::string() : std::string(env);
    const char* home = std::getenv("HOME");
    return home ? std::string(home) + "/.cache/starmap/batch_tune.txt" : std::string();
}

// The build's hash of the sources a tuning depends on (build.py); compiled
// without it, the time of compilation.
#ifndef STARMAP_BATCH_SOURCES
#define STARMAP_BATCH_SOURCES __DATE__ " " __TIME__
#endif

// FNV-1a over the batch kernel's sources, the device (name, SM count) and
// every instance's system, order, cells, boundaries and schedule.
std::string batch_signature(const starmap_config* cfgs, int count) {
    unsigned long long hsh = 1469598103934665603ull;
    auto mix = [&](const void* p, size_t n) {
        const unsigned char* c = static_cast<const unsigned char*>(p);
        for (size_t i = 0; i < n; ++i) { hsh ^= c[i]; hsh *= 1099511628211ull; }
    };
    mix(STARMAP_BATCH_SOURCES, sizeof(STARMAP_BATCH_SOURCES));
    int dev = 0;
    cudaDeviceProp prop;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaGetDeviceProperties(&prop, dev) == cudaSuccess) {
        mix(prop.name, std::strlen(prop.name));
        mix(&prop.multiProcessorCount, sizeof(int));
    }
    mix(&count, sizeof(int));
    for (int i = 0; i < count; ++i) {
        const starmap_config& c = cfgs[i];
        const int v[7] = {c.system, c.N, c.n[0], c.n[1], c.bc[0], c.bc[1], c.schedule};
        mix(v, sizeof(v));
    }
    char buf[32];
    std::snprintf(buf, sizeof(buf), "%016llx", hsh);
    return buf;
}

bool tune_cache_get(const std::string& sig, int* rows, int* strip) {
    const std::string path = tune_cache_path();
    if (path.empty()) return false;
    FILE* fp = std::fopen(path.c_str(), "r");
    if (!fp) return false;
    char s[64];
    int r, st;
    double ms;
    bool found = false;
    while (std::fscanf(fp, "%63s %d %d %lf", s, &r, &st, &ms) == 4)
        if (sig == s && (r == 10 || r == 5) && st >= 1 && st <= 4096) { *rows = r; *strip = st; found = true; }
    std::fclose(fp);
    return found;
}

void tune_cache_put(const std::string& sig, int rows, int strip, double ms) {
    const std::string path = tune_cache_path();
    if (path.empty()) return;
    const size_t slash = path.find_last_of('/');
    if (slash != std::string::npos && slash > 0) {
        std::string dir = path.substr(0, slash);
        for (size_t p = 1; p <= dir.size(); ++p)                  // mkdir -p
            if (p == dir.size() || dir[p] == '/') mkdir(dir.substr(0, p).c_str(), 0755);
    }
    FILE* fp = std::fopen(path.c_str(), "a");
    if (!fp) return;
    std::fprintf(fp, "%s %d %d %.6f\n", sig.c_str(), rows, strip, ms);
    std::fclose(fp);
}

}  // namespace

extern "C" {

int starmap_batch_create(const starmap_config* cfgs, int count, starmap_batch_t** out) {
    if (!out) return bfail(nullptr, STARMAP_E_ARG, "out is NULL");
    *out = nullptr;
    if (!cfgs || count < 1) return bfail(nullptr, STARMAP_E_ARG, "a batch needs at least one configuration");
    const int k = cfgs[0].kernel;
    if (k == STARMAP_KERNEL_TILED_TALL || k == STARMAP_KERNEL_TILED_SHORT)
        return batch_build(cfgs, count, k == STARMAP_KERNEL_TILED_SHORT ? 1 : 0, out);
    const std::string sig = batch_signature(cfgs, count);
    int rows = 0, strip = 0;
    if (tune_cache_get(sig, &rows, &strip)) {
        starmap_batch_t* b = nullptr;
        int rc = batch_build(cfgs, count, rows == 5 ? 1 : 0, &b);
        if (rc == STARMAP_OK && strip != b->strip) rc = batch_replan(b, strip);
        if (rc != STARMAP_OK) {
            if (b) g_batch_create_error = b->err;
            starmap_batch_destroy(b);
            return rc;
        }
        b->from_cache = true;
        *out = b;
        return STARMAP_OK;
    }
    // Autotuner: build the batch with each tile height and, for each, plan
    // the work units with strips of 96, 192 and 384 stages; time four steps
    // of every candidate (one step call: nine passes with the merged
    // schedule) on the freshly created (all-zero, source-free, vacuum) state
    // -- which the steps leave zero -- keep the fastest and cache the choice.
    static const int kStrips[3] = {192, 96, 384};
    starmap_batch_t* cand[2] = {nullptr, nullptr};
    double ms[2] = {-1.0, -1.0};
    int best_strip[2] = {192, 192};
    int rc = STARMAP_OK;
    for (int v = 0; v < 2 && rc == STARMAP_OK; ++v) {
        rc = batch_build(cfgs, count, v, &cand[v]);
        for (int s = 0; s < 3 && rc == STARMAP_OK; ++s) {
            if (cand[v]->strip != kStrips[s]) rc = batch_replan(cand[v], kStrips[s]);
            double t = 0.0;
            if (rc == STARMAP_OK) rc = batch_time(cand[v], 4, &t);
            if (rc == STARMAP_OK && (ms[v] < 0 || t < ms[v])) { ms[v] = t; best_strip[v] = kStrips[s]; }
        }
        if (rc == STARMAP_OK && cand[v]->strip != best_strip[v]) rc = batch_replan(cand[v], best_strip[v]);
        if (rc != STARMAP_OK && cand[v]) g_batch_create_error = cand[v]->err;
    }
    if (rc != STARMAP_OK) {
        for (starmap_batch_t* c : cand) starmap_batch_destroy(c);
        return rc;
    }
    const int best = ms[1] < ms[0] ? 1 : 0;
    starmap_batch_destroy(cand[1 - best]);
    starmap_batch_t* b = cand[best];
    b->tuned_ms[0] = ms[0];
    b->tuned_ms[1] = ms[1];
    batch_reset_clock(b);
    tune_cache_put(sig, best ? 5 : 10, b->strip, ms[best]);
    *out = b;
    return STARMAP_OK;
}

int starmap_batch_tuning(const starmap_batch_t* b, int* tile_rows, int* strip_stages, int* from_cache) {
    if (!b) return STARMAP_E_ARG;
    if (tile_rows) *tile_rows = b->variant ? 5 : 10;
    if (strip_stages) *strip_stages = b->strip;
    if (from_cache) *from_cache = b->from_cache ? 1 : 0;
    return STARMAP_OK;
}

int starmap_batch_tile_rows(const starmap_batch_t* b, double* ms_tall, double* ms_short) {
    if (!b) return 0;
    if (ms_tall) *ms_tall = b->tuned_ms[0];
    if (ms_short) *ms_short = b->tuned_ms[1];
    return b->variant ? 5 : 10;
}

void starmap_batch_destroy(starmap_batch_t* b) {
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    batch_release(b);
    delete b;
}

const char* starmap_batch_last_error(const starmap_batch_t* b) { return b ? b->err.c_str() : g_batch_create_error.c_str(); }

int starmap_batch_count(const starmap_batch_t* b) { return b ? (int)b->inst.size() : 0; }

starmap_t* starmap_batch_instance(starmap_batch_t* b, int i) {
    if (!b || i < 0 || i >= (int)b->inst.size()) return nullptr;
    return b->inst[i];
}

long starmap_batch_launches(const starmap_batch_t* b, long nsteps) {
    if (!b || nsteps <= 0) return 0;
    // one launch per pass
    return b->schedule == STARMAP_SCHEDULE_MERGED ? 2 * nsteps + 1 : 3 * nsteps;
}

int starmap_batch_step(starmap_batch_t* b, long nsteps) {
    if (!b) return STARMAP_E_ARG;
    if (nsteps < 0) return bfail(b, STARMAP_E_ARG, "negative step count");
    if (nsteps == 0) return STARMAP_OK;
    for (starmap_t* h : b->inst)
        if (h->ghosts_dirty) {
            int rc = fill_ghosts_all<float>(h);
            if (rc) return bfail(b, rc, h->err);
        }
    int rc = batch_sync_params(b);
    if (rc) return rc;
    cudaGraphExec_t exec = nullptr;
    for (auto& gx : b->graphs)
        if (gx.first == nsteps) exec = gx.second;
    if (!exec) {
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return bfail(b, STARMAP_E_CUDA, std::string("begin capture: ") + cudaGetErrorString(e));
        rc = batch_issue(b, nsteps);
        e = cudaStreamEndCapture(b->stream, &graph);
        if (rc || e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return bfail(b, STARMAP_E_CUDA, std::string("capture of the batch step: ") + cudaGetErrorString(e));
        }
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return bfail(b, STARMAP_E_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
        if (b->graphs.size() >= 8) {
            cudaGraphExecDestroy(b->graphs.front().second);
            b->graphs.erase(b->graphs.begin());
        }
        b->graphs.push_back({nsteps, exec});
    }
    cudaError_t e = cudaGraphLaunch(exec, b->stream);
    if (e != cudaSuccess) return bfail(b, STARMAP_E_CUDA, std::string("graph launch: ") + cudaGetErrorString(e));
    for (starmap_t* h : b->inst) {
        h->t += nsteps * h->dt;
        h->steps += nsteps;
        h->have_output = false;
    }
    return STARMAP_OK;
}

int starmap_batch_sync(starmap_batch_t* b) {
    if (!b) return STARMAP_E_ARG;
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bfail(b, STARMAP_E_CUDA, std::string("sync: ") + cudaGetErrorString(e));
    for (size_t i = 0; i < b->inst.size(); ++i) {
        int rc = poll_kernel(b->inst[i]);
        if (rc) return bfail(b, rc, "instance " + std::to_string(i) + ": " + b->inst[i]->err);
    }
    return STARMAP_OK;
}

}  // extern "C"
