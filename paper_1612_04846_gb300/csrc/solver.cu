// Host side of the C ABI: plan setup (scaling, multigrid hierarchy, Chebyshev smoother tables,
// device workspaces) and the solve drivers (FP64 multi-shift PCG, and FP32 PCG inside FP64
// iterative refinement), followed by the FP64 weighted sum u = sum_j c_j v_j (eq. (Rgeneral)).
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <atomic>
#include <mutex>
#include <shared_mutex>
#include <thread>
#include <vector>

#include "../../include/bura.h"
#include "guard.h"
#include "kernels.cuh"
#include "tma.cuh"

namespace bura {
std::shared_mutex& capture_guard() {
    static std::shared_mutex m;
    return m;
}
}  // namespace bura

using namespace bura;

namespace {

struct HostLevel {
    int n[3];            // nx, ny, nz (nz = 1 in 2D)
    long long N;
    double h[3];         // mesh sizes (h[2] unused in 2D)
    double w[3];         // constant weights 1/(h^2 Lambda)
    std::vector<double> a[3];  // unscaled face coefficients (variable coefficients only)
    double amax;         // max diagonal of the scaled level operator
    double lmin;         // lower bound on lambda_min of the scaled level operator
    // sparse operator (plan dim 0): the scaled matrix's rows (all entries, diagonal included), its diagonal
    // and absolute row sums; lmin = 0 when no lower bound on lambda_min is known
    std::vector<int> rowptr, col;
    std::vector<double> val, diag, rowsum;
};

// Kernel types for launch counting and per-kernel timing (fine level only).
enum KId { K_SPMV, K_CGUPD, K_CHEB0, K_CHEB, K_RESTRICT, K_PRE2, K_PROLONG, K_COARSE, K_DOT, K_BCAST, K_NORM,
           K_RES64, K_CAST, K_CORR64, K_WSUM, K_GATHER, K_CLUSTER, K_PRE2R, K_PROCHEB, K_RESDF, K_CASTDF, K_REDFIN,
           K_POST2, K_RESID, K_PUPD, K_FDIAG, K_POST2S, K_RESV, K_RES, K_RESOUT, K_NK };
// [kernel][f32][coarser level]
const char* const kNames[K_NK][2][2] = {
    {{"spmv_p_f64", "spmv_p_f64@coarse"}, {"spmv_p_f32", "spmv_p_f32@coarse"}},
    {{"cg_update_f64", "cg_update_f64@coarse"}, {"cg_update_f32", "cg_update_f32@coarse"}},
    {{"cheb_zero_f64", "cheb_zero_f64@coarse"}, {"cheb_zero_f32", "cheb_zero_f32@coarse"}},
    {{"cheb_step_f64", "cheb_step_f64@coarse"}, {"cheb_step_f32", "cheb_step_f32@coarse"}},
    {{"restrict_res_f64", "restrict_res_f64@coarse"}, {"restrict_res_f32", "restrict_res_f32@coarse"}},
    {{"cheb_pre2_f64", "cheb_pre2_f64@coarse"}, {"cheb_pre2_f32", "cheb_pre2_f32@coarse"}},
    {{"prolong_add_f64", "prolong_add_f64@coarse"}, {"prolong_add_f32", "prolong_add_f32@coarse"}},
    {{"coarse_cycle_f64", "coarse_cycle_f64@coarse"}, {"coarse_cycle_f32", "coarse_cycle_f32@coarse"}},
    {{"dot_f64", "dot_f64@coarse"}, {"dot_f32", "dot_f32@coarse"}},
    {{"broadcast_f64", "broadcast_f64"}, {"broadcast_f32", "broadcast_f32"}},
    {{"norm2", "norm2"}, {"norm2", "norm2"}},
    {{"residual64", "residual64"}, {"residual64", "residual64"}},
    {{"cast_scaled", "cast_scaled"}, {"cast_scaled", "cast_scaled"}},
    {{"correct64", "correct64"}, {"correct64", "correct64"}},
    {{"weighted_sum", "weighted_sum"}, {"weighted_sum", "weighted_sum"}},
    {{"gather_systems", "gather_systems"}, {"gather_systems", "gather_systems"}},
    {{"coarse_cluster_f64", "coarse_cluster_f64@coarse"}, {"coarse_cluster_f32", "coarse_cluster_f32@coarse"}},
    {{"pre2_restrict_f64", "pre2_restrict_f64@coarse"}, {"pre2_restrict_f32", "pre2_restrict_f32@coarse"}},
    {{"prolong_cheb_f64", "prolong_cheb_f64@coarse"}, {"prolong_cheb_f32", "prolong_cheb_f32@coarse"}},
    {{"update_residual_df", "update_residual_df"}, {"update_residual_df", "update_residual_df"}},
    {{"cast_f_df", "cast_f_df"}, {"cast_f_df", "cast_f_df"}},
    {{"red_finish_f64", "red_finish_f64"}, {"red_finish_f32", "red_finish_f32"}},
    {{"post2_f64", "post2_f64@coarse"}, {"post2_f32", "post2_f32@coarse"}},
    {{"residual_f64", "residual_f64@coarse"}, {"residual_f32", "residual_f32@coarse"}},
    {{"p_update_f64", "p_update_f64"}, {"p_update_f32", "p_update_f32"}},
    {{"coarse_fdiag_f64", "coarse_fdiag_f64@coarse"}, {"coarse_fdiag_f32", "coarse_fdiag_f32@coarse"}},
    {{"post2_strip_f64", "post2_strip_f64@coarse"}, {"post2_strip_f32", "post2_strip_f32@coarse"}},
    {{"coarse_resident_f64", "coarse_resident_f64@coarse"}, {"coarse_resident_f32", "coarse_resident_f32@coarse"}},
    {{"resident_solve_f64", "resident_solve_f64"}, {"resident_solve_f32", "resident_solve_f32"}},
    {{"resident_output", "resident_output"}, {"resident_output", "resident_output"}}};
constexpr int kSlots = K_NK * 4;

struct Tracer {
    bool on = false;
    std::vector<cudaEvent_t> ev;  // 2 per timed launch
    struct Rec { int slot; double bytes; };
    std::vector<Rec> pending;
    long long n[K_NK * 4] = {0};
    double ms[K_NK * 4] = {0};
    double bytes[K_NK * 4] = {0};
    long long launches = 0;  // every launch of the current solve
};
constexpr size_t kMaxTimed = 16384;
constexpr int kCoarseResident = 100;  // a coarse kind that only AUTO chooses

template <class T>
struct Work {
    int Kp = 0, W = 0, C = 0;
    std::vector<Launch> g;
    std::vector<Lev> L;
    Lev Lop{};                    // level 0 as the CG operator (FP32/FP64 faces even when L[0]'s are bf16)
    T *x = nullptr, *r = nullptr, *pa = nullptr, *pb = nullptr, *q = nullptr;
    std::vector<T*> b, xa, xb, dd;
    std::vector<T*> c1, c2;       // [level] -> deg rows of Kp coefficients, in the kernels' precision
    std::vector<int> deg;
    int lc = -1;                  // first level run by the coarse kernel (-1: none, grid kernels to the end)
    int coarse_kind = 0;          // BURA_COARSE_CLUSTER, BURA_COARSE_CTA, BURA_COARSE_FDIAG or kCoarseResident
    ResArgs rv{};                 // kCoarseResident: the V-cycle from level lc down (resident.cu)
    int csize = 0;                // CTAs of the cluster (cluster kind)
    int le = -1;                  // level solved exactly with dense inverses inside that kernel (-1: none)
    T* minv = nullptr;            // the inverses, [row][col][Kp]
    size_t coarse_smem = 0;       // shared-memory bytes of the single-CTA kind's vectors
    size_t minv_smem = 0;         // bytes of one chunk's inverses staged in its shared memory (0: not staged)
    Launch gc{};                  // launch shape of the coarse kernel (one CTA)
    // fast-diagonalization coarse solve (BURA_COARSE_FDIAG): level lc solved exactly, one cluster of fd_G
    // CTAs per system; sine bases and 1-D eigenvalues of level lc in the kernels' precision
    T *fd_img = nullptr, *fd_lx = nullptr, *fd_ly = nullptr;
    int fd_G = 0;
    size_t fd_smem = 0;
    T* dsh = nullptr;  // the shifts d_j (KMAXP entries) in the kernels' precision
    Scal* scal = nullptr;
    // TMA-staged sweeps (FP32, 2-D) of the levels above the coarse kernel's: tensor maps of the level's vectors, with a
    // halo box (stencil inputs) and a plain box
    struct TmaLev {
        bool on = false;
        TmaGeo geo{};
        struct Ent { int box; const void* buf; CUtensorMap map; };
        std::vector<Ent> maps;
        bool var = false;  // variable coefficients: the packed weights, boxed as each sweep's stencil input
        CUtensorMap w_rsrc, w_halo2, w_halo;
        const CUtensorMap* find(int box, const void* buf) const {
            for (const auto& e : maps)
                if (e.box == box && e.buf == buf) return &e.map;
            return nullptr;
        }
    };
    std::vector<TmaLev> tma;
    // TMA-staged sweeps of the large 3-D levels (FP32): geometry and the maps of the level's vectors by box
    struct S3Lev {
        bool on = false;
        Sweep3Lev geo{};
        std::vector<typename TmaLev::Ent> maps;
        const CUtensorMap* at(int box, const void* buf) const {  // null: no such map, and the sweep that asks reports it
            for (const auto& e : maps)
                if (e.box == box && e.buf == buf) return &e.map;
            return nullptr;
        }
    };
    std::vector<S3Lev> s3;
    bool ready = false;
    // the PCG loop captured once as a graph with a device-side conditional WHILE node
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphConditionalHandle cond = 0;
    long long body_launches = 0;
};

int ceil_to(int v, int m) { return (v + m - 1) / m * m; }

// Degree of the Chebyshev polynomial preconditioner of a sparse operator (one level, no coarse grids).
constexpr int kCsrDegree = 8;

// FP32 -> bfloat16 bits, rounded to nearest even (finite values).
unsigned short to_bf16(float f) {
    unsigned u;
    std::memcpy(&u, &f, 4);
    u += 0x7fffu + ((u >> 16) & 1u);
    return (unsigned short)(u >> 16);
}
float from_bf16(unsigned short h) {
    const unsigned u = (unsigned)h << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return f;
}


}  // namespace

struct bura_plan {
    int dev = 0, nsm = 152;
    bool cluster_ok = false;  // the device launches thread-block clusters
    int dim = 2;
    bool var = false;
    int k = 0, K = 0;
    double alpha = 0, E = 0, Lambda = 0, lambda_lo = 0;
    bool shifts_only = false;  // set up by bura_setup_shifts: caller-given weights and shifts, no alpha
    double out_scale = 1.0;    // factor of the weights in the output sum (Lambda^-alpha with opt.unscaled)
    long long wait_cycles = 0; // budget of the TMA ring waits (0: the kernels' default)
    std::vector<double> c, d;
    const int* csr_rowptr = nullptr;  // device copies of the sparse operator's row offsets and columns
    const int* csr_col = nullptr;
    bura_options opt{};
    std::vector<HostLevel> hl;
    Work<double> w64;
    Work<float> w32;
    double* v64 = nullptr;   // FP64 solutions (refinement accumulator), Kp64 layout
    double* r64 = nullptr;   // FP64 residuals, Kp64 layout
    double* cdev = nullptr;  // c_j, Kp64 entries
    double* partial = nullptr;
    unsigned int* tickets = nullptr;
    unsigned int* red_nblk = nullptr;  // grid size of a deferred reduction's producer (after the tickets)
    double* red_out = nullptr;  // [KMAXP]
    // mixed path: refinement accumulator v_j as FP32 pairs hi + lo (Kp32 layout, two ping-pong copies),
    // f as a pair, and the pair form of the level-0 operator's and the weighted sum's coefficients
    float* vh[2] = {nullptr, nullptr};
    float* vl[2] = {nullptr, nullptr};
    int vcur = 0;
    float* fh = nullptr;
    float* fl = nullptr;
    DfOpHost dfop;
    float* cwh = nullptr;  // c_j hi / lo, KMAXP entries
    float* cwl = nullptr;
    double* scale = nullptr;    // [KMAXP] refinement scales (FP64 refinement)
    double* invscale = nullptr;
    Scal* scal_outer = nullptr;
    Scal* hscal = nullptr;      // pinned host mirror
    double* hbuf = nullptr;     // pinned host scratch [4*KMAXP]
    double* fdev = nullptr;     // host-solve staging
    double* udev = nullptr;
    std::vector<void*> allocs;
    size_t dbytes = 0;           // sum of the allocations
    cudaEvent_t done = nullptr;  // recorded after the last kernel of every solve (bura_retarget waits on it)
    // device-driven solve: the whole FP64 or mixed/FP64-refinement solve as one graph (controller kernels
    // take the host's decisions); its outcome is copied to the pinned mirror hstate at the end of the solve
    OuterCfg* ocfg = nullptr;
    OuterState* ostate = nullptr;
    OuterState* hstate = nullptr;
    cudaGraph_t sgraph = nullptr;
    cudaGraphExec_t sexec = nullptr;
    long long s_fixed = 0, s_outer = 0, s_body = 0;  // launches: once, per refinement step, per PCG iteration
    cudaError_t sweep_err = cudaSuccess;  // a staged 3-D sweep that was not launched
    bool res_on = false;         // the whole solve is one launch (resident.cu)
    ResArgs res{};
    bool pending = false;        // a device-driven solve's outcome has not been read into st yet
    int last_status = BURA_OK;   // status of the last solve whose outcome was read
    bura_stats st{};
    Tracer tr;
    cudaStream_t cap = nullptr;  // private stream used only to capture the PCG loop graphs
};

namespace {

thread_local cudaError_t g_last = cudaSuccess;
// Stream capture of a PCG graph is invalidated by a device-synchronising call of another thread (a
// device-wide synchronisation, a free, a synchronous copy or memset).  The library's own such calls
// (plan setup, retargeting, destruction, the allocation-free entry point's first symbol lookup) hold
// this guard shared; a capture holds it exclusively.
std::shared_mutex& g_capture_guard = bura::capture_guard();
#define CK(call)                                  \
    do {                                          \
        cudaError_t e_ = (call);                  \
        if (e_ != cudaSuccess) {                  \
            g_last = e_;                          \
            return BURA_ECUDA;                    \
        }                                         \
    } while (0)
#define CKL() CK(cudaGetLastError())
#define CK_VOID(call)                             \
    do {                                          \
        cudaError_t e_ = (call);                  \
        if (e_ != cudaSuccess) g_last = e_;       \
    } while (0)

template <class P>
int dalloc(bura_plan* p, P** ptr, size_t bytes) {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
    if (e != cudaSuccess) {
        g_last = e;
        return e == cudaErrorMemoryAllocation ? BURA_ENOMEM : BURA_ECUDA;
    }
    p->allocs.push_back(q);
    p->dbytes += bytes > 0 ? bytes : 16;
    *ptr = reinterpret_cast<P*>(q);
    return BURA_OK;
}
#define CA(expr)                      \
    do {                              \
        int rc_ = (expr);             \
        if (rc_ != BURA_OK) return rc_; \
    } while (0)

// Count a launch; when profiling, bracket it by events (finest-level and coarser-level launches are
// accumulated separately).
template <class F>
void traced(bura_plan* p, int kid, bool is_f32, bool fine, double bytes, cudaStream_t s, F&& launch) {
    Tracer& t = p->tr;
    ++t.launches;
    const int slot = (kid * 2 + (is_f32 ? 1 : 0)) * 2 + (fine ? 0 : 1);
    const bool rec = t.on && t.pending.size() < kMaxTimed;
    if (rec) cudaEventRecord(t.ev[2 * t.pending.size()], s);
    launch();
    if (rec) {
        cudaEventRecord(t.ev[2 * t.pending.size() + 1], s);
        t.pending.push_back({slot, bytes});
    }
}

// The per-iteration reductions of the PCG (r.z, p.q, r.r) are deferred: the producing grid only stores
// block partials and a one-CTA k_red_finish sums them next on the stream, so the large grids end
// without fences, tickets or a serial last block.
Red deferred(const bura_plan* p, Red r) {
    r.defer = 1;
    r.nblk = p->red_nblk;
    return r;
}

void red_finish(bura_plan* p, const Red& r, int Kp, bool is_f32, cudaStream_t s) {
    traced(p, K_REDFIN, is_f32, true, 0.0, s, [&] { launch_red_finish(r, Kp, is_f32, s); });
}

// Fold the timed launches of the finished solve into the per-kernel totals (stream must be idle).
void collect_trace(bura_plan* p) {
    Tracer& t = p->tr;
    for (size_t i = 0; i < t.pending.size(); ++i) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, t.ev[2 * i], t.ev[2 * i + 1]) == cudaSuccess) {
            t.n[t.pending[i].slot] += 1;
            t.ms[t.pending[i].slot] += ms;
            t.bytes[t.pending[i].slot] += t.pending[i].bytes;
        }
    }
    t.pending.clear();
}

Launch make_launch(int Kp, int W, long long N, int nsm, int block_points, int blocks_per_sm) {
    Launch g;
    g.Kp = Kp;
    g.C = Kp / W;
    g.PPB = block_points > 0 ? std::max(block_points, W) : (g.C <= 4 ? 64 : 32);  // (a reduction takes a thread per system)
    if (g.PPB * g.C > kSweepThreads) g.PPB = kSweepThreads / g.C;
    long long tiles = (N + g.PPB - 1) / g.PPB;
    long long cap = (long long)nsm * (blocks_per_sm > 0 ? blocks_per_sm : 8);
    g.blocks = (int)std::max(1LL, std::min(tiles, cap));
    return g;
}

double harm(double a, double b) { return 2.0 / (1.0 / a + 1.0 / b); }

// Coarse face coefficients: harmonic mean of the two fine faces in series on the line through
// the coarse node (coarse node I sits on fine node 2I+1).
void coarsen_faces(const HostLevel& f, HostLevel& c, int dim) {
    const int fx = f.n[0], fy = f.n[1];
    const int cx = c.n[0], cy = c.n[1], cz = c.n[2];
    auto fidx = [&](int axis, int l, int j, int i) -> size_t {  // face arrays of the fine level
        if (axis == 0) return ((size_t)l * fy + j) * (fx + 1) + i;
        if (axis == 1) return ((size_t)l * (fy + 1) + j) * fx + i;
        return ((size_t)l * fy + j) * fx + i;
    };
    c.a[0].assign((size_t)cz * cy * (cx + 1), 0.0);
    c.a[1].assign((size_t)cz * (cy + 1) * cx, 0.0);
    if (dim == 3) c.a[2].assign((size_t)(cz + 1) * cy * cx, 0.0);
    for (int L = 0; L < cz; ++L) {
        const int l = dim == 3 ? 2 * L + 1 : 0;
        for (int J = 0; J < cy; ++J)
            for (int I = 0; I <= cx; ++I)
                c.a[0][((size_t)L * cy + J) * (cx + 1) + I] =
                    harm(f.a[0][fidx(0, l, 2 * J + 1, 2 * I)], f.a[0][fidx(0, l, 2 * J + 1, 2 * I + 1)]);
        for (int J = 0; J <= cy; ++J)
            for (int I = 0; I < cx; ++I)
                c.a[1][((size_t)L * (cy + 1) + J) * cx + I] =
                    harm(f.a[1][fidx(1, l, 2 * J, 2 * I + 1)], f.a[1][fidx(1, l, 2 * J + 1, 2 * I + 1)]);
    }
    if (dim == 3)
        for (int L = 0; L <= cz; ++L)
            for (int J = 0; J < cy; ++J)
                for (int I = 0; I < cx; ++I)
                    c.a[2][((size_t)L * cy + J) * cx + I] =
                        harm(f.a[2][fidx(2, 2 * L, 2 * J + 1, 2 * I + 1)], f.a[2][fidx(2, 2 * L + 1, 2 * J + 1, 2 * I + 1)]);
}

// Max diagonal of the scaled operator and min face value of a level (variable coefficients).
void level_bounds(HostLevel& h, int dim, bool var, double Lambda) {
    const int nx = h.n[0], ny = h.n[1], nz = h.n[2];
    double lc = 0.0;  // lambda_min of the constant-coefficient scaled operator on this level
    for (int a = 0; a < dim; ++a) {
        const double s = std::sin(M_PI * h.h[a] / 2.0);
        lc += 4.0 * h.w[a] * s * s;
    }
    if (!var) {
        h.amax = 2.0 * (h.w[0] + h.w[1] + (dim == 3 ? h.w[2] : 0.0));
        h.lmin = lc;
        return;
    }
    (void)Lambda;
    double amax = 0.0, amin = 1e300;
    for (int a = 0; a < dim; ++a)
        for (double v : h.a[a]) amin = std::min(amin, v);
    for (int l = 0; l < nz; ++l)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                double dg = (h.a[0][((size_t)l * ny + j) * (nx + 1) + i] + h.a[0][((size_t)l * ny + j) * (nx + 1) + i + 1]) * h.w[0];
                dg += (h.a[1][((size_t)l * (ny + 1) + j) * nx + i] + h.a[1][((size_t)l * (ny + 1) + j + 1) * nx + i]) * h.w[1];
                if (dim == 3)
                    dg += (h.a[2][((size_t)l * ny + j) * nx + i] + h.a[2][((size_t)(l + 1) * ny + j) * nx + i]) * h.w[2];
                amax = std::max(amax, dg);
            }
    h.amax = amax;
    h.lmin = amin * lc;
}

// Gershgorin bound max_P sum_Q |Atilde_PQ| of the unscaled fine operator.
double gershgorin(const HostLevel& h, int dim, bool var) {
    const int nx = h.n[0], ny = h.n[1], nz = h.n[2];
    if (!var) {
        double s = 0.0;
        for (int a = 0; a < dim; ++a) s += (2.0 + std::min(h.n[a] - 1, 2)) / (h.h[a] * h.h[a]);
        return s;
    }
    const double ix = 1.0 / (h.h[0] * h.h[0]), iy = 1.0 / (h.h[1] * h.h[1]), iz = dim == 3 ? 1.0 / (h.h[2] * h.h[2]) : 0.0;
    double best = 0.0;
    for (int l = 0; l < nz; ++l)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                const double xm = h.a[0][((size_t)l * ny + j) * (nx + 1) + i] * ix;
                const double xp = h.a[0][((size_t)l * ny + j) * (nx + 1) + i + 1] * ix;
                const double ym = h.a[1][((size_t)l * (ny + 1) + j) * nx + i] * iy;
                const double yp = h.a[1][((size_t)l * (ny + 1) + j + 1) * nx + i] * iy;
                double zm = 0, zp = 0;
                if (dim == 3) {
                    zm = h.a[2][((size_t)l * ny + j) * nx + i] * iz;
                    zp = h.a[2][((size_t)(l + 1) * ny + j) * nx + i] * iz;
                }
                double s = xm + xp + ym + yp + zm + zp;  // diagonal
                if (i > 0) s += xm;
                if (i < nx - 1) s += xp;
                if (j > 0) s += ym;
                if (j < ny - 1) s += yp;
                if (dim == 3) {
                    if (l > 0) s += zm;
                    if (l < nz - 1) s += zp;
                }
                best = std::max(best, s);
            }
    return best;
}

// Chebyshev step coefficients for one level and every system: eigenvalue interval [lo_s, hi_s] of
// Dinv (A - d_s I); c1/c2 per step as in the three-term Chebyshev semi-iteration.
void cheb_tables(const HostLevel& h, bool var, const std::vector<double>& d, int K, int Kp, int deg, double ratio,
                 bool coarse_solve, std::vector<std::vector<double>>& C1, std::vector<std::vector<double>>& C2) {
    C1.assign(deg, std::vector<double>(Kp, 0.0));
    C2.assign(deg, std::vector<double>(Kp, 0.0));
    for (int s = 0; s < K; ++s) {
        const double mds = -d[s];  // >= 0
        double hi = 1.0 + h.amax / (h.amax + mds);
        if (!h.rowsum.empty()) {  // sparse operator: Gershgorin bound of Dinv (A - dI) row by row
            hi = 0.0;
            for (size_t i = 0; i < h.rowsum.size(); ++i) hi = std::max(hi, (h.rowsum[i] + mds) / (h.diag[i] + mds));
        }
        // a sparse operator's polynomial preconditioner takes [hi / ratio, hi] even with a lambda_min bound:
        // lambda_min / max(diag) underestimates the bottom of Dinv A by the spread of the diagonal (a
        // coefficient jump), and the wide interval converges far more slowly (353 against 12 CG iterations
        // on the P1 half-cube matrix with mu = 1e-3, 15^3)
        double lo;
        if (coarse_solve && h.rowsum.empty()) lo = (h.lmin + mds) / (h.amax + mds);
        else lo = std::max(hi / ratio, mds / (h.amax + mds));
        lo = std::min(lo, hi * (1.0 - 1e-12));
        const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo);
        const double sigma = theta / delta;
        const double dinv = var ? 1.0 : 1.0 / (h.amax + mds);  // constant diagonal: amax == diag
        double rho = 1.0 / sigma;
        for (int m = 0; m < deg; ++m) {
            if (m == 0) {
                C1[m][s] = 0.0;
                C2[m][s] = dinv / theta;
            } else {
                const double rn = 1.0 / (2.0 * sigma - rho);
                C1[m][s] = rn * rho;
                C2[m][s] = dinv * 2.0 * rn / delta;
                rho = rn;
            }
        }
    }
}

// Dense (A_l - d_j I)^{-1} of a tiny level for every system j, laid out [row][col][Kp] (zero for the
// padding systems); Gauss-Jordan elimination with partial pivoting in FP64.
void dense_inverses(const HostLevel& h, int dim, bool var, const std::vector<double>& d, int K, int Kp,
                    std::vector<double>& out) {
    const int nx = h.n[0], ny = h.n[1], nz = h.n[2];
    const int n = (int)h.N;
    std::vector<double> A((size_t)n * n, 0.0);
    auto id = [&](int i, int j, int l) { return (l * ny + j) * nx + i; };
    for (int l = 0; l < nz; ++l)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                const int P = id(i, j, l);
                double w[6];
                if (var) {
                    w[0] = h.a[0][((size_t)l * ny + j) * (nx + 1) + i] * h.w[0];
                    w[1] = h.a[0][((size_t)l * ny + j) * (nx + 1) + i + 1] * h.w[0];
                    w[2] = h.a[1][((size_t)l * (ny + 1) + j) * nx + i] * h.w[1];
                    w[3] = h.a[1][((size_t)l * (ny + 1) + j + 1) * nx + i] * h.w[1];
                    w[4] = dim == 3 ? h.a[2][((size_t)l * ny + j) * nx + i] * h.w[2] : 0.0;
                    w[5] = dim == 3 ? h.a[2][((size_t)(l + 1) * ny + j) * nx + i] * h.w[2] : 0.0;
                } else {
                    w[0] = w[1] = h.w[0];
                    w[2] = w[3] = h.w[1];
                    w[4] = w[5] = dim == 3 ? h.w[2] : 0.0;
                }
                A[(size_t)P * n + P] = w[0] + w[1] + w[2] + w[3] + w[4] + w[5];
                if (i > 0) A[(size_t)P * n + id(i - 1, j, l)] = -w[0];
                if (i < nx - 1) A[(size_t)P * n + id(i + 1, j, l)] = -w[1];
                if (j > 0) A[(size_t)P * n + id(i, j - 1, l)] = -w[2];
                if (j < ny - 1) A[(size_t)P * n + id(i, j + 1, l)] = -w[3];
                if (l > 0) A[(size_t)P * n + id(i, j, l - 1)] = -w[4];
                if (l < nz - 1) A[(size_t)P * n + id(i, j, l + 1)] = -w[5];
            }
    out.assign((size_t)n * n * Kp, 0.0);
    std::vector<double> M((size_t)n * 2 * n);
    for (int s = 0; s < K; ++s) {
        for (int r = 0; r < n; ++r)
            for (int c = 0; c < 2 * n; ++c)
                M[(size_t)r * 2 * n + c] = c < n ? A[(size_t)r * n + c] - (r == c ? d[s] : 0.0) : (c - n == r ? 1.0 : 0.0);
        for (int c = 0; c < n; ++c) {
            int pr = c;
            for (int r = c + 1; r < n; ++r)
                if (std::fabs(M[(size_t)r * 2 * n + c]) > std::fabs(M[(size_t)pr * 2 * n + c])) pr = r;
            if (pr != c)
                for (int k2 = 0; k2 < 2 * n; ++k2) std::swap(M[(size_t)pr * 2 * n + k2], M[(size_t)c * 2 * n + k2]);
            const double piv = M[(size_t)c * 2 * n + c];
            for (int k2 = 0; k2 < 2 * n; ++k2) M[(size_t)c * 2 * n + k2] /= piv;
            for (int r = 0; r < n; ++r) {
                if (r == c) continue;
                const double fct = M[(size_t)r * 2 * n + c];
                if (fct == 0.0) continue;
                for (int k2 = 0; k2 < 2 * n; ++k2) M[(size_t)r * 2 * n + k2] -= fct * M[(size_t)c * 2 * n + k2];
            }
        }
        for (int r = 0; r < n; ++r)
            for (int c = 0; c < n; ++c) out[((size_t)r * n + c) * Kp + s] = M[(size_t)r * 2 * n + n + c];
    }
}

int coarse_degree_auto(const HostLevel& h, double d0) {
    if (h.N == 1) return 1;
    const double mds = -d0;
    const double hi = 1.0 + h.amax / (h.amax + mds);
    const double lo = (h.lmin + mds) / (h.amax + mds);
    const double sigma = (hi + lo) / (hi - lo);
    int m = (int)std::ceil(std::acosh(20.0) / std::acosh(sigma));
    return std::max(2, std::min(m, 400));
}

// The packed weights of a 2-D variable-coefficient level for the TMA-staged sweeps (from the stored ones, on the device:
// packing on the host made a 511^2 plan's setup 0.8 ms longer, an eighth of it), and their maps.
int pack_weights2(bura_plan* p, const Lev& L, CUtensorMap& rsrc, CUtensorMap& halo2, CUtensorMap& halo) {
    float* d = nullptr;
    CA(dalloc(p, &d, (size_t)(L.nx + 1) * (L.ny + 1) * 4 * sizeof(float)));
    CK(tma_pack_weights(L, d, nullptr));
    CK(tma_encode_weights(&rsrc, d, L.nx, L.ny, TB_RSRC));
    CK(tma_encode_weights(&halo2, d, L.nx, L.ny, TB_HALO2));
    CK(tma_encode_weights(&halo, d, L.nx, L.ny, TB_HALO));
    return BURA_OK;
}

// Tensor maps for the TMA-staged sweeps: FP32, 2-D, every level that the grid kernels would run (not the coarse kernel's).
template <class T>
int build_tma(bura_plan* p, Work<T>& w) {
    const int nlev = (int)p->hl.size();
    w.tma.assign(nlev, typename Work<T>::TmaLev());
    if (sizeof(T) != 4 || p->dim != 2 || p->opt.sweeps == BURA_SWEEP_GRID || !tma_supported(w.Kp)) return BURA_OK;
    // variable coefficients: the fused sweeps only (degree 2, FP32 weights); other options keep the grid sweeps
    if (p->var && (p->opt.smoother_degree != 2 || p->opt.post_smooth_split != 0 || p->opt.smoother_bf16)) return BURA_OK;
    bool any = false;
    for (int l = 0; l < nlev; ++l) {
        if (w.lc >= 0 && l >= w.lc) break;
        const bool has_coarse = l + 1 < nlev;
        if (p->var && !has_coarse) break;
        TmaGeo g = tma_geo(w.L[l], has_coarse ? &w.L[l + 1] : nullptr, w.Kp);
        if (p->opt.tma_stages > 0) g.stages = p->opt.tma_stages;
        // every grid level: even with fewer tiles than SMs the fused 3-launch V-cycle step beats the
        // 5 grid launches of a small level (measured on GB300: 255^2 ... 63^2 levels of a 1023^2 solve)
        auto& t = w.tma[l];
        t.geo = g;
        const void* bl = l == 0 ? (const void*)w.r : (const void*)w.b[l];
        struct Want { int box; const void* buf; int lev; };
        std::vector<Want> want = {{TB_HALO, bl, l}, {TB_HALO, w.xa[l], l}, {TB_HALO, w.xb[l], l},
                                  {TB_PLAIN, bl, l}, {TB_PLAIN, w.dd[l], l}, {TB_HALO2, w.xa[l], l}};
        if (l == 0) {
            want.push_back({TB_HALO, w.pa, 0});
            want.push_back({TB_HALO, w.pb, 0});
            // the CG update's pointwise tiles
            want.push_back({TB_PLAIN, w.x, 0});
            want.push_back({TB_PLAIN, w.pa, 0});
            want.push_back({TB_PLAIN, w.pb, 0});
            want.push_back({TB_PLAIN, w.q, 0});
        }
        if (has_coarse) {  // the fused transfers: b with a two-point halo, coarse results for prolongation
            want.push_back({TB_RSRC, bl, l});
            want.push_back({TB_CPRO, w.xa[l + 1], l + 1});
            want.push_back({TB_CPRO, w.xb[l + 1], l + 1});
            want.push_back({TB_CPRO2, w.xa[l + 1], l + 1});
            want.push_back({TB_CPRO2, w.xb[l + 1], l + 1});
        }
        bool ok = true;
        for (const Want& e : want) {
            typename Work<T>::TmaLev::Ent ent;
            ent.box = e.box;
            ent.buf = e.buf;
            if (tma_encode(&ent.map, reinterpret_cast<const float*>(e.buf), w.Kp, w.L[e.lev].nx, w.L[e.lev].ny,
                           e.box) != cudaSuccess) {
                ok = false;  // a map the driver does not accept: this level and the coarser ones stay on grid kernels
                break;
            }
            t.maps.push_back(ent);
        }
        if (!ok) {
            t = typename Work<T>::TmaLev();
            break;
        }
        if (p->var) CA(pack_weights2(p, w.L[l], t.w_rsrc, t.w_halo2, t.w_halo));
        t.var = p->var;
        t.on = true;
        any = true;
    }
    if (any) CK(tma_prepare(w.Kp));
    return BURA_OK;
}

// Chebyshev interval [lmax / ratio, lmax] of the smoother: the option, or (0 = auto) the upper quarter of
// the spectrum in 2-D and the upper eighth in 3-D, where full coarsening leaves a wider high-frequency
// band (the eigenvalues of D^-1 A over the modes that are oscillatory in at least one direction reach
// down to 1/dim of their maximum for the 7-point operator).
double smoother_ratio(const bura_plan* p) {
    if (p->opt.smoother_ratio > 0) return p->opt.smoother_ratio;
    if (p->dim == 0) return 30.0;  // sparse operator without a lambda_min bound: the polynomial preconditioner
    return p->dim == 3 ? 8.0 : 4.0;
}

// The fast-diagonalization tables of level lc (independent of the shifts): for each axis the orthonormal
// sine basis S_ik = sqrt(2/(n+1)) sin(pi (i+1)(k+1)/(n+1)) and the eigenvalues w (2 - 2 cos(pi (k+1)/(n+1)))
// = 4 w sin^2(pi (k+1) / (2 (n+1))) of w tridiag(-1, 2, -1), in FP64, rounded to T.
template <class T>
void sine_axis(const HostLevel& h, int a, std::vector<double>& S, std::vector<T>& lam) {
    const int n = h.n[a];
    const double pi = 3.14159265358979323846;
    const double sc = std::sqrt(2.0 / (n + 1));
    // sin of every angle pi m / (n+1) once, m = (i+1)(k+1) reduced modulo 2 (n+1): n^2 sines an axis, taken for the coarse
    // solve and again for the one-launch solve, were 0.1 ms of a 63^2 plan's 0.59
    const int period = 2 * (n + 1);
    std::vector<double> sine(period);
    for (int m = 0; m < period; ++m) sine[m] = sc * std::sin(pi * (double)m / (n + 1));
    S.resize((size_t)n * n);
    for (int i = 0; i < n; ++i)
        for (int k = 0, m = i + 1; k < n; ++k) {
            S[(size_t)i * n + k] = sine[m];
            m += i + 1;
            if (m >= period) m -= period;
        }
    lam.resize(n);
    for (int k = 0; k < n; ++k) {
        const double sk = std::sin(pi * (k + 1) / (2.0 * (n + 1)));
        lam[k] = (T)(4.0 * h.w[a] * sk * sk);
    }
}

template <class T>
int upload_fdiag(bura_plan* p, Work<T>& w) {
    const HostLevel& h = p->hl[w.lc];
    std::vector<double> S[2];
    T** dst_l[2] = {&w.fd_lx, &w.fd_ly};
    for (int a = 0; a < 2; ++a) {
        const int n = h.n[a];
        std::vector<T> lam;
        sine_axis<T>(h, a, S[a], lam);
        CA(dalloc(p, dst_l[a], (size_t)n * sizeof(T)));
        CK(cudaMemcpy(*dst_l[a], lam.data(), lam.size() * sizeof(T), cudaMemcpyHostToDevice));
    }
    std::vector<T> img;
    fdiag_image<T>(h.n[0], h.n[1], S[0].data(), S[1].data(), img);
    CA(dalloc(p, &w.fd_img, img.size() * sizeof(T)));
    CK(cudaMemcpy(w.fd_img, img.data(), img.size() * sizeof(T), cudaMemcpyHostToDevice));
    return BURA_OK;
}

// The shift-dependent tables of a work set, written into its existing buffers: per level the Chebyshev
// coefficients c1, c2 (deg x Kp), the shifts, and the dense inverses of the exact level.  Their sizes
// do not depend on the shifts (the coarsest degree depends on d_0 = 0 only), so a plan can be moved
// to another alpha without reallocating and without recapturing its PCG graph, whose kernels read
// these buffers.
template <class T>
int upload_tables(bura_plan* p, Work<T>& w) {
    const int nlev = (int)p->hl.size();
    for (int l = 0; l < (int)w.c1.size(); ++l) {
        if (!w.c1[l]) continue;
        const HostLevel& h = p->hl[l];
        const bool coarsest = (l == nlev - 1);
        const int deg = w.deg[l];
        std::vector<std::vector<double>> C1, C2;
        cheb_tables(h, p->var, p->d, p->K, w.Kp, deg, smoother_ratio(p), coarsest, C1, C2);
        if (coarsest && h.N == 1) {  // exact solve of the 1x1 system: x = b / (diag - d)
            for (int s = 0; s < p->K; ++s) C2[0][s] = p->var ? 1.0 : 1.0 / (h.amax - p->d[s]);
        }
        std::vector<T> t1((size_t)deg * w.Kp), t2((size_t)deg * w.Kp);
        for (int m = 0; m < deg; ++m)
            for (int s = 0; s < w.Kp; ++s) {
                t1[(size_t)m * w.Kp + s] = (T)C1[m][s];
                t2[(size_t)m * w.Kp + s] = (T)C2[m][s];
            }
        CK(cudaMemcpy(w.c1[l], t1.data(), t1.size() * sizeof(T), cudaMemcpyHostToDevice));
        CK(cudaMemcpy(w.c2[l], t2.data(), t2.size() * sizeof(T), cudaMemcpyHostToDevice));
    }
    std::vector<T> dsht(KMAXP, T(0));
    for (int s = 0; s < p->K; ++s) dsht[s] = (T)p->d[s];
    CK(cudaMemcpy(w.dsh, dsht.data(), KMAXP * sizeof(T), cudaMemcpyHostToDevice));
    if (w.minv) {
        std::vector<double> inv;
        dense_inverses(p->hl[w.le], p->dim, p->var, p->d, p->K, w.Kp, inv);
        const std::vector<T> tv(inv.begin(), inv.end());
        CK(cudaMemcpy(w.minv, tv.data(), tv.size() * sizeof(T), cudaMemcpyHostToDevice));
    }
    return BURA_OK;
}

// Face weights a / (h^2 Lambda) of a variable-coefficient level and its diagonal (the sum of a point's
// six stored weights, in FP64, rounded to T), as T or as bf16.
template <class T>
int upload_faces(bura_plan* p, const HostLevel& h, Lev& L, bool bf16) {
    const int nx = h.n[0], ny = h.n[1], nz = h.n[2];
    std::vector<double> stored[3];
    for (int a = 0; a < p->dim; ++a) {
        const size_t n = h.a[a].size();
        stored[a].resize(n);
        void* dptr = nullptr;
        if (bf16) {
            std::vector<unsigned short> v(n);
            for (size_t i = 0; i < n; ++i) {
                v[i] = to_bf16((float)(h.a[a][i] * h.w[a]));
                stored[a][i] = from_bf16(v[i]);
            }
            CA(dalloc(p, &dptr, n * sizeof(unsigned short)));
            CK(cudaMemcpy(dptr, v.data(), n * sizeof(unsigned short), cudaMemcpyHostToDevice));
        } else {
            std::vector<T> v(n);
            for (size_t i = 0; i < n; ++i) {
                v[i] = (T)(h.a[a][i] * h.w[a]);
                stored[a][i] = (double)v[i];
            }
            CA(dalloc(p, &dptr, n * sizeof(T)));
            CK(cudaMemcpy(dptr, v.data(), n * sizeof(T), cudaMemcpyHostToDevice));
        }
        if (a == 0) L.fx = dptr;
        else if (a == 1) L.fy = dptr;
        else L.fz = dptr;
    }
    std::vector<T> dg((size_t)h.N);
    for (int l = 0; l < nz; ++l)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                double s = stored[0][((size_t)l * ny + j) * (nx + 1) + i] + stored[0][((size_t)l * ny + j) * (nx + 1) + i + 1];
                s += stored[1][((size_t)l * (ny + 1) + j) * nx + i] + stored[1][((size_t)l * (ny + 1) + j + 1) * nx + i];
                if (p->dim == 3)
                    s += stored[2][((size_t)l * ny + j) * nx + i] + stored[2][((size_t)(l + 1) * ny + j) * nx + i];
                dg[((size_t)l * ny + j) * nx + i] = (T)s;
            }
    T* dptr = nullptr;
    CA(dalloc(p, &dptr, dg.size() * sizeof(T)));
    CK(cudaMemcpy(dptr, dg.data(), dg.size() * sizeof(T), cudaMemcpyHostToDevice));
    L.dg = dptr;
    L.cbf16 = bf16 ? 1 : 0;
    return BURA_OK;
}

// The packed weights of a variable-coefficient level for the staged 3-D sweeps: a float4 per point of the grid extended
// by one point along each axis (the faces below the point along x, y and z, and the diagonal summed from the stored
// weights as upload_faces does; zero where a face or a point does not exist), and its maps.
int upload_packed(bura_plan* p, const HostLevel& h, Sweep3Lev& g) {
    const int nx = h.n[0], ny = h.n[1], nz = h.n[2];
    std::vector<float> v((size_t)(nx + 1) * (ny + 1) * (nz + 1) * 4, 0.f);
    for (int l = 0; l <= nz; ++l)
        for (int j = 0; j <= ny; ++j) {
            float* o = &v[((size_t)l * (ny + 1) + j) * (nx + 1) * 4];
            const double* ax = h.a[0].data() + ((size_t)l * ny + j) * (nx + 1);  // read where the face exists only
            const double* ay = h.a[1].data() + ((size_t)l * (ny + 1) + j) * nx;
            const double* az = h.a[2].data() + ((size_t)l * ny + j) * nx;
            const size_t up = (size_t)ny * nx;
            for (int i = 0; i <= nx; ++i, o += 4) {
                const bool in = i < nx && j < ny && l < nz;
                if (j < ny && l < nz) o[0] = (float)(ax[i] * h.w[0]);
                if (i < nx && l < nz) o[1] = (float)(ay[i] * h.w[1]);
                if (i < nx && j < ny) o[2] = (float)(az[i] * h.w[2]);
                if (in) {
                    double s = (double)o[0] + (double)(float)(ax[i + 1] * h.w[0]);
                    s += (double)o[1] + (double)(float)(ay[i + nx] * h.w[1]);
                    s += (double)o[2] + (double)(float)(az[i + up] * h.w[2]);
                    o[3] = (float)s;
                }
            }
        }
    float* d = nullptr;
    CA(dalloc(p, &d, v.size() * sizeof(float)));
    CK(cudaMemcpy(d, v.data(), v.size() * sizeof(float), cudaMemcpyHostToDevice));
    for (int q = 0; q < 2; ++q) {
        int bx = 0, by = 0;
        sweep3_box(q ? S3B_RHALO : S3B_HALO, &bx, &by);
        CK(tma_encode3(q ? &g.wr : &g.w, d, (long long)(nx + 1) * 2, ny + 1, nz + 1, bx * 2, by));
    }
    return BURA_OK;
}

// Whether level l of an FP32 work set runs the staged 3-D sweeps (kSweep3MinN points along x, half that along the other
// axes: below, an item's fill of its ring costs more than the sweep saves), and its maps.  The buffers exist.  Plans that ask
// for the grid sweeps keep them.
template <class T>
int build_sweep3(bura_plan* p, Work<T>& w, int l) {
    const int nlev = (int)p->hl.size();
    const HostLevel& h = p->hl[l];
    auto& t = w.s3[l];
    if (sizeof(T) != 4 || p->dim != 3 || p->opt.sweeps == BURA_SWEEP_GRID || (p->var && p->opt.smoother_bf16) || w.Kp > 16 || l + 1 >= nlev || w.deg[l] < 2 ||
        h.n[0] < kSweep3MinN || std::min(h.n[1], h.n[2]) < kSweep3MinN / 2)
        return BURA_OK;
    const HostLevel& hc = p->hl[l + 1];
    Sweep3Lev& g = t.geo;
    g.nx = h.n[0]; g.ny = h.n[1]; g.nz = h.n[2];
    g.ncx = hc.n[0]; g.ncy = hc.n[1]; g.ncz = hc.n[2];
    g.Kp = w.Kp;
    g.nsm = p->nsm;
    g.var = p->var;
    g.wx = (float)h.w[0]; g.wy = (float)h.w[1]; g.wz = (float)h.w[2];
    const void* bl = l == 0 ? (const void*)w.r : (const void*)w.b[l];
    struct Want { int box; const void* buf; int lev; };
    std::vector<Want> want = {{S3B_HALO, bl, l}, {S3B_TILE, bl, l}, {S3B_RTILE, bl, l}, {S3B_TILE, w.dd[l], l},
                              {S3B_COARSE, w.xa[l + 1], l + 1}, {S3B_COARSE, w.xb[l + 1], l + 1}};
    for (const void* x : {(const void*)w.xa[l], (const void*)w.xb[l]}) {
        want.push_back({S3B_HALO, x, l});
        want.push_back({S3B_RHALO, x, l});
    }
    if (l == 0) {
        want.push_back({S3B_HALO, w.pa, 0});
        want.push_back({S3B_HALO, w.pb, 0});
    }
    for (const Want& e : want) {
        typename Work<T>::TmaLev::Ent ent;
        ent.box = e.box;
        ent.buf = e.buf;
        int bx = 0, by = 0;
        sweep3_box(e.box, &bx, &by);
        const HostLevel& q = p->hl[e.lev];
        if (tma_encode3(&ent.map, e.buf, (long long)q.n[0] * w.Kp / 2, q.n[1], q.n[2], bx * w.Kp / 2, by) != cudaSuccess) {
            t = typename Work<T>::S3Lev();
            return BURA_OK;  // a map the driver does not accept: the grid sweeps
        }
        t.maps.push_back(ent);
    }
    if (p->var) CA(upload_packed(p, h, g));
    CK(sweep3_prepare(w.Kp, p->var));
    t.on = true;
    return BURA_OK;
}

// The arguments of the resident kernels (resident.cu) for the 2-D hierarchy from level l0 down: geometry, tables,
// coefficients, and for constant ones the image of the exact level's sine bases.  False in *fits where the hierarchy has
// no such form: it has to reach a level of at most 63 points per axis (constant coefficients, solved by fast
// diagonalization) or, below a level of at most 31, one of at most kExactPoints points (dense inverses).
int resident_args(bura_plan* p, Work<float>& w, int l0, bool vonly, ResArgs& a, bool* fits) {
    *fits = false;
    const int nlev = (int)p->hl.size();
    auto size = [&](int l) { return std::max(p->hl[l].n[0], p->hl[l].n[1]); };
    int le = p->var ? l0 + 1 : l0;
    while (le < nlev && size(le) > (p->var ? 31 : kFdiagMaxN<float>)) ++le;
    if (le >= nlev) return BURA_OK;
    int ld = le;
    if (p->var) {
        while (ld < nlev && p->hl[ld].N > kExactPoints) ++ld;
        if (ld >= nlev || p->hl[l0].N <= kExactPoints || ld != w.le || !w.minv) return BURA_OK;
    }
    if (ld - l0 >= kResMaxLevels) return BURA_OK;
    a.var = p->var;
    a.vonly = vonly;
    a.le = le - l0;
    a.ld = ld - l0;
    a.ne = p->hl[le].n[1];
    a.Kp = w.Kp;
    a.N = (size_t)p->hl[l0].N;
    a.wx = p->hl[l0].w[0];
    a.wy = p->hl[l0].w[1];
    for (int l = l0; l <= ld; ++l) {
        ResLevel& L = a.lev[l - l0];
        L.nx = p->hl[l].n[0];
        L.ny = p->hl[l].n[1];
        L.wx = (float)p->hl[l].w[0];
        L.wy = (float)p->hl[l].w[1];
        L.c1 = w.c1[l];
        L.c2 = w.c2[l];
        L.fx = reinterpret_cast<const float*>(w.L[l].fx);
        L.fy = reinterpret_cast<const float*>(w.L[l].fy);
        L.dg = reinterpret_cast<const float*>(w.L[l].dg);
    }
    a.minv = w.minv;
    a.dsh = w.dsh;
    if (!resident_plan(a, p->K)) return BURA_OK;
    if (!p->var) {
        const int nx = p->hl[le].n[0], ny = p->hl[le].n[1];
        std::vector<double> S[2];
        std::vector<float> lam[2];
        for (int q = 0; q < 2; ++q) sine_axis<float>(p->hl[le], q, S[q], lam[q]);
        std::vector<float> img(res_image_floats(nx, ny));
        res_image(nx, ny, S[0].data(), S[1].data(), lam[0].data(), lam[1].data(), img.data());
        float* di = nullptr;
        CA(dalloc(p, &di, img.size() * sizeof(float)));
        CK(cudaMemcpy(di, img.data(), img.size() * sizeof(float), cudaMemcpyHostToDevice));
        a.img = di;
    }
    *fits = true;
    return BURA_OK;
}

// Plans that the resident kernels serve: 2-D FP32 work of a mixed plan with the default smoothing.  Options that ask for
// particular sweeps or coarse kernels keep them.
bool resident_options(const bura_plan* p) {
    const bura_options& o = p->opt;
    return p->dim == 2 && p->cluster_ok && o.precision == BURA_PREC_MIXED && o.sweeps == BURA_SWEEP_AUTO && !o.smoother_bf16;
}

// The one-launch solve of a small plan with FP64 refinement, whose slabs fit the shared memory of a cluster.  It keeps
// its solutions in the plan's v64 buffer, system by system.
int build_resident(bura_plan* p) {
    const bura_options& o = p->opt;
    Work<float>& w = p->w32;
    if (!resident_options(p) || o.refine != BURA_REFINE_FP64 || o.post_smooth_split != 0 || o.tma_stages != 0 ||
        o.max_outer > kResMaxOuter)
        return BURA_OK;
    if (!(o.coarse_kernel == BURA_COARSE_AUTO || (o.coarse_kernel == BURA_COARSE_FDIAG && !p->var))) return BURA_OK;
    const bool smooths = p->var || std::max(p->hl[0].n[0], p->hl[0].n[1]) > kFdiagMaxN<float>;
    if (smooths && o.smoother_degree != 2) return BURA_OK;
    ResArgs& a = p->res;
    CA(resident_args(p, w, 0, false, a, &p->res_on));
    if (!p->res_on) return BURA_OK;
    if (a.le > 0 && !p->var) tma_dot_blocks(tma_geo(w.L[0], &w.L[1], w.Kp), p->nsm, &a.blk_pq, &a.blk_rz);
    CA(dalloc(p, &a.out, (size_t)p->K * sizeof(ResOut)));
    a.cfg = p->ocfg;
    a.x = nullptr;
    if (a.o_x < 0)
        CA(dalloc(p, &a.x, (size_t)p->K * p->hl[0].n[1] * ((p->hl[0].n[0] + 1) / 2 * 2) * sizeof(float)));
    a.v = p->v64;
    const Lev& L64 = p->w64.L[0];
    a.fx64 = reinterpret_cast<const double*>(L64.fx);
    a.fy64 = reinterpret_cast<const double*>(L64.fy);
    a.dg64 = reinterpret_cast<const double*>(L64.dg);
    return BURA_OK;
}

// The lower part of a larger plan's V-cycle as one launch of a cluster per system: the first level (below the finest)
// that lets every system's cluster be resident at once.  Sets w.lc and the kind on success.
template <class T>
int build_resident_cycle(bura_plan* p, Work<T>& w) {
    if constexpr (sizeof(T) == 4) {
        if (!resident_options(p) || p->opt.coarse_kernel != BURA_COARSE_AUTO || p->opt.smoother_degree != 2) return BURA_OK;
        const int nlev = (int)p->hl.size();
        // (a grid that is the exact level itself is one exact solve)
        if (!p->var && std::max(p->hl[0].n[0], p->hl[0].n[1]) <= kFdiagMaxN<float>) return BURA_OK;
        for (int l = 1; l < nlev; ++l) {
            if (std::max(p->hl[l].n[0], p->hl[l].n[1]) > kResCycleMaxN) continue;
            bool fits = false;
            CA(resident_args(p, w, l, true, w.rv, &fits));
            if (!fits) continue;
            w.coarse_kind = kCoarseResident;
            w.lc = l;
            w.rv.vb = w.b[l];
            w.rv.vx = w.xa[l];
            w.rv.cfg = nullptr;  // (p->ocfg, once it exists)
            // the padding systems of the result are never written
            CK(cudaMemset(w.xa[l], 0, (size_t)p->hl[l].N * w.Kp * sizeof(T)));
            return BURA_OK;
        }
    }
    return BURA_OK;
}

// full = false: only what the mixed path's FP64 refinement and bura_apply_shifted use of the FP64 work
// (level-0 launch shape, geometry and face coefficients, the shifts); no hierarchy, no PCG buffers.
template <class T>
int build_work(bura_plan* p, Work<T>& w, bool full = true) {
    const int nlev = full ? (int)p->hl.size() : 1;
    w.W = VecT<T>::W;
    w.Kp = ceil_to(p->K, w.W);
    w.C = w.Kp / w.W;
    w.g.resize(nlev);
    w.L.resize(nlev);
    w.b.assign(nlev, nullptr);
    w.xa.assign(nlev, nullptr);
    w.xb.assign(nlev, nullptr);
    w.dd.assign(nlev, nullptr);
    w.c1.assign(nlev, nullptr);
    w.c2.assign(nlev, nullptr);
    w.deg.resize(nlev);
    w.s3.assign(nlev, typename Work<T>::S3Lev());
    if (full) {  // the level vectors, the smoothing degrees and the CG's vectors
        for (int l = 0; l < nlev; ++l) {
            const HostLevel& h = p->hl[l];
            const size_t vb = (size_t)h.N * w.Kp * sizeof(T);
            CA(dalloc(p, &w.b[l], vb));  // level 0 uses the CG residual instead; kept for the coarse CTA
            CA(dalloc(p, &w.xa[l], vb));
            CA(dalloc(p, &w.xb[l], vb));
            CA(dalloc(p, &w.dd[l], vb));
            int deg = p->opt.smoother_degree;
            if (l == nlev - 1)
                deg = h.N == 1 ? 1 : (p->opt.coarse_degree > 0 ? p->opt.coarse_degree
                                      : p->dim == 0 ? kCsrDegree : coarse_degree_auto(h, p->d[0]));
            w.deg[l] = deg;
            // the Chebyshev tables (deg x Kp each) depend on the shifts: filled by upload_tables
            CA(dalloc(p, &w.c1[l], (size_t)deg * w.Kp * sizeof(T)));
            CA(dalloc(p, &w.c2[l], (size_t)deg * w.Kp * sizeof(T)));
        }
        const size_t vb0 = (size_t)p->hl[0].N * w.Kp * sizeof(T);
        for (T** q : {&w.x, &w.r, &w.pa, &w.pb, &w.q}) CA(dalloc(p, q, vb0));
        CA(dalloc(p, &w.dsh, KMAXP * sizeof(T)));
    }
    for (int l = 0; l < nlev; ++l) {
        const HostLevel& h = p->hl[l];
        if (full) CA(build_sweep3(p, w, l));
        // a row segment of the 3-D column sweeps is a CTA's points: no more of them than a short row has
        int points = p->opt.block_points;
        if (points == 0 && l > 0 && p->dim == 3 && h.n[0] <= 32) points = h.n[0] <= 16 ? 16 : 32;
        w.g[l] = make_launch(w.Kp, w.W, h.N, p->nsm, points, p->opt.blocks_per_sm);
        Lev& L = w.L[l];
        L.nx = h.n[0];
        L.ny = h.n[1];
        L.nz = h.n[2];
        L.N = h.N;
        L.plane = (long long)h.n[0] * h.n[1];
        L.wx = h.w[0];
        L.wy = h.w[1];
        L.wz = p->dim == 3 ? h.w[2] : 0.0;
        L.wxf = (float)L.wx;
        L.wyf = (float)L.wy;
        L.wzf = (float)L.wz;
        L.fx = L.fy = L.fz = L.dg = nullptr;
        L.cbf16 = 0;
        L.rowptr = L.col = nullptr;
        L.val = nullptr;
        if (p->dim == 0) {  // the sparse operator: values and diagonal in T, shared row offsets and columns
            std::vector<T> v(h.val.size()), dg(h.diag.size());
            for (size_t i = 0; i < v.size(); ++i) v[i] = (T)h.val[i];
            for (size_t i = 0; i < dg.size(); ++i) dg[i] = (T)h.diag[i];
            T* dv = nullptr;
            T* dd = nullptr;
            CA(dalloc(p, &dv, v.size() * sizeof(T)));
            CA(dalloc(p, &dd, dg.size() * sizeof(T)));
            CK(cudaMemcpy(dv, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
            CK(cudaMemcpy(dd, dg.data(), dg.size() * sizeof(T), cudaMemcpyHostToDevice));
            L.rowptr = p->csr_rowptr;
            L.col = p->csr_col;
            L.val = dv;
            L.dg = dd;
            w.Lop = L;
        } else if (p->var) {
            // the CG operator's faces in T; the V-cycle's in bf16 when asked (FP32 path), with the diagonal
            // summed from the stored values so each level operator is the M-matrix of its stored faces
            const bool bf = sizeof(T) == 4 && p->opt.smoother_bf16;
            if (!w.s3[l].on && (!bf || l == 0)) CA(upload_faces<T>(p, h, L, false));
            if (l == 0) w.Lop = L;
            if (bf) CA(upload_faces<T>(p, h, L, true));
        }
        if (l == 0 && !p->var) w.Lop = L;
        if (!full) break;
    }
    if (!full) {
        CA(dalloc(p, &w.dsh, KMAXP * sizeof(T)));
        CA(upload_tables<T>(p, w));
        return BURA_OK;  // w.ready stays false: this work never runs a PCG
    }
    // the first level with at most kExactPoints points is solved exactly (dense inverses); the levels
    // below it are never visited
    w.le = -1;
    for (int l = 0; l < nlev && p->dim != 0; ++l)
        if (p->hl[l].N <= kExactPoints) { w.le = l; break; }
    const int last = w.le >= 0 ? w.le : nlev - 1;
    w.lc = -1;
    w.coarse_smem = 0;
    w.coarse_kind = p->opt.coarse_kernel;
    // 2-D constant coefficients: the exact fast-diagonalization solve of a level of up to kFdiagMaxN
    // points per axis replaces that level and every coarser one.  Otherwise, as measured on GB300 (2-D
    // 1023^2, k = 7), the single CTA over shared memory beats the cluster, whose sweeps each pay an L2
    // round trip and a cluster barrier (about 3 us of fixed cost per sweep).
    if (p->var && p->dim == 2 && w.le >= 0) {  // dense inverses, whichever of the kernels below runs the coarse levels
        const size_t n = (size_t)p->hl[w.le].N;
        CA(dalloc(p, &w.minv, n * n * w.Kp * sizeof(T)));
    }
    CA(build_resident_cycle<T>(p, w));
    if (w.coarse_kind == BURA_COARSE_AUTO)
        w.coarse_kind = (p->dim == 2 && !p->var && p->cluster_ok) ? BURA_COARSE_FDIAG : BURA_COARSE_CTA;
    if (p->dim == 0) w.coarse_kind = BURA_COARSE_NONE;  // one level: the polynomial preconditioner alone
    if (w.coarse_kind == BURA_COARSE_FDIAG) {
        for (int l = 0; l < nlev; ++l)
            if (std::max(p->hl[l].n[0], p->hl[l].n[1]) <= kFdiagMaxN<T>) { w.lc = l; break; }
        if (w.lc >= 0) {
            const int nx = p->hl[w.lc].n[0], ny = p->hl[w.lc].n[1];
            CK(fdiag_prepare<T>(nx, ny, w.Kp, &w.fd_G, &w.fd_smem));
            CA(upload_fdiag<T>(p, w));
        }
    } else if (w.coarse_kind == BURA_COARSE_CLUSTER) {
        // the small levels (at most kClusterPoints points each, L2 resident) run in one thread-block cluster
        for (int l = 0; l <= last; ++l)
            if (p->hl[l].N <= kClusterPoints && last - l + 1 <= kMaxCoarseLevels) { w.lc = l; break; }
        if (w.lc >= 0) {
            const int want = p->opt.cluster_size > 0 ? p->opt.cluster_size : 16;
            CK(Ops<T>::cluster_prepare(p->dim, p->var, kClusterThreads, want, &w.csize));
            if (w.csize < 2) w.lc = -1;
        }
    } else if (w.coarse_kind == BURA_COARSE_CTA) {
        // the smallest levels run together in one CTA with all their vectors in shared memory
        for (int l = 0; l <= last; ++l) {
            size_t bytes = 0;
            // one CTA per 16-byte chunk: each holds its chunk's W values per point
            for (int m = l; m <= last; ++m) bytes += 4 * (((size_t)p->hl[m].N * w.W * sizeof(T) + 15) / 16 * 16);
            if (bytes <= kCoarseSmem && last - l + 1 <= kMaxCoarseLevels) {
                w.lc = l;
                w.coarse_smem = bytes;
                break;
            }
        }
    }
    if (w.lc < 0 || w.coarse_kind == BURA_COARSE_FDIAG || (w.coarse_kind == kCoarseResident && !p->var))
        w.le = -1;  // no dense solve
    if (w.le < 0) w.minv = nullptr;
    if (w.le >= 0 && !w.minv) {  // [row][col][Kp] dense inverses of the exact level, filled by upload_tables
        const size_t n = (size_t)p->hl[w.le].N;
        CA(dalloc(p, &w.minv, n * n * w.Kp * sizeof(T)));
    }
    w.gc.Kp = w.Kp;
    w.gc.C = w.C;
    w.gc.PPB = (w.coarse_kind == BURA_COARSE_CLUSTER ? kClusterThreads : kCoarseThreads) / w.C;
    w.gc.blocks = 1;
    // the single-CTA kind stages its chunk of the dense inverses in shared memory when they fit
    w.minv_smem = 0;
    if (w.lc >= 0 && w.le >= 0 && w.coarse_kind == BURA_COARSE_CTA) {
        const size_t mb = (size_t)p->hl[w.le].N * p->hl[w.le].N * w.W * sizeof(T);
        if (w.coarse_smem + kCoarseTables + KMAXP * sizeof(double) + mb <= kCoarseSmemMax) w.minv_smem = mb;
    }
    if (w.lc >= 0 && w.coarse_kind == BURA_COARSE_CTA)
        CK(Ops<T>::prepare_coarse(p->dim, p->var,
                                  w.coarse_smem + kCoarseTables + KMAXP * sizeof(double) + w.minv_smem));
    CA(upload_tables<T>(p, w));
    CA(dalloc(p, &w.scal, sizeof(Scal)));
    CK(cudaMemset(w.scal, 0, sizeof(Scal)));
    CA(build_tma(p, w));
    if (sizeof(T) == 4 && p->dim == 2 && !p->var && w.Kp <= 16) CK(strip_prepare(w.Kp));
    w.ready = true;
    return BURA_OK;
}

// Algorithmic bytes of `vec` multi-shift vectors of level l (K systems, not the padding) plus,
// for variable coefficients, the face coefficients a stencil kernel reads.
template <class T>
double vbytes(const bura_plan* p, int l, double vec, bool stencil) {
    const double N = (double)p->hl[l].N;
    double b = vec * N * p->K * sizeof(T);
    if (stencil && p->dim == 0) b += (double)p->hl[0].val.size() * (4 + sizeof(T)) + N * (4 + sizeof(T));
    else if (stencil && p->var) b += N * p->dim * sizeof(T);
    return b;
}

// The TMA kernels are FP32 only: these views are taken only when T is float (w.tma[l].on is never set
// for the FP64 work), where they are the identity.
template <class T>
ChebStepT<float> f32_step(ChebStepT<T> c) {
    return ChebStepT<float>{reinterpret_cast<const float*>(c.c1), reinterpret_cast<const float*>(c.c2)};
}
template <class T>
const float* f32_ptr(const T* q) { return reinterpret_cast<const float*>(q); }

template <class T>
ChebStepT<T> step_of(const Work<T>& w, int l, int m, bool with_c1 = true) {
    return ChebStepT<T>{with_c1 ? w.c1[l] + (size_t)m * w.Kp : nullptr, w.c2[l] + (size_t)m * w.Kp};
}

// 3-D grids, variable coefficients and sparse operators run the first pre-smoothing step and the CG
// direction update as their own pointwise sweeps: re-evaluating them at every stencil neighbour (as the
// fused kernels do) costs more there than the extra vector pass.
bool split_sweeps(const bura_plan* p) { return p->dim != 2 || p->var; }

// Whether level l of the FP64 work takes the sweeps of sweep64.cu: any 2-D constant-coefficient level above the coarse
// solver with degree-2 smoothing (511^2, k = 7: the whole solve 4.02 -> 2.22 ms).  Levels of at
// least kLean64Stored values store the residual and restrict it (255^2, k = 7: 18 us of kernels against 22 for the single
// sweep, 511^2: 45 against 54); smaller ones save a launch (127^2: 10 us against 17).
constexpr long long kLean64Stored = 300000;
template <class T>
bool lean64(const bura_plan* p, const Work<T>& w, int l) {
    return sizeof(T) == 8 && p->dim == 2 && !p->var && w.deg[l] == 2 && l + 1 < (int)p->hl.size() &&
           p->opt.sweeps == BURA_SWEEP_AUTO;
}

// Launch the shared-memory V-cycle over levels w.lc..nlev-1 for the right-hand side b (global), one
// CTA per 16-byte chunk of systems; the result of level lc is written to w.xa[lc].  Inside a CTA every
// level has b, xa, xb, dd of its chunk in shared memory; a level's pre-smoothing (zero step + deg-1
// steps) ends in xa when deg-1 is even and its post-smoothing toggles deg more times (the coarsest
// level has no post-smoothing).
template <class T>
T* coarse_part(bura_plan* p, Work<T>& w, const T* b, cudaStream_t s) {
    const int nlev = (int)p->hl.size();
    CoarseArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nlev = (w.le >= 0 ? w.le : nlev - 1) - w.lc + 1;
    a.exact = w.le >= 0 ? w.le - w.lc : -1;
    a.minv = w.minv;
    a.Kp = w.Kp;
    a.dsh = w.dsh;
    a.b_in = b;
    a.x_out = w.xa[w.lc];
    unsigned int off = 0;
    unsigned int cof = (unsigned int)w.coarse_smem;  // small tables follow the vectors
    a.dsh_ofs = cof;
    cof += KMAXP * sizeof(double);
    for (int i = 0; i < a.nlev; ++i) {
        const int l = w.lc + i;
        const unsigned int vb = (unsigned int)((((size_t)p->hl[l].N * w.W * sizeof(T)) + 15) / 16 * 16);
        CoarseLevel& c = a.lev[i];
        c.L = w.L[l];
        c.b = off;
        c.xa = off + vb;
        c.xb = off + 2 * vb;
        c.dd = off + 3 * vb;
        off += 4 * vb;
        const int deg = w.deg[l];
        const unsigned int pre = ((deg - 1) % 2 == 0) ? c.xa : c.xb;
        const unsigned int other = pre == c.xa ? c.xb : c.xa;
        if (i == a.exact) c.result = c.xa;  // the dense solve writes xa
        else c.result = (l == nlev - 1 || deg % 2 == 0) ? pre : other;
        c.c1 = w.c1[l];
        c.c2 = w.c2[l];
        c.deg = deg;
        const unsigned int tb = (unsigned int)(2 * deg * w.W * sizeof(T));
        if (tb <= 4096 && cof + tb <= w.coarse_smem + KMAXP * sizeof(double) + kCoarseTables) {
            c.cofs = cof;
            cof += tb;
        } else {
            c.cofs = kNoCopy;
        }
    }
    a.minv_ofs = kNoCopy;
    if (w.minv_smem > 0) {
        a.minv_ofs = (unsigned int)(w.coarse_smem + KMAXP * sizeof(double) + kCoarseTables);
        cof = a.minv_ofs + (unsigned int)w.minv_smem;
    }
    a.smem_bytes = cof;
    traced(p, K_COARSE, sizeof(T) == 4, w.lc == 0, 0.0, s,
           [&] { Ops<T>::coarse_cycle(w.gc, p->dim, p->var, a, s); });
    return w.xa[w.lc];
}

// Launch the clustered V-cycle over levels w.lc..(w.le or nlev-1) for the right-hand side b; every
// level keeps its vectors in its own global buffers (L2 resident).  Returns the buffer holding the
// result of level lc (predicted exactly as the kernel leaves it: a level's pre-smoothing ends in xa
// when deg-1 is even, its post-smoothing toggles deg more times, the coarsest level has no
// post-smoothing and the dense solve writes xa).
template <class T>
T* cluster_part(bura_plan* p, Work<T>& w, const T* b, cudaStream_t s) {
    const int nlev = (int)p->hl.size();
    ClusterArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nlev = (w.le >= 0 ? w.le : nlev - 1) - w.lc + 1;
    a.exact = w.le >= 0 ? w.le - w.lc : -1;
    a.minv = w.minv;
    a.Kp = w.Kp;
    a.dsh = w.dsh;
    for (int i = 0; i < a.nlev; ++i) {
        const int l = w.lc + i;
        ClusterLevel& c = a.lev[i];
        c.L = w.L[l];
        c.b = i == 0 ? const_cast<T*>(b) : w.b[l];
        c.xa = w.xa[l];
        c.xb = w.xb[l];
        c.dd = w.dd[l];
        const int deg = w.deg[l];
        T* pre = ((deg - 1) % 2 == 0) ? w.xa[l] : w.xb[l];
        T* other = pre == w.xa[l] ? w.xb[l] : w.xa[l];
        if (i == a.exact) c.result = w.xa[l];
        else c.result = (l == nlev - 1 || deg % 2 == 0) ? pre : other;
        c.c1 = w.c1[l];
        c.c2 = w.c2[l];
        c.deg = deg;
    }
    traced(p, K_CLUSTER, sizeof(T) == 4, w.lc == 0, 0.0, s,
           [&] { (void)Ops<T>::coarse_cluster(w.gc, w.csize, p->dim, p->var, a, s); });  // errors: cudaGetLastError
    return reinterpret_cast<T*>(const_cast<void*>(a.lev[0].result));
}

// The exact solve of level lc by fast diagonalization for the right-hand side b; the result is written
// to w.xa[lc].
template <class T>
T* fdiag_part(bura_plan* p, Work<T>& w, const T* b, cudaStream_t s) {
    const HostLevel& h = p->hl[w.lc];
    FdiagArgs a;
    a.nx = h.n[0];
    a.ny = h.n[1];
    a.Kp = w.Kp;
    a.b = b;
    a.x = w.xa[w.lc];
    a.simg = w.fd_img;
    a.lx = w.fd_lx;
    a.ly = w.fd_ly;
    a.dsh = w.dsh;
    a.scal = w.scal;
    traced(p, K_FDIAG, sizeof(T) == 4, w.lc == 0, vbytes<T>(p, w.lc, 2.0, false), s,
           [&] { (void)fdiag_launch<T>(a, w.fd_G, w.fd_smem, w.Kp, s); });  // errors: cudaGetLastError
    return w.xa[w.lc];
}

// The V-cycle from level lc down as one launch (its right-hand side is that level's b).
template <class T>
T* resident_part(bura_plan* p, Work<T>& w, cudaStream_t s) {
    w.rv.cfg = p->ocfg;
    w.rv.scal = w.scal;
    traced(p, K_RESV, sizeof(T) == 4, w.lc == 0, vbytes<T>(p, w.lc, 2.0, false), s,
           [&] { (void)launch_resident(w.rv, p->K, nullptr, 0.0, s); });  // errors: cudaGetLastError
    return w.xa[w.lc];
}

// Symmetric V-cycle on level l for rhs b; returns the buffer holding the result.  With rz_fused
// (level 0 only) the last smoothing step also forms r^T z and the CG beta of every system.
template <class T>
T* vcycle(bura_plan* p, Work<T>& w, int l, const T* b, bool rz_fused, cudaStream_t s) {
    const int dim = p->dim;
    const bool var = p->var;
    const Launch& g = w.g[l];
    const Lev& L = w.L[l];
    const int deg = w.deg[l];
    const bool f32 = sizeof(T) == 4;
    const bool fine = (l == 0);
    Red none{p->partial, p->tickets, w.scal, nullptr, RED_NONE, 0};
    const Red beta = deferred(p, Red{p->partial, p->tickets, w.scal, nullptr, RED_BETA, 0});
    if (l == w.lc) {  // the rest of the hierarchy in one kernel
        T* res = w.coarse_kind == BURA_COARSE_CLUSTER ? cluster_part(p, w, b, s)
                 : w.coarse_kind == BURA_COARSE_FDIAG ? fdiag_part(p, w, b, s)
                 : w.coarse_kind == kCoarseResident   ? resident_part(p, w, s)
                                                      : coarse_part(p, w, b, s);
        if (rz_fused) {
            traced(p, K_DOT, f32, fine, vbytes<T>(p, l, 2.0, false), s, [&] { Ops<T>::dot(g, L.N, b, res, beta, s); });
            red_finish(p, beta, w.Kp, f32, s);
        }
        return res;
    }
    T* A = w.xa[l];
    T* B = w.xb[l];
    T* D = w.dd[l];
    T* cur = A;
    T* oth = B;
    bool rz_done = false;
    const auto& tl = w.tma[l];
    const auto& s3l = w.s3[l];
    const bool s3 = s3l.on;
    auto note = [&](cudaError_t e) { if (e != cudaSuccess) p->sweep_err = e; };
    // one Chebyshev step, TMA-staged where the level has tensor maps
    auto cheb = [&](const T* xin, const T* din, T* xout, T* dout, ChebStepT<T> cs, const Red& red) {
        const CUtensorMap* mx = tl.on ? tl.find(TB_HALO, xin) : nullptr;
        const CUtensorMap* md = tl.on && din ? tl.find(TB_PLAIN, din) : nullptr;
        const CUtensorMap* mb = tl.on ? tl.find(TB_PLAIN, b) : nullptr;
        if (mx && mb && (md || !din))
            (void)tma_cheb_step(tl.geo, p->nsm, *mx, md, *mb, reinterpret_cast<float*>(xout),
                                reinterpret_cast<float*>(dout), f32_step(cs), f32_ptr(w.dsh), red, s);
        else if (s3)
            note(sweep3_step(s3l.geo, s3l.at(S3B_HALO, xin), din != nullptr, din ? s3l.at(S3B_TILE, din) : nullptr,
                             s3l.at(S3B_TILE, b), reinterpret_cast<float*>(xout), reinterpret_cast<float*>(dout), f32_step(cs),
                             f32_ptr(w.dsh), red, s));
        else
            Ops<T>::cheb_step(g, L, dim, var, xin, din, b, xout, dout, cs, w.dsh, red, s);
    };
    if constexpr (sizeof(T) == 8) {
        if (lean64(p, w, l)) {
            const Lev& Lc = w.L[l + 1];
            traced(p, K_PRE2, f32, fine, vbytes<T>(p, l, 2.0, false), s,
                   [&] { sweep64_pre2(L, w.Kp, p->nsm, b, A, step_of(w, l, 0), step_of(w, l, 1), w.dsh, none, s); });
            if ((long long)w.Kp * L.N >= kLean64Stored) {
                traced(p, K_RESID, f32, fine, vbytes<T>(p, l, 3.0, false), s,
                       [&] { sweep64_residual(L, w.Kp, p->nsm, A, b, D, w.dsh, none, s); });
                traced(p, K_RESTRICT, f32, fine, vbytes<T>(p, l, 1.0, false) + vbytes<T>(p, l + 1, 1.0, false), s,
                       [&] { Ops<T>::restrict_r(w.g[l + 1], L, Lc, dim, D, w.b[l + 1], s); });
            } else {
                traced(p, K_RESTRICT, f32, fine, vbytes<T>(p, l, 2.0, false) + vbytes<T>(p, l + 1, 1.0, false), s,
                       [&] { sweep64_restrict(L, Lc, w.Kp, p->nsm, A, b, w.b[l + 1], w.dsh, s); });
            }
            const T* ec = vcycle<T>(p, w, l + 1, w.b[l + 1], false, s);
            traced(p, K_PROLONG, f32, fine, vbytes<T>(p, l, 2.0, false) + vbytes<T>(p, l + 1, 1.0, false), s,
                   [&] { sweep64_prolong(L, Lc, w.Kp, p->nsm, ec, A, s); });
            traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 3.0, false), s, [&] {
                sweep64_post1(L, w.Kp, p->nsm, A, B, b, step_of(w, l, 0), w.dsh, none, s);
            });
            traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 4.0, false), s, [&] {
                sweep64_post2(L, w.Kp, p->nsm, A, B, b, step_of(w, l, 1), w.dsh, rz_fused ? beta : none, s);
            });
            if (rz_fused) red_finish(p, beta, w.Kp, f32, s);
            return A;
        }
    }
    // TMA-staged level with degree-2 smoothing: pre-smoothing fused with the restriction of its
    // residual, the coarse levels, the first post-smoothing step fused with the prolongation, the last
    // post-smoothing step (with r.z and beta at the finest level)
    const CUtensorMap* m_rsrc = tl.on && deg == 2 ? tl.find(TB_RSRC, b) : nullptr;
    const CUtensorMap* m_ca = tl.on ? tl.find(TB_CPRO, w.xa[l + 1 < (int)p->hl.size() ? l + 1 : l]) : nullptr;
    const CUtensorMap* m_cb = tl.on ? tl.find(TB_CPRO, w.xb[l + 1 < (int)p->hl.size() ? l + 1 : l]) : nullptr;
    const CUtensorMap* m_xa = tl.on ? tl.find(TB_HALO, A) : nullptr;
    const CUtensorMap* m_bp = tl.on ? tl.find(TB_PLAIN, b) : nullptr;
    if (m_rsrc && m_ca && m_cb && m_xa && m_bp) {
        traced(p, K_PRE2R, f32, fine, vbytes<T>(p, l, 2.0, tl.var) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
            (void)tma_pre2_restrict(tl.geo, p->nsm, *m_rsrc, tl.var ? &tl.w_rsrc : nullptr, reinterpret_cast<float*>(A),
                                    reinterpret_cast<float*>(w.b[l + 1]), f32_step(step_of(w, l, 0)),
                                    f32_step(step_of(w, l, 1)), f32_ptr(w.dsh), none, s);
        });
        T* ec = vcycle<T>(p, w, l + 1, w.b[l + 1], false, s);
        // prolongation and both post-smoothing steps in one sweep: x (= A) on a two-point halo, ec, b in;
        // the smoothed result out to B
        const int lc1 = l + 1 < (int)p->hl.size() ? l + 1 : l;
        const CUtensorMap* mec2 = ec == w.xa[lc1] ? tl.find(TB_CPRO2, w.xa[lc1])
                                : ec == w.xb[lc1] ? tl.find(TB_CPRO2, w.xb[lc1]) : nullptr;
        const CUtensorMap* m_xa2 = tl.find(TB_HALO2, A);
        const CUtensorMap* m_bh = tl.find(TB_HALO, b);
        // the same as y-marching strips (no recomputed halo rows, the vertical neighbours in registers),
        // option post_smooth_split = 2
        const int pss = p->opt.post_smooth_split;
        if (pss == 2 && l + 1 < (int)p->hl.size()) {
            const Red& red = rz_fused ? beta : none;
            const StripGeo sg = strip_geo(L.nx, L.ny, w.L[l + 1].nx, w.L[l + 1].ny, w.Kp, L.wxf, L.wyf, p->nsm);
            traced(p, K_POST2S, f32, fine, vbytes<T>(p, l, 3.0, false) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
                (void)launch_post2_strip(sg, p->nsm, f32_ptr(A), f32_ptr(ec), f32_ptr(b), reinterpret_cast<float*>(B),
                                         f32_step(step_of(w, l, 0, false)), f32_step(step_of(w, l, 1)),
                                         f32_ptr(w.dsh), red, s);
            });
            if (rz_fused) red_finish(p, beta, w.Kp, f32, s);
            return B;
        }
        if (pss == 0 && mec2 && m_xa2 && m_bh) {
            const Red& red = rz_fused ? beta : none;
            traced(p, K_POST2, f32, fine, vbytes<T>(p, l, 3.0, false) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
                (void)tma_post2(tl.geo, p->nsm, *m_xa2, *mec2, *m_bh, tl.var ? &tl.w_halo2 : nullptr, reinterpret_cast<float*>(B),
                                f32_step(step_of(w, l, 0, false)), f32_step(step_of(w, l, 1)), f32_ptr(w.dsh), red, s);
            });
            if (rz_fused) red_finish(p, beta, w.Kp, f32, s);
            return B;
        }
        const CUtensorMap* mec = ec == w.xa[l + 1] ? m_ca : ec == w.xb[l + 1] ? m_cb : nullptr;
        if (mec) {
            traced(p, K_PROCHEB, f32, fine, vbytes<T>(p, l, 4.0, false) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
                (void)tma_prolong_cheb(tl.geo, p->nsm, *m_xa, *mec, *m_bp, reinterpret_cast<float*>(B),
                                       reinterpret_cast<float*>(D), f32_step(step_of(w, l, 0, false)), f32_ptr(w.dsh),
                                       none, s);
            });
        } else {  // a coarse result outside the level's two buffers: unfused correction and first step
            traced(p, K_PROLONG, f32, fine, vbytes<T>(p, l, 2.0, false) + vbytes<T>(p, l + 1, 1.0, false), s,
                   [&] { Ops<T>::prolong_add(g, L, w.L[l + 1], dim, ec, A, s); });
            traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 4.0, true), s,
                   [&] { cheb(A, nullptr, B, D, step_of(w, l, 0, false), none); });
        }
        const Red& red = rz_fused ? beta : none;
        traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 4.0, true), s,
               [&] { cheb(B, D, A, nullptr, step_of(w, l, 1), red); });
        if (rz_fused) red_finish(p, beta, w.Kp, f32, s);
        return A;
    }
    // pre-smoothing from a zero initial guess; the first two Chebyshev steps share one sweep (or, with
    // split sweeps, the first step is a pointwise sweep and the second reads it as its previous direction)
    if (deg == 1) {
        traced(p, K_CHEB0, f32, fine, vbytes<T>(p, l, 2.0, var), s,
               [&] { Ops<T>::cheb_zero(g, L, dim, var, b, A, step_of(w, l, 0), w.dsh, s); });
    } else if (s3) {  // both steps from zero in one staged sweep
        traced(p, K_PRE2, f32, fine, vbytes<T>(p, l, deg > 2 ? 3.0 : 2.0, true), s, [&] {
            note(sweep3_pre(s3l.geo, s3l.at(S3B_HALO, b), reinterpret_cast<float*>(A),
                            reinterpret_cast<float*>(deg > 2 ? D : nullptr), f32_step(step_of(w, l, 0)),
                            f32_step(step_of(w, l, 1)), f32_ptr(w.dsh), none, s));
        });
        for (int m = 2; m < deg; ++m) {
            T* dout = m < deg - 1 ? D : nullptr;
            traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 4.0 + (dout ? 1.0 : 0.0), true), s,
                   [&] { cheb(cur, D, oth, dout, step_of(w, l, m), none); });
            std::swap(cur, oth);
        }
    } else if (!tl.on && split_sweeps(p)) {
        traced(p, K_CHEB0, f32, fine, vbytes<T>(p, l, 2.0, var), s,
               [&] { Ops<T>::cheb_zero(g, L, dim, var, b, A, step_of(w, l, 0), w.dsh, s); });
        // d_1 = x_1 (the step from zero): the second step reads A as both iterate and direction
        traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, deg > 2 ? 4.0 : 3.0, true), s,
               [&] { cheb(A, A, B, deg > 2 ? D : nullptr, step_of(w, l, 1), none); });
        std::swap(cur, oth);
        for (int m = 2; m < deg; ++m) {
            T* dout = m < deg - 1 ? D : nullptr;
            // a single level's last step also forms r.z
            const bool dot = rz_fused && m == deg - 1 && l == (int)p->hl.size() - 1;
            traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 4.0 + (dout ? 1.0 : 0.0), true), s,
                   [&] { cheb(cur, D, oth, dout, step_of(w, l, m), dot ? beta : none); });
            rz_done |= dot;
            std::swap(cur, oth);
        }
    } else {
        traced(p, K_PRE2, f32, fine, vbytes<T>(p, l, deg > 2 ? 3.0 : 2.0, true), s, [&] {
            const CUtensorMap* mb = tl.on ? tl.find(TB_HALO, b) : nullptr;
            if (mb)
                (void)tma_pre2(tl.geo, p->nsm, *mb, reinterpret_cast<float*>(A),
                               reinterpret_cast<float*>(deg > 2 ? D : nullptr), f32_step(step_of(w, l, 0)),
                               f32_step(step_of(w, l, 1)), f32_ptr(w.dsh), none, s);
            else
                Ops<T>::cheb_pre2(g, L, dim, var, b, A, deg > 2 ? D : nullptr, step_of(w, l, 0), step_of(w, l, 1),
                                  w.dsh, s);
        });
        for (int m = 2; m < deg; ++m) {
            T* dout = m < deg - 1 ? D : nullptr;
            traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 4.0 + (dout ? 1.0 : 0.0), true), s,
                   [&] { cheb(cur, D, oth, dout, step_of(w, l, m), none); });
            std::swap(cur, oth);
        }
    }
    if (l == (int)p->hl.size() - 1) {  // coarsest level on the grid kernels: the Chebyshev solve above
        if (rz_fused) {
            if (!rz_done)
                traced(p, K_DOT, f32, fine, vbytes<T>(p, l, 2.0, false), s, [&] { Ops<T>::dot(g, L.N, b, cur, beta, s); });
            red_finish(p, beta, w.Kp, f32, s);
        }
        return cur;
    }
    // coarse-grid correction: residual + restriction, then the coarser levels.  In 3-D and with variable
    // coefficients the residual is stored (in D, free between pre- and post-smoothing) and restricted by a
    // second sweep: 27 (3-D) stencil evaluations per coarse point cost more than the extra vector pass.
    if (s3) {
        traced(p, K_RESTRICT, f32, fine, vbytes<T>(p, l, 2.0, true) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
            note(sweep3_residual_restrict(s3l.geo, s3l.at(S3B_RHALO, cur), s3l.at(S3B_RTILE, b),
                                          reinterpret_cast<float*>(w.b[l + 1]), f32_ptr(w.dsh), none, s));
        });
    } else if (dim == 3 || var) {
        traced(p, K_RESID, f32, fine, vbytes<T>(p, l, 3.0, true), s,
               [&] { Ops<T>::residual(g, L, dim, var, cur, b, D, w.dsh, s); });
        traced(p, K_RESTRICT, f32, fine, vbytes<T>(p, l, 1.0, false) + vbytes<T>(p, l + 1, 1.0, false), s,
               [&] { Ops<T>::restrict_r(w.g[l + 1], L, w.L[l + 1], dim, D, w.b[l + 1], s); });
    } else {
        traced(p, K_RESTRICT, f32, fine, vbytes<T>(p, l, 2.0, true) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
            Ops<T>::restrict_res(w.g[l + 1], L, w.L[l + 1], dim, var, cur, b, w.b[l + 1], w.dsh, s);
        });
    }
    T* ec = vcycle<T>(p, w, l + 1, w.b[l + 1], false, s);
    int m0 = 0;
    if (s3) {  // the correction and the first post-smoothing step in one staged sweep
        traced(p, K_PROCHEB, f32, fine, vbytes<T>(p, l, 4.0, true) + vbytes<T>(p, l + 1, 1.0, false), s, [&] {
            note(sweep3_prolong_step(s3l.geo, s3l.at(S3B_HALO, cur), s3l.at(S3B_COARSE, ec), s3l.at(S3B_TILE, b),
                                     reinterpret_cast<float*>(oth), reinterpret_cast<float*>(D),
                                     f32_step(step_of(w, l, 0, false)), f32_ptr(w.dsh), none, s));
        });
        std::swap(cur, oth);
        m0 = 1;
    } else {
        traced(p, K_PROLONG, f32, fine, vbytes<T>(p, l, 2.0, false) + vbytes<T>(p, l + 1, 1.0, false), s,
               [&] { Ops<T>::prolong_add(g, L, w.L[l + 1], dim, ec, cur, s); });
    }
    // post-smoothing with the same polynomial (symmetric preconditioner)
    for (int m = m0; m < deg; ++m) {
        const bool last = (m == deg - 1);
        T* din = m == 0 ? nullptr : D;
        T* dout = last ? nullptr : D;
        const Red& red = (rz_fused && last) ? beta : none;
        traced(p, K_CHEB, f32, fine, vbytes<T>(p, l, 3.0 + (din ? 1.0 : 0.0) + (dout ? 1.0 : 0.0), true), s,
               [&] { cheb(cur, din, oth, dout, step_of(w, l, m, m != 0), red); });
        std::swap(cur, oth);
    }
    if (rz_fused) red_finish(p, beta, w.Kp, f32, s);
    return cur;
}

// One PCG iteration body: z = M r (with r.z and beta), p = z + beta p and q = (A - dI) p (with p.q and
// alpha), x += alpha p, r -= alpha q (with r.r, convergence and loop control).
template <class T>
int pcg_body(bura_plan* p, Work<T>& w, unsigned long long cond, cudaStream_t s) {
    const Launch& g = w.g[0];
    const Lev& L = w.Lop;  // the CG operator (its faces never bf16)
    const bool f32 = sizeof(T) == 4;
    const Red ralpha = deferred(p, Red{p->partial, p->tickets, w.scal, nullptr, RED_ALPHA, 0});
    const Red rconv = deferred(p, Red{p->partial, p->tickets, w.scal, nullptr, RED_CONV, cond});
    T* z = vcycle<T>(p, w, 0, w.r, true, s);
    const auto& tl = w.tma[0];
    const auto& s3l = w.s3[0];
    const bool s3 = s3l.on;
    const bool lean = lean64(p, w, 0) && w.lc != 0;
    const bool split = !tl.on && !s3 && (split_sweeps(p) || lean);
    if (split)  // p = z + beta p as its own pointwise sweep
        traced(p, K_PUPD, f32, true, vbytes<T>(p, 0, 3.0, false), s,
               [&] { Ops<T>::pupdate(g, L.N, z, w.pa, w.pb, ralpha, s); });
    traced(p, K_SPMV, f32, true, vbytes<T>(p, 0, split ? 2.0 : 4.0, true), s, [&] {
        if constexpr (sizeof(T) == 8) {
            if (lean) return sweep64_spmv(L, w.Kp, p->nsm, w.pa, w.pb, w.q, ralpha, s);
        }
        const CUtensorMap* mz = tl.on ? tl.find(TB_HALO, z) : nullptr;
        const CUtensorMap* ma = tl.on ? tl.find(TB_HALO, w.pa) : nullptr;
        const CUtensorMap* mbb = tl.on ? tl.find(TB_HALO, w.pb) : nullptr;
        if (mz && ma && mbb)
            (void)tma_spmv_p(tl.geo, p->nsm, *mz, *ma, *mbb, tl.var ? &tl.w_halo : nullptr, reinterpret_cast<float*>(w.pa),
                             reinterpret_cast<float*>(w.pb), reinterpret_cast<float*>(w.q), ralpha, s);
        else if (s3) {
            const cudaError_t e = sweep3_spmv(s3l.geo, s3l.at(S3B_HALO, z), s3l.at(S3B_HALO, w.pa), s3l.at(S3B_HALO, w.pb),
                                              reinterpret_cast<float*>(w.pa), reinterpret_cast<float*>(w.pb),
                                              reinterpret_cast<float*>(w.q), ralpha, s);
            if (e != cudaSuccess) p->sweep_err = e;
        } else if (split_sweeps(p))
            Ops<T>::spmv_q(g, L, p->dim, p->var, w.pa, w.pb, w.q, ralpha, s);
        else
            Ops<T>::spmv_p(g, L, p->dim, p->var, z, w.pa, w.pb, w.q, ralpha, s);
    });
    red_finish(p, ralpha, w.Kp, f32, s);
    traced(p, K_CGUPD, f32, true, vbytes<T>(p, 0, 6.0, false), s, [&] {
        const CUtensorMap* mx = tl.on ? tl.find(TB_PLAIN, w.x) : nullptr;
        const CUtensorMap* mr = tl.on ? tl.find(TB_PLAIN, w.r) : nullptr;
        const CUtensorMap* mpa = tl.on ? tl.find(TB_PLAIN, w.pa) : nullptr;
        const CUtensorMap* mpb = tl.on ? tl.find(TB_PLAIN, w.pb) : nullptr;
        const CUtensorMap* mq = tl.on ? tl.find(TB_PLAIN, w.q) : nullptr;
        // the TMA-staged CG update (one CTA per SM, a 3-stage ring) measured no faster than the grid
        // kernel on GB300 (42.6 vs 41.3 us at 1023^2, k = 7); it is used only with a deeper ring requested
        if (mx && mr && mpa && mpb && mq && tma_cg_fits(w.Kp) && p->opt.tma_stages >= 3)
            (void)tma_cg_update(tl.geo, p->nsm, *mx, *mr, *mpa, *mpb, *mq, reinterpret_cast<float*>(w.x),
                                reinterpret_cast<float*>(w.r), rconv, s);
        else
            Ops<T>::cg_update(g, L.N, w.x, w.r, w.pa, w.pb, w.q, rconv, s);
    });
    red_finish(p, rconv, w.Kp, f32, s);
    CKL();
    const cudaError_t missed = p->sweep_err;
    p->sweep_err = cudaSuccess;
    CK(missed);
    return BURA_OK;
}

// Capture the PCG loop once: a conditional WHILE node whose body is one iteration; the k_red_finish
// after k_cg_update clears the condition when every system has converged, on breakdown, or at the cap.
template <class T>
int build_graph(bura_plan* p, Work<T>& w) {
    if (w.exec) return BURA_OK;
    // capture and instantiation happen once per plan, one plan at a time, and never beside the library's
    // own device-synchronising calls in other threads
    std::unique_lock<std::shared_mutex> lock(g_capture_guard);
    CK(cudaGraphCreate(&w.graph, 0));
    CK(cudaGraphConditionalHandleCreate(&w.cond, w.graph, 1u, cudaGraphCondAssignDefault));
    // the parameter struct holds a union with no default constructor: start from zeroed storage
    alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)] = {};
    cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = w.cond;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    CK(cudaGraphAddNode(&node, w.graph, nullptr, nullptr, 0, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    CK(cudaStreamBeginCaptureToGraph(p->cap, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    const long long before = p->tr.launches;
    const bool was_on = p->tr.on;
    p->tr.on = false;
    int rc = pcg_body<T>(p, w, (unsigned long long)w.cond, p->cap);
    p->tr.on = was_on;
    w.body_launches = p->tr.launches - before;
    p->tr.launches = before;
    cudaGraph_t captured = nullptr;
    cudaError_t e = cudaStreamEndCapture(p->cap, &captured);
    if (rc == BURA_OK && e == cudaSuccess) e = cudaGraphInstantiate(&w.exec, w.graph, 0);
    if (rc != BURA_OK || e != cudaSuccess) {
        // a capture that another thread invalidated leaves a graph the driver cannot always destroy
        // (observed: a crash in cudaGraphDestroy); it is left allocated and the next solve captures afresh
        cudaGetLastError();
        w.graph = nullptr;
        w.exec = nullptr;
        if (rc != BURA_OK) return rc;
        CK(e);
    }
    return BURA_OK;
}

// Multi-shift PCG on the work set w: r holds the right-hand sides, x = 0, pa = 0 and the Scal
// record is initialised by the caller.  Returns BURA_OK, BURA_ENOCONV or BURA_ENOTSPD.
template <class T>
int pcg(bura_plan* p, Work<T>& w, int* iters_out, cudaStream_t s) {
    if (p->tr.on) {  // per-kernel timing: the same iteration launched directly, one sync per iteration
        for (;;) {
            CA(pcg_body<T>(p, w, 0, s));
            CK(cudaMemcpyAsync(p->hscal, w.scal, sizeof(Scal), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            collect_trace(p);
            const Scal& h = *p->hscal;
            if (h.breakdown || h.fault || h.nactive == 0 || h.it >= h.max_it) break;
        }
    } else {
        int brc = build_graph<T>(p, w);
        for (int attempt = 1; brc == BURA_ECUDA && attempt < 3; ++attempt) brc = build_graph<T>(p, w);
        CA(brc);
        CK(cudaGraphLaunch(w.exec, s));
        CK(cudaMemcpyAsync(p->hscal, w.scal, sizeof(Scal), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        p->tr.launches += w.body_launches * p->hscal->it;
    }
    const Scal& h = *p->hscal;
    *iters_out = h.it;
    if (h.fault) return BURA_ETIMEOUT;
    if (h.breakdown) return BURA_ENOTSPD;
    return h.nactive == 0 ? BURA_OK : BURA_ENOCONV;
}

int init_scal(bura_plan* p, Scal* dev, const double* thr, const int* active, cudaStream_t s) {
    Scal h;
    std::memset(&h, 0, sizeof(h));
    int na = 0;
    for (int j = 0; j < KMAXP; ++j) {
        h.rz[j] = 1.0;
        h.beta[j] = 0.0;
        h.alpha[j] = 0.0;
        h.dsh[j] = j < p->K ? p->d[j] : 0.0;
        h.dshf[j] = (float)h.dsh[j];
        h.thr[j] = j < p->K ? thr[j] : 0.0;
        h.active[j] = (j < p->K && active[j]) ? 1 : 0;
        na += h.active[j];
    }
    h.nactive = na;
    h.ticket = 0u;
    h.it = 0;
    h.max_it = p->opt.max_iters;
    h.parity = 0;
    h.wait_cycles = p->wait_cycles;
    *p->hscal = h;
    CK(cudaMemcpyAsync(dev, p->hscal, sizeof(Scal), cudaMemcpyHostToDevice, s));
    return BURA_OK;
}

// Per-system absolute thresholds on ||r_j||^2 so that sum_j c_j ||r_j|| / (lambda_lo - d_j) <= tol ||f||.
// A sparse operator without a lower bound on lambda_min stops each system at ||r_j|| <= tol ||f|| (the
// relative residual criterion of the paper's PCG runs, Sec. 5.4).
void thresholds(const bura_plan* p, double tol, double fnorm2, double* thr) {
    for (int j = 0; j < p->K; ++j) {
        const double t = p->lambda_lo > 0 ? tol * (p->lambda_lo - p->d[j]) / (p->K * p->c[j]) : tol;
        thr[j] = t * t * fnorm2;
    }
}

void finish_stats(bura_plan* p, const double* rr, double fnorm2) {
    double eb = 0.0;
    const double fn = std::sqrt(fnorm2);
    for (int j = 0; j < p->K; ++j) {
        const double rn = std::sqrt(std::max(rr[j], 0.0));
        p->st.rel_res[j] = fn > 0 ? rn / fn : 0.0;
        eb += p->c[j] * rn / (p->lambda_lo - p->d[j]);
    }
    p->st.err_bound = p->lambda_lo > 0 ? (fn > 0 ? eb / fn : 0.0) : -1.0;
}

int solve_fp64(bura_plan* p, const double* f, double tol, cudaStream_t s) {
    Work<double>& w = p->w64;
    const long long N = p->hl[0].N;
    traced(p, K_BCAST, false, true, (double)N * 8 + vbytes<double>(p, 0, 3.0, false), s,
           [&] { Ops<double>::broadcast(w.g[0], f, N, p->K, w.r, w.x, w.pa, s); });
    Red store{p->partial, p->tickets, p->scal_outer, p->red_out, RED_STORE, 0};
    traced(p, K_NORM, false, true, (double)N * 8, s, [&] { launch_norm2(N, f, store, p->nsm, s); });
    CKL();
    CK(cudaMemcpyAsync(p->hbuf, p->red_out, KMAXP * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    double fnorm2 = 0.0;  // k_norm2 leaves KMAXP partial sums
    for (int i = 0; i < KMAXP; ++i) fnorm2 += p->hbuf[i];
    double thr[KMAXP] = {0};
    int act[KMAXP] = {0};
    thresholds(p, tol, fnorm2, thr);
    for (int j = 0; j < p->K; ++j) act[j] = fnorm2 > 0 ? 1 : 0;
    CA(init_scal(p, w.scal, thr, act, s));
    int it = 0;
    int rc = BURA_OK;
    if (fnorm2 > 0) rc = pcg<double>(p, w, &it, s);
    p->st.iters = it;
    p->st.outer = 1;
    for (int j = 0; j <= p->k; ++j) p->st.shift_iters[j] = fnorm2 > 0 ? p->hscal->iters[j] : 0;
    double rr[KMAXP] = {0};
    for (int j = 0; j < p->K; ++j) rr[j] = fnorm2 > 0 ? p->hscal->rr[j] : 0.0;
    finish_stats(p, rr, fnorm2);
    return rc;
}

// Mixed path with IEEE FP64 refinement: v_j (Kp64 layout) += scale_j * x_j after each FP32 inner solve,
// the true residual r_j = f - (A - d_j I) v_j in FP64, and the next inner rhs r_j / ||r_j|| in FP32.
int solve_mixed_fp64(bura_plan* p, const double* f, double tol, cudaStream_t s) {
    Work<float>& w = p->w32;
    const Launch& g64 = p->w64.g[0];
    const Lev& L64 = p->w64.L[0];
    const long long N = p->hl[0].N;
    CK(cudaMemsetAsync(p->v64, 0, (size_t)N * g64.Kp * sizeof(double), s));
    Red store{p->partial, p->tickets, p->scal_outer, p->red_out, RED_STORE, 0};
    // the residual of the zero initial guess is f itself: only its norm is needed
    traced(p, K_NORM, false, true, (double)N * 8, s, [&] { launch_norm2(N, f, store, p->nsm, s); });
    CKL();
    CK(cudaMemcpyAsync(p->hbuf, p->red_out, KMAXP * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    double fnorm2 = 0.0;  // k_norm2 leaves KMAXP partial sums
    for (int i = 0; i < KMAXP; ++i) fnorm2 += p->hbuf[i];
    double thr64[KMAXP] = {0};
    double rr[KMAXP] = {0};
    thresholds(p, tol, fnorm2, thr64);
    for (int j = 0; j < p->K; ++j) rr[j] = fnorm2;
    // Plan the refinement: system j needs its residual reduced by need_j = sqrt(thr64_j) / ||f||; one
    // FP32 inner solve is asked for at most a reduction of inner_rtol, so n_j = ceil(log need_j /
    // log inner_rtol) steps are needed and each takes the even share need_j^(1/n_j).
    double step_target[KMAXP] = {0};
    for (int j = 0; j < p->K; ++j) {
        const double need = fnorm2 > 0 ? std::sqrt(thr64[j] / fnorm2) : 1.0;
        if (need >= 1.0) { step_target[j] = 1.0; continue; }
        const int n = std::max(1, (int)std::ceil(std::log(need) / std::log(p->opt.inner_rtol) - 1e-9));
        step_target[j] = std::pow(need, 1.0 / n);
    }
    int total_it = 0, outer = 0;
    int rc = BURA_ENOCONV;
    int siters[KMAXP] = {0};
    for (;;) {
        if (outer > 0) {
            traced(p, K_RES64, false, true, (double)N * 8 + vbytes<double>(p, 0, 2.0, true), s,
                   [&] { launch_residual64(g64, L64, p->dim, p->var, f, p->v64, p->r64, store, s); });
            CKL();
            CK(cudaMemcpyAsync(p->hbuf, p->red_out, KMAXP * sizeof(double), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            for (int j = 0; j < p->K; ++j) rr[j] = p->hbuf[j];
        }
        int act[KMAXP] = {0};
        int na = 0;
        for (int j = 0; j < p->K; ++j) {
            if (!std::isfinite(rr[j])) return BURA_ENOTSPD;
            act[j] = rr[j] > thr64[j] ? 1 : 0;
            na += act[j];
        }
        if (na == 0) { rc = BURA_OK; break; }
        if (outer >= p->opt.max_outer) { rc = BURA_ENOCONV; break; }
        double* hs = p->hbuf + KMAXP;
        double* his = p->hbuf + 2 * KMAXP;
        double thr[KMAXP] = {0};
        for (int j = 0; j < KMAXP; ++j) {
            const bool a = j < p->K && act[j];
            hs[j] = a ? std::sqrt(rr[j]) : 0.0;
            his[j] = a ? 1.0 / hs[j] : 0.0;
            if (a) {
                // relative target of this inner solve (the scaled rhs has unit norm): the planned
                // share, or less if that already meets the FP64 threshold (with a margin of 2)
                const double need = 0.5 * std::sqrt(thr64[j] / rr[j]);
                const double t = std::max(step_target[j] * 0.5, need);
                thr[j] = t * t;
            }
        }
        CK(cudaMemcpyAsync(p->scale, hs, KMAXP * sizeof(double), cudaMemcpyHostToDevice, s));
        CK(cudaMemcpyAsync(p->invscale, his, KMAXP * sizeof(double), cudaMemcpyHostToDevice, s));
        if (outer == 0)
            traced(p, K_CAST, false, true, (double)N * 8 + vbytes<float>(p, 0, 3.0, false), s,
                   [&] { launch_cast_f(w.g[0], N, p->K, f, p->invscale, w.r, w.x, w.pa, s); });
        else
            traced(p, K_CAST, false, true, vbytes<double>(p, 0, 1.0, false) + vbytes<float>(p, 0, 3.0, false), s,
                   [&] { launch_cast_scaled(g64, w.g[0], N, p->K, p->r64, p->invscale, w.r, w.x, w.pa, s); });
        CKL();
        CA(init_scal(p, w.scal, thr, act, s));
        int it = 0;
        int irc = pcg<float>(p, w, &it, s);
        if (irc == BURA_ENOTSPD || irc == BURA_ETIMEOUT) return irc;
        for (int j = 0; j < p->K; ++j) siters[j] += p->hscal->iters[j];
        total_it += it;
        traced(p, K_CORR64, false, true, vbytes<double>(p, 0, 2.0, false) + vbytes<float>(p, 0, 1.0, false), s,
               [&] { launch_correct64(g64, w.g[0], N, p->K, p->v64, w.x, p->scale, s); });
        CKL();
        ++outer;
    }
    p->st.iters = total_it;
    p->st.outer = outer;
    for (int j = 0; j <= p->k; ++j) p->st.shift_iters[j] = siters[j];
    finish_stats(p, rr, fnorm2);
    return rc;
}

// Mixed path with double-float refinement (BURA_REFINE_DF): v_j kept as FP32 pairs, correction and true
// residual fused in one FP32-pipe kernel.
int solve_mixed_df(bura_plan* p, const double* f, double tol, cudaStream_t s) {
    Work<float>& w = p->w32;
    const Launch& g32 = w.g[0];
    const Lev& L32 = w.L[0];
    const long long N = p->hl[0].N;
    const size_t vb = (size_t)N * w.Kp * sizeof(float);
    p->vcur = 0;
    CK(cudaMemsetAsync(p->vh[0], 0, vb, s));
    CK(cudaMemsetAsync(p->vl[0], 0, vb, s));
    Red store{p->partial, p->tickets, p->scal_outer, p->red_out, RED_STORE, 0};
    // the residual of the zero initial guess is f itself: only its norm is needed
    traced(p, K_NORM, false, true, (double)N * 8, s, [&] { launch_norm2(N, f, store, p->nsm, s); });
    CKL();
    CK(cudaMemcpyAsync(p->hbuf, p->red_out, KMAXP * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    double fnorm2 = 0.0;  // k_norm2 leaves KMAXP partial sums
    for (int i = 0; i < KMAXP; ++i) fnorm2 += p->hbuf[i];
    if (!std::isfinite(fnorm2)) return BURA_ENOTSPD;
    // The inner FP32 solves work on sf * residual with sf a power of two that brings f's typical entry
    // near 1 (exact scaling, no FP32 range trouble); their thresholds are in the same units.
    const double sf = fnorm2 > 0 ? std::ldexp(1.0, -(int)std::lround(0.5 * std::log2(fnorm2 / (double)N))) : 1.0;
    double thr64[KMAXP] = {0};
    double rr[KMAXP] = {0};
    thresholds(p, tol, fnorm2, thr64);
    for (int j = 0; j < p->K; ++j) rr[j] = fnorm2;
    // Plan the refinement: system j needs its residual reduced by need_j = sqrt(thr64_j) / ||f||; one
    // FP32 inner solve is asked for at most a reduction of inner_rtol, so n_j = ceil(log need_j /
    // log inner_rtol) steps are needed and each takes the even share need_j^(1/n_j).
    double step_target[KMAXP] = {0};
    for (int j = 0; j < p->K; ++j) {
        const double need = fnorm2 > 0 ? std::sqrt(thr64[j] / fnorm2) : 1.0;
        if (need >= 1.0) { step_target[j] = 1.0; continue; }
        const int n = std::max(1, (int)std::ceil(std::log(need) / std::log(p->opt.inner_rtol) - 1e-9));
        step_target[j] = std::pow(need, 1.0 / n);
    }
    int total_it = 0, outer = 0;
    int rc = BURA_ENOCONV;
    int siters[KMAXP] = {0};
    for (;;) {
        if (outer > 0) {
            // v <- v + x / sf and the next scaled right-hand side sf (f - (A - d_j I) v), in FP32 pairs
            const int nxt = p->vcur ^ 1;
            traced(p, K_RESDF, true, true, vbytes<float>(p, 0, 6.0, true) + (double)N * 8, s, [&] {
                launch_update_residual_df(g32, L32, p->dim, p->var, p->dfop, p->fh, p->fl, p->vh[p->vcur],
                                          p->vl[p->vcur], w.x, p->vh[nxt], p->vl[nxt], w.r, (float)sf, store, s);
            });
            CKL();
            p->vcur = nxt;
            CK(cudaMemcpyAsync(p->hbuf, p->red_out, KMAXP * sizeof(double), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            for (int j = 0; j < p->K; ++j) rr[j] = p->hbuf[j] / (sf * sf);
        }
        int act[KMAXP] = {0};
        int na = 0;
        for (int j = 0; j < p->K; ++j) {
            if (!std::isfinite(rr[j])) return BURA_ENOTSPD;
            act[j] = rr[j] > thr64[j] ? 1 : 0;
            na += act[j];
        }
        if (na == 0) { rc = BURA_OK; break; }
        if (outer >= p->opt.max_outer) { rc = BURA_ENOCONV; break; }
        double thr[KMAXP] = {0};
        for (int j = 0; j < KMAXP; ++j) {
            if (!(j < p->K && act[j])) continue;
            // relative target of this inner solve: the planned share, or less if that already meets the
            // FP64 threshold (with a margin of 2); absolute in the scaled units of the inner solve
            const double need = 0.5 * std::sqrt(thr64[j] / rr[j]);
            const double t = std::max(step_target[j] * 0.5, need);
            thr[j] = t * t * rr[j] * sf * sf;
        }
        if (outer == 0) {
            traced(p, K_CASTDF, false, true, (double)N * 8 + vbytes<float>(p, 0, 3.0, false) + (double)N * 8, s,
                   [&] { launch_cast_f_df(g32, N, p->K, f, sf, w.r, w.x, w.pa, p->fh, p->fl, s); });
            CKL();
        } else {
            // zero iterate and direction of the next inner solve (the residual kernel wrote its rhs)
            CK(cudaMemsetAsync(w.x, 0, vb, s));
            CK(cudaMemsetAsync(w.pa, 0, vb, s));
        }
        CA(init_scal(p, w.scal, thr, act, s));
        int it = 0;
        int irc = pcg<float>(p, w, &it, s);
        if (irc == BURA_ENOTSPD || irc == BURA_ETIMEOUT) return irc;
        for (int j = 0; j < p->K; ++j) siters[j] += p->hscal->iters[j];
        total_it += it;
        ++outer;
    }
    p->st.iters = total_it;
    p->st.outer = outer;
    for (int j = 0; j <= p->k; ++j) p->st.shift_iters[j] = siters[j];
    finish_stats(p, rr, fnorm2);
    return rc;
}

int solve_core(bura_plan* p, const double* f, double tol, cudaStream_t s) {
    if (!(tol > 0)) return BURA_EINVAL;
    CK(cudaSetDevice(p->dev));
    p->tr.launches = 0;
    std::memset(p->st.shift_iters, 0, sizeof(p->st.shift_iters));
    std::memset(p->st.rel_res, 0, sizeof(p->st.rel_res));
    if (p->opt.precision == BURA_PREC_FP64) return solve_fp64(p, f, tol, s);
    return p->opt.refine == BURA_REFINE_DF ? solve_mixed_df(p, f, tol, s) : solve_mixed_fp64(p, f, tol, s);
}

// Split x into FP32 parts hi + lo with hi = fl32(x) and lo = fl32(x - hi) (x - hi is exact in FP64).
void split_df(double x, float* hi, float* lo) {
    *hi = (float)x;
    *lo = (float)(x - (double)*hi);
}

// Buffers and coefficient tables of the double-float refinement of the mixed path.
// The double-float refinement's per-system tables (KMAXP entries each, zero in the padding): diag - d_j,
// d_j, c_j as (hi, lo) pairs, written into the buffer that starts at dfop.ch.
int upload_df_tables(bura_plan* p) {
    const HostLevel& h = p->hl[0];
    std::vector<float> t(6 * KMAXP, 0.f);
    const double diag = 2.0 * (h.w[0] + h.w[1] + (p->dim == 3 ? h.w[2] : 0.0));
    for (int j = 0; j < p->K; ++j) {
        split_df(diag - p->d[j], &t[j], &t[KMAXP + j]);
        split_df(p->d[j], &t[2 * KMAXP + j], &t[3 * KMAXP + j]);
        split_df(p->c[j] * p->out_scale, &t[4 * KMAXP + j], &t[5 * KMAXP + j]);
    }
    CK(cudaMemcpy(const_cast<float*>(p->dfop.ch), t.data(), t.size() * sizeof(float), cudaMemcpyHostToDevice));
    return BURA_OK;
}

int build_df(bura_plan* p) {
    const long long N = p->hl[0].N;
    const int Kp = p->w32.Kp;
    const size_t vb = (size_t)N * Kp * sizeof(float);
    for (int i = 0; i < 2; ++i) {
        CA(dalloc(p, &p->vh[i], vb));
        CA(dalloc(p, &p->vl[i], vb));
    }
    CA(dalloc(p, &p->fh, (size_t)N * sizeof(float)));
    CA(dalloc(p, &p->fl, (size_t)N * sizeof(float)));
    const HostLevel& h = p->hl[0];
    DfOpHost& op = p->dfop;
    for (int a = 0; a < 3; ++a) split_df(a < p->dim ? h.w[a] : 0.0, &op.w[a][0], &op.w[a][1]);
    float* dt = nullptr;
    CA(dalloc(p, &dt, 6 * KMAXP * sizeof(float)));
    op.ch = dt;
    op.cl = dt + KMAXP;
    op.dh = dt + 2 * KMAXP;
    op.dl = dt + 3 * KMAXP;
    p->cwh = dt + 4 * KMAXP;
    p->cwl = dt + 5 * KMAXP;
    CA(upload_df_tables(p));
    if (p->var) {
        for (int a = 0; a < p->dim; ++a) {
            std::vector<float> fh(h.a[a].size()), fl(h.a[a].size());
            for (size_t i = 0; i < fh.size(); ++i) split_df(h.a[a][i] * h.w[a], &fh[i], &fl[i]);
            float *dh = nullptr, *dl = nullptr;
            CA(dalloc(p, &dh, fh.size() * sizeof(float)));
            CA(dalloc(p, &dl, fl.size() * sizeof(float)));
            CK(cudaMemcpy(dh, fh.data(), fh.size() * sizeof(float), cudaMemcpyHostToDevice));
            CK(cudaMemcpy(dl, fl.data(), fl.size() * sizeof(float), cudaMemcpyHostToDevice));
            op.fh[a] = dh;
            op.fl[a] = dl;
        }
    }
    return BURA_OK;
}

// The weights c_j (times the output scale) of the output sum and the shifts of the outer (refinement) CG state record.
int upload_outer(bura_plan* p) {
    std::vector<double> cc(KMAXP, 0.0);
    for (int j = 0; j < p->K; ++j) cc[j] = p->c[j] * p->out_scale;
    CK(cudaMemcpy(p->cdev, cc.data(), KMAXP * sizeof(double), cudaMemcpyHostToDevice));
    Scal so;
    std::memset(&so, 0, sizeof(so));
    for (int j = 0; j < p->K; ++j) so.dsh[j] = p->d[j];
    CK(cudaMemcpy(p->scal_outer, &so, sizeof(Scal), cudaMemcpyHostToDevice));
    if (p->ocfg) {
        OuterCfg oc;
        std::memset(&oc, 0, sizeof(oc));
        for (int j = 0; j < p->K; ++j) {
            oc.c[j] = p->c[j];
            oc.d[j] = p->d[j];
        }
        oc.lambda_lo = p->lambda_lo;
        oc.inner_rtol = p->opt.inner_rtol;
        oc.rtol_slack = std::pow(p->opt.inner_rtol, 1e-9);
        oc.log_rtol = std::log(p->opt.inner_rtol);
        oc.wait_cycles = p->wait_cycles;
        oc.K = p->K;
        oc.max_outer = p->opt.max_outer;
        oc.max_iters = p->opt.max_iters;
        CK(cudaMemcpy(p->ocfg, &oc, sizeof(oc), cudaMemcpyHostToDevice));
    }
    return BURA_OK;
}

// The device-driven solve applies to the FP64 path and to the mixed path with FP64 refinement, outside
// per-kernel profiling (which times launches one by one).
bool device_driven(const bura_plan* p) {
    return !p->tr.on && (p->opt.precision == BURA_PREC_FP64 || p->opt.refine == BURA_REFINE_FP64);
}

// Add a WHILE node after the current capture dependencies of stream s, with a new condition handle of
// the graph being captured (reset to `dflt` at every launch); capture continues after the node.
int capture_while(cudaStream_t s, unsigned dflt, cudaGraphConditionalHandle* h, cudaGraph_t* body) {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    CK(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd));
    if (cs != cudaStreamCaptureStatusActive || !g) return BURA_ECUDA;
    CK(cudaGraphConditionalHandleCreate(h, g, dflt, cudaGraphCondAssignDefault));
    alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)] = {};
    cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = *h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    CK(cudaGraphAddNode(&node, g, deps, nullptr, nd, &cp));
    *body = cp.conditional.phGraph_out[0];
    CK(cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    return BURA_OK;
}

// A condition handle of the graph that stream s is capturing into (to pass to a kernel before the node
// that uses it is added).
int capture_handle(cudaStream_t s, unsigned dflt, cudaGraphConditionalHandle* h) {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    CK(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, nullptr, nullptr, nullptr));
    if (cs != cudaStreamCaptureStatusActive || !g) return BURA_ECUDA;
    CK(cudaGraphConditionalHandleCreate(h, g, dflt, cudaGraphCondAssignDefault));
    return BURA_OK;
}

// The WHILE node of an existing handle (created before its setter kernel was captured).
int capture_while_h(cudaStream_t s, cudaGraphConditionalHandle h, cudaGraph_t* body) {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    CK(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd));
    if (cs != cudaStreamCaptureStatusActive || !g) return BURA_ECUDA;
    alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)] = {};
    cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    CK(cudaGraphAddNode(&node, g, deps, nullptr, nd, &cp));
    *body = cp.conditional.phGraph_out[0];
    CK(cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    return BURA_OK;
}

// The device-driven solve is captured level by level: the top level into the graph that a stream is
// capturing into, each WHILE body afterwards into its own body graph.
struct BodyTask {
    bura_plan* p;
    cudaGraph_t body;
    int kind;                          // 0: one PCG iteration; 1: one refinement step of the mixed path
    cudaGraphConditionalHandle cond;   // the WHILE condition of this body
};

// Top level of one solve of plan p, captured on s (which is capturing): the FP64 path is ||f||, the
// controller, WHILE(PCG), the outcome; the mixed path is zero v, ||f||, the controller, WHILE(refinement
// step).  The right-hand side is read through the plan's solve record.  Bodies are queued in tasks.
int capture_solve_top(bura_plan* p, cudaStream_t s, std::vector<BodyTask>& tasks) {
    const long long N = p->hl[0].N;
    const double* const* fpp =
        reinterpret_cast<const double* const*>(reinterpret_cast<const char*>(p->ostate) + offsetof(OuterState, f));
    Red store{p->partial, p->tickets, p->scal_outer, p->red_out, RED_STORE, 0};
    cudaGraphConditionalHandle h = 0;
    cudaGraph_t body = nullptr;
    if (p->opt.precision == BURA_PREC_FP64) {
        Work<double>& w = p->w64;
        Ops<double>::broadcast(w.g[0], nullptr, N, p->K, w.r, w.x, w.pa, s, fpp);
        launch_norm2(N, nullptr, store, p->nsm, s, fpp);
        CA(capture_handle(s, 0u, &h));
        launch_outer_begin(p->ocfg, p->ostate, p->red_out, w.scal, p->scale, p->invscale, 0ull, (unsigned long long)h, 1, s);
        CA(capture_while_h(s, h, &body));
        launch_outer_end_fp64(p->ocfg, p->ostate, w.scal, s);
        p->s_fixed += 4;
        tasks.push_back({p, body, 0, h});
    } else {
        Work<float>& w = p->w32;
        CK(cudaMemsetAsync(p->v64, 0, (size_t)N * p->w64.g[0].Kp * sizeof(double), s));
        launch_norm2(N, nullptr, store, p->nsm, s, fpp);
        CA(capture_handle(s, 0u, &h));
        launch_outer_begin(p->ocfg, p->ostate, p->red_out, w.scal, p->scale, p->invscale, (unsigned long long)h, 0ull, 0, s);
        CA(capture_while_h(s, h, &body));
        p->s_fixed += 2;
        tasks.push_back({p, body, 1, h});
    }
    CK(cudaGetLastError());
    return BURA_OK;
}

// Capture one queued body (and queue the bodies it contains) on the plan's private capture stream.
int capture_body(const BodyTask& t, std::vector<BodyTask>& tasks) {
    bura_plan* p = t.p;
    cudaStream_t s = p->cap;
    const long long N = p->hl[0].N;
    CK(cudaStreamBeginCaptureToGraph(s, t.body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    int rc = BURA_OK;
    const long long b0 = p->tr.launches;
    if (t.kind == 0) {
        rc = p->opt.precision == BURA_PREC_FP64 ? pcg_body<double>(p, p->w64, (unsigned long long)t.cond, s)
                                                : pcg_body<float>(p, p->w32, (unsigned long long)t.cond, s);
        p->s_body = p->tr.launches - b0;
    } else {
        // one refinement step: the inner right-hand side (arming the inner loop), WHILE(PCG), the correction,
        // the FP64 residual and the controller, which clears the outer condition when the solve is decided
        Work<float>& w = p->w32;
        const Launch& g64 = p->w64.g[0];
        Red store{p->partial, p->tickets, p->scal_outer, p->red_out, RED_STORE, 0};
        const double* const* fpp =
            reinterpret_cast<const double* const*>(reinterpret_cast<const char*>(p->ostate) + offsetof(OuterState, f));
        cudaGraphConditionalHandle hin = 0;
        cudaGraph_t ibody = nullptr;
        rc = capture_handle(s, 1u, &hin);
        if (rc == BURA_OK) {
            launch_cast_outer(g64, w.g[0], N, p->K, p->ostate, p->r64, p->invscale, w.r, w.x, w.pa,
                              (unsigned long long)hin, s);
            rc = capture_while_h(s, hin, &ibody);
        }
        if (rc == BURA_OK) {
            launch_correct64(g64, w.g[0], N, p->K, p->v64, w.x, p->scale, s);
            launch_residual64(g64, p->w64.L[0], p->dim, p->var, nullptr, p->v64, p->r64, store, s, fpp);
            launch_outer_next(p->ocfg, p->ostate, p->red_out, w.scal, p->scale, p->invscale, (unsigned long long)t.cond,
                              s);
            p->s_outer += 4;
            tasks.push_back({p, ibody, 0, hin});
        }
    }
    cudaGraph_t done = nullptr;
    const cudaError_t e = cudaStreamEndCapture(s, &done);
    if (rc == BURA_OK && e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    return rc;
}

// Capture every queued body (depth first); profiling is off while capturing and launches are not counted.
int capture_bodies(std::vector<BodyTask>& tasks) {
    while (!tasks.empty()) {
        const BodyTask t = tasks.back();
        tasks.pop_back();
        const bool was_on = t.p->tr.on;
        const long long before = t.p->tr.launches;
        t.p->tr.on = false;
        const int rc = capture_body(t, tasks);
        t.p->tr.on = was_on;
        t.p->tr.launches = before;
        if (rc != BURA_OK) return rc;
    }
    return BURA_OK;
}

// Build and instantiate the plan's device-driven solve graph once (capture under the exclusive guard).
int build_solve_graph(bura_plan* p) {
    if (p->sexec) return BURA_OK;
    std::unique_lock<std::shared_mutex> lock(g_capture_guard);
    cudaGraph_t g = nullptr;
    CK(cudaGraphCreate(&g, 0));
    p->s_fixed = p->s_outer = p->s_body = 0;
    int rc = BURA_OK;
    std::vector<BodyTask> tasks;
    cudaError_t e = cudaStreamBeginCaptureToGraph(p->cap, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    if (rc == BURA_OK) {
        const bool was_on = p->tr.on;
        const long long before = p->tr.launches;
        p->tr.on = false;
        rc = capture_solve_top(p, p->cap, tasks);
        p->tr.on = was_on;
        p->tr.launches = before;
        cudaGraph_t done = nullptr;
        e = cudaStreamEndCapture(p->cap, &done);
        if (rc == BURA_OK && e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    }
    if (rc == BURA_OK) rc = capture_bodies(tasks);
    cudaGraphExec_t ex = nullptr;
    if (rc == BURA_OK) {
        e = cudaGraphInstantiate(&ex, g, 0);
        if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    }
    if (rc != BURA_OK) {
        cudaGetLastError();  // a failed capture's partial graph is left allocated (see build_graph)
        return rc;
    }
    p->sgraph = g;
    p->sexec = ex;
    return BURA_OK;
}

// Enqueue the device-driven solve of f on s (no host synchronisation); the outcome is copied to the
// pinned mirror after the output stage by the caller.
int solve_device(bura_plan* p, const double* f, double tol, cudaStream_t s) {
    int rc = build_solve_graph(p);
    for (int attempt = 1; rc == BURA_ECUDA && attempt < 3; ++attempt) rc = build_solve_graph(p);
    CA(rc);
    launch_solve_params(p->ostate, f, tol, s);
    CK(cudaGetLastError());
    CK(cudaGraphLaunch(p->sexec, s));
    return BURA_OK;
}

// The outcome of the last device-driven solve (waits for it): statistics and its status.
int read_outcome(bura_plan* p) {
    CK(cudaEventSynchronize(p->done));
    if (!p->pending) return p->last_status;
    p->pending = false;
    const OuterState& o = *p->hstate;
    p->st.iters = o.total_it;
    p->st.outer = o.outer;
    for (int j = 0; j <= p->k; ++j) p->st.shift_iters[j] = o.siters[j];
    double rr[KMAXP] = {0};
    for (int j = 0; j < p->K; ++j) rr[j] = o.rr[j];
    finish_stats(p, rr, o.fnorm2);
    p->st.launches = p->res_on ? 2 : 2 + p->s_fixed + (long long)o.outer * p->s_outer + (long long)o.total_it * p->s_body;
    p->last_status = o.status;
    return o.status;
}

// Where the solutions are: FP64 path w64.x, mixed path with FP64 refinement v64 (both Kp64 layout),
// mixed path with double-float refinement the FP32 pairs vh/vl[vcur] (Kp32 layout).
bool df_solution(const bura_plan* p) {
    return p->opt.precision != BURA_PREC_FP64 && p->opt.refine == BURA_REFINE_DF;
}
const double* solution_vectors(const bura_plan* p) {
    return p->opt.precision == BURA_PREC_FP64 ? p->w64.x : p->v64;
}

// Frees every device and host resource of the plan (the body of bura_destroy, without its guard).
int destroy_plan(bura_plan* p) {
    cudaSetDevice(p->dev);
    for (auto& e : p->tr.ev) cudaEventDestroy(e);
    if (p->done) cudaEventDestroy(p->done);
    if (p->w64.exec) cudaGraphExecDestroy(p->w64.exec);
    if (p->w64.graph) cudaGraphDestroy(p->w64.graph);
    if (p->w32.exec) cudaGraphExecDestroy(p->w32.exec);
    if (p->w32.graph) cudaGraphDestroy(p->w32.graph);
    if (p->sexec) cudaGraphExecDestroy(p->sexec);
    if (p->sgraph) cudaGraphDestroy(p->sgraph);
    if (p->cap) cudaStreamDestroy(p->cap);
    for (void* q : p->allocs) cudaFree(q);
    if (p->hstate) cudaFreeHost(p->hstate);
    if (p->hscal) cudaFreeHost(p->hscal);
    if (p->hbuf) cudaFreeHost(p->hbuf);
    delete p;
    return BURA_OK;
}

}  // namespace

extern "C" {

void bura_default_options(bura_options* opt) {
    if (!opt) return;
    std::memset(opt, 0, sizeof(*opt));
    opt->precision = BURA_PREC_MIXED;
    opt->smoother_degree = 2;
    opt->smoother_ratio = 0.0;
    opt->max_iters = 200;
    opt->max_outer = 12;
    opt->inner_rtol = 1e-5;
    opt->coarse_degree = 0;
    opt->unscaled = 0;
    opt->tma_wait_cycles = 0;
    opt->smoother_bf16 = 0;
}


}  // extern "C"

namespace {

// Grid and coefficient checks shared by the setup entry points; *N receives the number of points.
int check_grid(const bura_grid* grid, const double* const* faces, long long* N) {
    if (!grid) return BURA_EINVAL;
    if (grid->dim != 2 && grid->dim != 3) return BURA_EINVAL;
    if (grid->coef_kind != BURA_COEF_CONSTANT && grid->coef_kind != BURA_COEF_FACES) return BURA_EINVAL;
    long long n = 1;
    for (int a = 0; a < grid->dim; ++a) {
        if (grid->n[a] < 1) return BURA_EINVAL;
        n *= grid->n[a];
    }
    if (grid->coef_kind == BURA_COEF_FACES && !faces) return BURA_EINVAL;
    if (n * 16 >= (1LL << 31)) return BURA_ERANGE;
    *N = n;
    return BURA_OK;
}

int check_options(const bura_options& o) {
    if (o.precision != BURA_PREC_FP64 && o.precision != BURA_PREC_MIXED) return BURA_EINVAL;
    if (o.smoother_degree < 1 || o.smoother_degree > 16 || !(o.smoother_ratio == 0 || o.smoother_ratio > 1) || o.max_iters < 1 ||
        o.max_outer < 1 || !(o.inner_rtol > 0 && o.inner_rtol < 1) || o.coarse_degree < 0 || o.coarse_degree > 1000 ||
        o.block_points < 0 || o.block_points > 1024 || o.blocks_per_sm < 0 || o.blocks_per_sm > 64 ||
        o.coarse_kernel < BURA_COARSE_AUTO || o.coarse_kernel > BURA_COARSE_FDIAG ||
        !(o.cluster_size == 0 || o.cluster_size == 2 || o.cluster_size == 4 || o.cluster_size == 8 ||
          o.cluster_size == 16) ||
        o.sweeps < BURA_SWEEP_AUTO || o.sweeps > BURA_SWEEP_GRID || o.refine < BURA_REFINE_FP64 ||
        o.refine > BURA_REFINE_DF || o.tma_stages < 0 || o.tma_stages > 4 || o.post_smooth_split < 0 ||
        o.post_smooth_split > 2 || o.unscaled < 0 || o.unscaled > 1 || o.tma_wait_cycles < 0 ||
        o.smoother_bf16 < 0 || o.smoother_bf16 > 1)
        return BURA_EINVAL;
    return BURA_OK;
}

// The device part of a plan's setup (after its levels and coefficients are on the host): workspaces,
// tables, tensor maps, refinement buffers.  Frees the plan on failure.
int setup_device(bura_plan* p, long long N, bura_plan** out) {
    auto fail = [&](int rc) { destroy_plan(p); return rc; };
    const bura_options& o = p->opt;
    int rc = BURA_OK;
    if (cudaGetDevice(&p->dev) != cudaSuccess) return fail(BURA_ECUDA);
    if (cudaStreamCreateWithFlags(&p->cap, cudaStreamNonBlocking) != cudaSuccess) {
        p->cap = nullptr;
        return fail(BURA_ECUDA);
    }
    int nsm = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->dev) != cudaSuccess || nsm <= 0)
        return fail(BURA_ECUDA);
    p->nsm = nsm;
    int cl = 0;
    p->cluster_ok = cudaDeviceGetAttribute(&cl, cudaDevAttrClusterLaunch, p->dev) == cudaSuccess && cl != 0;
    if ((o.coarse_kernel == BURA_COARSE_CLUSTER || o.coarse_kernel == BURA_COARSE_FDIAG) && !p->cluster_ok)
        return fail(BURA_EINVAL);
    if (p->dim == 0) {  // the sparse operator's row offsets and columns, shared by both precisions
        const HostLevel& h = p->hl[0];
        int* rp = nullptr;
        int* ci = nullptr;
        if ((rc = dalloc(p, &rp, h.rowptr.size() * sizeof(int))) != BURA_OK) return fail(rc);
        if ((rc = dalloc(p, &ci, h.col.size() * sizeof(int))) != BURA_OK) return fail(rc);
        if (cudaMemcpy(rp, h.rowptr.data(), h.rowptr.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(ci, h.col.data(), h.col.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
            return fail(BURA_ECUDA);
        p->csr_rowptr = rp;
        p->csr_col = ci;
    }

    rc = build_work<double>(p, p->w64, o.precision == BURA_PREC_FP64);
    if (rc != BURA_OK) return fail(rc);
    if (o.precision == BURA_PREC_MIXED) {
        rc = build_work<float>(p, p->w32);
        if (rc != BURA_OK) return fail(rc);
    }
    const size_t v64b = (size_t)N * p->w64.Kp * sizeof(double);
    if ((rc = dalloc(p, &p->v64, v64b)) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->r64, v64b)) != BURA_OK) return fail(rc);
    const size_t max_blocks = (size_t)nsm * std::max(8, o.blocks_per_sm);
    const size_t max_groups = (max_blocks + kRedGroup - 1) / kRedGroup;
    // block partials (FP32 data: half as much again for the third words), or block and group partials
    const size_t max_partials = max_blocks + std::max(max_groups, (max_blocks + 1) / 2);
    if ((rc = dalloc(p, &p->partial, max_partials * KMAXP * sizeof(double))) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->tickets, (max_groups + 2) * sizeof(unsigned int))) != BURA_OK) return fail(rc);
    if (cudaMemset(p->tickets, 0, (max_groups + 2) * sizeof(unsigned int)) != cudaSuccess) return fail(BURA_ECUDA);
    p->red_nblk = p->tickets + max_groups + 1;
    if ((rc = dalloc(p, &p->red_out, KMAXP * sizeof(double))) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->scale, KMAXP * sizeof(double))) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->invscale, KMAXP * sizeof(double))) != BURA_OK) return fail(rc);
    if (o.precision == BURA_PREC_MIXED && o.refine == BURA_REFINE_DF && (rc = build_df(p)) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->scal_outer, sizeof(Scal))) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->cdev, KMAXP * sizeof(double))) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->ocfg, sizeof(OuterCfg))) != BURA_OK) return fail(rc);
    if ((rc = dalloc(p, &p->ostate, sizeof(OuterState))) != BURA_OK) return fail(rc);
    if (cudaMemset(p->ostate, 0, sizeof(OuterState)) != cudaSuccess) return fail(BURA_ECUDA);
    if (cudaMallocHost(&p->hstate, sizeof(OuterState)) != cudaSuccess) { p->hstate = nullptr; return fail(BURA_ENOMEM); }
    std::memset(p->hstate, 0, sizeof(OuterState));
    if ((rc = upload_outer(p)) != BURA_OK) return fail(rc);
    if ((rc = build_resident(p)) != BURA_OK) return fail(rc);
    if (cudaEventCreateWithFlags(&p->done, cudaEventDisableTiming) != cudaSuccess) {
        p->done = nullptr;
        return fail(BURA_ECUDA);
    }
    if (cudaMallocHost(&p->hscal, sizeof(Scal)) != cudaSuccess) { p->hscal = nullptr; return fail(BURA_ENOMEM); }
    if (cudaMallocHost(&p->hbuf, 4 * KMAXP * sizeof(double)) != cudaSuccess) { p->hbuf = nullptr; return fail(BURA_ENOMEM); }
    if (cudaDeviceSynchronize() != cudaSuccess) return fail(BURA_ECUDA);
    p->st.Lambda = p->Lambda;
    p->st.E = p->E;
    p->st.k = p->K - 1;
    p->st.levels = (int)p->hl.size();
    p->st.lambda_lo = p->lambda_lo;
    *out = p;
    return BURA_OK;
}

// A plan for the K weights c and shifts d (d[0] >= d[1] >= ... , all <= 0, c > 0) of a partial-fraction
// sum u = sum_j c_j (A - d_j I)^{-1} f on the grid: scaling, multigrid hierarchy, tables, workspaces.
int setup_plan(const bura_grid* grid, const double* const* faces, long long N, int K, const double* c,
               const double* d, double E, double alpha, bool shifts_only, const bura_options& o, bura_plan** out) {
    const int dim = grid->dim;
    const bool var = grid->coef_kind == BURA_COEF_FACES;
    if (o.coarse_kernel == BURA_COARSE_FDIAG && (dim != 2 || var)) return BURA_EINVAL;
    std::shared_lock<std::shared_mutex> guard(g_capture_guard);
    bura_plan* p = new (std::nothrow) bura_plan();
    if (!p) return BURA_ENOMEM;
    auto fail = [&](int rc) { destroy_plan(p); return rc; };
    p->dim = dim;
    p->var = var;
    p->k = K - 1;
    p->K = K;
    p->alpha = alpha;
    p->shifts_only = shifts_only;
    p->opt = o;
    p->wait_cycles = o.tma_wait_cycles;
    p->c.assign(c, c + K);
    p->d.assign(d, d + K);
    p->E = E;
    int rc = BURA_OK;
    // fine level
    HostLevel h0;
    h0.n[0] = grid->n[0];
    h0.n[1] = grid->n[1];
    h0.n[2] = dim == 3 ? grid->n[2] : 1;
    h0.N = N;
    for (int a = 0; a < 3; ++a) h0.h[a] = 1.0 / (h0.n[a] + 1);
    if (var) {
        const size_t sz[3] = {(size_t)h0.n[2] * h0.n[1] * (h0.n[0] + 1), (size_t)h0.n[2] * (h0.n[1] + 1) * h0.n[0],
                              (size_t)(h0.n[2] + 1) * h0.n[1] * h0.n[0]};
        for (int a = 0; a < dim; ++a) {
            if (!faces[a]) return fail(BURA_EINVAL);
            h0.a[a].assign(faces[a], faces[a] + sz[a]);
            for (double v : h0.a[a])
                if (!(v > 0) || !std::isfinite(v)) return fail(BURA_EINVAL);
        }
    }
    p->Lambda = gershgorin(h0, dim, var);
    p->hl.push_back(h0);
    for (;;) {  // coarsen while every size is odd and >= 3
        const HostLevel& f = p->hl.back();
        bool ok = true;
        for (int a = 0; a < dim; ++a) ok = ok && (f.n[a] >= 3) && (f.n[a] % 2 == 1);
        if (!ok) break;
        HostLevel c;
        for (int a = 0; a < 3; ++a) c.n[a] = (a < dim) ? (f.n[a] - 1) / 2 : 1;
        c.N = (long long)c.n[0] * c.n[1] * c.n[2];
        for (int a = 0; a < 3; ++a) c.h[a] = 1.0 / (c.n[a] + 1);
        if (var) coarsen_faces(f, c, dim);
        p->hl.push_back(std::move(c));
    }
    for (auto& h : p->hl) {
        for (int a = 0; a < 3; ++a) h.w[a] = (a < dim) ? 1.0 / (h.h[a] * h.h[a] * p->Lambda) : 0.0;
        level_bounds(h, dim, var, p->Lambda);
    }
    p->lambda_lo = p->hl[0].lmin * (1.0 - 1e-12);
    p->out_scale = o.unscaled ? std::pow(p->Lambda, -alpha) : 1.0;

    return setup_device(p, N, out);
}


}  // namespace

extern "C" {

int bura_setup(const bura_grid* grid, const double* const* faces, double alpha, int k, const bura_options* opt,
               bura_plan** out) {
    if (!out) return BURA_EINVAL;
    *out = nullptr;
    long long N = 0;
    CA(check_grid(grid, faces, &N));
    if (!(alpha > 0 && alpha < 1) || k < 1 || k > BURA_MAX_K) return BURA_EINVAL;
    bura_options o;
    bura_default_options(&o);
    if (opt) o = *opt;
    CA(check_options(o));
    std::vector<double> c(k + 1, 0.0), d(k + 1, 0.0);
    double E = 0.0;
    CA(bura_rational(alpha, k, c.data(), d.data(), &E));
    return setup_plan(grid, faces, N, k + 1, c.data(), d.data(), E, alpha, false, o, out);
}

int bura_setup_csr(const bura_csr* A, double alpha, int k, const bura_options* opt, bura_plan** out) {
    if (!out) return BURA_EINVAL;
    *out = nullptr;
    if (!A || !A->row_ptr || !A->col || !A->val || A->n < 1 || A->nnz < A->n) return BURA_EINVAL;
    if (!(alpha > 0 && alpha < 1) || k < 1 || k > BURA_MAX_K) return BURA_EINVAL;
    if ((long long)A->n * 16 >= (1LL << 31) || A->nnz >= (1LL << 31)) return BURA_ERANGE;
    if (!(A->lambda_min >= 0) || !std::isfinite(A->lambda_min)) return BURA_EINVAL;
    bura_options o;
    bura_default_options(&o);
    if (opt) o = *opt;
    CA(check_options(o));
    if (o.refine == BURA_REFINE_DF) return BURA_EINVAL;  // double-float refinement: grids only
    if (o.coarse_kernel == BURA_COARSE_FDIAG) return BURA_EINVAL;  // a grid operator's coarse solve
    // structure: offsets from 0 to nnz, columns in range, finite values, a positive diagonal in every row,
    // and symmetry (the entries sorted by (row, col) and by (col, row) must agree)
    const int n = A->n;
    const long long nnz = A->nnz;
    if (A->row_ptr[0] != 0 || A->row_ptr[n] != nnz) return BURA_EINVAL;
    HostLevel h0;
    h0.n[0] = n;
    h0.n[1] = h0.n[2] = 1;
    h0.N = n;
    h0.h[0] = h0.h[1] = h0.h[2] = 0.0;
    h0.w[0] = h0.w[1] = h0.w[2] = 0.0;
    h0.rowptr.assign(A->row_ptr, A->row_ptr + n + 1);
    h0.col.assign(A->col, A->col + nnz);
    h0.diag.assign(n, 0.0);
    h0.rowsum.assign(n, 0.0);
    std::vector<long long> ord((size_t)nnz);
    for (int i = 0; i < n; ++i) {
        if (A->row_ptr[i + 1] < A->row_ptr[i]) return BURA_EINVAL;
        for (int q = A->row_ptr[i]; q < A->row_ptr[i + 1]; ++q) {
            const int j = A->col[q];
            const double v = A->val[q];
            if (j < 0 || j >= n || !std::isfinite(v)) return BURA_EINVAL;
            if (j == i) h0.diag[i] += v;
            h0.rowsum[i] += std::fabs(v);
        }
    }
    for (int i = 0; i < n; ++i)
        if (!(h0.diag[i] > 0)) return BURA_EINVAL;
    {
        struct E { int r, c; double v; };
        std::vector<E> a, t;
        a.reserve((size_t)nnz);
        t.reserve((size_t)nnz);
        for (int i = 0; i < n; ++i)
            for (int q = A->row_ptr[i]; q < A->row_ptr[i + 1]; ++q) {
                a.push_back({i, A->col[q], A->val[q]});
                t.push_back({A->col[q], i, A->val[q]});
            }
        auto lt = [](const E& x, const E& y) { return x.r != y.r ? x.r < y.r : x.c < y.c; };
        std::sort(a.begin(), a.end(), lt);
        std::sort(t.begin(), t.end(), lt);
        double amax = 0.0;
        for (const E& e : a) amax = std::max(amax, std::fabs(e.v));
        for (size_t q = 0; q < a.size(); ++q)
            if (a[q].r != t[q].r || a[q].c != t[q].c || std::fabs(a[q].v - t[q].v) > 1e-14 * amax) return BURA_EINVAL;
    }
    double Lambda = 0.0;
    for (int i = 0; i < n; ++i) Lambda = std::max(Lambda, h0.rowsum[i]);
    h0.val.resize((size_t)nnz);
    for (long long q = 0; q < nnz; ++q) h0.val[q] = A->val[q] / Lambda;
    double dmax = 0.0;
    for (int i = 0; i < n; ++i) {
        h0.diag[i] /= Lambda;
        h0.rowsum[i] /= Lambda;
        dmax = std::max(dmax, h0.diag[i]);
    }
    h0.amax = dmax;
    h0.lmin = A->lambda_min / Lambda;
    std::vector<double> c(k + 1, 0.0), d(k + 1, 0.0);
    double E = 0.0;
    CA(bura_rational(alpha, k, c.data(), d.data(), &E));
    std::shared_lock<std::shared_mutex> guard(g_capture_guard);
    bura_plan* p = new (std::nothrow) bura_plan();
    if (!p) return BURA_ENOMEM;
    p->dim = 0;
    p->var = true;
    p->k = k;
    p->K = k + 1;
    p->alpha = alpha;
    p->opt = o;
    p->wait_cycles = o.tma_wait_cycles;
    p->c = c;
    p->d = d;
    p->E = E;
    p->Lambda = Lambda;
    p->lambda_lo = h0.lmin > 0 ? h0.lmin * (1.0 - 1e-12) : 0.0;
    p->out_scale = o.unscaled ? std::pow(Lambda, -alpha) : 1.0;
    p->hl.push_back(std::move(h0));
    return setup_device(p, n, out);
}

int bura_scale(const bura_grid* grid, const double* const* faces, double* Lambda) {
    long long N = 0;
    if (!Lambda) return BURA_EINVAL;
    CA(check_grid(grid, faces, &N));
    const int dim = grid->dim;
    const bool var = grid->coef_kind == BURA_COEF_FACES;
    HostLevel h0;
    h0.n[0] = grid->n[0];
    h0.n[1] = grid->n[1];
    h0.n[2] = dim == 3 ? grid->n[2] : 1;
    h0.N = N;
    for (int a = 0; a < 3; ++a) h0.h[a] = 1.0 / (h0.n[a] + 1);
    if (var) {
        const size_t sz[3] = {(size_t)h0.n[2] * h0.n[1] * (h0.n[0] + 1), (size_t)h0.n[2] * (h0.n[1] + 1) * h0.n[0],
                              (size_t)(h0.n[2] + 1) * h0.n[1] * h0.n[0]};
        for (int a = 0; a < dim; ++a) {
            if (!faces[a]) return BURA_EINVAL;
            h0.a[a].assign(faces[a], faces[a] + sz[a]);
            for (double v : h0.a[a])
                if (!(v > 0) || !std::isfinite(v)) return BURA_EINVAL;
        }
    }
    *Lambda = gershgorin(h0, dim, var);
    return BURA_OK;
}

int bura_quadrature_bp15(double alpha, double kprime, double Lambda, int cap, double* c, double* d, int* n) {
    if (!n || !(alpha > 0 && alpha < 1) || !(kprime > 0) || !std::isfinite(kprime) || !(Lambda > 0) ||
        !std::isfinite(Lambda) || cap < 0 || (cap > 0 && (!c || !d)))
        return BURA_EINVAL;
    // node counts below and above l = 0 that balance the three error terms of the quadrature
    const double lo = std::ceil(M_PI * M_PI / (4.0 * alpha * kprime * kprime));
    const double hi = std::ceil(M_PI * M_PI / (4.0 * (1.0 - alpha) * kprime * kprime));
    if (lo + hi + 1 > 1e6) return BURA_ERANGE;
    const int m = (int)lo, M = (int)hi;
    *n = m + M + 1;
    if (*n > cap) return BURA_ERANGE;
    const double pre = 2.0 * kprime * std::sin(M_PI * alpha) / M_PI * std::pow(Lambda, alpha - 1.0);
    for (int l = -m; l <= M; ++l) {
        // (e^{-2lk'} I + Atilde)^{-1} = Lambda^{-1} (A - d_l I)^{-1} with d_l = -e^{-2lk'} / Lambda
        c[l + m] = pre * std::exp(2.0 * (alpha - 1.0) * l * kprime);
        d[l + m] = -std::exp(-2.0 * l * kprime) / Lambda;
    }
    return BURA_OK;
}

int bura_setup_shifts(const bura_grid* grid, const double* const* faces, int nsys, const double* c, const double* d,
                      const bura_options* opt, bura_plan** out) {
    if (!out) return BURA_EINVAL;
    *out = nullptr;
    long long N = 0;
    CA(check_grid(grid, faces, &N));
    if (!c || !d || nsys < 1) return BURA_EINVAL;
    if (nsys > BURA_MAX_K + 1) return BURA_ERANGE;
    bura_options o;
    bura_default_options(&o);
    if (opt) o = *opt;
    CA(check_options(o));
    if (o.unscaled) return BURA_EINVAL;  // no fractional power to undo the scaling with
    std::vector<std::pair<double, double>> cd;
    for (int j = 0; j < nsys; ++j) {
        if (!(c[j] > 0) || !std::isfinite(c[j]) || !(d[j] <= 0) || !std::isfinite(d[j])) return BURA_EINVAL;
        cd.push_back({d[j], c[j]});
    }
    // the system nearest d = 0 (the hardest) first, as the BURA poles d_0 = 0 > d_1 > ...
    std::stable_sort(cd.begin(), cd.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    std::vector<double> cs(nsys), ds(nsys);
    for (int j = 0; j < nsys; ++j) {
        ds[j] = cd[j].first;
        cs[j] = cd[j].second;
    }
    return setup_plan(grid, faces, N, nsys, cs.data(), ds.data(), 0.0, 0.0, true, o, out);
}

}  // extern "C"

namespace {

// The output stage of the device-driven solve and its outcome copy: u = sum_j c_j v_j (or the systems)
// after the solve graph, then the solve record into the pinned mirror, then the plan's event.
int enqueue_device_solve(bura_plan* p, const double* f, double* u, double* V, double tol, cudaStream_t s, int accumulate) {
    if (!(tol > 0)) return BURA_EINVAL;
    CK(cudaSetDevice(p->dev));
    if (p->res_on) {
        const double N = (double)p->hl[0].N, vb = N * p->K * 8.0;
        cudaError_t e = cudaSuccess;
        p->tr.launches = 0;
        traced(p, K_RES, true, true, N * 8.0 + vb, s, [&] { e = launch_resident(p->res, p->K, f, tol, s); });
        CK(e);
        traced(p, K_RESOUT, false, true, V ? 2.0 * vb : vb + N * 8.0 * (accumulate ? 2.0 : 1.0), s,
               [&] { e = launch_resident_out(p->res, p->K, p->cdev, u, V, accumulate, p->hstate, s); });
        CK(e);
        CK(cudaEventRecord(p->done, s));
        p->pending = true;
        return BURA_OK;
    }
    CA(solve_device(p, f, tol, s));
    const long long N = p->hl[0].N;
    if (V) launch_gather_systems(N, p->w64.Kp, p->K, solution_vectors(p), V, s);
    else launch_weighted_sum(N, p->w64.Kp, p->K, solution_vectors(p), p->cdev, u, accumulate, s);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(p->hstate, p->ostate, sizeof(OuterState), cudaMemcpyDeviceToHost, s));
    CK(cudaEventRecord(p->done, s));
    p->pending = true;
    return BURA_OK;
}

// The same, to its end.  A one-launch solve is this with profiling on too (its launches timed), so that a profile is of
// the kernels that the plan's solves run.
int run_device_solve(bura_plan* p, const double* f, double* u, double* V, double tol, cudaStream_t s, int accumulate) {
    CA(enqueue_device_solve(p, f, u, V, tol, s, accumulate));
    const int rc = read_outcome(p);
    if (p->tr.on) {
        CK(cudaStreamSynchronize(s));
        collect_trace(p);
    }
    return rc;
}

// The solve and the output sum u = sum_j c_j v_j (accumulate = 1: u += ...), stream-ordered on s.
int solve_into(bura_plan* p, const double* f, double* u, double tol, cudaStream_t s, int accumulate) {
    if (device_driven(p) || p->res_on) return run_device_solve(p, f, u, nullptr, tol, s, accumulate);
    int rc = solve_core(p, f, tol, s);
    if (rc != BURA_OK && rc != BURA_ENOCONV) return rc;
    const double N = (double)p->hl[0].N;
    const double wbytes = N * p->K * 8.0 + N * 8.0 * (accumulate ? 2.0 : 1.0);
    if (df_solution(p))
        traced(p, K_WSUM, false, true, wbytes, s, [&] {
            launch_weighted_sum_df(p->hl[0].N, p->w32.Kp, p->K, p->vh[p->vcur], p->vl[p->vcur], p->cwh, p->cwl, u,
                                   accumulate, s);
        });
    else
        traced(p, K_WSUM, false, true, wbytes, s,
               [&] { launch_weighted_sum(p->hl[0].N, p->w64.Kp, p->K, solution_vectors(p), p->cdev, u, accumulate, s); });
    CKL();
    CK(cudaEventRecord(p->done, s));
    p->st.launches = p->tr.launches;
    if (p->tr.on) {
        CK(cudaStreamSynchronize(s));
        collect_trace(p);
    }
    return rc;
}

// Plans of one grid and operator on one device (bura_solve_chain, bura_solve_sum).
bool same_operator(const bura_plan* a, const bura_plan* b) {
    return a->dim == b->dim && a->var == b->var && a->hl[0].n[0] == b->hl[0].n[0] && a->hl[0].n[1] == b->hl[0].n[1] &&
           a->hl[0].n[2] == b->hl[0].n[2] && a->dev == b->dev;
}

}  // namespace

extern "C" {

int bura_solve(bura_plan* p, const double* f, double* u, double tol, void* stream) {
    if (!p || !f || !u) return BURA_EINVAL;
    return solve_into(p, f, u, tol, reinterpret_cast<cudaStream_t>(stream), 0);
}

int bura_solve_async(bura_plan* p, const double* f, double* u, double tol, void* stream) {
    if (!p || !f || !u) return BURA_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (!device_driven(p)) {  // host-driven paths (double-float refinement, profiling) finish in the call
        const int rc = solve_into(p, f, u, tol, s, 0);
        p->st.launches = p->tr.launches;
        return rc == BURA_ENOCONV ? BURA_OK : rc;
    }
    return enqueue_device_solve(p, f, u, nullptr, tol, s, 0);
}

int bura_solve_wait(bura_plan* p) {
    if (!p) return BURA_EINVAL;
    if (!p->pending) return p->last_status;
    p->last_status = read_outcome(p);
    return p->last_status;
}

int bura_solve_sum(bura_plan* const* plans, int n, const double* f, double* u, double tol, void* stream) {
    if (!plans || n < 1 || !f || !u || !(tol > 0)) return BURA_EINVAL;
    for (int i = 0; i < n; ++i)
        if (!plans[i] || !same_operator(plans[i], plans[0])) return BURA_EINVAL;
    if (f == u && n > 1) return BURA_EINVAL;  // every term reads f after the first has written u
    int out = BURA_OK;
    for (int i = 0; i < n; ++i) {
        const int rc = solve_into(plans[i], f, u, tol, reinterpret_cast<cudaStream_t>(stream), i > 0 ? 1 : 0);
        if (rc != BURA_OK && rc != BURA_ENOCONV) return rc;
        if (rc == BURA_ENOCONV) out = BURA_ENOCONV;
    }
    return out;
}

int bura_set_tma_wait_cycles(bura_plan* p, long long cycles) {
    if (!p || cycles < 0) return BURA_EINVAL;
    p->wait_cycles = cycles;  // read by the next solve's CG state records (host-driven) or controller (captured)
    std::shared_lock<std::shared_mutex> guard(g_capture_guard);
    CK(cudaSetDevice(p->dev));
    CK(cudaEventSynchronize(p->done));
    return upload_outer(p);
}

int bura_solve_chain(bura_plan* const* plans, int n, const double* f, double* u, double tol, void* stream) {
    if (!plans || n < 1 || !f || !u || !(tol > 0)) return BURA_EINVAL;
    for (int i = 0; i < n; ++i)
        if (!plans[i] || !same_operator(plans[i], plans[0])) return BURA_EINVAL;
    int out = BURA_OK;
    const double* in = f;
    for (int i = 0; i < n; ++i) {
        const int rc = bura_solve(plans[i], in, u, tol, stream);  // bura_solve reads f before writing u
        if (rc != BURA_OK && rc != BURA_ENOCONV) return rc;
        if (rc == BURA_ENOCONV) out = BURA_ENOCONV;
        in = u;
    }
    return out;
}

int bura_solve_host(bura_plan* p, const double* f, double* u, double tol, void* stream) {
    if (!p || !f || !u) return BURA_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const size_t nb = (size_t)p->hl[0].N * sizeof(double);
    CK(cudaSetDevice(p->dev));
    if (!p->fdev) {
        std::shared_lock<std::shared_mutex> guard(g_capture_guard);
        CA(dalloc(p, &p->fdev, nb));
        CA(dalloc(p, &p->udev, nb));
    }
    CK(cudaMemcpyAsync(p->fdev, f, nb, cudaMemcpyHostToDevice, s));
    int rc = bura_solve(p, p->fdev, p->udev, tol, stream);
    if (rc != BURA_OK && rc != BURA_ENOCONV) return rc;
    CK(cudaMemcpyAsync(u, p->udev, nb, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    return rc;
}

int bura_solve_systems(bura_plan* p, const double* f, double* V, double tol, void* stream) {
    if (!p || !f || !V) return BURA_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (device_driven(p) || p->res_on) return run_device_solve(p, f, nullptr, V, tol, s, 0);
    int rc = solve_core(p, f, tol, s);
    if (rc != BURA_OK && rc != BURA_ENOCONV) return rc;
    traced(p, K_GATHER, false, true, 2.0 * p->hl[0].N * p->K * 8.0, s, [&] {
        if (df_solution(p)) launch_gather_df(p->hl[0].N, p->w32.Kp, p->K, p->vh[p->vcur], p->vl[p->vcur], V, s);
        else launch_gather_systems(p->hl[0].N, p->w64.Kp, p->K, solution_vectors(p), V, s);
    });
    CKL();
    CK(cudaEventRecord(p->done, s));
    p->st.launches = p->tr.launches;
    if (p->tr.on) {
        CK(cudaStreamSynchronize(s));
        collect_trace(p);
    }
    return rc;
}

}  // extern "C"

struct bura_batch {
    int dev = 0;
    std::vector<bura_plan*> plans;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<cudaStream_t> streams;
    cudaEvent_t fork = nullptr;
    std::vector<cudaEvent_t> joins;
};

namespace {

void free_batch(bura_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (cudaEvent_t e : b->joins) cudaEventDestroy(e);
    if (b->fork) cudaEventDestroy(b->fork);
    for (cudaStream_t s : b->streams) cudaStreamDestroy(s);
    delete b;
}

// Capture every problem of the batch into one graph: branch i % S of S parallel branches holds problem
// i's whole device-driven solve (its solve record, ||f||, controller, WHILE loops, output sum and outcome
// copy), so one launch of the graph solves them all, S at a time.
int build_batch(bura_batch* b, const double* const* f, double* const* u, double tol, int S) {
    std::unique_lock<std::shared_mutex> lock(g_capture_guard);
    const int n = (int)b->plans.size();
    b->streams.assign(S, nullptr);
    for (int i = 0; i < S; ++i) CK(cudaStreamCreateWithFlags(&b->streams[i], cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming));
    b->joins.assign(S, nullptr);
    for (int i = 0; i < S; ++i) CK(cudaEventCreateWithFlags(&b->joins[i], cudaEventDisableTiming));
    CK(cudaGraphCreate(&b->graph, 0));
    cudaStream_t s0 = b->streams[0];
    std::vector<BodyTask> tasks;
    for (bura_plan* p : b->plans) p->s_fixed = p->s_outer = p->s_body = 0;
    CK(cudaStreamBeginCaptureToGraph(s0, b->graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    int rc = BURA_OK;
    cudaError_t e = cudaEventRecord(b->fork, s0);
    for (int i = 1; i < S && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(b->streams[i], b->fork, 0);
    if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    for (int i = 0; i < n && rc == BURA_OK; ++i) {
        bura_plan* p = b->plans[i];
        cudaStream_t s = b->streams[i % S];
        const bool was_on = p->tr.on;
        const long long before = p->tr.launches;
        p->tr.on = false;
        if (p->res_on) {
            e = launch_resident(p->res, p->K, f[i], tol, s);
            if (e == cudaSuccess) e = launch_resident_out(p->res, p->K, p->cdev, u[i], nullptr, 0, p->hstate, s);
            p->tr.on = was_on;
            if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
            continue;
        }
        launch_solve_params(p->ostate, f[i], tol, s);
        rc = capture_solve_top(p, s, tasks);
        p->tr.on = was_on;
        p->tr.launches = before;
        if (rc != BURA_OK) break;
        launch_weighted_sum(p->hl[0].N, p->w64.Kp, p->K, solution_vectors(p), p->cdev, u[i], 0, s);
        e = cudaMemcpyAsync(p->hstate, p->ostate, sizeof(OuterState), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    }
    for (int i = 1; i < S && rc == BURA_OK; ++i) {
        e = cudaEventRecord(b->joins[i], b->streams[i]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s0, b->joins[i], 0);
        if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    }
    cudaGraph_t done = nullptr;
    e = cudaStreamEndCapture(s0, &done);
    if (rc == BURA_OK && e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
    if (rc == BURA_OK) rc = capture_bodies(tasks);
    if (rc == BURA_OK) {
        e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; b->exec = nullptr; }
    }
    if (rc != BURA_OK) {
        cudaGetLastError();
        b->graph = nullptr;  // a failed capture's partial graph is left allocated (see build_graph)
    }
    return rc;
}

}  // namespace

extern "C" {

int bura_autotune(const bura_grid* grid, const double* const* faces, double alpha, int k, const bura_options* base,
                  double tol, int trials, bura_options* best, double* best_ms) {
    if (!grid || !best || !(alpha > 0 && alpha < 1) || k < 1 || k > BURA_MAX_K || !(tol > 0) || trials < 1)
        return BURA_EINVAL;
    long long N = 0;
    CA(check_grid(grid, faces, &N));
    bura_options b0;
    bura_default_options(&b0);
    if (base) b0 = *base;
    CA(check_options(b0));
    // candidates: smoother degree 2 or 3, the Chebyshev interval by dimension or twice as wide, and on 2-D
    // constant-coefficient grids the TMA-staged tiles or the grid-stride sweeps
    std::vector<bura_options> cand;
    const double r0 = b0.smoother_ratio > 0 ? b0.smoother_ratio : (grid->dim == 3 ? 8.0 : 4.0);
    const bool tiles = grid->dim == 2 && grid->coef_kind == BURA_COEF_CONSTANT && b0.precision == BURA_PREC_MIXED;
    for (int deg = 2; deg <= 3; ++deg)
        for (int wide = 0; wide <= 1; ++wide)
            for (int sw = 0; sw <= (tiles ? 1 : 0); ++sw) {
                bura_options o = b0;
                o.smoother_degree = deg;
                o.smoother_ratio = wide ? 2.0 * r0 : r0;
                o.sweeps = sw ? BURA_SWEEP_GRID : BURA_SWEEP_AUTO;
                cand.push_back(o);
            }
    // a fixed pseudo-random right-hand side in [-1, 1] (the timing does not depend on its values)
    std::vector<double> fh((size_t)N);
    unsigned long long x = 0x9e3779b97f4a7c15ull;
    for (auto& v : fh) {
        x = x * 6364136223846793005ull + 1442695040888963407ull;
        v = (double)(x >> 11) / 9007199254740992.0 * 2.0 - 1.0;
    }
    double* fd = nullptr;
    double* ud = nullptr;
    cudaStream_t s = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    auto cleanup = [&]() {
        if (fd) cudaFree(fd);
        if (ud) cudaFree(ud);
        if (s) cudaStreamDestroy(s);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
    };
    {
        std::shared_lock<std::shared_mutex> guard(g_capture_guard);
        if (cudaMalloc(&fd, N * sizeof(double)) != cudaSuccess || cudaMalloc(&ud, N * sizeof(double)) != cudaSuccess ||
            cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
            cudaEventCreate(&e1) != cudaSuccess ||
            cudaMemcpy(fd, fh.data(), N * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess) {
            cleanup();
            return BURA_ENOMEM;
        }
    }
    double bms = 1e300;
    int found = 0;
    for (const bura_options& o : cand) {
        bura_plan* p = nullptr;
        if (bura_setup(grid, faces, alpha, k, &o, &p) != BURA_OK) continue;
        bool ok = bura_solve(p, fd, ud, tol, s) == BURA_OK;  // warm-up: captures the graphs
        std::vector<float> t;
        for (int i = 0; ok && i < trials; ++i) {
            float ms = 0.f;
            ok = cudaEventRecord(e0, s) == cudaSuccess && bura_solve_async(p, fd, ud, tol, s) == BURA_OK &&
                 cudaEventRecord(e1, s) == cudaSuccess && bura_solve_wait(p) == BURA_OK &&
                 cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
            t.push_back(ms);
        }
        bura_destroy(p);
        if (!ok) continue;
        std::sort(t.begin(), t.end());
        const double med = t[t.size() / 2];
        if (med < bms) {
            bms = med;
            *best = o;
            found = 1;
        }
    }
    cleanup();
    if (!found) return BURA_ENOCONV;
    if (best_ms) *best_ms = bms;
    return BURA_OK;
}

int bura_batch_create(bura_plan* const* plans, const double* const* f, double* const* u, int n, double tol,
                      int branches, bura_batch** out) {
    if (!out) return BURA_EINVAL;
    *out = nullptr;
    if (n < 1 || !plans || !f || !u || !(tol > 0) || branches < 0) return BURA_EINVAL;
    for (int i = 0; i < n; ++i) {
        if (!plans[i] || !f[i] || !u[i]) return BURA_EINVAL;
        if (!device_driven(plans[i]) || plans[i]->dev != plans[0]->dev) return BURA_EINVAL;
        for (int j = 0; j < i; ++j)
            if (plans[j] == plans[i]) return BURA_EINVAL;
    }
    bura_batch* b = new (std::nothrow) bura_batch();
    if (!b) return BURA_ENOMEM;
    b->dev = plans[0]->dev;
    b->plans.assign(plans, plans + n);
    cudaError_t e = cudaSetDevice(b->dev);
    if (e != cudaSuccess) { g_last = e; delete b; return BURA_ECUDA; }
    const int S = std::max(1, std::min(branches > 0 ? branches : 64, n));
    const int rc = build_batch(b, f, u, tol, S);
    if (rc != BURA_OK) { free_batch(b); return rc; }
    *out = b;
    return BURA_OK;
}

int bura_batch_run(bura_batch* b, void* stream) {
    if (!b) return BURA_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CK(cudaSetDevice(b->dev));
    CK(cudaGraphLaunch(b->exec, s));
    for (bura_plan* p : b->plans) {
        CK(cudaEventRecord(p->done, s));
        p->pending = true;
    }
    return BURA_OK;
}

int bura_batch_wait(bura_batch* b, int* status) {
    if (!b) return BURA_EINVAL;
    int rc = BURA_OK;
    for (size_t i = 0; i < b->plans.size(); ++i) {
        const int st = read_outcome(b->plans[i]);
        if (status) status[i] = st;
        if (st != BURA_OK && (rc == BURA_OK || rc == BURA_ENOCONV)) rc = st;
    }
    return rc;
}

int bura_batch_destroy(bura_batch* b) {
    if (!b) return BURA_OK;
    std::shared_lock<std::shared_mutex> guard(g_capture_guard);
    cudaSetDevice(b->dev);
    for (bura_plan* p : b->plans) cudaEventSynchronize(p->done);
    free_batch(b);
    return BURA_OK;
}

int bura_solve_batch(bura_plan* const* plans, const double* const* f, double* const* u, int n, double tol,
                     int nworkers, int* status) {
    if (n < 0 || nworkers < 0 || (n > 0 && (!plans || !f || !u))) return BURA_EINVAL;
    for (int i = 0; i < n; ++i) {
        if (!plans[i] || !f[i] || !u[i]) return BURA_EINVAL;
        for (int j = 0; j < i; ++j)
            if (plans[j] == plans[i]) return BURA_EINVAL;  // a plan's buffers serve one solve at a time
    }
    if (n == 0) return BURA_OK;
    bool graphable = tol > 0;
    for (int i = 0; i < n; ++i) graphable = graphable && device_driven(plans[i]) && plans[i]->dev == plans[0]->dev;
    if (graphable) {  // one graph: every problem a branch of device-driven solves
        bura_batch* b = nullptr;
        int rc = bura_batch_create(plans, f, u, n, tol, nworkers, &b);
        if (rc == BURA_OK) {
            cudaStream_t s = nullptr;
            cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, s);
            if (e == cudaSuccess)
                for (bura_plan* p : b->plans) {
                    cudaEventRecord(p->done, s);
                    p->pending = true;
                }
            if (e != cudaSuccess) { g_last = e; rc = BURA_ECUDA; }
            else rc = bura_batch_wait(b, status);
            if (s) { cudaStreamSynchronize(s); cudaStreamDestroy(s); }
            bura_batch_destroy(b);
        }
        return rc;
    }
    const int nw = std::max(1, std::min(nworkers > 0 ? nworkers : 16, n));
    std::vector<int> st(n, BURA_OK);
    std::atomic<int> next(0);
    std::mutex err_mutex;
    cudaError_t first_err = cudaSuccess;  // reported to the calling thread by bura_last_cuda_error
    auto worker = [&]() {
        // one stream per worker; the plans are taken in list order, each solved exactly as bura_solve
        // does it alone (its own buffers, deterministic reductions), so its result does not depend on
        // which other solves run beside it
        cudaStream_t s = nullptr;
        int dev = -1;
        for (;;) {
            const int i = next.fetch_add(1);
            if (i >= n) break;
            bura_plan* p = plans[i];
            if (p->dev != dev) {
                if (s) {
                    cudaStreamSynchronize(s);
                    cudaStreamDestroy(s);
                    s = nullptr;
                }
                cudaError_t e = cudaSetDevice(p->dev);
                if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
                if (e != cudaSuccess) {
                    s = nullptr;
                    g_last = e;
                    st[i] = BURA_ECUDA;
                    std::lock_guard<std::mutex> lock(err_mutex);
                    if (first_err == cudaSuccess) first_err = e;
                    continue;
                }
                dev = p->dev;
            }
            st[i] = bura_solve(p, f[i], u[i], tol, s);
            if (st[i] == BURA_ECUDA) {
                std::lock_guard<std::mutex> lock(err_mutex);
                if (first_err == cudaSuccess) first_err = g_last;
            }
        }
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
    };
    std::vector<std::thread> pool;
    pool.reserve(nw);
    for (int w = 0; w < nw; ++w) pool.emplace_back(worker);
    for (auto& t : pool) t.join();
    if (first_err != cudaSuccess) g_last = first_err;
    int rc = BURA_OK;
    for (int i = 0; i < n; ++i) {
        if (status) status[i] = st[i];
        if (st[i] != BURA_OK && (rc == BURA_OK || rc == BURA_ENOCONV)) rc = st[i];
    }
    return rc;
}

int bura_apply_shifted(bura_plan* p, const double* x, double* y, void* stream) {
    if (!p || !x || !y) return BURA_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CK(cudaSetDevice(p->dev));
    const long long N = p->hl[0].N;
    launch_scatter_systems(N, p->w64.Kp, p->K, x, p->v64, s);
    Ops<double>::apply_shifted(p->w64.g[0], p->w64.L[0], p->dim, p->var, p->v64, p->r64, p->w64.dsh, s);
    launch_gather_systems(N, p->w64.Kp, p->K, p->r64, y, s);
    CKL();
    return BURA_OK;
}

int bura_get_rational(const bura_plan* p, double* c, double* d, double* E) {
    if (!p || !c || !d) return BURA_EINVAL;
    for (int j = 0; j < p->K; ++j) { c[j] = p->c[j]; d[j] = p->d[j]; }
    if (E) *E = p->E;
    return BURA_OK;
}

int bura_get_stats(const bura_plan* cp, bura_stats* st) {
    if (!cp || !st) return BURA_EINVAL;
    bura_plan* p = const_cast<bura_plan*>(cp);  // reading a finished solve's outcome updates the cached stats
    if (p->pending) read_outcome(p);
    *st = p->st;
    st->device_bytes = p->dbytes;
    return BURA_OK;
}

int bura_set_profiling(bura_plan* p, int enable) {
    if (!p) return BURA_EINVAL;
    CK(cudaSetDevice(p->dev));
    Tracer& t = p->tr;
    if (enable && t.ev.empty()) {
        t.ev.resize(2 * kMaxTimed);
        for (auto& e : t.ev) CK(cudaEventCreate(&e));
    }
    t.on = enable != 0;
    t.pending.clear();
    if (enable) {
        std::memset(t.n, 0, sizeof(t.n));
        std::memset(t.ms, 0, sizeof(t.ms));
        std::memset(t.bytes, 0, sizeof(t.bytes));
    }
    return BURA_OK;
}

int bura_get_profile(const bura_plan* p, int max_entries, bura_kernel_prof* out, int* n_out) {
    if (!p || !n_out || (max_entries > 0 && !out)) return BURA_EINVAL;
    int n = 0;
    for (int slot = 0; slot < kSlots && n < max_entries; ++slot) {
        if (p->tr.n[slot] == 0) continue;
        out[n].name = kNames[slot / 4][(slot / 2) % 2][slot % 2];
        out[n].launches = p->tr.n[slot];
        out[n].ms = p->tr.ms[slot];
        out[n].bytes = p->tr.bytes[slot];
        ++n;
    }
    *n_out = n;
    return BURA_OK;
}

int bura_destroy(bura_plan* p) {
    if (!p) return BURA_OK;
    std::shared_lock<std::shared_mutex> guard(g_capture_guard);
    return destroy_plan(p);
}


int bura_retarget(bura_plan* p, double alpha) {
    if (!p || !(alpha > 0 && alpha < 1) || p->shifts_only) return BURA_EINVAL;
    std::vector<double> c(p->K, 0.0), d(p->K, 0.0);
    double E = 0.0;
    int rc = bura_rational(alpha, p->k, c.data(), d.data(), &E);
    if (rc != BURA_OK) return rc;
    if (d[0] != p->d[0]) return BURA_EREMEZ;  // d_0 = 0 fixes the coarsest smoothing degree
    std::shared_lock<std::shared_mutex> guard(g_capture_guard);
    CK(cudaSetDevice(p->dev));
    CK(cudaEventSynchronize(p->done));  // the last solve's kernels read the tables being replaced
    p->alpha = alpha;
    p->c = c;
    p->d = d;
    p->E = E;
    if (p->opt.unscaled) p->out_scale = std::pow(p->Lambda, -alpha);
    CA(upload_tables<double>(p, p->w64));
    if (p->opt.precision == BURA_PREC_MIXED) CA(upload_tables<float>(p, p->w32));
    if (p->dfop.ch) CA(upload_df_tables(p));
    CA(upload_outer(p));
    p->st.E = E;
    return BURA_OK;
}

const char* bura_last_cuda_error(void) {
    static thread_local char buf[256];
    snprintf(buf, sizeof(buf), "%s: %s", cudaGetErrorName(g_last), cudaGetErrorString(g_last));
    return buf;
}

const char* bura_strerror(int status) {
    switch (status) {
        case BURA_OK: return "success";
        case BURA_EINVAL: return "invalid argument";
        case BURA_ENOMEM: return "out of memory";
        case BURA_EREMEZ: return "rational approximation did not converge";
        case BURA_ENOTSPD: return "CG breakdown (operator not SPD or non-finite values)";
        case BURA_ENOCONV: return "tolerance not reached within the iteration caps";
        case BURA_ETIMEOUT: return "device-side wait timed out";
        case BURA_ECUDA: return "CUDA runtime error";
        case BURA_ERANGE: return "size above the supported maximum";
        default: return "unknown status";
    }
}

}  // extern "C"
