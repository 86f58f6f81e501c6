// A whole mixed-precision solve of a small 2-D plan in one launch, with every vector of the inner solver resident in
// shared memory (constant and variable coefficients), and the lower part of a larger 2-D plan's V-cycle as one launch.
//
// The shifted systems never exchange values, so each system gets a thread-block cluster of G CTAs of its own
// that runs the refinement loop, the multigrid-preconditioned CG inside it and all their decisions: the
// formulas are those of the grid kernels (kernels_tma.cu, fdiag.cu), of the reductions (kernels_impl.cuh) and
// of the controller (outer.cu), point by point; only the grouping of the dot products' sums differs (except in the first
// iteration: see grid_dot).
//
// Why: on grids of up to about 10^5 points the graph of grid kernels is bound by its own launches.  A 383 x 255,
// k = 8 solve is 108 launches in 812 us, 7.5 us each, for about 1 us of work each.  Here a vector is read from
// and written to shared memory, and a phase ends in an exchange of its edge rows.
//
// Layout: CTA g owns a slab of grid rows on every level: rows [a, b) of the exact level le and, on a level s
// levels above it, rows [a 2^s, b 2^s) (the last slab also the rows above (ny_le) 2^s), so that a coarse row and
// the fine rows 2J, 2J + 1 it sits on have one owner.  A vector is rows of ld floats (zero columns on either
// side, column 0 on an 8-byte boundary: a thread takes pairs of columns, with packed FP32 arithmetic) with halo
// rows: R (right-hand side, 3), X (pre-smoothed iterate, 2), Y (scratch, 1), D (direction and result, 2), and on
// level 0 the CG direction P (1).  With these halos the way down a level (both pre-smoothing steps, residual,
// restriction) and the way up (prolongation, both post-smoothing steps) need no other slab's values: halo rows
// are recomputed.
//
// Exchanges: what a phase produces is also stored into the halo rows of the slabs around it with st.async, which
// counts its bytes on an mbarrier of the receiver; a phase waits for the bytes of its own halo rows only (about
// 500 SM clocks less per exchange than a cluster barrier behind ordinary remote stores: 690 against 1196 measured
// with 16 CTAs of 512 threads).  Every (buffer, level) has an mbarrier of its own, used once per CG iteration;
// the reductions alternate between two.  A sender is never two uses ahead of a receiver: between two uses of a
// barrier lies a reduction, which needs every CTA's contribution.  For the same reason a halo row is only
// written when its last readers are done.  Every wait is bounded, and a wait that ran out is looked at before the sum it
// was for is used and once more at the end: the outcome is then BURA_ETIMEOUT.
//
// The exact solve of level le is fdiag.cu's fast diagonalization, every sum in the same order.
//
// Measured (GB300, one call of bura_solve, alpha = 0.5, tol 1e-6, graph of kernels -> here): 63^2, k = 5: 168 -> 49 us; 127^2,
// k = 6: 418 -> 120; 255^2, k = 7: 539 -> 233; 383 x 255, k = 8: 883 -> 405.  What is left is latency: a 127^2 iteration is
// some 10 us, of which the exact solve's four products and three exchanges take 3.6; the warps issue in 18 % of the cycles.
//
// Variable coefficients: every level's face and diagonal weights stay in the owner's shared memory too (three floats a
// point, so the largest grid is about 2 / 3 as wide), copied in while the first residual is taken.  The exact level is one
// dense product per system; grids above 31 put their last levels on the cluster's first CTA, which then runs them without
// an exchange (a boundary at 15 instead: 127^2 7 % slower, and 191^2 no longer fits).  63^2, k = 5: 945 -> 211 us; 127^2,
// k = 6: 1240 -> 276; 191^2: 1919 -> 387.
//
// V-cycle only: an iteration of a larger plan launches its levels from the first one of at most kResCycleMaxN points a
// side here.  About 10 of the launch's 25 us are its start (loading weights and tables), so it takes the place of five or
// more launches only: var 511^2, k = 7: 4.72 -> 3.79 ms; constant 511^2, three problems: 3.05 -> 2.96; 1023^2: 1.985 -> 1.964.
#include <cooperative_groups.h>

#include <algorithm>
#include <array>
#include <map>
#include <mutex>

#include "kernels_impl.cuh"
#include "refine_plan.h"
#include "tma.cuh"

namespace cg = cooperative_groups;

namespace bura {

namespace {

constexpr int kResMostWarps = 16;
constexpr int kHR = 3, kHX = 2, kHY = 1, kHD = 2, kHP = 1;  // halo rows of R, X, Y, D, P
constexpr int kSP = 64;                                     // leading dimension of the sine bases
constexpr int kStrip = 4;                                   // most rows a thread takes at a time

// The CG's sums and scalars are three-word sums (sum3.h): a scalar FP64 step that all 16 warps execute costs 256 SM clocks.

__device__ __forceinline__ unsigned map_rank(const void* p, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
// Asynchronous stores into CTA `rank`'s copy of *p, counted on its copy of *bar.
__device__ __forceinline__ void put(float* p, int rank, uint64_t* bar, float v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(map_rank(p, rank)),
                 "f"(v), "r"(map_rank(bar, rank))
                 : "memory");
}
__device__ __forceinline__ void put2(void* p, int rank, uint64_t* bar, float v0, float v1) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                     map_rank(p, rank)),
                 "f"(v0), "f"(v1), "r"(map_rank(bar, rank))
                 : "memory");
}
__device__ __forceinline__ void put4(float4* p, int rank, uint64_t* bar, float v0, float v1, float v2) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                     map_rank(p, rank)),
                 "f"(v0), "f"(v1), "f"(v2), "f"(0.f), "r"(map_rank(bar, rank))
                 : "memory");
}
// Wait for a phase whose bytes other CTAs of the cluster store; false if they have not come within `budget`.
__device__ __forceinline__ bool wait_bytes(uint64_t* bar, unsigned parity, long long budget) {
    const long long t0 = clock64();
    for (;;) {
        unsigned ok;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > budget) return false;
    }
}
// The same under a budget of the caller's: a phase that takes longer sets *late, and is waited for all the same, so that no
// store is in flight into a buffer that is in use again and the CTAs of a cluster stay together.  (Not inlined: 127^2 113.2 ->
// 112.6 us, with variable coefficients 268.7 -> 267.0.)
__device__ __noinline__ bool wait_timed(uint64_t* bar, unsigned parity, long long budget, int* late) {
    const long long t0 = clock64();
    const bool come = wait_bytes(bar, parity, max(budget, kTmaWaitCycles));
    if (clock64() - t0 > budget) *late = 1;
    return come;
}
// One float from global to shared memory, asynchronously; copies_done() waits for this thread's.
__device__ __forceinline__ void copy4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void st2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// Rows [y0, y1) of a level with ny rows, sh levels above the exact level (ne rows, re rows per slab), that
// slab t owns (empty for a slab past the last row).
__device__ __forceinline__ void slab(int t, int re, int ne, int sh, int ny, int& y0, int& y1) {
    const int a = min(t * re, ne), b = min(a + re, ne);
    y0 = a < ne ? a << sh : ny;
    y1 = b < ne ? b << sh : ny;
}

__host__ __device__ constexpr int even(int v) { return (v + 1) / 2 * 2; }
// Floats per row: two in front of column 0 and at least one zero column after the last.
__host__ __device__ constexpr int row_floats(int nx) { return 2 + even(nx + 1); }

struct Slab {
    int y0, y1;  // own rows
    int nx, ny, ld;
    __device__ __forceinline__ bool some() const { return y1 > y0; }
    // bytes of the rows that fill this slab's H halo rows
    __device__ __forceinline__ unsigned halo_bytes(int H) const {
        return some() ? (unsigned)((min(H, y0) + min(H, ny - y1)) * even(nx) * 4) : 0u;
    }
};

// A x at the column pair c of a row (u above, w below, l and r the values beside the pair), diag = 2 wx + 2 wy: the
// grid kernels' order of multiply-adds.
__device__ __forceinline__ float2 stencil2(float wx, float wy, float diag, float2 c, float l, float r, float2 u, float2 w) {
    float2 t = __fmul2_rn(dup(diag), c);
    t.x = fmaf(-wx, l, t.x);
    t.y = fmaf(-wx, c.x, t.y);
    t.x = fmaf(-wx, c.y, t.x);
    t.y = fmaf(-wx, r, t.y);
    t = __ffma2_rn(dup(-wy), u, t);
    return __ffma2_rn(dup(-wy), w, t);
}

// How a level's row sweeps are split over the warps: items of h rows x 64 columns, h the number (up to kStrip) whose
// rounds of items take the fewest row steps, for the own rows (kind 0) and with 1, 2 and 4 rows more (1, 2, 3).
template <int kResWarps>
struct Split {
    // (bytes: the static arrays take from the 227 KB of a CTA)
    unsigned char nch, q, m;  // column chunks; a warp's next item lies q rows of items and m chunks on
    unsigned char h[4];
    unsigned char s[kResWarps], ch[kResWarps];  // a warp's first item
};

template <int kResWarps>
struct Ctx {
    const ResArgs* a;
    float* sm;
    int g, G, warp, lane;
    // the pair v at (y, x) of level l's buffer `ofs` with H halo rows, stored into the other slabs whose halo rows
    // include y
    __device__ __forceinline__ void share(int l, int ofs, int H, const Slab& s, uint64_t* bar, int y, int x, float2 v) const {
        if (y < s.y0 + H)
            for (int t = g - 1; t >= 0; --t) {
                int u0, u1;
                slab(t, a->re, a->ne, a->le - l, s.ny, u0, u1);
                if (y >= u1 + H) break;
                put2(sm + ofs + (y - u0 + H) * s.ld + x + 2, t, bar, v.x, v.y);
            }
        if (y >= s.y1 - H)
            for (int t = g + 1; t < G; ++t) {
                int u0, u1;
                slab(t, a->re, a->ne, a->le - l, s.ny, u0, u1);
                if (u0 >= s.ny || y < u0 - H) break;
                put2(sm + ofs + (y - u0 + H) * s.ld + x + 2, t, bar, v.x, v.y);
            }
    }
    // f(first row, rows, first column of a pair) over rows [r0, r1) of a level whose work is split as in sp: a warp takes
    // 64 columns of up to h = sp.h[kind] rows at a time
    template <class F>
    __device__ __forceinline__ void strips(const Split<kResWarps>& sp, int kind, int r0, int r1, int nx, F&& f) const {
        const int h = sp.h[kind], nch = sp.nch, m = sp.m;
        int ch = sp.ch[warp];
        for (int y = r0 + sp.s[warp] * h; y < r1;) {
            const int x = (ch << 6) + 2 * lane;
            if (x < nx) f(y, min(h, r1 - y), x);
            ch += m;
            y += sp.q * h;
            if (ch >= nch) { ch -= nch; y += h; }
        }
    }
};

}  // namespace

// VAR: variable coefficients.  VONLY: one V-cycle from level 0 of the arguments for the interleaved right-hand side a.vb
// into a.vx, instead of the whole solve.
template <int kResThreads, bool VAR, bool VONLY>
__global__ void __launch_bounds__(kResThreads, 512 / kResThreads) k_resident(const __grid_constant__ ResArgs a, const double* f, double tol) {
    constexpr int kResWarps = kResThreads / 32;
    extern __shared__ __align__(16) float rsm[];
    float* const sm = rsm;
    __shared__ __align__(16) float4 slots[2][16];  // a reduction's partial sums of every CTA (a Sum3, or an FP64 value)
    __shared__ union {
        Limbs sum[kResWarps];            // a reduction's sums of the warps
        int late_in[16];                 // before the first one: each CTA's copy timed out
    } wb;
    __shared__ double bc[6];             // FP64 scalars that one warp computes for all
    __shared__ Sum3 thr_s;               // the inner threshold
    __shared__ float2 sum_r;             // a reduction's result
    __shared__ Split<kResWarps> split[kResMaxLevels], tsplit[VAR ? kResMaxLevels : 1];  // of the slabs; of the tail's levels
    __shared__ float coef[kResMaxLevels][3];  // c2 of the first Chebyshev step, c1 and c2 of the second
    __shared__ __align__(8) uint64_t bimg, bR[kResMaxLevels], bD[kResMaxLevels], bC, bB, bV, bS[2];
    __shared__ int late;                 // a wait outlasted the caller's budget
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x;
    const int G = (int)cl.num_blocks(), g = (int)cl.block_rank();
    const int sys = blockIdx.x / G;
    Ctx<kResWarps> cx{&a, sm, g, G, tid >> 5, tid & 31};
    const int le = a.le;
    const float d = a.dsh[sys];
    const long long* const budget = &a.cfg->wait_cycles;  // the caller's, 0: the default
    const bool timed = *budget > 0;
    if (tid == 0) {
        mbar_init(&bimg, 1);
        for (int l = 0; l <= le; ++l) {
            mbar_init(&bR[l], 1);
            mbar_init(&bD[l], 1);
        }
        mbar_init(&bC, 1);
        mbar_init(&bB, 1);
        mbar_init(&bV, 1);
        mbar_init(&bS[0], 1);
        mbar_init(&bS[1], 1);
        mbar_fence_init();
        if (VAR) {
            late = 0;
        } else {
            mbar_expect_tx(&bimg, a.img_bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(sm + a.o_sx)), "l"(a.img), "r"(a.img_bytes), "r"(smem_u32(&bimg))
                         : "memory");
            // a wait budget of the caller's starts at the copy's issue; the default one after the buffers are cleared
            late = timed && !mbar_wait_bounded(&bimg, 0, *budget);
        }
    }
    __syncthreads();
    const int lend = VAR ? a.ld : le;  // the last level
    if (tid < 8 * (lend + 1)) {  // thread (level, slabs or tail, kind)
        const int l = tid >> 3, k = tid & 3, nch = (a.lev[l].nx + 63) >> 6;
        const bool tail = (tid & 4) != 0;
        if (tail ? VAR && l >= le : l <= le) {
            int y0 = 0, y1 = a.lev[l].ny;
            if (!tail) slab(g, a.re, a.ne, le - l, a.lev[l].ny, y0, y1);
            const int rows = y1 - y0 + (k == 3 ? 4 : k);
            int h = 1, best = 1 << 30;
            for (int q = 1; q <= kStrip; ++q) {
                const int cost = (((rows + q - 1) / q) * nch + kResWarps - 1) / kResWarps * (q + 1);
                if (cost < best) { best = cost; h = q; }
            }
            Split<kResWarps>& sp = tail ? tsplit[VAR ? l : 0] : split[l];
            sp.h[k] = (unsigned char)h;
            for (int w = k; w < kResWarps; w += 4) {
                sp.s[w] = (unsigned char)(w / nch);
                sp.ch[w] = (unsigned char)(w % nch);
            }
            if (k == 0) {
                sp.nch = (unsigned char)nch;
                sp.q = (unsigned char)(kResWarps / nch);
                sp.m = (unsigned char)(kResWarps % nch);
            }
        }
        if (!tail && l < lend && k < 3)
            coef[l][k] = k == 0 ? a.lev[l].c2[sys] : k == 1 ? a.lev[l].c1[a.Kp + sys] : a.lev[l].c2[a.Kp + sys];
    }
    // everything but the bases starts at zero: the zero columns and the rows outside the grid stay zero
    for (int i = a.o_zero / 4 + tid; i < a.floats / 4; i += kResThreads)
        reinterpret_cast<float4*>(sm)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!VAR && !mbar_wait_bounded(&bimg, 0, max(*budget, kTmaWaitCycles))) late = 1;  // (it lands before the kernel goes on)
    __syncthreads();
    int faulted = late;
    if constexpr (VAR) {
        // the weights (faces negated) of the own rows and three halo rows, the tail's whole levels and its dense inverse in
        // CTA 0; 1 on the diagonal where there is no point
        auto weights = [&](const ResLevel& L, int y0, int y1) {
            const int ld = row_floats(L.nx), rows = y1 - y0 + 2 * kHR, nx = L.nx;
            float *wx = sm + L.oW, *wy = wx + L.wsz, *wd = wy + L.wsz;
            for (int r = cx.warp; r <= rows; r += kResWarps) {
                const int y = y0 - kHR + r;
                const bool iny = y >= 0 && y < L.ny;
                for (int x = cx.lane; x <= nx; x += 32) {
                    const int i = r * ld + x + 2;
                    if (iny && r < rows) copy4(wx + i, L.fx + (size_t)y * (nx + 1) + x);
                    if (x < nx && y >= 0 && y <= L.ny) copy4(wy + i, L.fy + (size_t)y * nx + x);
                    if (x < nx && iny && r < rows) copy4(wd + i, L.dg + (size_t)y * nx + x);
                }
            }
        };
        auto each = [&](auto&& fn) {  // fn(level, first row, end) for every level whose weights this CTA keeps
            for (int l = 0; l < le; ++l) {
                int y0, y1;
                slab(g, a.re, a.ne, le - l, a.lev[l].ny, y0, y1);
                if (y1 > y0) fn(a.lev[l], y0, y1);
            }
            if (g == 0)
                for (int l = le; l < lend; ++l) fn(a.tail[l], 0, a.tail[l].ny);
        };
        each([&](const ResLevel& L, int, int) {
            for (int i = tid; i < L.wsz; i += kResThreads) sm[L.oW + 2 * L.wsz + i] = 1.f;
        });
        __syncthreads();
        each(weights);
        if (g == 0) {
            const int n = a.tail[lend].nx * a.tail[lend].ny;
            for (int i = tid; i < n * n; i += kResThreads) copy4(sm + a.o_inv + i, a.minv + (size_t)i * a.Kp + sys);
        }
        copies_done();
        __syncthreads();
        each([&](const ResLevel& L, int, int) {
            for (int i = tid; i < 2 * L.wsz; i += kResThreads) sm[L.oW + i] = -sm[L.oW + i];
        });
        __syncthreads();
    }
    if (VONLY) pdl_wait();  // what is read so far does not depend on the kernel before
    cl.sync();  // every CTA runs and has cleared its buffers and barriers before the first remote store

    unsigned uR = 0, uD = 0, uC = 0, uB = 0, uV = 0, uS = 0;  // the parity of each barrier's next phase
    bool lost = false;  // what a wait of this thread was for did not come
    int gone = 0;       // ... of this CTA, as of its last reduction
    // arm (thread 0) and await one phase; local values of the phase are published by the caller's barrier
    auto arm = [&](uint64_t* bar, unsigned bytes) {
        if (tid == 0) mbar_expect_tx(bar, bytes);
    };
    auto await = [&](uint64_t* bar, unsigned& bits, int at) {
        if (!lost && !(timed ? wait_timed(bar, (bits >> at) & 1u, *budget, &late) : wait_bytes(bar, (bits >> at) & 1u, kTmaWaitCycles)))
            lost = true;
        bits ^= 1u << at;
    };
    auto range = [&](int l) {
        Slab s;
        slab(g, a.re, a.ne, le - l, a.lev[l].ny, s.y0, s.y1);
        s.nx = a.lev[l].nx;
        s.ny = a.lev[l].ny;
        s.ld = row_floats(s.nx);
        return s;
    };
    auto whole = [&](int l) { return Slab{0, a.lev[l].ny, a.lev[l].nx, a.lev[l].ny, row_floats(a.lev[l].nx)}; };
    // (y, x) of a buffer at base + y * ld + x
    auto at = [&](int ofs, int H, const Slab& s) { return sm + ofs + (H - s.y0) * s.ld + 2; };
    int flip = 0;
    auto tree = [](Sum3& v, int most) {  // the sum over the lanes that differ in the bits up to `most`
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (o <= most) v.add(sum3_shfl_xor(v, o));
    };
    // the sum over the cluster of every thread's v, formed by warp 0 of each CTA, with the same bits: use(sum) is called there
    // and its result, and the sum rounded to FP32, are returned in every thread
    auto all_sum = [&](Sum3 v, auto&& use) {
        arm(&bS[flip], 16u * G);
        Limbs l = to_limbs(v, __reduce_max_sync(0xffffffffu, limb_top(v)));
#pragma unroll
        for (int i = 0; i < 3; ++i) l.w[i] = __reduce_add_sync(0xffffffffu, l.w[i]);
        if (cx.lane == 0) wb.sum[cx.warp] = l;
        __syncthreads();
        if (cx.warp == 0) {
            Sum3 t = from_limbs(wb.sum[cx.lane & (kResWarps - 1)]);
            tree(t, kResWarps / 2);
            if (cx.lane < G) put4(&slots[flip][g], cx.lane, &bS[flip], t.s, t.c, t.e);
            await(&bS[flip], uS, flip);
            const float4 w = slots[flip][cx.lane & 15];
            t = (cx.lane & 15) < G ? Sum3{w.x, w.y, w.z} : Sum3{};
            tree(t, 8);
            const float r = use(t);
            if (cx.lane == 0) sum_r = make_float2(r, t.s);
        } else {
            uS ^= 1u << flip;
        }
        gone = __syncthreads_or(lost);
        flip ^= 1;
        return sum_r;
    };
    // a reduction of nothing: every CTA has come here
    auto meet = [&]() {
        arm(&bS[flip], 16u * G);
        __syncthreads();
        if (cx.warp == 0) {
            if (cx.lane < G) put4(&slots[flip][g], cx.lane, &bS[flip], 0.f, 0.f, 0.f);
            await(&bS[flip], uS, flip);
        } else {
            uS ^= 1u << flip;
        }
        gone = __syncthreads_or(lost);
        flip ^= 1;
    };
    // This thread's share of a . b (level 0) in the groups that other kernels of the same solve sum in FP32, so that a plan's
    // result does not depend on which of the two solves it.  A system that ends after
    // one iteration returns alpha p, so another grouping, which may round alpha the other way, would show in the result's
    // eighth digit (small powers, whose largest shifts converge at once: one plan of 32 in ten batches).  Taken in the first
    // iteration only, later ones correct such a difference (the cost: 63^2 47 -> 48 us, 383 x 255, k = 8, 282 -> 330, 32
    // mixed problems 2.51 -> 2.81 ms).  A group's values are read from the CTAs
    // that own their rows, behind a reduction used as a barrier: unlike a cluster barrier it is bounded, and a CTA that gave
    // up keeps its shared memory until all are done.  A change of the other kernels' tiles, blocks or threads changes their
    // groups: tests/test_gpu_resident_groups.py compares the two.
    //   one exact solve: points P and P + 64, P in the even runs of 64 (the grid kernels of the graph, whose whole cycle is
    //     that solve)
    //   variable coefficients: the same, the groups of the grid sweeps (BURA_SWEEP_GRID).  Larger variable-coefficient plans
    //     run the TMA-staged sweeps, whose groups are other ones: with a ring depth set (which keeps the graph) a small plan
    //     takes those, and such a system may differ by 4e-8
    //   else: the points of a thread of k_spmv_tma, or, with rz, of k_post2_tma, up to eight at a time
    auto grid_dot = [&](int oa, int Ha, int ob, int Hb, bool rz) {
        const Slab s = range(0);
        const int nx = s.nx, ny = s.ny, N = nx * ny;
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
        meet();
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
        Sum3 t{};
        float v = 0.f;
        int n = 0;
        auto flush = [&]() {
            t.add(v);
            v = 0.f;
            n = 0;
        };
        // up to four terms in order, all their values loaded first; where(i, y, x) says whether term i exists
        auto four = [&](auto&& where) {
            float av[4], bv[4];
            bool on[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                int y = 0, x = 0;
                on[i] = where(i, y, x);
                if (on[i]) {
                    const int rank = min(y >> le, a.ne - 1) / a.re;
                    const int k = (y - ((rank * a.re) << le)) * s.ld + 2 + x;
                    const float *pa = sm + oa + Ha * s.ld + k, *pb = sm + ob + Hb * s.ld + k;
                    av[i] = rank == g ? *pa : *cl.map_shared_rank(pa, rank);
                    bv[i] = rank == g ? *pb : *cl.map_shared_rank(pb, rank);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (on[i]) {
                    v = fmaf(av[i], bv[i], v);
                    if (++n == 8) flush();
                }
        };
        // a CTA takes the groups that start in its own rows (another CTA's shared memory is some 50 clocks a warp's load)
        if (VAR || le == 0) {
            for (int c = s.y0 * nx + tid; c < s.y1 * nx; c += kResThreads) {
                if (c & 64) continue;
                four([&](int i, int& y, int& x) {
                    const int P = c + 64 * i;
                    y = P / nx;
                    x = P - y * nx;
                    return i < 2 && P < N;
                });
                flush();
            }
        } else {
            const int R = 256 / (a.Kp / 4), blocks = rz ? a.blk_rz : a.blk_pq;  // thread rows a CTA, CTAs
            const int ntx = (nx + kTX - 1) / kTX, tiles = ntx * ((ny + kTY - 1) / kTY);
            const int lo = (s.y0 + kTY - 1) / kTY * ntx, hi = min((s.y1 + kTY - 1) / kTY * ntx, blocks);
            for (int c = tid; c < (hi - lo) * R; c += kResThreads) {
                const int c0 = c / R, row = c - c0 * R;
                for (int tile = lo + c0; tile < tiles; tile += blocks) {
                    const int ty = tile / ntx, x0 = (tile - ty * ntx) * kTX, y0 = ty * kTY;
                    four([&](int i, int& y, int& x) {
                        const int p = row + (rz ? i / 2 : i) * R;
                        x = x0 + p % kTX;
                        y = y0 + (rz ? p / kTX * 2 + (i & 1) : p / kTX);
                        return p < (rz ? kTX * kTY / 2 : kTX * kTY) && x < nx && y < ny;
                    });
                }
                flush();
            }
        }
        return t;
    };
    // the same in FP64 (norms of the refinement): warp 0 adds the partials; the sum is returned in warp 0 only.
    // `extra` more bytes are due on the barrier.
    auto all_sum64 = [&](double v, unsigned extra) {
        arm(&bS[flip], 8u * G + extra);
        double* const pd = reinterpret_cast<double*>(sm + a.o_d);
        pd[tid] = v;
        gone = __syncthreads_or(lost);
        if (cx.warp == 0) {
            double t = 0.0;
#pragma unroll
            for (int k = 0; k < kResWarps; k += 4)
                t += (pd[k * 32 + cx.lane] + pd[(k + 1) * 32 + cx.lane]) + (pd[(k + 2) * 32 + cx.lane] + pd[(k + 3) * 32 + cx.lane]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (cx.lane < G)
                put2(&slots[flip][g], cx.lane, &bS[flip], __int_as_float(__double2loint(t)), __int_as_float(__double2hiint(t)));
        }
        await(&bS[flip], uS, flip);
        double t = 0.0;
        if (cx.warp == 0) {
            t = cx.lane < G ? *reinterpret_cast<const double*>(&slots[flip][cx.lane]) : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            t = __shfl_sync(0xffffffffu, t, 0);
        }
        flip ^= 1;
        return t;
    };

    // ---- pieces of the V-cycle, on slabs or (loc) on the tail's whole levels in CTA 0
    // the operator at pair index k of a level: A c (no shift) and the pair's diagonal (variable coefficients)
    struct Op {
        const float *fx, *fy, *dg;
        int ld;
        float wx, wy, diag;
        __device__ __forceinline__ float2 apply(int k, float2 c, float l, float r, float2 u, float2 w, float2& dv) const {
            if constexpr (VAR) {
                const float2 xm = ld2(fx + k), ym = ld2(fy + k), yp = ld2(fy + k + ld);
                dv = ld2(dg + k);
                float2 t = __fmul2_rn(dv, c);
                t.x = fmaf(xm.x, l, t.x);
                t.y = fmaf(xm.y, c.x, t.y);
                t.x = fmaf(xm.y, c.y, t.x);
                t.y = fmaf(fx[k + 2], r, t.y);
                t = __ffma2_rn(ym, u, t);
                return __ffma2_rn(yp, w, t);
            } else {
                return stencil2(wx, wy, diag, c, l, r, u, w);
            }
        }
    };
    auto op_of = [&](const ResLevel& L, const Slab& s) {
        Op o;
        o.ld = s.ld;
        o.wx = L.wx;
        o.wy = L.wy;
        o.diag = L.wx + L.wx + L.wy + L.wy;
        o.fx = sm + L.oW + (kHR - s.y0) * s.ld + 2;
        o.fy = o.fx + L.wsz;
        o.dg = o.fy + L.wsz;
        return o;
    };
    // the Jacobi scaling: the constant operator's is part of the coefficients
    auto jac = [&](float2 v, float2 dv) { return VAR ? make_float2(jdiv(v.x, dv.x - d), jdiv(v.y, dv.y - d)) : v; };
    auto jac1 = [&](float v, const float* dg) { return VAR ? jdiv(v, *dg - d) : v; };
    // way down level l: x2 (both pre-smoothing steps from zero) on the own rows and two halo rows, the residual
    // in Y on the fine rows the slab restricts, its full weighting into R of level l + 1
    auto down = [&](int l, bool loc) {
        const ResLevel &L = loc ? a.tail[VAR ? l : 0] : a.lev[l];
        const Slab s = loc ? whole(l) : range(l), sc = loc ? whole(l + 1) : range(l + 1);
        const Split<kResWarps>&sp = loc ? tsplit[VAR ? l : 0] : split[l], &spc = loc ? tsplit[VAR ? l + 1 : 0] : split[l + 1];
        const int ld = s.ld, nx = s.nx;
        const Op A = op_of(L, s);
        const float c20 = coef[l][0], c1 = coef[l][1], c2 = coef[l][2];
        const bool more = !loc && l + 1 < le;  // the last slab level's readers take their own rows only
        if (more) arm(&bR[l + 1], sc.halo_bytes(kHR));
        if (VAR && !loc && l + 1 == le && g == 0) arm(&bC, (unsigned)(sc.ny * even(sc.nx) * 4));
        if (s.some()) {
            const float* R = at(L.oR, kHR, s);
            float* X = at(L.oX, kHX, s);
            cx.strips(sp, 3, max(0, s.y0 - 2), min(s.ny, s.y1 + 2), nx, [&](int y, int n, int x) {
                int k = y * ld + x;
                const float* q = R + k;
                float* o = X + k;
                const bool last = x + 1 >= nx;
                auto first = [&](float2 b, int kk) { return jac(__fmul2_rn(dup(c20), b), VAR ? ld2(A.dg + kk) : b); };
                float2 b = ld2(q), c = first(b, k), u = first(ld2(q - ld), k - ld);
                for (int i = 0; i < n; ++i, q += ld, o += ld, k += ld) {
                    const float2 bn = ld2(q + ld), w = first(bn, k + ld);
                    float2 dv;
                    const float2 t = A.apply(k, c, jac1(c20 * q[-1], A.dg + k - 1), jac1(c20 * q[2], A.dg + k + 2), u, w, dv);
                    const float2 tt = __ffma2_rn(dup(-d), c, t);
                    const float2 res = make_float2(b.x - tt.x, b.y - tt.y);
                    float2 v = __fadd2_rn(c, __ffma2_rn(dup(c1), c, jac(__fmul2_rn(dup(c2), res), dv)));
                    if (last) v.y = 0.f;
                    st2(o, v);
                    u = c; c = w; b = bn;
                }
            });
        }
        __syncthreads();
        if (s.some()) {
            const float *R = at(L.oR, kHR, s), *X = at(L.oX, kHX, s);
            float* Y = at(L.oY, kHY, s);
            cx.strips(sp, 1, s.y0, min(s.ny, s.y1 + 1), nx, [&](int y, int n, int x) {
                int k = y * ld + x;
                const float *q = X + k, *rb = R + k;
                float* o = Y + k;
                float2 u = ld2(q - ld), c = ld2(q);
                for (int i = 0; i < n; ++i, q += ld, rb += ld, o += ld, k += ld) {
                    const float2 w = ld2(q + ld);
                    float2 dv;
                    const float2 t = __ffma2_rn(dup(-d), c, A.apply(k, c, q[-1], q[2], u, w, dv));
                    const float2 b = ld2(rb);
                    st2(o, make_float2(b.x - t.x, b.y - t.y));
                    u = c; c = w;
                }
            });
        }
        __syncthreads();
        if (sc.some()) {
            const float* Y = at(L.oY, kHY, s);
            const int oRc = loc ? a.tail[VAR ? l + 1 : 0].oR : a.lev[l + 1].oR;
            float* Rc = at(oRc, kHR, sc);
            cx.strips(spc, 0, sc.y0, sc.y1, sc.nx, [&](int J, int n, int I) {
                const float* q = Y + 2 * J * ld + 2 * I;
                const bool last = I + 1 >= sc.nx;
                for (int i = 0; i < n; ++i, ++J, q += 2 * ld) {
                    float2 t = make_float2(0.f, 0.f);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {  // columns 2I .. 2I + 4 of rows 2J .. 2J + 2
                        const float2 p = ld2(q + k * ld), m = ld2(q + k * ld + 2);
                        const float e = q[k * ld + 4];
                        const float w0 = k == 1 ? 0.125f : 0.0625f, w1 = k == 1 ? 0.25f : 0.125f;
                        t.x = fmaf(w0, m.x, fmaf(w1, p.y, fmaf(w0, p.x, t.x)));
                        t.y = fmaf(w0, e, fmaf(w1, m.y, fmaf(w0, m.x, t.y)));
                    }
                    if (last) t.y = 0.f;
                    if (VAR && !loc && l + 1 == le) {  // into CTA 0's whole level
                        put2(sm + a.tail[le].oR + (J + kHR) * sc.ld + I + 2, 0, &bC, t.x, t.y);
                    } else {
                        st2(Rc + J * sc.ld + I, t);
                        if (more) cx.share(l + 1, oRc, kHR, sc, &bR[l + 1], J, I, t);
                    }
                }
            });
        }
        __syncthreads();
        if (more) await(&bR[l + 1], uR, l + 1);
    };
    // way up level l: x2 + P (result of level l + 1) on two halo rows, the first post-smoothing step on one, the
    // second on the own rows into D; returns this thread's part of r.z
    auto up = [&](int l, bool loc) {
        const ResLevel &L = loc ? a.tail[VAR ? l : 0] : a.lev[l];
        const Slab s = loc ? whole(l) : range(l), sc = loc ? whole(l + 1) : range(l + 1);
        const Split<kResWarps>& sp = loc ? tsplit[VAR ? l : 0] : split[l];
        const int ld = s.ld, ldc = sc.ld, nx = s.nx;
        const Op A = op_of(L, s);
        const float c20 = coef[l][0], c1 = coef[l][1], c2 = coef[l][2];
        const float* R = at(L.oR, kHR, s);
        float *X = at(L.oX, kHX, s), *Y = at(L.oY, kHY, s), *D = at(L.oD, kHD, s);
        const float* E = at(loc ? a.tail[VAR ? l + 1 : 0].oD : a.lev[l + 1].oD, kHD, sc);
        Sum3 tot{};
        if (!loc) arm(&bD[l], s.halo_bytes(kHD));
        if (s.some()) {
            cx.strips(sp, 3, max(0, s.y0 - 2), min(s.ny, s.y1 + 2), nx, [&](int y, int n, int x) {
                const bool last = x + 1 >= nx;
                float* o = X + y * ld + x;
                for (int i = 0; i < n; ++i, ++y, o += ld) {
                    // column x reads coarse columns x/2 - 1 and x/2, column x + 1 reads x/2
                    const float* e = E + ((y & 1) ? y >> 1 : (y >> 1) - 1) * ldc + (x >> 1);
                    const float e0 = e[-1], e1 = e[0];
                    float2 t;
                    if (y & 1) {
                        t.x = fmaf(0.5f, e1, 0.5f * e0);
                        t.y = e1;
                    } else {
                        const float f0 = e[ldc - 1], f1 = e[ldc];
                        t.x = fmaf(0.25f, f1, fmaf(0.25f, f0, fmaf(0.25f, e1, 0.25f * e0)));
                        t.y = fmaf(0.5f, f1, 0.5f * e1);
                    }
                    if (last) t.y = 0.f;
                    st2(o, __fadd2_rn(ld2(o), t));
                }
            });
        }
        __syncthreads();
        if (s.some()) {
            cx.strips(sp, 2, max(0, s.y0 - 1), min(s.ny, s.y1 + 1), nx, [&](int y, int n, int x) {
                const bool last = x + 1 >= nx;
                int k = y * ld + x;
                const float *q = X + k, *rb = R + k;
                float *oy = Y + k, *od = D + k;
                float2 u = ld2(q - ld), c = ld2(q);
                for (int i = 0; i < n; ++i, q += ld, rb += ld, oy += ld, od += ld, k += ld) {
                    const float2 w = ld2(q + ld), b = ld2(rb);
                    float2 dg;
                    const float2 t = __ffma2_rn(dup(-d), c, A.apply(k, c, q[-1], q[2], u, w, dg));
                    float2 dv = jac(__fmul2_rn(dup(c20), make_float2(b.x - t.x, b.y - t.y)), dg);
                    if (last) dv.y = 0.f;
                    st2(oy, __fadd2_rn(c, dv));
                    if (y + i >= s.y0 && y + i < s.y1) st2(od, dv);
                    u = c; c = w;
                }
            });
        }
        __syncthreads();
        if (s.some()) {
            cx.strips(sp, 0, s.y0, s.y1, nx, [&](int y, int n, int x) {
                const bool last = x + 1 >= nx;
                int k = y * ld + x;
                const float *q = Y + k, *rb = R + k;
                float* od = D + k;
                float2 u = ld2(q - ld), c = ld2(q), p2 = make_float2(0.f, 0.f);
                for (int i = 0; i < n; ++i, q += ld, rb += ld, od += ld, k += ld) {
                    const float2 w = ld2(q + ld), b = ld2(rb);
                    float2 dg;
                    const float2 t = __ffma2_rn(dup(-d), c, A.apply(k, c, q[-1], q[2], u, w, dg));
                    const float2 res = make_float2(b.x - t.x, b.y - t.y);
                    float2 z = __fadd2_rn(c, __ffma2_rn(dup(c1), ld2(od), jac(__fmul2_rn(dup(c2), res), dg)));
                    if (last) z.y = 0.f;
                    st2(od, z);
                    if (!loc) cx.share(l, L.oD, kHD, s, &bD[l], y + i, x, z);
                    p2 = __ffma2_rn(b, z, p2);
                    u = c; c = w;
                }
                tot.add(p2.x + p2.y);
            });
        }
        __syncthreads();
        if (!loc) await(&bD[l], uD, l);
        return tot;
    };
    // variable coefficients: CTA 0 runs the V-cycle of levels le .. lend (dense inverse on the last) on whole levels and
    // sends every slab its rows of the result with two halo rows
    auto tail = [&]() {
        const Slab s = whole(le), mine = range(le);
        if (mine.some()) arm(&bB, (unsigned)((min(mine.ny, mine.y1 + kHD) - max(0, mine.y0 - kHD)) * even(s.nx) * 4));
        if (g == 0) {
            await(&bC, uC, 0);
            __syncthreads();
            for (int l = le; l < lend; ++l) down(l, true);
            const ResLevel& L = a.tail[lend];
            const int nx = L.nx, n = nx * L.ny, ld = row_floats(nx);
            float* const b = sm + a.o_bt;
            for (int i = tid; i < n; i += kResThreads) b[i] = sm[L.oR + (i / nx + kHR) * ld + i % nx + 2];
            __syncthreads();
            if (tid < n) {
                const float* m = sm + a.o_inv + tid * n;
                float v = 0.f;
                for (int j = 0; j < n; ++j) v = fmaf(m[j], b[j], v);
                sm[L.oD + (tid / nx + kHD) * ld + tid % nx + 2] = v;
            }
            __syncthreads();
            for (int l = lend - 1; l >= le; --l) (void)up(l, true);
            const float* D = at(a.tail[le].oD, kHD, s);
            const int half = even(s.nx) / 2;
            for (int i = tid; i < s.ny * half; i += kResThreads) {
                const int y = i / half, x = 2 * (i - y * half);
                const float2 v = ld2(D + y * s.ld + x);
                for (int t = max(0, (y - kHD) / a.re - 1); t < G; ++t) {
                    int u0, u1;
                    slab(t, a.re, a.ne, 0, s.ny, u0, u1);
                    if (u0 >= s.ny || y < u0 - kHD) break;
                    if (y < u1 + kHD) put2(sm + a.lev[le].oD + (y - u0 + kHD) * s.ld + x + 2, t, &bB, v.x, v.y);
                }
            }
        } else {
            uC ^= 1u;
        }
        if (mine.some()) await(&bB, uB, 0);
        else uB ^= 1u;
        __syncthreads();
    };
    // out[q][m] = sum_k S[k][m] C[q][k] (k in increasing order) for m < M, q < Q, handed to epi(q, value) by a thread with
    // tid mod kSP = m; C has rows of kSP floats, zero from Kd on (so that k may run on to a multiple of 4: the bases are
    // followed by finite values).  A thread takes two q, so a value of S is loaded once for both; a warp shares them, so
    // its loads of C are broadcasts of four at a time.
    const int m = tid & (kSP - 1);
    const int own_c = m / a.ce, own_r = m / a.re;  // the slabs that own column and row m of the exact level
    auto product = [&](const float* S, const float* C, int Kd, int M, int Q, auto&& epi) {
        if (m >= M) return;
        const float* Sm = S + m;
        for (int q = 2 * (tid / kSP); q < Q; q += 2 * (kResThreads / kSP)) {
            const bool two = q + 1 < Q;
            const float4 *A4 = reinterpret_cast<const float4*>(C + q * kSP), *B4 = A4 + (two ? kSP / 4 : 0);
            float v = 0.f, w = 0.f;
#pragma unroll 4
            for (int k = 0; k < Kd; k += 4) {
                const float4 c = A4[k >> 2], e = B4[k >> 2];
                const float s0 = Sm[k * kSP], s1 = Sm[(k + 1) * kSP], s2 = Sm[(k + 2) * kSP], s3 = Sm[(k + 3) * kSP];
                v = fmaf(s0, c.x, v);
                w = fmaf(s0, e.x, w);
                v = fmaf(s1, c.y, v);
                w = fmaf(s1, e.y, w);
                v = fmaf(s2, c.z, v);
                w = fmaf(s2, e.z, w);
                v = fmaf(s3, c.w, v);
                w = fmaf(s3, e.w, w);
            }
            epi(q, v);
            if (two) epi(q + 1, w);
        }
    };
    // exact solve of level le: D = (A - d I)^{-1} R there; returns this thread's part of R.D (the CG r.z when le = 0)
    auto exact = [&]() {
        const ResLevel& L = a.lev[le];
        const Slab s = range(le);
        const int ld = s.ld, nx = s.nx, ny = s.ny, rows = s.y1 - s.y0;
        const float* R = at(L.oR, kHR, s);
        float* D = at(L.oD, kHD, s);
        const float *SX = sm + a.o_sx, *SY = sm + a.o_sy;
        float *Bt = sm + a.o_bt, *Br = sm + a.o_br, *Cc = sm + a.o_cc, *Cd = sm + a.o_cd;
        const int c0 = min(nx, g * a.ce), cw = min(nx, c0 + a.ce) - c0;
        arm(&bC, 4u * ny * cw);
        arm(&bB, 4u * rows * nx);
        arm(&bD[le], s.halo_bytes(kHD));
        for (int i = tid; i < rows * kSP; i += kResThreads) {
            const int r = i / kSP, k = i & (kSP - 1);
            Bt[i] = k < nx ? R[(s.y0 + r) * ld + k] : 0.f;
        }
        __syncthreads();
        // rows of R S_x, each value to the slab that owns its column
        product(SX, Bt, nx, nx, rows, [&](int r, float v) {
            put(Cc + (m - own_c * a.ce) * kSP + s.y0 + r, own_c, &bC, v);
        });
        await(&bC, uC, 0);
        product(SY, Cc, ny, ny, cw, [&](int c, float v) {
            Cd[c * kSP + m] = v / ((sm[a.o_lam + c0 + c] + sm[a.o_lam + kSP + m]) - d);
        });
        __syncthreads();
        product(SY, Cd, ny, ny, cw, [&](int c, float v) {
            put(Br + (m - own_r * a.re) * kSP + c0 + c, own_r, &bB, v);
        });
        await(&bB, uB, 0);
        Sum3 tot{};
        product(SX, Br, nx, nx, rows, [&](int r, float v) {
            const int y = s.y0 + r;
            D[y * ld + m] = v;
            tot.add(v * R[y * ld + m]);
        });
        __syncthreads();
        if (s.some())  // the edge rows, in pairs
            for (int i = tid; i < rows * (kSP / 2); i += kResThreads) {
                const int r = i / (kSP / 2), x = 2 * (i & (kSP / 2 - 1));
                if (x < nx && (r < kHD || r >= rows - kHD)) cx.share(le, L.oD, kHD, s, &bD[le], s.y0 + r, x, ld2(D + (s.y0 + r) * ld + x));
            }
        await(&bD[le], uD, le);
        return tot;
    };

    // z = M r into D of level 0; returns this thread's part of r.z
    auto cycle = [&]() {
        Sum3 t{};
        for (int l = 0; l < le; ++l) down(l, false);
        if constexpr (VAR) tail();
        else t = exact();
        for (int l = le - 1; l >= 0; --l) t = up(l, false);
        return t;
    };

    if constexpr (VONLY) {
        // the right-hand side on the own rows and the halo rows, one V-cycle, the result's own rows
        const Slab s = range(0);
        float* const R = at(a.lev[0].oR, kHR, s);
        const float* const D = at(a.lev[0].oD, kHD, s);
        if (s.some()) {
            for (int y = max(0, s.y0 - kHR) + cx.warp; y < min(s.ny, s.y1 + kHR); y += kResWarps)
                for (int x = cx.lane; x < s.nx; x += 32) copy4(R + y * s.ld + x, a.vb + ((size_t)y * s.nx + x) * a.Kp + sys);
        }
        copies_done();
        __syncthreads();
        (void)cycle();
        if (s.some())
            for (int y = s.y0 + cx.warp; y < s.y1; y += kResWarps)
                for (int x = cx.lane; x < s.nx; x += 32) a.vx[((size_t)y * s.nx + x) * a.Kp + sys] = D[y * s.ld + x];
        if (lost || late || faulted) atomicExch(&a.scal->fault, 1);
        pdl_trigger();
        cl.sync();  // no CTA leaves while another may still store into its shared memory
        return;
    }

    // ---- the whole solve
    const Slab s0 = range(0);
    const int np = (s0.y1 - s0.y0) * s0.nx;  // own points of level 0, numbered along the rows
    const int ld0 = s0.ld, ldx = even(s0.nx);
    float* const R0 = at(a.lev[0].oR, kHR, s0);
    float* const P0 = at(a.o_p, kHP, s0);
    double* const r64 = reinterpret_cast<double*>(sm + a.o_r64);     // own points (over P, X, Y, D: free between inner solves)
    double* const vg = a.v + (size_t)sys * a.N;
    double* const vs = reinterpret_cast<double*>(sm + a.o_vs);       // v of the own points for the residual
    double* const vh = reinterpret_cast<double*>(sm + a.o_vh);       // v on the rows below and above the slab
    // x of the own points, rows of ldx
    float* const xs = (a.o_x >= 0 ? sm + a.o_x : a.x + ((size_t)sys * s0.ny + s0.y0) * ldx) - (size_t)s0.y0 * ldx;
    const size_t gofs = (size_t)s0.y0 * s0.nx;

    if (cx.warp == kResWarps - 1) {
        // this system's relative threshold need_j, reached in n_j steps of need_j^(1/n_j) each
        const OuterCfg& c = *a.cfg;
        const double t = c.lambda_lo > 0 ? tol * (c.lambda_lo - c.d[sys]) / (c.K * c.c[sys]) : tol;
        double st2 = 1.0;  // the square of a step's share
        if (t < 1.0) {
            const double n = plan_steps(t, c.inner_rtol, c.rtol_slack, c.log_rtol);
            st2 = n == 1.0 ? t * t : n == 2.0 ? t : pow(t, 2.0 / n);
        }
        if (cx.lane == 0) {
            bc[5] = t;
            bc[2] = 0.25 * st2;
        }
    }
    // ||f||^2
    double part = 0.0;
    for (int i = tid; i < np; i += kResThreads) {
        const double v = __ldg(f + gofs + i);
        part = fma(v, v, part);
    }
    if (tid < G) put(reinterpret_cast<float*>(&wb.late_in[g]), tid, &bS[0], __int_as_float(faulted));
    const double sum_f = all_sum64(part, 4u * G);
    for (int t = 0; t < G; ++t) faulted |= wb.late_in[t];
    if (tid == 0) {
        bc[0] = sum_f;
        bc[1] = bc[5] * bc[5] * sum_f;
    }
    if (__syncthreads_or(lost)) faulted = gone = 1;
    const double fn2 = bc[0], thr64 = bc[1];
    const int max_outer = a.cfg->max_outer, max_iters = a.cfg->max_iters;

    // ---- the refinement loop
    const double d64 = a.cfg->d[sys], c0_64 = 2.0 * (a.wx + a.wy) - d64;
    double rr64 = fn2;  // uniform: every decision below is taken alike by all threads of the cluster
    int outer = 0, siters = 0, status = -5;
    if (faulted) status = -6;
    ResOut& out = a.out[sys];
    const ResLevel& L0 = a.lev[0];
    for (; !faulted;) {
        if (!isfinite(rr64)) { status = -4; break; }
        if (!(rr64 > thr64)) { status = 0; break; }
        if (outer >= max_outer) break;
        // the scale, its reciprocal and the inner target on ||r||^2 (a step's share or what is left, with a margin of 2), by
        // a warp each: FP64 roots and divisions are long chains on GB300
        if (cx.warp == 0) {
            const double h = sqrt(rr64);
            if (cx.lane == 0) bc[3] = h;
        } else if (cx.warp == 1) {
            const double h = rsqrt(rr64);
            if (cx.lane == 0) bc[4] = h;
        } else if (cx.warp == 2) {
            const double t = fmax(bc[2], 0.25 * (thr64 / rr64));
            if (cx.lane == 0) thr_s = sum3_of(t);
        }
        arm(&bR[0], s0.halo_bytes(kHR));
        __syncthreads();
        const double hs = bc[3], is = bc[4];
        // the inner right-hand side r / ||r|| in FP32, with its halo rows
        if (s0.some())
            cx.strips(split[0], 0, s0.y0, s0.y1, s0.nx, [&](int y, int n, int x) {
                const bool last = x + 1 >= s0.nx;
                for (int i = 0; i < n; ++i, ++y) {
                    const int k = (y - s0.y0) * s0.nx + x;
                    const double* src = outer == 0 ? f + gofs : r64;
                    float2 v;
                    v.x = (float)(src[k] * is);
                    v.y = last ? 0.f : (float)(src[k + 1] * is);
                    st2(R0 + y * ld0 + x, v);
                    cx.share(0, L0.oR, kHR, s0, &bR[0], y, x, v);
                }
            });
        // P, X, Y, D held the FP64 residual and the norm's partials: their zero columns and rows are restored
        __syncthreads();
        for (int i = a.o_r64 / 4 + tid; i < a.o_r64_end / 4; i += kResThreads)
            reinterpret_cast<float4*>(sm)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        await(&bR[0], uR, 0);
        Sum3 rz{1.f, 0.f, 0.f};  // (warp 0's)
        int it = 0, breakdown = 0;
        for (;;) {
            // z = M r into D
            Sum3 t = cycle();
            if (siters == 0) t = grid_dot(L0.oR, kHR, L0.oD, kHD, true);
            const float2 zr = all_sum(t, [&](const Sum3& s) {
                const float q = sum3_div(s, rz);
                rz = s;
                return q;
            });
            if (!isfinite(zr.y)) breakdown = 1;
            const float beta = zr.x;
            // p = z + beta p on the own rows and one halo row, q = (A - d I) p into Y
            const float* Z = at(L0.oD, kHD, s0);
            float* Q = at(L0.oY, kHY, s0);
            if (s0.some())
                cx.strips(split[0], 2, max(0, s0.y0 - 1), min(s0.ny, s0.y1 + 1), s0.nx, [&](int y, int n, int x) {
                    const int k = y * ld0 + x;
                    const float* z = Z + k;
                    float* o = P0 + k;
                    for (int i = 0; i < n; ++i, z += ld0, o += ld0)
                        st2(o, it == 0 ? ld2(z) : __ffma2_rn(dup(beta), ld2(o), ld2(z)));
                });
            __syncthreads();
            t = Sum3{};
            if (s0.some()) {
                const Op A = op_of(L0, s0);
                cx.strips(split[0], 0, s0.y0, s0.y1, s0.nx, [&](int y, int n, int x) {
                    int k = y * ld0 + x;
                    const float* q = P0 + k;
                    float* o = Q + k;
                    float2 u = ld2(q - ld0), c = ld2(q), p2 = make_float2(0.f, 0.f);
                    for (int i = 0; i < n; ++i, q += ld0, o += ld0, k += ld0) {
                        const float2 w = ld2(q + ld0);
                        float2 dv;
                        const float2 v = __ffma2_rn(dup(-d), c, A.apply(k, c, q[-1], q[2], u, w, dv));
                        st2(o, v);
                        p2 = __ffma2_rn(c, v, p2);  // c is zero in the padding column
                        u = c; c = w;
                    }
                    t.add(p2.x + p2.y);
                });
            }
            if (siters == 0) t = grid_dot(a.o_p, kHP, L0.oY, kHY, false);
            const float2 pq = all_sum(t, [&](const Sum3& s) { return sum3_div(rz, s); });
            float af = 0.f;
            if (!(pq.y > 0.f) || !isfinite(pq.y)) breakdown = 1;
            else af = pq.x;
            // x += alpha p, r -= alpha q with the halo rows of r
            arm(&bR[0], s0.halo_bytes(kHR));
            t = Sum3{};
            if (s0.some())
                cx.strips(split[0], 0, s0.y0, s0.y1, s0.nx, [&](int y, int n, int x) {
                    const bool last = x + 1 >= s0.nx;
                    const int k = y * ld0 + x;
                    const float *p = P0 + k, *q = Q + k;
                    float *r = R0 + k, *xp = xs + y * ldx + x;
                    float2 p2 = make_float2(0.f, 0.f);
                    for (int i = 0; i < n; ++i, p += ld0, q += ld0, r += ld0, xp += ldx) {
                        const float2 pv = ld2(p);
                        st2(xp, it == 0 ? __fmul2_rn(dup(af), pv) : __ffma2_rn(dup(af), pv, ld2(xp)));
                        float2 rv = __ffma2_rn(dup(-af), ld2(q), ld2(r));
                        if (last) rv.y = 0.f;
                        st2(r, rv);
                        cx.share(0, L0.oR, kHR, s0, &bR[0], y + i, x, rv);
                        p2 = __ffma2_rn(rv, rv, p2);
                    }
                    t.add(p2.x + p2.y);
                });
            const float2 rr = all_sum(t, [&](const Sum3& s) { return sum3_le(s, thr_s) ? 1.f : 0.f; });
            await(&bR[0], uR, 0);
            ++it;
            ++siters;
            if (!isfinite(rr.y)) breakdown = 1;
            if (rr.x != 0.f || breakdown || it >= max_iters || gone) break;
        }
        if (tid == 0 && g == 0) out.its[outer] = it;
        ++outer;
        if (gone) { status = -6; break; }
        if (breakdown) { status = -4; break; }
        // v += ||r|| x, its edge rows into the neighbours' vh, then the true residual f - (A - d I) v and its norm, in FP64
        arm(&bV, s0.some() ? (unsigned)((s0.y0 > 0) + (s0.y1 < s0.ny)) * s0.nx * 8u : 0u);
        __syncthreads();
        for (int i = tid; i < np; i += kResThreads) {
            const int r = i / s0.nx, x = i - r * s0.nx;
            const double xv = (double)xs[(s0.y0 + r) * ldx + x];
            const double v = outer == 1 ? hs * xv : fma(hs, xv, vg[gofs + i]);
            vg[gofs + i] = v;
            vs[i] = v;
            if (r == 0 && s0.y0 > 0) put2(vh + s0.nx + x, g - 1, &bV, __int_as_float(__double2loint(v)), __int_as_float(__double2hiint(v)));
            if (r == s0.y1 - s0.y0 - 1 && s0.y1 < s0.ny)
                put2(vh + x, g + 1, &bV, __int_as_float(__double2loint(v)), __int_as_float(__double2hiint(v)));
        }
        __syncthreads();
        await(&bV, uV, 0);
        double t = 0.0;
        for (int i = tid; i < np; i += kResThreads) {
            const int r = i / s0.nx, x = i - r * s0.nx, y = s0.y0 + r;
            const double* q = vs + i;
            const double lo = y == 0 ? 0.0 : r == 0 ? vh[x] : q[-s0.nx];
            const double hi = y == s0.ny - 1 ? 0.0 : y == s0.y1 - 1 ? vh[s0.nx + x] : q[s0.nx];
            const double fv = __ldg(f + gofs + i);
            double v;
            if constexpr (VAR) {  // f - (A - d I) v, the grid kernel's order
                const size_t P = gofs + i, F = (size_t)y * (s0.nx + 1) + x;
                v = __ldg(a.dg64 + P) * q[0];
                v = fma(-__ldg(a.fx64 + F), x > 0 ? q[-1] : 0.0, v);
                v = fma(-__ldg(a.fx64 + F + 1), x < s0.nx - 1 ? q[1] : 0.0, v);
                v = fma(-__ldg(a.fy64 + P), lo, v);
                v = fma(-__ldg(a.fy64 + P + s0.nx), hi, v);
                v = fv - fma(-d64, q[0], v);
            } else {
                const double sx = (x > 0 ? q[-1] : 0.0) + (x < s0.nx - 1 ? q[1] : 0.0);
                v = fma(-c0_64, q[0], fv);
                v = fma(a.wx, sx, v);
                v = fma(a.wy, lo + hi, v);
            }
            r64[i] = v;
            t = fma(v, v, t);
        }
        t = all_sum64(t, 0u);
        if (tid == 0) bc[0] = t;
        gone = __syncthreads_or(lost);
        if (gone) { status = -6; break; }  // (the sum lacks what did not come)
        rr64 = bc[0];
    }
    if (outer == 0)
        for (int i = tid; i < np; i += kResThreads) vg[gofs + i] = 0.0;
    if (tid == 0 && g == 0) {
        out.rr = rr64;
        out.fnorm2 = fn2;
        out.outer = outer;
        out.siters = siters;
    }
    if (tid == 0 && g == 0) out.status = status;
    gone = __syncthreads_or(lost || late);
    cl.sync();  // no CTA leaves while another may still store into its shared memory
    if (tid == 0 && gone) out.status = -6;
}

// The output stage: u = sum_j c_j v_j (FP64, j = 0..K-1 in order) or the systems themselves into V, and the solve's
// outcome from the systems' records (page-locked host memory): the counts of the lockstep solve, in which a
// refinement step lasts as long as its slowest system.
__global__ void k_resident_out(ResArgs a, int K, const double* c, double* u, double* V, int accumulate, OuterState* st) {
    pdl_wait();
    const size_t N = a.N;
    if (blockIdx.x == 0 && threadIdx.x < 32) {  // lane j: system j
        const int j = threadIdx.x;
        const bool on = j < K;
        const ResOut& o = a.out[on ? j : 0];
        const int mine = o.outer;
        int rank = o.status == -6 ? 3 : o.status == -4 ? 2 : o.status == -5 ? 1 : 0, outer = mine;
        for (int w = 16; w > 0; w >>= 1) {
            rank = max(rank, __shfl_xor_sync(0xffffffffu, rank, w));
            outer = max(outer, __shfl_xor_sync(0xffffffffu, outer, w));
        }
        int total = 0;
        for (int q = 0; q < outer; ++q) {
            int m = q < mine ? o.its[q] : 0;
            for (int w = 16; w > 0; w >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, w));
            total += m;
        }
        if (on) {
            st->siters[j] = o.siters;
            st->rr[j] = o.rr;
        }
        if (j == 0) {
            st->fnorm2 = o.fnorm2;
            st->outer = outer;
            st->total_it = total;
            st->status = rank == 3 ? -6 : rank == 2 ? -4 : rank == 1 ? -5 : 0;
            st->done = 1;
        }
    }
    for (size_t P = blockIdx.x * (size_t)blockDim.x + threadIdx.x; P < N; P += (size_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int j = 0; j < K; ++j) {
            const double v = a.v[j * N + P];
            if (V) V[j * N + P] = v;
            s = fma(c[j], v, s);
        }
        if (u) u[P] = accumulate ? u[P] + s : s;
    }
}

namespace {

int up4(int v) { return (v + 3) / 4 * 4; }

// Shared-memory layout of one CTA for clusters of G; false if it does not fit (or has no rows to give a CTA).
bool res_layout(ResArgs& a, int G) {
    a.re = (a.ne + G - 1) / G;
    a.ce = (a.lev[a.le].nx + G - 1) / G;
    const int nxe = a.lev[a.le].nx;
    const int last = a.ne - a.re * ((a.ne + a.re - 1) / a.re - 1);  // rows of the exact level in the last slab
    long long own0 = 0;
    int o = 0;
    auto take = [&](long long n) {
        const int at = o;
        o = (int)std::min<long long>(1 << 28, up4((int)std::min<long long>(1 << 28, o + n)));
        return at;
    };
    if (!a.var) {
        a.o_sx = take((long long)nxe * kSP);
        a.o_sy = take((long long)a.ne * kSP);
        a.o_lam = take(2 * kSP);
        a.img_bytes = (unsigned)(res_image_floats(nxe, a.ne) * sizeof(float));
    }
    a.o_zero = o;
    for (int l = 0; l <= a.le; ++l) {
        ResLevel& L = a.lev[l];
        const int ld = row_floats(L.nx);
        const int sh = a.le - l;
        const int tail = ((last << sh) + (1 << sh) - 1);  // the last slab's rows
        const int most = std::min(std::max(a.re << sh, tail), L.ny);
        const bool smoothed = l < a.le, cg = l == 0 && !a.vonly;
        L.oR = smoothed || !a.var ? take((long long)(most + 2 * kHR) * ld) : o;
        if (cg) {
            a.o_r64 = o;
            a.o_p = take((long long)(most + 2 * kHP) * ld);
        }
        L.oX = smoothed ? take((long long)(most + 2 * kHX) * ld) : o;
        L.oY = smoothed || cg ? take((long long)(most + 2 * kHY) * ld) : o;
        L.oD = take((long long)(most + 2 * kHD) * ld);
        if (cg) {  // between inner solves: the FP64 residual, v with its neighbours' edge rows, the partials of a norm
            own0 = (long long)most * even(L.nx);
            const int end = o;
            o = a.o_r64;
            take(2 * own0);
            a.o_vs = take(2 * own0);
            a.o_vh = take(4 * L.nx);
            a.o_d = take(2 * 32 * kResMostWarps);
            a.o_r64_end = o = std::max(o, end);
        }
        L.wsz = (most + 2 * kHR + 1) * ld;
        if (a.var && smoothed) L.oW = take(3LL * L.wsz);
    }
    if (a.var) {  // the tail's whole levels, the dense inverse of its last one
        for (int l = a.le; l <= a.ld; ++l) {
            ResLevel& L = a.tail[l];
            L = a.lev[l];
            const int ld = row_floats(L.nx);
            L.oR = take((long long)(L.ny + 2 * kHR) * ld);
            L.oD = take((long long)(L.ny + 2 * kHD) * ld);
            if (l == a.ld) break;
            L.oX = take((long long)(L.ny + 2 * kHX) * ld);
            L.oY = take((long long)(L.ny + 2 * kHY) * ld);
            L.wsz = (L.ny + 2 * kHR + 1) * ld;
            L.oW = take(3LL * L.wsz);
        }
        const int n = a.lev[a.ld].nx * a.lev[a.ld].ny;
        a.o_inv = take((long long)n * n);
        a.o_bt = take(n);
    } else {
        a.o_bt = take((long long)a.re * kSP);
        a.o_br = take((long long)a.re * kSP);
        a.o_cc = take((long long)a.ce * kSP);
        a.o_cd = take((long long)a.ce * kSP);
    }
    a.floats = o;
    a.o_x = -1;
    const size_t room = (size_t)o * sizeof(float) <= kResSmemHalf ? kResSmemHalf : kResSmemMax;
    if ((size_t)(o + own0) * sizeof(float) <= room) {
        a.o_x = take(own0);
        a.floats = o;
    }
    return (size_t)a.floats * sizeof(float) <= kResSmemMax;
}

using ResKernel = void (*)(const ResArgs, const double*, double);
template <bool VAR, bool VONLY>
ResKernel res_kernel_t(const ResArgs& a) { return a.threads == 256 ? k_resident<256, VAR, VONLY> : k_resident<512, VAR, VONLY>; }
ResKernel res_kernel(const ResArgs& a) {
    return a.var ? (a.vonly ? res_kernel_t<true, true>(a) : res_kernel_t<true, false>(a))
                 : (a.vonly ? res_kernel_t<false, true>(a) : res_kernel_t<false, false>(a));
}

cudaLaunchConfig_t res_config(const ResArgs& a, int blocks, cudaLaunchAttribute* attr, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(a.threads);
    cfg.dynamicSmemBytes = (size_t)a.floats * sizeof(float);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.vonly) {  // within a chain of dependent launches: the setup overlaps the kernel before
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.numAttrs = 2;
    }
    return cfg;
}

}  // namespace

size_t res_image_floats(int nx, int ny) { return (size_t)(nx + ny + 2) * kSP; }

void res_image(int nx, int ny, const double* sx, const double* sy, const float* lx, const float* ly, float* img) {
    std::fill(img, img + res_image_floats(nx, ny), 0.f);
    for (int i = 0; i < nx; ++i)
        for (int k = 0; k < nx; ++k) img[(size_t)i * kSP + k] = (float)sx[(size_t)i * nx + k];
    for (int i = 0; i < ny; ++i)
        for (int k = 0; k < ny; ++k) img[(size_t)(nx + i) * kSP + k] = (float)sy[(size_t)i * ny + k];
    std::copy(lx, lx + nx, img + (size_t)(nx + ny) * kSP);
    std::copy(ly, ly + ny, img + (size_t)(nx + ny + 1) * kSP);
}

// Clusters of a plan's shape that the current device holds at once (0: none), after setting the kernel's limits, which are
// properties of the function: always the largest, whatever a plan takes.  The counts are kept: a query costs more than the
// rest of a small plan's setup, and there are few shapes.
int resident_clusters(const ResArgs& a) {
    static std::mutex m;
    static std::map<std::array<int, 5>, int> known;
    const ResKernel k = res_kernel(a);
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmemMax) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const std::array<int, 5> key = {dev, (a.var ? 2 : 0) + (a.vonly ? 1 : 0), a.threads, a.G, a.floats};
    std::lock_guard<std::mutex> lock(m);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = res_config(a, a.G, attr, nullptr);
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (known.size() < 4096) known[key] = n;
    return n;
}

// The largest cluster of up to 16 CTAs (the device holds 7 clusters of 16 at one CTA per SM; more systems than that
// run as the first clusters finish: 255^2 with 13 systems 989 -> 420 us).  Slabs small enough for two CTAs per SM
// take 256 threads each, so that 14 clusters are resident (63^2, k = 9: 80 us with 512 threads, 49 with 256; 32
// problems of up to 127^2 as one batch: 1772 and 993 us); larger ones take 512 (255^2, k = 5: 173 us, 189 with 256).
bool resident_plan(ResArgs& a, int K) {
    for (int G = 16; G >= 1; G /= 2) {
        if (G > a.ne || G > a.lev[a.le].nx) continue;
        if (!res_layout(a, G)) return false;
        a.G = G;
        a.threads = (size_t)a.floats * sizeof(float) <= kResSmemHalf ? 256 : 512;
        const int n = resident_clusters(a);
        if (n >= (a.vonly ? K : 1)) return true;  // a V-cycle inside an iteration takes one round of clusters
    }
    return false;
}

cudaError_t launch_resident(const ResArgs& a, int K, const double* f, double tol, cudaStream_t s) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = res_config(a, K * a.G, attr, s);
    return cudaLaunchKernelEx(&cfg, res_kernel(a), a, f, tol);
}

cudaError_t launch_resident_out(const ResArgs& a, int K, const double* c, double* u, double* V, int accumulate,
                                OuterState* st, cudaStream_t s) {
    const long long b = ((long long)a.N + 255) / 256;
    launch_pdl(k_resident_out, dim3((unsigned)std::min<long long>(b, 152 * 8)), dim3(256), 0, s, a, K, c, u, V, accumulate, st);
    return cudaGetLastError();
}

}  // namespace bura
