// FP64 sweeps of 2-D constant-coefficient levels with the fewest FP64 operations.
//
// GB300 executes about 1.7 FP64 operations per SM and clock, so these sweeps are bound by their operation count, not by
// memory (one operation per value of a 511^2, 8-system vector takes 4.3 us, reading it 2.5).  Every sweep is therefore
// written as one combination of the neighbours' pair sums l + r and u + d with coefficients that are formed once per CTA:
//
//   pre-smoothing, both steps    k0 b + kx (l + r) + ky (u + d) of b            15 -> 5 operations a value
//   residual and restriction     the residual stored, or formed 3 / 2 times, not 9 / 4   18 -> 7 or 10
//   x += P ec                    per 2 x 2 fine points from 4 coarse ones        9 -> 2
//   post-smoothing step          k0 x + k1 (b + wx (l + r) + wy (u + d))        10 -> 6; the second + k2 x_in  11 -> 8
//   q = (A - d I) p, p.q         p updated by its own sweep, not 5 times        12 -> 6 (+ 1)
//
// counting from the general sweeps of kernels_impl.cuh, which these are algebraically equal to.
#include <algorithm>
#include <cstddef>

#include "kernels_impl.cuh"

namespace bura {

namespace {

constexpr int kThreads = 256;
constexpr int kCtas = 3;  // per SM
constexpr int kRestrictThreads = 128;

enum Mode64 { M_PRE, M_RES, M_POST1, M_POST2, M_SPMV };

__device__ __forceinline__ double2 ld2(const double* p) { return *reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ double2 ld2_if(bool c, const double* p) { return c ? ld2(p) : make_double2(0.0, 0.0); }
__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) { return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)); }
__device__ __forceinline__ double2 fma2(double a, double2 b, double2 c) { return make_double2(fma(a, b.x, c.x), fma(a, b.y, c.y)); }
__device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }

struct Args64 {
    const double *x, *b, *xin;  // the stencil's input; right-hand side; M_POST2: the iterate before the first step
    double* out;
    const double *c20, *c1, *c2;  // M_PRE: c2 of step 0, c1 and c2 of step 1; M_POST*: c1 (M_POST2) and c2 of the step
    const double* dsh;
};

// Coefficients of one system: {k0, kx, ky} (M_PRE), {k0, k1, k2} (M_POST*), {diag - d} (M_SPMV, M_RES).
template <int MODE>
__device__ __forceinline__ void coefs(const Lev& L, const Args64& a, int s, double (&k)[3]) {
    const double dg = 2.0 * (L.wx + L.wy) - a.dsh[s];
    if constexpr (MODE == M_PRE) {
        const double c20 = a.c20[s], c = a.c2[s] * c20;
        k[0] = fma(c20, 1.0 + a.c1[s], fma(-c, dg, a.c2[s]));
        k[1] = c * L.wx;
        k[2] = c * L.wy;
    } else if constexpr (MODE == M_SPMV || MODE == M_RES) {
        k[0] = MODE == M_RES ? -dg : dg;
        k[1] = k[2] = 0.0;
    } else {
        const double c1 = MODE == M_POST2 ? a.c1[s] : 0.0, c2 = a.c2[s];
        k[0] = 1.0 + c1 - c2 * dg;
        k[1] = c2;
        k[2] = -c1;
    }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, kCtas) k_sweep64(Lev L, int Kp, Args64 a, const double* pa, const double* pb, Red red) {
    __shared__ double ks[3][KMAXP];
    pdl_wait();
    const int off = threadIdx.x * 2;
    if (threadIdx.y == 0)
        for (int v = 0; v < 2; ++v) {
            double k[3];
            coefs<MODE>(L, a, off + v, k);
            for (int q = 0; q < 3; ++q) ks[q][off + v] = k[q];
        }
    __syncthreads();
    double2 k[3];
    for (int q = 0; q < 3; ++q) k[q] = make_double2(ks[q][off], ks[q][off + 1]);
    const double* __restrict__ x = MODE == M_SPMV ? (red.scal->parity ? pa : pb) : a.x;
    const size_t sy = (size_t)L.nx * Kp;
    Accum<double> acc;
    struct St {
        double2 c, h, w, b, e;
    };
    sweep_u<St>(
        L.N, blockIdx.x, gridDim.x,
        [&](int P, St& st) {
            const Coord q = coord<2>(L, P);
            const size_t base = (size_t)P * Kp + off;
            st.c = ld2(x + base);
            st.h = ld2_if(q.i > 0, x + base - Kp) + ld2_if(q.i < L.nx - 1, x + base + Kp);
            st.w = ld2_if(q.j > 0, x + base - sy) + ld2_if(q.j < L.ny - 1, x + base + sy);
            if (MODE == M_RES || MODE == M_POST1 || MODE == M_POST2) st.b = ld2(a.b + base);
            if (MODE == M_POST2) st.e = ld2(a.xin + base);
        },
        [&](int P, St& st) {
            const size_t base = (size_t)P * Kp + off;
            double2 o;
            if constexpr (MODE == M_PRE) {
                o = fma2(k[2], st.w, fma2(k[1], st.h, mul2(k[0], st.c)));
            } else if constexpr (MODE == M_RES) {
                o = fma2(L.wy, st.w, fma2(L.wx, st.h, fma2(k[0], st.c, st.b)));
            } else if constexpr (MODE == M_SPMV) {
                o = fma2(-L.wy, st.w, fma2(-L.wx, st.h, mul2(k[0], st.c)));
            } else {
                o = fma2(k[1], fma2(L.wy, st.w, fma2(L.wx, st.h, st.b)), mul2(k[0], st.c));
                if (MODE == M_POST2) o = fma2(k[2], st.e, o);
            }
            *reinterpret_cast<double2*>(a.out + base) = o;
            if (MODE == M_SPMV || (MODE == M_POST2 && red.op != RED_NONE)) {
                const double u[2] = {o.x, o.y}, v[2] = {MODE == M_SPMV ? st.c.x : st.b.x, MODE == M_SPMV ? st.c.y : st.b.y};
                acc.add(v, u);
            }
        });
    pdl_trigger();
    if (red.op != RED_NONE) reduce_finish<double>(acc, red, Kp);
}

// bc = R (b - (A - d I) x), full weighting, in one sweep.  A thread takes a coarse column and a run of coarse rows and
// forms, fine row by fine row, the residual on the column's three fine points, its x-weighted sum, and of three such rows
// the coarse value.
__global__ void __launch_bounds__(kRestrictThreads, 4) k_restrict64(Lev Lf, Lev Lc, int Kp, int run, const double* __restrict__ x,
                                                                    const double* __restrict__ b, double* __restrict__ bc,
                                                                    const double* __restrict__ dsh) {
    pdl_wait();
    const int off = threadIdx.x * 2;
    const double dg = 2.0 * (Lf.wx + Lf.wy);
    const double2 k0 = make_double2(dsh[off] - dg, dsh[off + 1] - dg);
    const int runs = (Lc.ny + run - 1) / run;
    const size_t sy = (size_t)Lf.nx * Kp;
    const long long it = (long long)blockIdx.x * blockDim.y + threadIdx.y;
    if (it >= (long long)runs * Lc.nx) return;
    const int rn = (int)(it / Lc.nx), I = (int)(it - (long long)rn * Lc.nx);
    const int J0 = rn * run, J1 = min(Lc.ny, J0 + run);
    // r(2I) + 2 r(2I + 1) + r(2I + 2) of fine row j
    auto row = [&](int j) {
        const size_t base = ((size_t)j * Lf.nx + 2 * I) * Kp + off;
        double2 c[5], r[3];
        c[0] = ld2_if(I > 0, x + base - Kp);
        for (int q = 0; q < 3; ++q) c[q + 1] = ld2(x + base + (size_t)q * Kp);
        c[4] = ld2_if(2 * I + 3 < Lf.nx, x + base + (size_t)3 * Kp);
        for (int q = 0; q < 3; ++q) {
            const size_t o = base + (size_t)q * Kp;
            const double2 w = ld2_if(j > 0, x + o - sy) + ld2_if(j < Lf.ny - 1, x + o + sy);
            r[q] = fma2(Lf.wy, w, fma2(Lf.wx, c[q] + c[q + 2], fma2(k0, c[q + 1], ld2(b + o))));
        }
        return fma2(2.0, r[1], r[0] + r[2]);
    };
    double2 lo = row(2 * J0);
    for (int J = J0; J < J1; ++J) {
        const double2 m = row(2 * J + 1), hi = row(2 * J + 2);
        double2 s = fma2(2.0, m, lo + hi);
        s.x *= 0.0625;
        s.y *= 0.0625;
        *reinterpret_cast<double2*>(bc + ((size_t)J * Lc.nx + I) * Kp + off) = s;
        lo = hi;
    }
}

// x += P ec (bilinear).  A thread takes the 2 x 2 fine points (2I, 2J) .. (2I + 1, 2J + 1), which lie between the coarse
// points I - 1, I and J - 1, J.
__global__ void __launch_bounds__(kThreads, kCtas) k_prolong64(Lev Lf, Lev Lc, int Kp, const double* __restrict__ ec, double* __restrict__ x) {
    pdl_wait();
    const int off = threadIdx.x * 2;
    const int cx = Lc.nx + 1;
    const long long items = (long long)cx * (Lc.ny + 1);
    for (long long it = (long long)blockIdx.x * blockDim.y + threadIdx.y; it < items; it += (long long)gridDim.x * blockDim.y) {
        const int J = (int)(it / cx), I = (int)(it - (long long)J * cx);
        const bool xl = I > 0, xh = I < Lc.nx, yl = J > 0, yh = J < Lc.ny;
        const double* e = ec + ((long long)J * Lc.nx + I) * Kp + off;  // coarse (I, J)
        const ptrdiff_t ey = (ptrdiff_t)Lc.nx * Kp;
        const double2 e11 = ld2_if(xh && yh, e), e01 = ld2_if(xl && yh, e - Kp);
        const double2 e10 = ld2_if(xh && yl, e - ey), e00 = ld2_if(xl && yl, e - ey - Kp);
        double* o = x + ((size_t)(2 * J) * Lf.nx + 2 * I) * Kp + off;
        double* o1 = o + (size_t)Lf.nx * Kp;
        const double2 top = e01 + e11;
        const double2 x00 = ld2(o), x01 = ld2_if(xh, o + Kp), x10 = ld2_if(yh, o1), x11 = ld2_if(xh && yh, o1 + Kp);
        auto put = [](double* p, double2 v) { *reinterpret_cast<double2*>(p) = v; };
        put(o, fma2(0.25, top + (e00 + e10), x00));
        if (xh) put(o + Kp, fma2(0.5, e10 + e11, x01));
        if (yh) put(o1, fma2(0.5, top, x10));
        if (xh && yh) put(o1 + Kp, x11 + e11);
    }
}

dim3 block64(int Kp, int threads = kThreads) { return dim3((unsigned)(Kp / 2), (unsigned)(threads / (Kp / 2))); }

template <int MODE>
void sweep(const Lev& L, int Kp, int nsm, const Args64& a, const double* pa, const double* pb, const Red& red, cudaStream_t s) {
    const dim3 blk = block64(Kp);
    const long long tiles = (L.N + blk.y - 1) / blk.y;
    const size_t smem = red.op != RED_NONE ? (size_t)blk.x * blk.y * 2 * sizeof(double) : 0;
    launch_pdl(k_sweep64<MODE>, dim3((unsigned)std::min<long long>(tiles, (long long)nsm * kCtas)), blk, smem, s, L, Kp, a, pa, pb, red);
}

}  // namespace

void sweep64_pre2(const Lev& L, int Kp, int nsm, const double* b, double* x, ChebStepT<double> c0, ChebStepT<double> c1,
                  const double* dsh, const Red& none, cudaStream_t s) {
    sweep<M_PRE>(L, Kp, nsm, Args64{b, nullptr, nullptr, x, c0.c2, c1.c1, c1.c2, dsh}, nullptr, nullptr, none, s);
}

void sweep64_residual(const Lev& L, int Kp, int nsm, const double* x, const double* b, double* r, const double* dsh,
                      const Red& none, cudaStream_t s) {
    sweep<M_RES>(L, Kp, nsm, Args64{x, b, nullptr, r, nullptr, nullptr, nullptr, dsh}, nullptr, nullptr, none, s);
}

void sweep64_restrict(const Lev& Lf, const Lev& Lc, int Kp, int nsm, const double* x, const double* b, double* bc,
                      const double* dsh, cudaStream_t s) {
    const dim3 blk = block64(Kp, kRestrictThreads);
    // runs of up to 8 coarse rows (a run forms one fine row more than it owns), shorter ones where fewer than four CTAs
    // per SM would come of them
    const int run = (int)std::max(1LL, std::min(8LL, Lc.N / ((long long)nsm * 4 * blk.y)));
    const long long items = (long long)((Lc.ny + run - 1) / run) * Lc.nx;
    launch_pdl(k_restrict64, dim3((unsigned)((items + blk.y - 1) / blk.y)), blk, 0, s, Lf, Lc, Kp, run, x, b, bc, dsh);
}

void sweep64_prolong(const Lev& Lf, const Lev& Lc, int Kp, int nsm, const double* ec, double* x, cudaStream_t s) {
    const dim3 blk = block64(Kp);
    const long long items = (long long)(Lc.nx + 1) * (Lc.ny + 1);
    launch_pdl(k_prolong64, dim3((unsigned)std::min<long long>((items + blk.y - 1) / blk.y, (long long)nsm * kCtas)), blk, 0, s, Lf, Lc, Kp,
               ec, x);
}

void sweep64_post1(const Lev& L, int Kp, int nsm, const double* x, double* x1, const double* b, ChebStepT<double> c0,
                   const double* dsh, const Red& none, cudaStream_t s) {
    sweep<M_POST1>(L, Kp, nsm, Args64{x, b, nullptr, x1, nullptr, nullptr, c0.c2, dsh}, nullptr, nullptr, none, s);
}

void sweep64_post2(const Lev& L, int Kp, int nsm, double* x, const double* x1, const double* b, ChebStepT<double> c1,
                   const double* dsh, const Red& red, cudaStream_t s) {
    sweep<M_POST2>(L, Kp, nsm, Args64{x1, b, x, x, nullptr, c1.c1, c1.c2, dsh}, nullptr, nullptr, red, s);
}

void sweep64_spmv(const Lev& L, int Kp, int nsm, const double* pa, const double* pb, double* q, const Red& red, cudaStream_t s) {
    const double* dsh = reinterpret_cast<const double*>(reinterpret_cast<const char*>(red.scal) + offsetof(Scal, dsh));
    sweep<M_SPMV>(L, Kp, nsm, Args64{nullptr, nullptr, nullptr, q, nullptr, nullptr, nullptr, dsh}, pa, pb, red, s);
}

}  // namespace bura
