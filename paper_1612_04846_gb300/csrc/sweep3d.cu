// The 3-D sweeps of the multigrid-preconditioned CG (FP32) with their inputs staged in shared memory by TMA, each
// fused with the pointwise or grid-transfer pass before or after it:
//   STEP   one Chebyshev step                      x, b, d in; x, d out (and b . x)
//   PRE    both pre-smoothing steps from zero      b in; x2 out
//   RESR   the residual and its full weighting     x, b in; the coarse right-hand side out
//   PROL   prolongation and first post-smoothing   x, ec, b in; x1, d1 out
//   SPMV   p = z + beta p and q = (A - d_j I) p    z, p in; p, q out (and p . q)
//
// A work item is a tile of kPX x kPY points of the (x, y) plane over pz consecutive planes.  A CTA of Kp/4 x RX x RY
// threads (one 16-byte chunk of one point each) marches the item along z: a ring of kPRing plane slots in shared
// memory holds, per plane, the vectors a stencil reads with a one-point halo, the pointwise ones, and for variable
// coefficients the packed weights (a float4 per point: the faces below it along x, y, z and its diagonal).  One thread
// fills a slot with one tiled TMA load per vector, kPRing - 2 planes ahead of the plane being computed; zero fill
// outside the grid is the homogeneous Dirichlet boundary.  Where the stencil reads a value that is not stored (the
// first iterate c2 Dinv b of PRE, x + P ec of PROL, z + beta p of SPMV), it is formed once per point of the tile and
// its halo into a ring of three planes; one CTA barrier per plane publishes it and frees the oldest slots.  x on the
// plane below and on the current one stays in registers; per point the arithmetic is the z-marching sweep's (zmarch in
// kernels_impl.cuh), operation for operation, in packed pairs.
// RESR computes the residual on the 17 x 9 points that the tile's 8 x 4 coarse points read, sums it along z in
// registers (1/4, 1/2, 1/4) and, every second plane, along y and x through shared memory.
//
// Measured on the fine level of a 255^3, k = 9 solve with variable coefficients (one vector is 796 MB with its padding),
// one launch, against the passes each replaces (per-thread cp.async staging or grid sweeps): PRE 0.48 ms (0.27 + 0.60),
// RESR 0.44 (0.52 + 0.21), PROL 0.63 (0.37 + 0.60), STEP 0.53 (0.65), SPMV 0.57 (0.37 + 0.59); the solve 148.5 -> 107.3 ms.
// STEP, PROL and SPMV run at 5.7 to 6.7 TB/s of DRAM traffic (ncu; a plain copy 6.8); PRE and RESR, with half the vectors
// per point, move 3.3 to 4.6 and wait for shared memory and the plane's barrier (half to 58 % of the issue slots taken).
// With the copies and their addresses done by the threads the same five passes issued 3 to 4 times the instructions (PRE
// 460 per warp and chunk) and were no faster than the passes they replace.
#include "kernels_impl.cuh"
#include "tma.cuh"

namespace bura {

namespace {

constexpr int kPX = 16, kPY = 8;      // tile points along x and y
#ifndef BURA_3S_PZ
#define BURA_3S_PZ 128
#endif
constexpr int kPZ = BURA_3S_PZ;       // planes per work item on levels whose items fill the grid
constexpr int kPRing = 4;             // plane slots of the ring
constexpr int kVRing = 3;             // planes of formed values
constexpr int kCX = kPX / 2 + 2, kCY = kPY / 2 + 2;  // coarse points that the tile and its halo interpolate from
constexpr int kCRing = 4;             // coarse planes held by PROL

__host__ __device__ constexpr int up128(int bytes) { return (bytes + 127) / 128 * 128; }

// Points a mode computes per plane, and the byte offsets of a slot.
template <int MODE, bool VAR>
struct Geo {
    static constexpr int RX = MODE == S3_RESR ? kPX + 1 : kPX, RY = MODE == S3_RESR ? kPY + 1 : kPY;
    static constexpr int HX = RX + 2, HY = RY + 2;  // with the one-point halo
    static constexpr int pts = RX * RY, halo = HX * HY;
    static constexpr bool form = MODE == S3_PRE || MODE == S3_PROL || MODE == S3_SPMV;  // the stencil's value is formed
    static constexpr bool second = MODE == S3_SPMV;                      // a second vector with its halo (p)
    static constexpr bool tile_b = MODE != S3_SPMV && MODE != S3_PRE;    // b on the tile (PRE reads it from the halo box)
    static constexpr bool tile_d = MODE == S3_STEP;                      // the previous direction on the tile
    __host__ __device__ static constexpr int hb(int Kp) { return up128(halo * Kp * 4); }
    __host__ __device__ static constexpr int tb(int Kp) { return up128(pts * Kp * 4); }
    __host__ __device__ static constexpr int o_p(int Kp) { return hb(Kp); }
    __host__ __device__ static constexpr int o_b(int Kp) { return o_p(Kp) + (second ? hb(Kp) : 0); }
    __host__ __device__ static constexpr int o_d(int Kp) { return o_b(Kp) + (tile_b ? tb(Kp) : 0); }
    __host__ __device__ static constexpr int o_w(int Kp) { return o_d(Kp) + (tile_d ? tb(Kp) : 0); }
    __host__ __device__ static constexpr int slot(int Kp) { return o_w(Kp) + (VAR ? up128(halo * 16) : 0); }
    // after the ring: the formed planes, then PROL's coarse planes or RESR's sums along z
    __host__ __device__ static constexpr int o_v(int Kp) { return kPRing * slot(Kp); }
    __host__ __device__ static constexpr int o_e(int Kp) { return o_v(Kp) + (form ? kVRing * hb(Kp) : 0); }
    __host__ __device__ static constexpr int eb(int Kp) { return up128(kCX * kCY * Kp * 4); }
    __host__ __device__ static constexpr int bytes(int Kp) {
        return o_e(Kp) + (MODE == S3_PROL ? kCRing * eb(Kp) : MODE == S3_RESR ? tb(Kp) : 0);
    }
    // bytes that TMA brings per plane (without PROL's coarse plane)
    __host__ __device__ static constexpr unsigned due(int Kp, bool din) {
        return (unsigned)(halo * Kp * 4 * (second ? 2 : 1) + (tile_b ? pts * Kp * 4 : 0) + (tile_d && din ? pts * Kp * 4 : 0) +
                          (VAR ? halo * 16 : 0));
    }
    static size_t smem(int Kp) { return (size_t)bytes(Kp) + 128; }  // + the alignment of the first slot
};

struct P4 {
    float2 a, b;
};
__device__ __forceinline__ P4 ldp(const void* q) {
    const float4 v = *reinterpret_cast<const float4*>(q);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void stp(void* q, P4 v) { *reinterpret_cast<float4*>(q) = make_float4(v.a.x, v.a.y, v.b.x, v.b.y); }
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ P4 mul(float s, P4 x) { return {__fmul2_rn(dup2(s), x.a), __fmul2_rn(dup2(s), x.b)}; }
__device__ __forceinline__ P4 mul(P4 s, P4 x) { return {__fmul2_rn(s.a, x.a), __fmul2_rn(s.b, x.b)}; }
__device__ __forceinline__ P4 mad(float s, P4 x, P4 y) { return {__ffma2_rn(dup2(s), x.a, y.a), __ffma2_rn(dup2(s), x.b, y.b)}; }
__device__ __forceinline__ P4 mad(P4 s, P4 x, P4 y) { return {__ffma2_rn(s.a, x.a, y.a), __ffma2_rn(s.b, x.b, y.b)}; }
__device__ __forceinline__ P4 add(P4 x, P4 y) { return {__fadd2_rn(x.a, y.a), __fadd2_rn(x.b, y.b)}; }
__device__ __forceinline__ P4 neg(P4 x) { return {make_float2(-x.a.x, -x.a.y), make_float2(-x.b.x, -x.b.y)}; }
__device__ __forceinline__ P4 sub(P4 x, P4 y) {
    return {make_float2(x.a.x - y.a.x, x.a.y - y.a.y), make_float2(x.b.x - y.b.x, x.b.y - y.b.y)};
}
__device__ __forceinline__ P4 jdiv4(P4 x, float dp, P4 d) {
    return {make_float2(jdiv(x.a.x, dp - d.a.x), jdiv(x.a.y, dp - d.a.y)), make_float2(jdiv(x.b.x, dp - d.b.x), jdiv(x.b.y, dp - d.b.y))};
}

}  // namespace

// The arguments of a launch.  Maps: v (halo box), p's two buffers (SPMV, halo boxes), b and din (tile boxes), ec, weights.
struct Sweep3 {
    CUtensorMap v, p0, p1, b, d, e, w;
    float *out, *out2, *pa, *pb;
    const float* din;         // null: no previous direction
    ChebStepT<float> c0, c1;  // PRE: first and second step; else c1
    const float* dsh;
    int nx, ny, nz;
    int ncx, ncy, ncz;        // the coarse level of RESR and PROL
    int pz;                   // planes (RESR: coarse planes) per item
    float wx, wy, wz;         // constant coefficients
};

template <int C, bool VAR, int MODE>
__global__ void __launch_bounds__(C * Geo<MODE, VAR>::pts, C <= 3 ? 2 : 1) k_sweep3s(const __grid_constant__ Sweep3 a, Red red) {
    pdl_wait();
    using G = Geo<MODE, VAR>;
    constexpr int Kp = 4 * C, nthr = C * G::pts, Pb = Kp * 4;  // Pb: bytes of a point
    extern __shared__ __align__(128) unsigned char raw3[];
    __shared__ __align__(8) uint64_t bars[kPRing], bar_e;
    unsigned char* const ring = raw3 + ((128u - (smem_u32(raw3) & 127u)) & 127u);
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int c = threadIdx.x, p = threadIdx.y;
    const int off = c * 4;
    const int px = p % G::RX, py = p / G::RX;
    const int tid = p * C + c;
    float* __restrict__ pout = nullptr;
    const CUtensorMap* mpin = &a.p0;            // SPMV: the previous direction
    P4 c20, c1, c2, d;                          // c20: the first step's c2 (PRE), beta (SPMV)
    if constexpr (MODE == S3_SPMV) {
        const int par = red.scal->parity;
        mpin = par ? &a.p1 : &a.p0;
        pout = par ? a.pa : a.pb;
        c20 = ldp(red.scal->betaf + off);
        d = ldp(red.scal->dshf + off);
    } else {
        if (MODE == S3_PRE) c20 = ldp(a.c0.c2 + off);
        if (MODE != S3_RESR) {
            c1 = a.c1.c1 ? ldp(a.c1.c1 + off) : P4{dup2(0.f), dup2(0.f)};
            c2 = ldp(a.c1.c2 + off);
        }
        d = ldp(a.dsh + off);
    }
    const bool dot = (MODE == S3_STEP && red.op != RED_NONE) || MODE == S3_SPMV;
    const bool has_d = MODE == S3_STEP && a.din != nullptr;
    const unsigned due = G::due(Kp, has_d);
    const long long budget = red.scal->wait_cycles > 0 ? red.scal->wait_cycles : kTmaWaitCycles;
    Accum<float> acc;
    if (tid == 0) {
        for (int q = 0; q < kPRing; ++q) mbar_init(&bars[q], 1);
        mbar_init(&bar_e, 1);
        mbar_fence_init();
    }
    __syncthreads();
    const int ntx = MODE == S3_RESR ? (a.ncx + kPX / 2 - 1) / (kPX / 2) : (nx + kPX - 1) / kPX;
    const int nty = MODE == S3_RESR ? (a.ncy + kPY / 2 - 1) / (kPY / 2) : (ny + kPY - 1) / kPY;
    const int nzs = ((MODE == S3_RESR ? a.ncz : nz) + a.pz - 1) / a.pz;
    const int items = ntx * nty * nzs;
    const size_t pv = (size_t)nx * ny * Kp;  // floats per plane of a vector
    // the chunks of the halo that this thread forms: tid and tid + nthr (chunk offset c in both); their point, and for
    // PROL the coarse point they interpolate from and the steps to its neighbours (0: an odd fine coordinate)
    const int h0 = tid / C, h1 = (tid + nthr) / C;
    const bool second = tid + nthr < G::halo * C;
    const int hc = (py + 1) * G::HX + px + 1;  // the own point in the halo box
    unsigned fill = 0;                         // planes fetched so far by this CTA: slot fill % kPRing, phase fill / kPRing
    unsigned nex = 0;                          // uses of bar_e
    bool ok = true;
    for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const int tz = item / (ntx * nty);
        const int rem = item - tz * ntx * nty;
        const int ty = rem / ntx, tx = rem - ty * ntx;
        const int X0 = tx * kPX, Y0 = ty * kPY;
        // planes [l0, l1) computed (RESR: both ends of its coarse planes' footprint); l0 - 1 .. l1 fetched
        const int l0 = MODE == S3_RESR ? 2 * tz * a.pz : tz * a.pz;
        const int l1 = MODE == S3_RESR ? 2 * min(a.ncz, (tz + 1) * a.pz) + 1 : min(nz, l0 + a.pz);
        const unsigned f0 = fill;                // plane l is the fetch f0 + l - (l0 - 1)
        auto fetch = [&](int l) {                // thread 0
            const unsigned n = f0 + (unsigned)(l - l0 + 1);
            unsigned char* S = ring + (n % kPRing) * G::slot(Kp);
            uint64_t* bar = &bars[n % kPRing];
            // PROL: coarse plane m with fine plane 2m - 1, two barriers before plane 2m is formed
            const bool with_e = MODE == S3_PROL && (l & 1) && l > l0;
            mbar_expect_tx(bar, due + (with_e ? (unsigned)(kCX * kCY * Pb) : 0u));
            tma_load_3d(S, &a.v, (X0 - 1) * (Kp / 2), Y0 - 1, l, bar);
            if (G::second) tma_load_3d(S + G::o_p(Kp), mpin, (X0 - 1) * (Kp / 2), Y0 - 1, l, bar);
            if (G::tile_b) tma_load_3d(S + G::o_b(Kp), &a.b, X0 * (Kp / 2), Y0, l, bar);
            if (G::tile_d && has_d) tma_load_3d(S + G::o_d(Kp), &a.d, X0 * (Kp / 2), Y0, l, bar);
            if (VAR) tma_load_3d(S + G::o_w(Kp), &a.w, (X0 - 1) * 2, Y0 - 1, l, bar);
            if (with_e) {
                const int m = (l + 1) >> 1;
                tma_load_3d(ring + G::o_e(Kp) + (m % kCRing) * G::eb(Kp), &a.e, (X0 / 2 - 1) * (Kp / 2), Y0 / 2 - 1, m, bar);
            }
        };
        auto wait = [&](int l) {
            const unsigned n = f0 + (unsigned)(l - l0 + 1);
            return mbar_wait_bounded(&bars[n % kPRing], (n / kPRing) & 1u, budget);
        };
        auto slot = [&](int l) { return ring + ((f0 + (unsigned)(l - l0 + 1)) % kPRing) * G::slot(Kp); };
        auto vslot = [&](int l) { return G::form ? ring + G::o_v(Kp) + ((l + kVRing) % kVRing) * G::hb(Kp) : slot(l); };
        // the value that the stencil reads at halo chunk i (point h), from plane l's landed slot
        auto form_at = [&](int l, const unsigned char* S, unsigned char* V, int i, int h) {
            P4 v = ldp(S + 16 * i);
            if constexpr (MODE == S3_PRE) {
                if (VAR) {
                    const float dp = *reinterpret_cast<const float*>(S + G::o_w(Kp) + 16 * h + 12);
                    v = mul(c20, v);
                    v = dp > 0.f ? jdiv4(v, dp, d) : P4{dup2(0.f), dup2(0.f)};  // zero outside the grid
                } else {
                    v = mul(c20, v);
                }
            } else if constexpr (MODE == S3_SPMV) {
                v = mad(c20, ldp(S + G::o_p(Kp) + 16 * i), v);
            } else if constexpr (MODE == S3_PROL) {
                const int hx = h % G::HX, hy = h / G::HX;  // fine point (X0 - 1 + hx, Y0 - 1 + hy), X0 and Y0 even
                const int gx = X0 - 1 + hx, gy = Y0 - 1 + hy;
                if (gx >= 0 && gx < nx && gy >= 0 && gy < ny && l >= 0 && l < nz) {
                    const int e0 = ((hy >> 1) * kCX + (hx >> 1)) * Pb + off * 4;  // hx even: an odd fine column
                    const int ex = (hx & 1) * Pb, ey = (hy & 1) * kCX * Pb;
                    auto bil = [&](int m) {
                        const unsigned char* E = ring + G::o_e(Kp) + ((m + kCRing) % kCRing) * G::eb(Kp) + e0;
                        return mad(0.25f, ldp(E + ex + ey), mad(0.25f, ldp(E + ey), mad(0.25f, ldp(E + ex), mul(0.25f, ldp(E)))));
                    };
                    if (l & 1) v = add(v, bil(l >> 1));
                    else v = add(v, mad(0.5f, bil(l >> 1), mul(0.5f, bil((l >> 1) - 1))));
                }
            }
            stp(V + 16 * i, v);
        };
        auto form = [&](int l) {
            if constexpr (G::form) {
                const unsigned char* S = slot(l);
                unsigned char* V = vslot(l);
                form_at(l, S, V, tid, h0);
                if (second) form_at(l, S, V, tid + nthr, h1);
            }
        };
        if (tid == 0) {
            if (MODE == S3_PROL) {  // the coarse planes of planes l0 - 1 and l0 (l0 even); fetch() brings the later ones
                mbar_expect_tx(&bar_e, 2u * kCX * kCY * Pb);
                for (int m = (l0 >> 1) - 1; m <= (l0 >> 1); ++m)
                    tma_load_3d(ring + G::o_e(Kp) + ((m + kCRing) % kCRing) * G::eb(Kp), &a.e, (X0 / 2 - 1) * (Kp / 2), Y0 / 2 - 1,
                                m, &bar_e);
            }
            for (int l = l0 - 1; l < l0 + kPRing - 1 && l <= l1; ++l) fetch(l);
        }
        bool got = true;
        if (MODE == S3_PROL) got = mbar_wait_bounded(&bar_e, nex & 1u, budget);
        ++nex;
        got = got && wait(l0 - 1) && wait(l0);
        if (got) {
            form(l0 - 1);
            form(l0);
        }
        const int gx = X0 + px, gy = Y0 + py;
        const bool mine = gx < nx && gy < ny;
        const size_t g0 = mine ? ((size_t)gy * nx + gx) * Kp + off : 0;
        P4 xm1, x0;
        if (G::form) __syncthreads();  // planes l0 - 1 and l0 are formed
        xm1 = ldp(vslot(l0 - 1) + hc * Pb + off * 4);
        x0 = ldp(vslot(l0) + hc * Pb + off * 4);
        float wzm = VAR ? *reinterpret_cast<const float*>(slot(l0) + G::o_w(Kp) + 16 * hc + 8) : a.wz;
        P4 rs{dup2(0.f), dup2(0.f)};           // RESR: the sum along z of the open coarse plane
        unsigned char* const sums = ring + G::o_e(Kp);
        auto emit = [&](int Lc) {              // RESR: coarse plane Lc from the sums along z
            if (p < (kPX / 2) * (kPY / 2)) {
                const int ix = p % (kPX / 2), iy = p / (kPX / 2);
                const int I = X0 / 2 + ix, J = Y0 / 2 + iy;
                if (I < a.ncx && J < a.ncy) {
                    P4 t{dup2(0.f), dup2(0.f)};
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
                            t = mad((dx == 1 ? 0.5f : 0.25f) * (dy == 1 ? 0.5f : 0.25f),
                                    ldp(sums + ((2 * iy + dy) * G::RX + 2 * ix + dx) * Pb + off * 4), t);
                    stp(a.out + (((size_t)Lc * a.ncy + J) * a.ncx + I) * Kp + off, t);
                }
            }
        };
        int l = l0;
        for (; l < l1; ++l) {
            got = got && wait(l + 1);
            if (got) form(l + 1);
            // plane l + 1 is formed; every thread is done with plane l - 1 (and its slot)
            if (__syncthreads_or(!got)) { ok = false; break; }
            if (tid == 0 && l + kPRing - 1 <= l1) fetch(l + kPRing - 1);
            if constexpr (MODE == S3_RESR)
                if ((l & 1) && l > l0 + 1) emit((l - 3) >> 1);  // the plane that the last even plane closed
            const unsigned char* S = slot(l);
            const unsigned char* Vc = vslot(l) + hc * Pb + off * 4;
            P4 wp = ldp(vslot(l + 1) + hc * Pb + off * 4);  // x on the plane above
            float wxm, wxp, wym, wyp, wzp, diag;
            if (VAR) {
                const float4 w = *reinterpret_cast<const float4*>(S + G::o_w(Kp) + 16 * hc);
                wxm = w.x;
                wym = w.y;
                diag = w.w;
                wxp = *reinterpret_cast<const float*>(S + G::o_w(Kp) + 16 * (hc + 1));
                wyp = *reinterpret_cast<const float*>(S + G::o_w(Kp) + 16 * (hc + G::HX) + 4);
                wzp = *reinterpret_cast<const float*>(slot(l + 1) + G::o_w(Kp) + 16 * hc + 8);
            } else {
                wxm = wxp = a.wx;
                wym = wyp = a.wy;
                wzp = a.wz;
                diag = wxm + wxp + wym + wyp;
                diag += wzm + wzp;
            }
            P4 t = mul(diag, x0);
            t = mad(-wxm, ldp(Vc - Pb), t);
            t = mad(-wxp, ldp(Vc + Pb), t);
            t = mad(-wym, ldp(Vc - G::HX * Pb), t);
            t = mad(-wyp, ldp(Vc + G::HX * Pb), t);
            t = mad(-wzm, xm1, t);
            t = mad(-wzp, wp, t);
            const P4 ax = mad(neg(d), x0, t);
            const size_t go = (size_t)l * pv + g0;
            if constexpr (MODE == S3_SPMV) {
                if (mine) {
                    stp(pout + go, x0);
                    stp(a.out + go, ax);
                    const float pa4[4] = {x0.a.x, x0.a.y, x0.b.x, x0.b.y}, qa4[4] = {ax.a.x, ax.a.y, ax.b.x, ax.b.y};
                    acc.add(pa4, qa4);
                }
            } else {
                const P4 bv = MODE == S3_PRE ? ldp(S + hc * Pb + off * 4) : ldp(S + G::o_b(Kp) + p * Pb + off * 4);
                const P4 res = sub(bv, ax);
                if constexpr (MODE == S3_RESR) {
                    if (l & 1) {
                        rs = mad(0.5f, res, rs);
                    } else {
                        rs = mad(0.25f, res, rs);
                        if (l > l0) stp(sums + p * Pb + off * 4, rs);
                        rs = mul(0.25f, res);
                    }
                } else {
                    P4 g = mul(c2, res);
                    if (VAR) g = jdiv4(g, diag, d);
                    P4 dv;
                    if (MODE == S3_PRE) dv = mad(c1, x0, g);
                    else if (MODE == S3_STEP && has_d) dv = mad(c1, ldp(S + G::o_d(Kp) + p * Pb + off * 4), g);
                    else dv = g;
                    const P4 xo = add(x0, dv);
                    if (mine) {
                        stp(a.out + go, xo);
                        if (a.out2) stp(a.out2 + go, dv);
                        if (MODE == S3_STEP && dot) {
                            const float ba[4] = {bv.a.x, bv.a.y, bv.b.x, bv.b.y}, xa4[4] = {xo.a.x, xo.a.y, xo.b.x, xo.b.y};
                            acc.add(ba, xa4);
                        }
                    }
                }
            }
            xm1 = x0;
            x0 = wp;
            wzm = wzp;
        }
        fill = f0 + (unsigned)(l1 - l0 + 2);
        if (!ok) {  // the copies in flight (planes l - 1 .. l + 2) land before the CTA exits
            for (int q = l - 1; q < l + kPRing - 1 && q <= l1; ++q) {
                const unsigned n = f0 + (unsigned)(q - l0 + 1);
                (void)mbar_wait_bounded(&bars[n % kPRing], (n / kPRing) & 1u, kTmaWaitCycles);
            }
            if (MODE == S3_PROL) (void)mbar_wait_bounded(&bar_e, (nex - 1) & 1u, kTmaWaitCycles);
            if (tid == 0) atomicExch(&red.scal->fault, 1);
        }
        __syncthreads();  // every thread is done with the item's slots before the next item refills them
        if constexpr (MODE == S3_RESR) {
            if (ok) emit((l1 - 3) >> 1);
            __syncthreads();
        }
    }
    pdl_trigger();
    if (dot) reduce_finish<float>(acc, red, Kp);
}

namespace {

// Work items of a level: kPZ planes each where that fills the CTA slots; smaller levels take the height (64 down to 8
// planes) whose rounds of items over the slots march the fewest planes, with kWarm planes per item to fill its ring.
// cols: tiles of a plane; planes: along z.
constexpr int kWarm = 4;
int item_grid(long long cols, int planes, long long slots, int& pz) {
    pz = kPZ;
    if (cols * ((planes + pz - 1) / pz) < slots) {
        long long best = 1LL << 60;
        for (int q = kPZ; q >= 8; q /= 2) {
            const long long cost = (cols * ((planes + q - 1) / q) + slots - 1) / slots * (std::min(q, planes) + kWarm);
            if (cost < best) { best = cost; pz = q; }
        }
    }
    return (int)std::min<long long>(cols * ((planes + pz - 1) / pz), slots);
}

template <int C, bool VAR, int MODE>
cudaError_t prepare3() {
    return cudaFuncSetAttribute(k_sweep3s<C, VAR, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Geo<MODE, VAR>::smem(4 * C));
}

}  // namespace

#define BURA_3S_SWITCH(Kp, var, CALL)                                         \
    switch (Kp) {                                                             \
        case 4: if (var) { constexpr int C = 1; constexpr bool V = true; CALL; } else { constexpr int C = 1; constexpr bool V = false; CALL; } break; \
        case 8: if (var) { constexpr int C = 2; constexpr bool V = true; CALL; } else { constexpr int C = 2; constexpr bool V = false; CALL; } break; \
        case 12: if (var) { constexpr int C = 3; constexpr bool V = true; CALL; } else { constexpr int C = 3; constexpr bool V = false; CALL; } break; \
        case 16: if (var) { constexpr int C = 4; constexpr bool V = true; CALL; } else { constexpr int C = 4; constexpr bool V = false; CALL; } break; \
        default: return cudaErrorInvalidValue;                                \
    }

cudaError_t sweep3_prepare(int Kp, bool var) {
    cudaError_t e = cudaSuccess;
    auto first = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    BURA_3S_SWITCH(Kp, var, (first(prepare3<C, V, S3_STEP>()), first(prepare3<C, V, S3_PRE>()), first(prepare3<C, V, S3_RESR>()),
                             first(prepare3<C, V, S3_PROL>()), first(prepare3<C, V, S3_SPMV>())))
    return e;
}

void sweep3_box(int box, int* bx, int* by) {
    switch (box) {
        case S3B_HALO: *bx = kPX + 2; *by = kPY + 2; break;
        case S3B_TILE: *bx = kPX; *by = kPY; break;
        case S3B_RHALO: *bx = kPX + 3; *by = kPY + 3; break;
        case S3B_RTILE: *bx = kPX + 1; *by = kPY + 1; break;
        default: *bx = kCX; *by = kCY; break;
    }
}

namespace {

template <int MODE>
cudaError_t launch3(const Sweep3Lev& g, Sweep3 a, const Red& red, cudaStream_t s) {
    a.nx = g.nx; a.ny = g.ny; a.nz = g.nz;
    a.ncx = g.ncx; a.ncy = g.ncy; a.ncz = g.ncz;
    a.wx = g.wx; a.wy = g.wy; a.wz = g.wz;
    const long long cols = MODE == S3_RESR ? (long long)((a.ncx + kPX / 2 - 1) / (kPX / 2)) * ((a.ncy + kPY / 2 - 1) / (kPY / 2))
                                           : (long long)((a.nx + kPX - 1) / kPX) * ((a.ny + kPY - 1) / kPY);
    const long long slots = (long long)(g.Kp <= 12 ? 2 : 1) * g.nsm;
    const int grid = item_grid(cols, MODE == S3_RESR ? a.ncz : a.nz, slots, a.pz);
    BURA_3S_SWITCH(g.Kp, g.var, launch_pdl(k_sweep3s<C, V, MODE>, dim3(grid), dim3(C, Geo<MODE, V>::pts),
                                           Geo<MODE, V>::smem(4 * C), s, a, red))
    return cudaGetLastError();
}

}  // namespace

cudaError_t sweep3_step(const Sweep3Lev& g, const CUtensorMap* x, bool has_din, const CUtensorMap* din, const CUtensorMap* b,
                        float* xout, float* dout, ChebStepT<float> cs, const float* dsh, const Red& red, cudaStream_t s) {
    Sweep3 a{};
    if (!x || !b || (has_din && !din)) return cudaErrorInvalidValue;
    a.v = *x; a.b = *b; a.out = xout; a.out2 = dout; a.c1 = cs; a.dsh = dsh; a.w = g.w;
    a.d = has_din ? *din : *b;
    a.din = has_din ? dsh : nullptr;  // (a flag)
    return launch3<S3_STEP>(g, a, red, s);
}
cudaError_t sweep3_pre(const Sweep3Lev& g, const CUtensorMap* b, float* xout, float* dout, ChebStepT<float> c0,
                       ChebStepT<float> c1, const float* dsh, const Red& none, cudaStream_t s) {
    Sweep3 a{};
    if (!b) return cudaErrorInvalidValue;
    a.v = *b; a.out = xout; a.out2 = dout; a.c0 = c0; a.c1 = c1; a.dsh = dsh; a.w = g.w;
    return launch3<S3_PRE>(g, a, none, s);
}
cudaError_t sweep3_residual_restrict(const Sweep3Lev& g, const CUtensorMap* x, const CUtensorMap* b, float* bc, const float* dsh,
                                     const Red& none, cudaStream_t s) {
    Sweep3 a{};
    if (!x || !b) return cudaErrorInvalidValue;
    a.v = *x; a.b = *b; a.out = bc; a.dsh = dsh; a.w = g.wr;
    return launch3<S3_RESR>(g, a, none, s);
}
cudaError_t sweep3_prolong_step(const Sweep3Lev& g, const CUtensorMap* x, const CUtensorMap* ec, const CUtensorMap* b,
                                float* xout, float* dout, ChebStepT<float> cs, const float* dsh, const Red& none,
                                cudaStream_t s) {
    Sweep3 a{};
    if (!x || !ec || !b) return cudaErrorInvalidValue;
    a.v = *x; a.e = *ec; a.b = *b; a.out = xout; a.out2 = dout; a.c1 = cs; a.dsh = dsh; a.w = g.w;
    return launch3<S3_PROL>(g, a, none, s);
}
cudaError_t sweep3_spmv(const Sweep3Lev& g, const CUtensorMap* z, const CUtensorMap* mpa, const CUtensorMap* mpb, float* pa,
                        float* pb, float* q, const Red& red, cudaStream_t s) {
    Sweep3 a{};
    if (!z || !mpa || !mpb) return cudaErrorInvalidValue;
    a.v = *z; a.p0 = *mpa; a.p1 = *mpb; a.pa = pa; a.pb = pb; a.out = q; a.w = g.w;
    return launch3<S3_SPMV>(g, a, red, s);
}

}  // namespace bura
