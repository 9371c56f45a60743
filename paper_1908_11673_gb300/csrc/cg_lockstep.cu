// Conjugate gradients of several right-hand sides in lockstep, scalars on the device
// (Sec. 4.4 CG; the correction solves of the multi-shift CG, App. A.2, and the normal-equation
// solves that take over where restarted GCR stalls).
//
//   shifted:  (Dhat^+ Dhat + sigma_j) e_j = b_j, stopped at |r_j| <= rtol_j |b_j|
//   normal:   min |b_j - Dhat e_j| (CG on the normal equations, tracking s = b - Dhat e),
//             stopped at |s_j| <= rtol_j |b_j|
//
// FP32 half-lattice fields, the right-hand sides one after the other.  Every right-hand side
// has its own scalars in device memory; one that has stopped is left alone (its blocks return
// at once), so that an iteration is a fixed sequence of launches without a host round trip:
//
//   t = A_oo^-1 H_oe p;  w = A_ee p - H_eo t = Dhat p, |w|^2
//   shifted:  t = A_oo^-1 H_oe g5 w;  r -= alpha (Dhat^+ w + sigma p), |r|^2
//             (alpha = |r|^2 / (|w|^2 + sigma |p|^2); Dhat^+ w is not stored)
//             e += alpha p;  p = r + beta p, |p|^2
//   normal:   s -= alpha w, |s|^2;  t = A_oo^-1 H_oe g5 s;  z = Dhat^+ s, |z|^2
//             e += alpha p;  p = z + beta p
//
// The host looks at the stopping flags after every kChunk iterations, one chunk behind the
// launches.  Sums: FP32 over a site, FP64 beyond, blocks in a fixed order.
//
// Why: one right-hand side at a time with a host round trip for each scalar took nine
// launches and two synchronisations per iteration, and every right-hand side read the links
// again.  Ten shifts on 32 x 16^3 (604 iterations in all): 85 -> 33 ms; four right-hand
// sides on 32 x 32 x 16 x 16 with C*: 0.83 -> 0.30 ms per iteration of the four.  Bound by
// the FP32 pipe and load latency of the hops.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "blas.h"
#include "hop.cuh"
#include "ops.h"

namespace qxd {

namespace {

constexpr int kCgMax = 32;      // right-hand sides of a state
constexpr int kCgThreads = 128;
constexpr int kChunk = 8;       // iterations between two looks at the flags

struct CgState {
    double rr[2][kCgMax];  // |r|^2 (normal: |z|^2) before and after the iteration, by parity of the iteration
    double ww[kCgMax], pp[kCgMax];
    double thr[kCgMax];    // stop at this |r|^2 (normal: |s|^2)
    double sig[kCgMax];
    int conv[kCgMax];      // iteration in which it stopped (-1: nothing to do), INT_MAX while it runs
    int bad[kCgMax];       // 1 non-finite, 2 breakdown
    unsigned ticket[kCgMax];
};

struct CgDev {
    CgState* s;
    double* partials;  // [B][tiles]
    int B, tiles;
};

// sum of v over all blocks of right-hand side j: true in thread 0 of the block that
// finishes last, with the sum in *total (partial sums in block order)
__device__ bool rhs_sum(const CgDev& c, int j, int tile, float v, double* total) {
    __shared__ double sh[kCgThreads / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double x = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) sh[warp] = x;
    __syncthreads();
    double* part = c.partials + (size_t)j * c.tiles;
    if (threadIdx.x == 0) {
        for (int w = 1; w < kCgThreads / 32; ++w) x += sh[w];
        part[tile] = x;
        __threadfence();
        last = atomicAdd(&c.s->ticket[j], 1u) == (unsigned)c.tiles - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    x = 0.0;
    for (int b = threadIdx.x; b < c.tiles; b += kCgThreads) x += __ldcg(part + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    __syncthreads();
    if (lane == 0) sh[warp] = x;
    __syncthreads();
    if (threadIdx.x != 0) return false;
    for (int w = 1; w < kCgThreads / 32; ++w) x += sh[w];
    c.s->ticket[j] = 0u;
    *total = x;
    return true;
}

__device__ __forceinline__ float site_norm(const cplx<float> v[12]) {
    float f = 0.f;
#pragma unroll
    for (int k = 0; k < 12; ++k) f = fmaf(v[k].re, v[k].re, fmaf(v[k].im, v[k].im, f));
    return f;
}

// the step length of iteration it: |r|^2 / <p, A p> (0 if that is not positive)
__device__ __forceinline__ double cg_alpha(const CgState* s, int j, int it, bool* broken) {
    const double q = s->ww[j] + s->sig[j] * s->pp[j];
    *broken = !(q > 0.0);
    return *broken ? 0.0 : s->rr[it & 1][j] / q;
}

// r = p = b, e = 0 (normal: s = b, e = 0) and |b|^2
template <bool NORMAL>
__global__ void __launch_bounds__(kCgThreads) k_cg_init(int Vh, CgDev c, const float4* __restrict__ b,
                                                        float4* __restrict__ e, float4* __restrict__ r,
                                                        float4* __restrict__ p) {
    const int j = blockIdx.x % c.B, tile = blockIdx.x / c.B;
    const int h = tile * kCgThreads + threadIdx.x;
    const size_t f = (size_t)j * 6 * Vh;
    float n = 0.f;
    if (h < Vh) {
        cplx<float> v[12];
        load_spinor<1>(b + f, Vh, h, v);
        n = site_norm(v);
        store_spinor<1>(r + f, Vh, h, v);
        if (!NORMAL) store_spinor<1>(p + f, Vh, h, v);
#pragma unroll
        for (int k = 0; k < 6; ++k) e[f + (size_t)k * Vh + h] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    double bb;
    if (rhs_sum(c, j, tile, n, &bb)) {
        CgState* s = c.s;
        s->rr[0][j] = s->rr[1][j] = bb;
        s->pp[j] = bb;
        s->thr[j] *= bb;  // rtol^2 before
        if (s->conv[j] == INT_MAX && !isfinite(bb)) s->bad[j] = 1;
        if (!(bb > 0.0) || !isfinite(bb)) s->conv[j] = -1;
    }
}

// t = A_oo^-1 H_oe (gamma5) in
// one warp per block and a bound of 256 threads: as many loads in flight as the registers allow
// (59 -> 50 us for four right-hand sides on 32 x 32 x 16 x 16; k_cg_hop2 69 -> 62 us with 170)
__global__ void __launch_bounds__(256, 1) k_cg_hop1(Geo g, HopDev a, CgDev c, int last, const float4* __restrict__ in,
                                                        float4* __restrict__ out) {
    const int j = blockIdx.x % c.B;
    if (c.s->conv[j] <= last) return;
    const int h = (blockIdx.x / c.B) * 32 + threadIdx.x;
    const int Vh = g.Vh;
    if (h >= Vh) return;
    const size_t f = (size_t)j * 6 * Vh;
    int x[4];
    site_coords(g, 1, h, x);
    cplx<float> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = {0.f, 0.f};
    hop_dir<1, 0>(g, a, in + f, x, h, acc);
    hop_dir<1, 1>(g, a, in + f, x, h, acc);
    hop_dir<1, 2>(g, a, in + f, x, h, acc);
    hop_dir<1, 3>(g, a, in + f, x, h, acc);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = -0.5f * acc[k];
    float d[72];
    load_diag<1>(a.diaginv, Vh, h, d);
    apply_diag(d, acc);
    store_spinor<1>(out + f, Vh, h, acc);
}

// v = (gamma5) [A_ee (gamma5) self - H_eo t], then by KIND
//   0: out = v (w = Dhat p), ww = |v|^2
//   1: out = r - alpha (v + sigma p), rr of the next iteration (shifted; out = r)
//   2: out = v (z = Dhat^+ s), rr of the next iteration (normal)
template <int KIND>
__global__ void __launch_bounds__(kCgThreads, 3) k_cg_hop2(Geo g, HopDev a, CgDev c, int it, int last,
                                                        const float4* __restrict__ t, const float4* __restrict__ self,
                                                        const float4* __restrict__ p, float4* out) {
    constexpr bool G5 = KIND != 0;
    const int j = blockIdx.x % c.B, tile = blockIdx.x / c.B;
    CgState* s = c.s;
    if (s->conv[j] <= last) return;
    const int h = tile * kCgThreads + threadIdx.x;
    const int Vh = g.Vh;
    const size_t f = (size_t)j * 6 * Vh;
    bool broken = false;
    const double alpha = KIND == 1 ? cg_alpha(s, j, it, &broken) : 0.0;
    float n = 0.f;
    if (h < Vh) {
        int x[4];
        site_coords(g, 0, h, x);
        cplx<float> acc[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = {0.f, 0.f};
        hop_dir<1, 0>(g, a, t + f, x, h, acc);
        hop_dir<1, 1>(g, a, t + f, x, h, acc);
        hop_dir<1, 2>(g, a, t + f, x, h, acc);
        hop_dir<1, 3>(g, a, t + f, x, h, acc);
        cplx<float> v[12];
        load_spinor<1>(self + f, Vh, h, v);
        if (G5) {
#pragma unroll
            for (int k = 6; k < 12; ++k) v[k] = -v[k];
        }
        float d[72];
        load_diag<1>(a.diag, Vh, h, d);
        apply_diag(d, v);
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = v[k] + 0.5f * acc[k];
        if (G5) {
#pragma unroll
            for (int k = 6; k < 12; ++k) v[k] = -v[k];
        }
        if (KIND == 1) {
            const float al = (float)alpha, sg = (float)s->sig[j];
            cplx<float> q[12], r[12];
            load_spinor<1>(p + f, Vh, h, q);
#pragma unroll
            for (int k = 0; k < 6; ++k) {  // r, which this thread alone updates
                const float4 u = out[f + (size_t)k * Vh + h];
                r[2 * k] = {u.x, u.y};
                r[2 * k + 1] = {u.z, u.w};
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                v[k].re = fmaf(-al, fmaf(sg, q[k].re, v[k].re), r[k].re);
                v[k].im = fmaf(-al, fmaf(sg, q[k].im, v[k].im), r[k].im);
            }
        }
        n = site_norm(v);
        store_spinor<1>(out + f, Vh, h, v);
    }
    double sum;
    if (rhs_sum(c, j, tile, n, &sum)) {
        if (KIND == 0) {
            s->ww[j] = sum;
            if (!isfinite(sum)) {
                s->bad[j] = 1;
                s->conv[j] = it;
            }
        } else {
            s->rr[(it + 1) & 1][j] = sum;
            if (s->bad[j]) {
                s->conv[j] = it;
            } else if (!isfinite(sum)) {
                s->bad[j] = 1;
                s->conv[j] = it;
            } else if (KIND == 1 && broken) {
                s->bad[j] = 2;
                s->conv[j] = it;
            } else if (KIND == 1 ? sum <= s->thr[j] : sum == 0.0) {
                s->conv[j] = it;
            }
        }
    }
}

// normal: s -= alpha w, |s|^2
__global__ void __launch_bounds__(kCgThreads) k_cg_residual(int Vh, CgDev c, int it, const float4* __restrict__ w,
                                                            float4* __restrict__ r) {
    const int j = blockIdx.x % c.B, tile = blockIdx.x / c.B;
    CgState* s = c.s;
    if (s->conv[j] < it || s->bad[j]) return;
    const int h = tile * kCgThreads + threadIdx.x;
    const size_t f = (size_t)j * 6 * Vh;
    bool broken;
    const float al = (float)cg_alpha(s, j, it, &broken);
    float n = 0.f;
    if (h < Vh) {
        float4 x[6], y[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            x[k] = QXD_LDG(w + f + (size_t)k * Vh + h);
            y[k] = r[f + (size_t)k * Vh + h];
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            y[k].x = fmaf(-al, x[k].x, y[k].x);
            y[k].y = fmaf(-al, x[k].y, y[k].y);
            y[k].z = fmaf(-al, x[k].z, y[k].z);
            y[k].w = fmaf(-al, x[k].w, y[k].w);
            n = fmaf(y[k].x, y[k].x, fmaf(y[k].y, y[k].y, fmaf(y[k].z, y[k].z, fmaf(y[k].w, y[k].w, n))));
            r[f + (size_t)k * Vh + h] = y[k];
        }
    }
    double sum;
    if (rhs_sum(c, j, tile, n, &sum)) {
        if (!isfinite(sum)) s->bad[j] = 1;
        if (broken || !isfinite(sum) || sum <= s->thr[j]) s->conv[j] = it;
    }
}

// e += alpha p;  p = r + beta p, |p|^2 (it = -1: p = r)
__global__ void __launch_bounds__(kCgThreads) k_cg_direction(int Vh, CgDev c, int it, const float4* __restrict__ r,
                                                             float4* __restrict__ e, float4* __restrict__ p) {
    const int j = blockIdx.x % c.B, tile = blockIdx.x / c.B;
    CgState* s = c.s;
    if (s->conv[j] < it || s->bad[j]) return;
    const int h = tile * kCgThreads + threadIdx.x;
    const size_t f = (size_t)j * 6 * Vh;
    bool broken;
    const float al = it < 0 ? 0.f : (float)cg_alpha(s, j, it, &broken);
    const double r0 = s->rr[it & 1][j];
    const float be = it < 0 || !(r0 > 0.0) ? 0.f : (float)(s->rr[(it + 1) & 1][j] / r0);
    float n = 0.f;
    if (h < Vh) {
        float4 x[6], y[6], z[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            x[k] = QXD_LDG(r + f + (size_t)k * Vh + h);
            if (it >= 0) {
                y[k] = p[f + (size_t)k * Vh + h];
                z[k] = e[f + (size_t)k * Vh + h];
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            if (it >= 0) {
                z[k].x = fmaf(al, y[k].x, z[k].x);
                z[k].y = fmaf(al, y[k].y, z[k].y);
                z[k].z = fmaf(al, y[k].z, z[k].z);
                z[k].w = fmaf(al, y[k].w, z[k].w);
                e[f + (size_t)k * Vh + h] = z[k];
                x[k].x = fmaf(be, y[k].x, x[k].x);
                x[k].y = fmaf(be, y[k].y, x[k].y);
                x[k].z = fmaf(be, y[k].z, x[k].z);
                x[k].w = fmaf(be, y[k].w, x[k].w);
            }
            n = fmaf(x[k].x, x[k].x, fmaf(x[k].y, x[k].y, fmaf(x[k].z, x[k].z, fmaf(x[k].w, x[k].w, n))));
            p[f + (size_t)k * Vh + h] = x[k];
        }
    }
    double sum;
    if (rhs_sum(c, j, tile, n, &sum)) s->pp[j] = sum;
}

}  // namespace

int cg_lockstep(qxd_ctx* ctx, int fl, int B, bool normal, const double* sigma, const double* rtol, const void* bv,
                void* ev, const CgFields& work, long long budget, int each, int* iters, cudaStream_t st) {
    if (B < 1 || B > kCgMax) return qxd_fail(ctx, QXD_EARG, "lockstep CG: 1 to 32 right-hand sides");
    const Geo& g = ctx->g;
    const QxdFlavour& F = ctx->fl[fl];
    const int Vh = g.Vh;
    const int tiles = nblocks(Vh, kCgThreads);
    void *sv, *pv;
    QXD_TRY(qxd_ws(ctx, WS_CG, sizeof(CgState), &sv));
    QXD_TRY(qxd_ws(ctx, WS_CG + 1, sizeof(double) * (size_t)B * tiles, &pv));
    CgDev c{static_cast<CgState*>(sv), static_cast<double*>(pv), B, tiles};
    CgState h{};
    int running = 0;
    for (int j = 0; j < B; ++j) {
        h.thr[j] = rtol[j] * rtol[j];
        h.sig[j] = sigma ? sigma[j] : 0.0;
        h.conv[j] = rtol[j] < 1.0 ? INT_MAX : -1;
        running += rtol[j] < 1.0;
    }
    QXD_CUDA(ctx, cudaMemcpyAsync(c.s, &h, sizeof h, cudaMemcpyHostToDevice, st));
    const float4* b = static_cast<const float4*>(bv);
    float4* e = static_cast<float4*>(ev);
    float4 *r = static_cast<float4*>(work.r), *z = static_cast<float4*>(work.z), *p = static_cast<float4*>(work.p),
           *w = static_cast<float4*>(work.w), *t = static_cast<float4*>(work.t);
    // links and site-diagonal terms of the two halves of Dhat (odd, then even output sites)
    auto dev = [&](int po, bool g5) {
        HopDev d{};
        d.U32_out = ctx->U32 + (size_t)po * 12 * Vh;
        d.U32_in = ctx->U32 + (size_t)(1 - po) * 12 * Vh;
        d.Z32_out = F.Z32 + (size_t)po * 2 * Vh;
        d.Z32_in = F.Z32 + (size_t)(1 - po) * 2 * Vh;
        d.diag = F.C32[0] + (size_t)po * 18 * Vh;
        d.diaginv = F.C32[1] + (size_t)po * 18 * Vh;
        d.g5_nb = g5;
        return d;
    };
    const HopDev d1 = dev(1, false), d1g = dev(1, true), d2 = dev(0, false);
    const unsigned grid = (unsigned)tiles * B, grid1 = (unsigned)nblocks(Vh, 32) * B;
    const double fb = 96.0 * Vh * B;                       // a field of every right-hand side
    const double h1 = (448.0 + 288.0) * Vh + 2 * fb, h2 = (448.0 + 288.0) * Vh;
    // an iteration it (-1: what the normal equations need before the first)
    auto dagger = [&](int it) {
        {
            ProfScope prof(ctx, "cg_hop1", h1, st);
            k_cg_hop1<<<grid1, 32, 0, st>>>(g, d1g, c, it, r, t);
        }
        ProfScope prof(ctx, "cg_hop2", h2 + 3 * fb, st);
        k_cg_hop2<2><<<grid, kCgThreads, 0, st>>>(g, d2, c, it, it, t, r, nullptr, z);
    };
    auto direction = [&](int it) {
        ProfScope prof(ctx, "cg_direction", 5 * fb, st);
        k_cg_direction<<<grid, kCgThreads, 0, st>>>(Vh, c, it, normal ? z : r, e, p);
    };
    auto iteration = [&](int it) {
        {
            ProfScope prof(ctx, "cg_hop1", h1, st);
            k_cg_hop1<<<grid1, 32, 0, st>>>(g, d1, c, it - 1, p, t);
        }
        {
            ProfScope prof(ctx, "cg_hop2", h2 + 3 * fb, st);
            k_cg_hop2<0><<<grid, kCgThreads, 0, st>>>(g, d2, c, it, it - 1, t, p, nullptr, w);
        }
        if (normal) {
            {
                ProfScope prof(ctx, "cg_residual", 3 * fb, st);
                k_cg_residual<<<grid, kCgThreads, 0, st>>>(Vh, c, it, w, r);
            }
            dagger(it);
        } else {
            {
                ProfScope prof(ctx, "cg_hop1", h1, st);
                k_cg_hop1<<<grid1, 32, 0, st>>>(g, d1g, c, it - 1, w, t);
            }
            ProfScope prof(ctx, "cg_hop2", h2 + 5 * fb, st);
            k_cg_hop2<1><<<grid, kCgThreads, 0, st>>>(g, d2, c, it, it - 1, t, w, p, r);
        }
        direction(it);
    };
    if (normal) {
        k_cg_init<true><<<grid, kCgThreads, 0, st>>>(Vh, c, b, e, r, p);
        dagger(-1);
        direction(-1);
    } else {
        k_cg_init<false><<<grid, kCgThreads, 0, st>>>(Vh, c, b, e, r, p);
    }
    QXD_CUDA(ctx, cudaGetLastError());
    // the flags go to the pinned mirror in two turns, each waited for one chunk later
    static_assert(2 * sizeof(int) * 2 * kCgMax <= kRedSlots * sizeof(double), "flags fit the pinned mirror");
    int* flags[2] = {reinterpret_cast<int*>(ctx->red_host), reinterpret_cast<int*>(ctx->red_host) + 2 * kCgMax};
    cudaEvent_t ev2[2] = {nullptr, nullptr};
    int rc = QXD_OK;
    for (auto& x : ev2)
        if (cudaEventCreateWithFlags(&x, cudaEventDisableTiming) != cudaSuccess)
            rc = qxd_fail(ctx, QXD_ECUDA, "lockstep CG: event creation failed");
    // iterations launched (it), and up to a chunk whose flags were read: made in all, running
    int it = 0, seen = 0, launched[2] = {0, 0};
    long long total = 0;
    std::vector<int> done(B, 0);
    std::vector<char> runs(B);
    for (int j = 0; j < B; ++j) runs[j] = rtol[j] < 1.0;
    auto look = [&](int turn) -> int {
        if (cudaEventSynchronize(ev2[turn]) != cudaSuccess) return qxd_fail(ctx, QXD_ECUDA, "lockstep CG: wait failed");
        seen = launched[turn];
        total = 0;
        running = 0;
        for (int j = 0; j < B; ++j) {
            const int cv = flags[turn][j], bad = flags[turn][kCgMax + j];
            if (bad == 1) return qxd_fail(ctx, QXD_ENAN, "non-finite value in CG");
            if (bad == 2) return qxd_fail(ctx, QXD_EBREAKDOWN, "shifted CG: <p, A p> <= 0");
            runs[j] = cv == INT_MAX;
            done[j] = runs[j] ? seen : cv + 1;
            total += done[j];
            running += runs[j];
        }
        return QXD_OK;
    };
    int chunk = 0, looked = 0;  // chunks launched and looked at
    while (rc == QXD_OK && running > 0 && it < each) {  // what still runs has made `it` iterations
        long long left = budget - total - (long long)(it - seen) * running;
        if (left < running && looked < chunk) {  // count what was really made
            rc = look(looked++ & 1);
            continue;
        }
        if (left <= 0) break;
        const int stop = it - 1;
        for (int j = B - 1; j >= 0 && left < running; --j) {  // not one more iteration for all of them
            if (!runs[j]) continue;
            runs[j] = 0;
            running -= 1;
            if (cudaMemcpyAsync(c.s->conv + j, &stop, sizeof stop, cudaMemcpyHostToDevice, st) != cudaSuccess)
                rc = qxd_fail(ctx, QXD_ECUDA, "lockstep CG: copy failed");
        }
        if (rc != QXD_OK) break;
        const int n = (int)std::max<long long>(1, std::min<long long>({kChunk, left / running, each - it}));
        for (int k = 0; k < n; ++k) iteration(it++);
        const int turn = chunk++ & 1;
        launched[turn] = it;
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(flags[turn], c.s->conv, sizeof(int) * 2 * kCgMax, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaEventRecord(ev2[turn], st) != cudaSuccess)
            rc = qxd_fail(ctx, QXD_ECUDA, "lockstep CG: launch failed");
        else if (chunk - looked > 1) rc = look(looked++ & 1);
    }
    while (rc == QXD_OK && looked < chunk) rc = look(looked++ & 1);
    if (rc != QXD_OK) cudaStreamSynchronize(st);  // what is still queued uses the workspaces
    for (auto& x : ev2)
        if (x) cudaEventDestroy(x);
    for (int j = 0; j < B; ++j) iters[j] = done[j];
    return rc;
}

}  // namespace qxd
