// Operator kernels that read and write the caller's canonical spinor fields
// ([site][4][3] complex, Sec. 2.3 operator), without a pass that converts them to
// the internal structure-of-arrays layout and back.
//
//   kDw     out = D in on the full lattice, both parities in the same launch
//   kDhat1  t_o = A_oo^-1 H_oe in_e, canonical even field in, internal odd field out
//   kDhat2  out_e = A_ee in_e - H_eo t_o, internal odd field and canonical even field in,
//           canonical even field out
//
// A site's twelve complex numbers are contiguous (96 or 192 bytes, whole 32-byte
// sectors), so a spinor is three or six 256-bit accesses per thread; links and
// site-diagonal terms keep the internal layout.  The arithmetic is that of the internal
// kernels, in the same order.
//
// Why: the conversion passes move four spinors per site and right-hand side (384 bytes in
// FP32, more than the operator itself with many right-hand sides) and cost two to four
// launches.  Time per call, conversion passes -> here (FP32 unless said): Dhat 8^4 24.6 ->
// 16.1 us, Dhat^+ 24^3x48 147 -> 126 us, Dhat 32^3x64 C* 771 -> 685 us, D_w 24^3x48 with 12
// right-hand sides 1521 -> 1102 us, D_w 24^3x48 FP64 1677 -> 1336 us (FP64-pipe bound: one
// launch over both parities also ends in one tail instead of two).
#include <cstdio>

#include "hop.cuh"
#include "ops.h"

namespace qxd {

namespace {

enum { kDw = 0, kDhat1 = 1, kDhat2 = 2 };

struct CanonDev {
    const void* nb;    // neighbour input
    const void* self;  // self input (canonical)
    void* out;
    const double2* V64;  // [p][36][Vh]
    const float4* U32;   // [p][12][Vh]
    const float4* Z32;   // [p][2][Vh]
    const void* diag;    // [p][36 or 18][Vh], the inverse for kDhat1
    int dagger;
};

__device__ __forceinline__ void ld32(const float* p, float v[8]) {
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
        : "l"(p));
}
__device__ __forceinline__ void ld32(const double* p, double v[4]) {
    asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
}
// of an array that the same launch writes (each thread its own site): not the read-only path
__device__ __forceinline__ void ld32_rw(const float* p, float v[8]) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void ld32_rw(const double* p, double v[4]) {
    asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st32(float* p, const float v[8]) {
    asm volatile("st.global.v8.f32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                 "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st32(double* p, const double v[4]) {
    asm volatile("st.global.v4.f64 [%4], {%0,%1,%2,%3};" ::"d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]), "l"(p)
                 : "memory");
}

// bfloat16 storage: the values that a field of that precision would hold
__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

template <int P, bool RW>
__device__ __forceinline__ void load_canon(const void* base, long long site, cplx<typename Prec<P>::real> s[12]) {
    using R = typename Prec<P>::real;
    constexpr int NV = 32 / sizeof(R), NL = 24 / NV;
    const R* p = static_cast<const R*>(base) + site * 24;
    R v[24];
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        if constexpr (RW) ld32_rw(p + NV * k, v + NV * k);
        else ld32(p + NV * k, v + NV * k);
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        if constexpr (P == 2) s[k] = {round_bf16(v[2 * k]), round_bf16(v[2 * k + 1])};
        else s[k] = {v[2 * k], v[2 * k + 1]};
    }
}

template <int P>
__device__ __forceinline__ void store_canon(void* base, long long site, const cplx<typename Prec<P>::real> s[12]) {
    using R = typename Prec<P>::real;
    constexpr int NV = 32 / sizeof(R), NL = 24 / NV;
    R* p = static_cast<R*>(base) + site * 24;
    R v[24];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        v[2 * k] = P == 2 ? (R)round_bf16((float)s[k].re) : s[k].re;
        v[2 * k + 1] = P == 2 ? (R)round_bf16((float)s[k].im) : s[k].im;
    }
#pragma unroll
    for (int k = 0; k < NL; ++k) st32(p + NV * k, v + NV * k);
}

template <int P, int MODE, int MU, bool FWD, typename R>
__device__ __forceinline__ void canon_hop(const Geo& g, const CanonDev& a, const void* nb, const int x[4], int p,
                                          int h, bool g5, cplx<R> acc[12]) {
    const int Vh = g.Vh;
    const int y = neighbour_lex(g, x, MU, FWD ? +1 : -1);
    cplx<R> s[12];
    Half<R> hp, r;
    Mat3<R> m;
    if constexpr (MODE == kDw) load_canon<P, false>(nb, y, s);
    else if constexpr (MODE == kDhat1) load_canon<P, false>(nb, y >> 1, s);
    else load_spinor<P>(static_cast<const typename Prec<P>::chunk*>(nb), Vh, y >> 1, s);
    if (MODE == kDhat1 && g5) {
#pragma unroll
        for (int k = 6; k < 12; ++k) s[k] = -s[k];
    }
    project<MU, FWD>(s, hp);
    const int pl = FWD ? p : 1 - p, hl = FWD ? h : y >> 1;
    if constexpr (P == 0) {
        load_link64(a.V64 + (size_t)pl * 36 * Vh, Vh, MU, hl, m);
        mul_half<!FWD>(m, hp, r);
    } else {
        cplx<float> z;
        load_link32(a.U32 + (size_t)pl * 12 * Vh, a.Z32 + (size_t)pl * 2 * Vh, Vh, MU, hl, m, z);
        mul_half<!FWD>(m, hp, r);
#pragma unroll
        for (int sp = 0; sp < 2; ++sp)
#pragma unroll
            for (int c = 0; c < 3; ++c) r.a[sp][c] = FWD ? z * r.a[sp][c] : cmul_conj(z, r.a[sp][c]);
    }
    reconstruct<MU, FWD>(r, acc);
}

// One thread per site and right-hand side, one warp per block; block b covers right-hand
// side b % nrhs of the site tile b / nrhs, so that the links and diagonal terms that the
// first of them brings into L2 serve the others.
//
// Latency-bound: what counts is loads in flight per thread, not warps.  The launch bound
// names 256 threads although a block has 32: with it the compiler spends 146 to 165
// registers (12 warps per SM) and starts several directions' loads early; with bounds
// that let it use 96 to 128 the same kernel is slower, as is an explicit prefetch of the
// next direction, two or four right-hand sides per thread (one link load for all), or
// blocks that hold four right-hand sides.  Measured (us; blocks of 4 right-hand sides or
// 128 sites -> here): D_w 24^3x48, 12 right-hand sides 1102 -> 761, Dhat^+ 24^3x48 126 ->
// 104, Dhat 32^3x64 C* 685 -> 585 (1952 bytes per even site at 7.0 TB/s).  With many
// right-hand sides the L1 data pipe is 76 % busy: a 96-byte stride takes two passes per
// 256-bit load where the internal layout takes one.
constexpr int kCanonThreads = 32;

template <int P, int MODE>
__global__ void __launch_bounds__(256, 1) k_hop_canon(Geo g, CanonDev a, int nrhs, int first, int end) {
    using R = typename Prec<P>::real;
    const int rhs = blockIdx.x % nrhs;
    const int i = first + (blockIdx.x / nrhs) * kCanonThreads + threadIdx.x;
    const int Vh = g.Vh;
    if (i >= end) return;
    int x[4], p, h;
    if constexpr (MODE == kDw) {
        int r = i;
        x[3] = r % g.N[3];
        r /= g.N[3];
        x[2] = r % g.N[2];
        r /= g.N[2];
        x[1] = r % g.N[1];
        x[0] = r / g.N[1];
        p = (x[0] + x[1] + x[2] + x[3]) & 1;
        h = i >> 1;
    } else {
        p = MODE == kDhat1 ? 1 : 0;
        h = i;
        site_coords(g, p, h, x);
    }
    // fields of this right-hand side
    const size_t canon = (size_t)rhs * (MODE == kDw ? (size_t)g.V : (size_t)Vh) * 24;   // reals
    const size_t inner = (size_t)rhs * Prec<P>::nchunk * Vh;                           // chunks
    using CH = typename Prec<P>::chunk;
    const void* nb = MODE == kDhat2 ? (const void*)(static_cast<const CH*>(a.nb) + inner)
                                    : (const void*)(static_cast<const R*>(a.nb) + canon);
    const bool dg = a.dagger != 0;
    cplx<R> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = {R(0), R(0)};
    canon_hop<P, MODE, 0, true>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 0, false>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 1, true>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 1, false>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 2, true>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 2, false>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 3, true>(g, a, nb, x, p, h, dg, acc);
    canon_hop<P, MODE, 3, false>(g, a, nb, x, p, h, dg, acc);
    const R c = MODE == kDhat2 ? R(0.5) : R(-0.5);  // -1/2 times the sign of the hopping term
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = c * acc[k];
    R d[72];
    constexpr int DP = P == 0 ? 0 : 1;
    constexpr size_t dsz = P == 0 ? 36 : 18;
    const void* dg_ptr = P == 0 ? (const void*)(static_cast<const double2*>(a.diag) + (size_t)p * dsz * Vh)
                                : (const void*)(static_cast<const float4*>(a.diag) + (size_t)p * dsz * Vh);
    if constexpr (MODE == kDhat1) {
        load_diag<DP>(dg_ptr, Vh, h, d);
        apply_diag(d, acc);
        store_spinor<P>(static_cast<CH*>(a.out) + inner, Vh, h, acc);
    } else {
        cplx<R> s[12];
        if constexpr (MODE == kDw) load_canon<P, false>(static_cast<const R*>(a.self) + canon, i, s);
        else load_canon<P, true>(static_cast<const R*>(a.self) + canon, i, s);
        if (MODE == kDhat2 && dg) {
#pragma unroll
            for (int k = 6; k < 12; ++k) s[k] = -s[k];
        }
        load_diag<DP>(dg_ptr, Vh, h, d);
        apply_diag(d, s);
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = acc[k] + s[k];
        if (MODE == kDhat2 && dg) {
#pragma unroll
            for (int k = 6; k < 12; ++k) acc[k] = -acc[k];
        }
        store_canon<P>(static_cast<R*>(a.out) + canon, i, acc);
    }
}

template <int MODE>
int launch_canon(qxd_ctx* ctx, int fl, int prec, const void* nb, const void* self, void* out, int dagger, int nrhs,
                 cudaStream_t st) {
    const Geo& g = ctx->g;
    const QxdFlavour& F = ctx->fl[fl];
    const int inv = MODE == kDhat1 ? 1 : 0;
    CanonDev a{nb, self, out, F.V64, ctx->U32, F.Z32, prec == QXD_FP64 ? (const void*)F.C64[inv] : F.C32[inv], dagger};
    const char* mode = MODE == kDw ? "dw" : MODE == kDhat1 ? "dhat1" : "dhat2";
    const double sp = prec == QXD_FP64 ? 192 : 96, si = prec == QXD_FP64 ? 192 : (prec == QXD_FP32 ? 96 : 48);
    const double link = prec == QXD_FP64 ? 8 * 144 : 8 * 56, dg = prec == QXD_FP64 ? 576 : 288;
    const double per = MODE == kDw ? 2 * (2 * sp) : MODE == kDhat1 ? sp + si : si + 2 * sp;
    char name[48];
    std::snprintf(name, sizeof name, "hop_%s_%s%s", prec == QXD_FP64 ? "fp64" : prec == QXD_FP32 ? "fp32" : "bf16", mode,
                  nrhs > 1 ? "_mrhs" : "");
    // D_w of several right-hand sides goes over the sites in two launches (the first and the
    // second half), as many as the half-lattice kernels take; one right-hand side in one
    const int sites = MODE == kDw ? (int)g.V : g.Vh;
    const int parts = MODE == kDw && nrhs > 1 ? 2 : 1;
    for (int k = 0; k < parts; ++k) {
        const int first = k * (sites / parts), end = k + 1 == parts ? sites : (k + 1) * (sites / parts);
        ProfScope prof(ctx, name, (double)g.Vh * ((MODE == kDw ? link + 2 * dg : link + dg) + per * nrhs) / parts, st);
        const int grid = nblocks(end - first, kCanonThreads) * nrhs;
        if (prec == QXD_FP64) k_hop_canon<0, MODE><<<grid, kCanonThreads, 0, st>>>(g, a, nrhs, first, end);
        else if (prec == QXD_FP32) k_hop_canon<1, MODE><<<grid, kCanonThreads, 0, st>>>(g, a, nrhs, first, end);
        else k_hop_canon<2, MODE><<<grid, kCanonThreads, 0, st>>>(g, a, nrhs, first, end);
        QXD_CUDA(ctx, cudaGetLastError());
    }
    return QXD_OK;
}

}  // namespace

// 256-bit accesses need 32-byte aligned fields
bool canon_fits(const void* in, const void* out, size_t bytes, bool in_place) {
    const uintptr_t i = reinterpret_cast<uintptr_t>(in), o = reinterpret_cast<uintptr_t>(out);
    if ((i | o) & 31) return false;
    if (i == o) return in_place;
    return i + bytes <= o || o + bytes <= i;
}

int op_Dw_canon(qxd_ctx* ctx, int fl, int P, const void* in, void* out, int nrhs, cudaStream_t st) {
    return launch_canon<kDw>(ctx, fl, P, in, in, out, 0, nrhs, st);
}

int op_Dhat_canon(qxd_ctx* ctx, int fl, int P, int dagger, const void* in_e, void* out_e, void* tmp_o, int nrhs,
                  cudaStream_t st) {
    QXD_TRY(launch_canon<kDhat1>(ctx, fl, P, in_e, nullptr, tmp_o, dagger, nrhs, st));
    return launch_canon<kDhat2>(ctx, fl, P, tmp_o, in_e, out_e, dagger, nrhs, st);
}

}  // namespace qxd
