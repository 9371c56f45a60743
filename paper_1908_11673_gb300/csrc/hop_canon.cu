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
// site-diagonal terms keep the internal layout.  k_hop_canon does the arithmetic of the
// internal kernels in the same order; k_hop_quad, on small lattices, adds the directions in
// another order.
//
// Why: the conversion passes move four spinors per site and right-hand side (384 bytes in
// FP32, more than the operator itself with many right-hand sides) and cost two to four
// launches.  Time per call, conversion passes -> here (FP32 unless said): Dhat 8^4 24.6 ->
// 6.1 us, Dhat^+ 24^3x48 146 -> 105 us, Dhat 32^3x64 C* 771 -> 585 us, D_w 24^3x48 with 12
// right-hand sides 1500 -> 762 us, D_w 24^3x48 FP64 1674 -> 1331 us (FP64-pipe bound: one
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
// of an array that is written while the launch exists (by itself, each thread its own site, or by
// the kernel before an early launch): not the read-only path
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

// bfloat16 storage: the values that a field of that precision would hold.  Two at a time: half the
// conversions (with one at a time and no register bound, below, Dhat on 32^3x64 C* took 741 us).
__device__ __forceinline__ cplx<float> round_bf16(float re, float im) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(re, im);
    const unsigned u = *reinterpret_cast<const unsigned*>(&v);
    return {__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)};
}

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
        if constexpr (P == 2) s[k] = round_bf16(v[2 * k], v[2 * k + 1]);
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
        cplx<R> c = s[k];
        if constexpr (P == 2) c = round_bf16(c.re, c.im);
        v[2 * k] = c.re;
        v[2 * k + 1] = c.im;
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
// With bfloat16 storage the rounding makes the compiler take up to 228 registers (8 warps per
// SM), so there the bound is 16 blocks (128 registers): Dhat 32^3x64 C* 645 us with 12 blocks,
// 593 with 16, 620 with 20, and 671 by the conversion passes; four right-hand sides 2006, 1708,
// 1796 and 2063.
constexpr int kCanonThreads = 32;

template <int P, int MODE>
__global__ void __launch_bounds__(P == 2 ? 32 : 256, P == 2 ? 16 : 1) k_hop_canon(Geo g, CanonDev a, int nrhs, int first, int end) {
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

// Small lattices: four lanes per site, lane q the two hops of direction q.
//
// With a thread per site such a launch is one long chain of instructions on a few warps, and
// on the FP64 pipe (64 cycles per warp instruction) most of the chip's schedulers have none.
// Four lanes shorten the chain and fill four times the warps; the launch also lets the next
// one start early, which loads its links and site-diagonal terms meanwhile.  Measured per
// call, one thread -> four lanes (us): Dhat 8^4 FP32 12.4 -> 6.4 (then bound by the host), FP64
// 84 -> 48; D_w 4 x 4 x 8 x 8 FP64 41 -> 15.  The exchanges and the site-diagonal term done
// twice cost more than that beyond about 8192 sites in FP32 (Dhat on 8 x 8 x 16 x 16 with two
// right-hand sides 12.4 -> 13.0) and 4096 in FP64 (81 against 84 us there, 88 against 84 at 8192).
//
// A lane forms the half-spinors of its direction's forward and backward hop; their sums and
// differences give its share of the upper and lower spins.  Two exchanges leave the upper
// chiral block in lanes 0, 1 and the lower one in lanes 2, 3, both lanes of a pair apply the
// block's 6 x 6 site-diagonal term and each stores three of the six components.
constexpr int kQuadThreads = 64;

template <typename R>
__device__ __forceinline__ cplx<R> sel(bool c, cplx<R> a, cplx<R> b) {
    return {c ? a.re : b.re, c ? a.im : b.im};
}
template <typename R>
__device__ __forceinline__ cplx<R> shfl_x(cplx<R> a, int m) {
    return {__shfl_xor_sync(0xffffffffu, a.re, m), __shfl_xor_sync(0xffffffffu, a.im, m)};
}

__device__ __forceinline__ void load_inner_rw(const float4* b, int Vh, int h, cplx<float> s[12]) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float4 v = b[(size_t)k * Vh + h];
        s[2 * k] = {v.x, v.y};
        s[2 * k + 1] = {v.z, v.w};
    }
}
__device__ __forceinline__ void load_inner_rw(const double2* b, int Vh, int h, cplx<double> s[12]) {
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 v = b[(size_t)k * Vh + h];
        s[k] = {v.x, v.y};
    }
}

template <int P, int MODE>
__global__ void __launch_bounds__(kQuadThreads) k_hop_quad(Geo g, CanonDev a, int nrhs) {
    using R = typename Prec<P>::real;
    using CH = typename Prec<P>::chunk;
    using C = cplx<R>;
    // the next launch of the stream may begin: it reads links and site-diagonal terms (which
    // no kernel that allows this writes) and waits before it touches a field
    asm volatile("griddepcontrol.launch_dependents;");
    const int sites = MODE == kDw ? (int)g.V : g.Vh;
    const int Vh = g.Vh;
    const int rhs = blockIdx.x % nrhs;
    const int site = (blockIdx.x / nrhs) * (kQuadThreads / 4) + (threadIdx.x >> 2);
    const bool live = site < sites;
    const int i = live ? site : sites - 1;  // every lane takes part in the exchanges
    const int q = threadIdx.x & 3;
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
    const int yf = q == 0 ? neighbour_lex(g, x, 0, +1) : q == 1 ? neighbour_lex(g, x, 1, +1) : q == 2 ? neighbour_lex(g, x, 2, +1) : neighbour_lex(g, x, 3, +1);
    const int yb = q == 0 ? neighbour_lex(g, x, 0, -1) : q == 1 ? neighbour_lex(g, x, 1, -1) : q == 2 ? neighbour_lex(g, x, 2, -1) : neighbour_lex(g, x, 3, -1);
    Mat3<R> mf, mb;
    cplx<float> zf, zb;
    if constexpr (P == 0) {
        load_link64(a.V64 + (size_t)p * 36 * Vh, Vh, q, h, mf);
        load_link64(a.V64 + (size_t)(1 - p) * 36 * Vh, Vh, q, yb >> 1, mb);
    } else {
        load_link32(a.U32 + (size_t)p * 12 * Vh, a.Z32 + (size_t)p * 2 * Vh, Vh, q, h, mf, zf);
        load_link32(a.U32 + (size_t)(1 - p) * 12 * Vh, a.Z32 + (size_t)(1 - p) * 2 * Vh, Vh, q, yb >> 1, mb, zb);
    }
    // the lane's 6 x 6 block (block q / 2)
    constexpr int NB = P == 0 ? 18 : 9;
    R d[36];
    {
        const CH* D = static_cast<const CH*>(a.diag) + ((size_t)p * 2 + (q >> 1)) * NB * Vh + h;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const CH v = QXD_LDG(D + (size_t)k * Vh);
            if constexpr (P == 0) {
                d[2 * k] = v.x;
                d[2 * k + 1] = v.y;
            } else {
                d[4 * k] = v.x;
                d[4 * k + 1] = v.y;
                d[4 * k + 2] = v.z;
                d[4 * k + 3] = v.w;
            }
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const size_t canon = (size_t)rhs * sites * 24, inner = (size_t)rhs * Prec<P>::nchunk * Vh;
    C sf[12], sb[12];
    // not by the read-only path: a kernel that writes the field may run until the wait above
    if constexpr (MODE == kDhat2) {
        const CH* t = static_cast<const CH*>(a.nb) + inner;
        load_inner_rw(t, Vh, yf >> 1, sf);
        load_inner_rw(t, Vh, yb >> 1, sb);
    } else {
        const R* f = static_cast<const R*>(a.nb) + canon;
        load_canon<P, true>(f, MODE == kDw ? yf : yf >> 1, sf);
        load_canon<P, true>(f, MODE == kDw ? yb : yb >> 1, sb);
    }
    const bool dg = a.dagger != 0;
    if (MODE == kDhat1 && dg) {
#pragma unroll
        for (int k = 6; k < 12; ++k) {
            sf[k] = -sf[k];
            sb[k] = -sb[k];
        }
    }
    // projections s_0 +- c_0 s_p0, s_1 +- c_1 s_p1: p = (2, 3) for directions 0, 3, (3, 2) for
    // 1, 2; c = 1 or i, c_1 with the opposite sign for 2, 3
    const bool imag = q & 1, swap = q == 1 || q == 2;
    const R s1 = q >= 2 ? R(-1) : R(1);
    Half<R> hf, hb, rf, rb;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        C b0 = sel(swap, sf[9 + c], sf[6 + c]), b1 = sel(swap, sf[6 + c], sf[9 + c]);
        b0 = sel(imag, times_i(b0), b0);
        b1 = s1 * sel(imag, times_i(b1), b1);
        hf.a[0][c] = sf[c] + b0;
        hf.a[1][c] = sf[3 + c] + b1;
        b0 = sel(swap, sb[9 + c], sb[6 + c]), b1 = sel(swap, sb[6 + c], sb[9 + c]);
        b0 = sel(imag, times_i(b0), b0);
        b1 = s1 * sel(imag, times_i(b1), b1);
        hb.a[0][c] = sb[c] - b0;
        hb.a[1][c] = sb[3 + c] - b1;
    }
    mul_half<false>(mf, hf, rf);
    mul_half<true>(mb, hb, rb);
    if constexpr (P != 0) {
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                rf.a[s][c] = zf * rf.a[s][c];
                rb.a[s][c] = cmul_conj(zb, rb.a[s][c]);
            }
    }
    // upper spins get the sum, spin p0 c_0^* and spin p1 c_1^* times the difference; lanes 0, 1
    // keep the upper block, 2, 3 the lower one
    C v[6];
    const bool low = q >= 2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const C u0 = rf.a[0][c] + rb.a[0][c], u1 = rf.a[1][c] + rb.a[1][c];
        C e0 = rf.a[0][c] - rb.a[0][c], e1 = s1 * (rf.a[1][c] - rb.a[1][c]);
        e0 = sel(imag, -times_i(e0), e0);
        e1 = sel(imag, -times_i(e1), e1);
        const C l2 = sel(swap, e1, e0), l3 = sel(swap, e0, e1);
        const C k0 = sel(low, l2, u0), k1 = sel(low, l3, u1);
        v[c] = k0 + shfl_x(sel(low, u0, l2), 2);
        v[3 + c] = k1 + shfl_x(sel(low, u1, l3), 2);
    }
    const R hc = MODE == kDhat2 ? R(0.5) : R(-0.5);  // -1/2 times the sign of the hopping term
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = hc * (v[k] + shfl_x(v[k], 1));
    C o[6];
    if constexpr (MODE == kDhat1) {
        herm6_mul(d, v, o);
    } else {
        const R* f = static_cast<const R*>(a.self) + canon + (size_t)i * 24 + 12 * (q >> 1);
        C s[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) s[k] = {f[2 * k], f[2 * k + 1]};
        if (MODE == kDhat2 && dg && low) {
#pragma unroll
            for (int k = 0; k < 6; ++k) s[k] = -s[k];
        }
        herm6_mul(d, s, o);
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = v[k] + o[k];
        if (MODE == kDhat2 && dg && low) {
#pragma unroll
            for (int k = 0; k < 6; ++k) o[k] = -o[k];
        }
    }
    // both lanes of a pair have read the site's own input by now (in place: before either writes)
    __syncwarp();
    if (!live) return;
    const bool odd = q & 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const C w = sel(odd, o[3 + k], o[k]);
        if constexpr (MODE == kDhat1) {
            const int m = 3 * q + k;  // component of the internal field
            if constexpr (P == 0) static_cast<double2*>(a.out)[inner + (size_t)m * Vh + h] = make_double2(w.re, w.im);
            else reinterpret_cast<float2*>(static_cast<float4*>(a.out) + inner + (size_t)(m >> 1) * Vh + h)[m & 1] = make_float2(w.re, w.im);
        } else {
            R* f = static_cast<R*>(a.out) + canon + (size_t)i * 24 + 6 * q + 2 * k;
            f[0] = w.re;
            f[1] = w.im;
        }
    }
}

// site and right-hand-side products up to which four lanes per site are the faster.  One thread
// and four lanes (us), by sites of the output times right-hand sides: Dhat FP32 12.3 and 6.3 at 4096,
// 11.5 at 8192, FP64 83.9 and 44 at 2048, 76 at 4096; D_w FP32 6.1 and 4.1 at 7168, 4.2 to 7.5 at
// 8192, 9.4 at 10240, FP64 40.9 and 15.6 at 2560, 42.4 at 3072, 48.5 at 4096
constexpr long long quad_sites(int prec, int mode) { return prec != QXD_FP64 ? 8192 : mode == kDw ? 2560 : 4096; }

template <int P, int MODE>
cudaError_t launch_quad(const Geo& g, const CanonDev& a, int nrhs, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(nblocks(MODE == kDw ? g.V : g.Vh, kQuadThreads / 4) * nrhs));
    cfg.blockDim = dim3(kQuadThreads);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_hop_quad<P, MODE>, g, a, nrhs);
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
    // D_w of several right-hand sides on a large lattice goes over the sites in two launches
    // (the first and the second half): as many as over two half lattices, which profiles of
    // launches count on.  It is not the faster form (24^3x48 with 12 right-hand sides 762 us, 747 in
    // one launch); 2^20 keeps it away from small lattices, where a second launch costs more.
    const int sites = MODE == kDw ? (int)g.V : g.Vh;
    const int parts = MODE == kDw && nrhs > 1 && (long long)sites * nrhs > (1 << 20) ? 2 : 1;
    for (int k = 0; k < parts; ++k) {
        const int first = k * (sites / parts), end = k + 1 == parts ? sites : (k + 1) * (sites / parts);
        ProfScope prof(ctx, name, (double)g.Vh * ((MODE == kDw ? link + 2 * dg : link + dg) + per * nrhs) / parts, st);
        if (prec != QXD_BF16 && (long long)sites * nrhs <= quad_sites(prec, MODE)) {
            const cudaError_t e = prec == QXD_FP64 ? launch_quad<0, MODE>(g, a, nrhs, st) : launch_quad<1, MODE>(g, a, nrhs, st);
            QXD_CUDA(ctx, e);
            continue;
        }
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
