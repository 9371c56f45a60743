// Schwarz alternating procedure (SAP) preconditioner (Sec. 4.1 and 4.4: SAP+GCR,
// blocks of 4^4 sites, ncy cycles, nmr minimal-residual steps per block).
//
// Blocks of 4^4 sites tile the simulated lattice and are coloured like a
// checkerboard by the parity of the block coordinates.  The block operator is
// D with Dirichlet block boundaries (hops leaving the block dropped).  One
// application M eta: psi = 0, rho = eta; ncy times, for each colour: every block
// of that colour solves its block system approximately (even-odd system of the
// block, nmr minimal-residual steps from zero) for the current residual
// rho = eta - D psi restricted to the block, and psi += d on the block.  As a
// preconditioner of Dhat: z_e = (M (r_e, 0))_e.  Every extent must hold an even
// number of blocks, so that blocks of one colour never touch, across the
// periodic boundary included.
//
// GPU layout: one launch per colour sweep, one CTA per block, 256 threads; the lane
// pair (2u, 2u + 1) owns the u-th even and the u-th odd site of the block, lane h
// the chiral block (spins 2h, 2h + 1) of every field, so that a lane keeps half a
// spinor per field and applies one 6 x 6 block of the site-diagonal terms (128
// registers, two CTAs and 16 warps per SM).  The block's links, V = U z^qhat in full, are
// staged in shared memory once per sweep, so the 2 nmr + 2 block hops of the
// minimal-residual steps read links and neighbour spinors from shared memory only.
// The sweep also computes the block residual rho = eta - D psi itself (the
// other colour's psi on the one-site halo comes from global memory), so no
// full-lattice residual is formed between colours.  Site-diagonal terms are
// streamed from global memory.  FP32 throughout, block sums in FP32.
//
// Bound by latency and shared-memory loads (35 % of the issue slots, 49 % of the LSU; the
// site-diagonal terms of each step come from L2).  Per lane and direction a colour product is
// 18 packed multiply-adds, (Re, Im) of a link entry times a duplicated part of the
// half-spinor (half the instructions).  Directions are unrolled with the
// half's signs as factors: a run-time loop with selects took 2.6 times the instructions.
// Sweep of 24^3x48 with nmr = 5: 499 us so, 496 us with few instructions but strided reads
// and bank conflicts, 276 us with the blocks' own copies and spins interleaved.
#include <cmath>
#include <cstdlib>

#include "blas.h"
#include "block.cuh"
#include "hop.cuh"
#include "ops.h"
#include "qxd_internal.h"

namespace qxd {

constexpr int kSapB = kBlk;
constexpr int kSapThreads = kBlkThreads;
constexpr int kSapSites = kBlkSites;
constexpr int kSapLanes = 2 * kSapThreads;  // threads of a sweep CTA: two lanes per (even, odd) site pair

struct SapDev {
    int nb[4];              // blocks per direction
    const float4* U32[2];   // links per parity
    const float4* Z32[2];   // phases per parity
    const float4* A[2];     // site-diagonal term per parity
    const float4* Aoo_inv;  // its inverse, odd sites
    const float4* eta;      // source, full field (even half, odd half)
    float4* psi;            // solution, full field
    const struct SapBlock* blocks;  // the blocks' own copies (null: not built)
    int nmr;
};

// the block's links: entries 0 .. 7 of V = U z^qhat per direction and local site, then entry 8
struct SapLinks {
    float4 lk4[4][4][kSapSites];
    float2 lk2[4][kSapSites];
};

// What a sweep streams of one block, in the order in which its threads read it (built once per
// flavour by k_sap_blocks): the fields themselves hold two sites of a block, 32 bytes, side by
// side, and the sites next to them belong to a block of the other colour, so that a sweep
// fetched twice its bytes from memory and each warp load touched 16 lines.
struct SapBlock {
    SapLinks lk;
    float4 diag[3][9][kSapLanes];  // A_ee, A_oo^-1, A_oo: chunk k of the lane's 6x6 block
};

// a spinor buffer of one parity: [colour][spins 2g, 2g + 1][site][spin & 1], so that the two
// lanes of a site pair read neighbouring banks
using SapSpinor = float2[3][2][kSapThreads][2];

// shared memory of one block: its links, two half-block spinor buffers and the odd residual
struct SapShared {
    SapLinks lk;
    SapSpinor sp[2];               // spinor buffers by parity
    float2 rho_o[6][kSapLanes];    // residual on the odd sites
    float red[3 * kSapLanes / 32];
};

__device__ __forceinline__ unsigned long long f2_bits(float2 a) { return *reinterpret_cast<unsigned long long*>(&a); }
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 f2_dup(float a) { return make_float2(a, a); }

// A pair of adjacent lanes (2u, 2u + 1) owns the u-th even and the u-th odd site
// of the block; lane `half` holds the spins 2 half, 2 half + 1 (its chiral block,
// complex components 6 half .. 6 half + 5) of every field it keeps.
__device__ __forceinline__ void store6_sm(SapSpinor& sm, int u, int half, const float2 v[6]) {
#pragma unroll
    for (int c = 0; c < 3; ++c)  // spins 2 half, 2 half + 1
        *reinterpret_cast<float4*>(&sm[c][half][u][0]) = make_float4(v[c].x, v[c].y, v[3 + c].x, v[3 + c].y);
}
// the chiral block of a global FP32 field: complex 6 half + k is in chunk 3 half + k / 2
__device__ __forceinline__ void load6_glob(const float4* __restrict__ b, int Vh, int h, int half, float2 v[6]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float4 f = QXD_LDG(b + (size_t)(3 * half + c) * Vh + h);
        v[2 * c] = make_float2(f.x, f.y);
        v[2 * c + 1] = make_float2(f.z, f.w);
    }
}
__device__ __forceinline__ void store6_glob(float4* __restrict__ b, int Vh, int h, int half, const float2 v[6]) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
        b[(size_t)(3 * half + c) * Vh + h] = make_float4(v[2 * c].x, v[2 * c].y, v[2 * c + 1].x, v[2 * c + 1].y);
}
// spin sp (three colours) of a site
__device__ __forceinline__ void load_spin_sm(const SapSpinor& sm, int u, int sp, float2 v[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = sm[c][sp >> 1][u][sp & 1];
}
__device__ __forceinline__ void load_spin_glob(const float4* __restrict__ b, int Vh, int h, int sp, float2 v[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int k = 3 * sp + c;
        const float4 f = QXD_LDG(b + (size_t)(k >> 1) * Vh + h);
        v[c] = (k & 1) ? make_float2(f.z, f.w) : make_float2(f.x, f.y);
    }
}

// V = U z^qhat of direction mu at the block's local site sid (= parity * 128 + slot)
__device__ __forceinline__ void link_sm(const SapShared& S, int mu, int sid, float2 m[9]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 v = S.lk.lk4[mu][k][sid];
        m[2 * k] = make_float2(v.x, v.y);
        m[2 * k + 1] = make_float2(v.z, v.w);
    }
    m[8] = S.lk.lk2[mu][sid];
}
__device__ __forceinline__ void link_glob(const float4* __restrict__ U32, const float4* __restrict__ Z32, int Vh, int mu,
                                          int h, float2 m[9]) {
    Mat3<float> u;
    cplx<float> z;
    load_link32(U32, Z32, Vh, mu, h, u, z);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const cplx<float> v = z * u.a[k / 3][k % 3];
        m[k] = make_float2(v.re, v.im);
    }
}

// what a lane sums over the hops: spin `half` of the output (o), and the lower spins that its
// half-spinor component feeds: spin 2 + half (p, times i: pi) in directions 0 and 3, spin
// 3 - half (q, times i: qi) in directions 2 and 1
struct HopSum {
    float2 o[3], p[3], pi[3], q[3], qi[3];
};

// One hop of direction MU: the half-spinor component `half` of the projection (spins half and
// its partner), times the link (V forwards, V^+ backwards), added to the sums.  hs = +1 for
// half 0, -1 for half 1: signs that depend on the half come as a factor, so the pair's lanes
// run the same instructions.
template <int MU, bool FWD>
__device__ __forceinline__ void hop_one(const float2 sa[3], const float2 sb[3], const float2 m[9], float hs,
                                        HopSum& H) {
    // projection (1 -+ gamma_mu): s_half + f s_partner, f = +-1 (MU 0, 2) or +-i (MU 1, 3)
    const float f = MU < 2 ? (FWD ? 1.f : -1.f) : (FWD ? hs : -hs);
    float2 A[3], B[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        float2 h;
        if (MU & 1) h = make_float2(fmaf(-f, sb[j].y, sa[j].x), fmaf(f, sb[j].x, sa[j].y));
        else h = f2_fma(sb[j], f2_dup(f), sa[j]);
        const float2 hr = f2_dup(h.x), hi = f2_dup(h.y);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float2 e = FWD ? m[3 * i + j] : m[3 * j + i];
            A[i] = j == 0 ? f2_mul(e, hr) : f2_fma(e, hr, A[i]);
            B[i] = j == 0 ? f2_mul(e, hi) : f2_fma(e, hi, B[i]);
        }
    }
    const float g = MU == 0 ? (FWD ? 1.f : -1.f) : MU == 1 ? (FWD ? -1.f : 1.f) : MU == 2 ? (FWD ? hs : -hs) : (FWD ? -hs : hs);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float2 r = FWD ? make_float2(A[i].x - B[i].y, A[i].y + B[i].x) : make_float2(A[i].x + B[i].y, B[i].x - A[i].y);
        H.o[i] = f2_add(H.o[i], r);
        float2& t = MU == 0 ? H.p[i] : MU == 1 ? H.qi[i] : MU == 2 ? H.q[i] : H.pi[i];
        t = f2_fma(r, f2_dup(g), t);
    }
}

// one direction at site s of parity P, local coordinates l, slot t (see hop_pair)
template <int P, bool HALO, int MU, bool FWD>
__device__ __forceinline__ void hop_dir_pair(const Geo& g, const SapDev& a, const SapShared& S, const SiteRef& s, int t,
                                             const SapSpinor& nb, const float4* nb_glob, int half, float hs,
                                             HopSum& H) {
    const int partner = (MU == 0 || MU == 3) ? 2 + half : 3 - half;
    const bool inside = FWD ? s.l[MU] + 1 < kSapB : s.l[MU] > 0;
    if (!HALO && !inside) return;
    float2 sa[3], sb[3], m[9];
    if (inside) {
        constexpr int st = MU == 0 ? 32 : MU == 1 ? 8 : MU == 2 ? 2 : 0;
        const int tn = MU < 3 ? (FWD ? t + st : t - st) : (FWD ? t + (s.l[3] & 1) : t - ((s.l[3] & 1) ^ 1));
        load_spin_sm(nb, tn, half, sa);
        load_spin_sm(nb, tn, partner, sb);
        link_sm(S, MU, FWD ? P * kSapThreads + t : (1 - P) * kSapThreads + tn, m);
    } else {
        const int hn = neighbour_lex(g, s.x, MU, FWD ? +1 : -1) >> 1;
        load_spin_glob(nb_glob, g.Vh, hn, half, sa);
        load_spin_glob(nb_glob, g.Vh, hn, partner, sb);
        if (FWD) link_sm(S, MU, P * kSapThreads + t, m);
        else link_glob(a.U32[1 - P], a.Z32[1 - P], g.Vh, MU, hn, m);
    }
    hop_one<MU, FWD>(sa, sb, m, hs, H);
}

// This lane's chiral block of
//   out = -1/2 sum_mu [(1 - gamma_mu) V(x,mu) f(x+mu) + (1 + gamma_mu) V(x-mu,mu)^+ f(x-mu)]
// at site s (slot t) of parity P, f the opposite-parity spinors in the buffer nb.  HALO = false:
// hops leaving the block are dropped (block operator); HALO = true: they take the
// spinor of the neighbouring site from the global field nb_glob and, backwards, its
// link from global memory.  The two lanes then exchange their partial sums.
template <int P, bool HALO>
__device__ __forceinline__ void hop_pair(const Geo& g, const SapDev& a, const SapShared& S, const SiteRef& s, int t,
                                         const SapSpinor& nb, const float4* nb_glob, int half, float2 out[6]) {
    HopSum H;
#pragma unroll
    for (int c = 0; c < 3; ++c) H.o[c] = H.p[c] = H.pi[c] = H.q[c] = H.qi[c] = make_float2(0.f, 0.f);
    const float hs = half ? -1.f : 1.f;
    hop_dir_pair<P, HALO, 0, true>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 0, false>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 1, true>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 1, false>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 2, true>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 2, false>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 3, true>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    hop_dir_pair<P, HALO, 3, false>(g, a, S, s, t, nb, nb_glob, half, hs, H);
    // lane 0 takes spins 0 (own o) and 1 (partner's o); lane 1 spin 2 (lane 0's p + own q)
    // and spin 3 (lane 0's q + own p)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 p = make_float2(H.p[c].x - H.pi[c].y, H.p[c].y + H.pi[c].x);
        const float2 q = make_float2(H.q[c].x - H.qi[c].y, H.q[c].y + H.qi[c].x);
        // lane 0 sends p and q, lane 1 its o: two exchanges
        const float2 x = half ? H.o[c] : p;
        const float2 rx = make_float2(__shfl_xor_sync(0xffffffffu, x.x, 1), __shfl_xor_sync(0xffffffffu, x.y, 1));
        const float2 rq = make_float2(__shfl_xor_sync(0xffffffffu, q.x, 1), __shfl_xor_sync(0xffffffffu, q.y, 1));
        const float2 s0 = half == 0 ? H.o[c] : f2_add(rx, q);
        const float2 s1 = half == 0 ? rx : f2_add(rq, p);
        out[c] = f2_mul(s0, f2_dup(-0.5f));
        out[3 + c] = f2_mul(s1, f2_dup(-0.5f));
    }
}

// v = D v for this lane's chiral block of a packed site-diagonal term (one
// Hermitian 6x6 block, 9 float4 `stride` apart), streamed from global memory.  An upper entry e = (Re, Im)
// enters row i as e v_j and row j as e^* v_i: packed products of e with duplicated parts.
__device__ __forceinline__ void diag6(const float4* __restrict__ D, size_t stride, float2 v[6]) {
    float2 d[18];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float4 f = QXD_LDG(D + k * stride);
        d[2 * k] = make_float2(f.x, f.y);
        d[2 * k + 1] = make_float2(f.z, f.w);
    }
    float2 out[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) out[i] = f2_mul(f2_dup((i & 1) ? d[i / 2].y : d[i / 2].x), v[i]);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        // row i: sum_{j > i} e_ij v_j  and  sum_{j < i} e_ji^* v_j
        float2 A = make_float2(0.f, 0.f), B = A, C = A, E = A;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j == i) continue;
            const float2 e = d[3 + herm_off(i < j ? i : j, i < j ? j : i)];
            if (j > i) {
                A = f2_fma(e, f2_dup(v[j].x), A);
                B = f2_fma(e, f2_dup(v[j].y), B);
            } else {
                C = f2_fma(e, f2_dup(v[j].x), C);
                E = f2_fma(e, f2_dup(v[j].y), E);
            }
        }
        out[i].x += (A.x - B.y) + (C.x + E.y);
        out[i].y += (A.y + B.x) + (E.x - C.y);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) v[i] = out[i];
}

// sum over the CTA of three floats (the caller synchronises before sh is used again)
__device__ __forceinline__ void cta_sum3(float v[3], float* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane == 0)
        for (int k = 0; k < 3; ++k) sh[warp * 3 + k] = v[k];
    __syncthreads();
    for (int k = 0; k < 3; ++k) {
        float s = 0.f;
        for (int w = 0; w < kSapLanes / 32; ++w) s += sh[w * 3 + k];
        v[k] = s;
    }
}

__device__ __forceinline__ void sub6(float2 a[6], const float2 b[6]) {
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k] = f2_fma(b[k], f2_dup(-1.f), a[k]);
}

// the block's links into lk: lane `half` takes directions 2 half, 2 half + 1
__device__ __forceinline__ void stage_links(const SapDev& a, SapLinks& lk, int Vh, const SiteRef& se, const SiteRef& so,
                                            int u, int half) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int h = p == 0 ? se.h : so.h;
        const int sid = p * kSapThreads + u;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int mu = 2 * half + q;
            float2 m[9];
            link_glob(a.U32[p], a.Z32[p], Vh, mu, h, m);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                lk.lk4[mu][k][sid] = make_float4(m[2 * k].x, m[2 * k].y, m[2 * k + 1].x, m[2 * k + 1].y);
            lk.lk2[mu][sid] = m[8];
        }
    }
}

// a block's own copy of its links and site-diagonal terms, one CTA per block
__global__ void __launch_bounds__(kSapLanes) k_sap_blocks(Geo g, SapDev a, SapBlock* __restrict__ blocks) {
    int bc[4];
    block_coords(blockIdx.x, a.nb, bc);
    const int u = threadIdx.x >> 1;
    const int half = threadIdx.x & 1;
    SiteRef se, so;
    block_site(g, bc, 0, u, se);
    block_site(g, bc, 1, u, so);
    SapBlock& B = blocks[blockIdx.x];
    stage_links(a, B.lk, g.Vh, se, so, u, half);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const size_t o = (size_t)(half * 9 + k) * g.Vh;
        B.diag[0][k][threadIdx.x] = a.A[0][o + se.h];
        B.diag[1][k][threadIdx.x] = a.Aoo_inv[o + so.h];
        B.diag[2][k][threadIdx.x] = a.A[1][o + so.h];
    }
}

// One colour sweep of SAP: every block of colour `colour` (one CTA each) takes
// its residual rho = eta - D psi (FIRST: psi = 0, so rho = eta), solves its
// Dirichlet block system approximately by nmr minimal-residual steps on the
// block's even-odd system, and adds the block solution to psi.  Blocks of one
// colour never touch, so every CTA reads the other colour's psi on its halo
// and writes its own sites only.  Two lanes per site pair (one chiral block each).
// BLK: links and site-diagonal terms from the blocks' own copies (SapBlock), else from the fields.
template <bool FIRST, bool BLK>
__global__ void __launch_bounds__(kSapLanes, 2) k_sap_sweep(Geo g, SapDev a, int colour) {
    extern __shared__ __align__(16) unsigned char sap_smem[];
    SapShared& S = *reinterpret_cast<SapShared*>(sap_smem);
    // block blockIdx.x of the colour: bc3 takes every second value
    int bc[4];
    {
        const int n3 = a.nb[3] / 2;
        int b = blockIdx.x / n3;
        bc[2] = b % a.nb[2];
        b /= a.nb[2];
        bc[1] = b % a.nb[1];
        bc[0] = b / a.nb[1];
        bc[3] = 2 * (blockIdx.x % n3) + ((colour + bc[0] + bc[1] + bc[2]) & 1);
    }
    const int u = threadIdx.x >> 1;
    const int half = threadIdx.x & 1;
    const int Vh = g.Vh;
    SiteRef se, so;
    block_site(g, bc, 0, u, se);
    block_site(g, bc, 1, u, so);
    // this lane's 6x6 blocks of A_ee, A_oo^-1 and A_oo
    const float4 *Aee, *Aoi, *Aoo;
    size_t ds;
    if constexpr (BLK) {
        const SapBlock* blk = a.blocks + ((bc[0] * a.nb[1] + bc[1]) * a.nb[2] + bc[2]) * a.nb[3] + bc[3];
        const float4* src = reinterpret_cast<const float4*>(&blk->lk);
        float4* dst = reinterpret_cast<float4*>(&S.lk);
        constexpr int n = sizeof(SapLinks) / 16 / kSapLanes;
#pragma unroll
        for (int k = 0; k < n; ++k)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             static_cast<uint32_t>(__cvta_generic_to_shared(dst + k * kSapLanes + threadIdx.x))),
                         "l"(src + k * kSapLanes + threadIdx.x)
                         : "memory");
        asm volatile("cp.async.wait_all;" ::: "memory");
        Aee = &blk->diag[0][0][threadIdx.x];
        Aoi = &blk->diag[1][0][threadIdx.x];
        Aoo = &blk->diag[2][0][threadIdx.x];
        ds = kSapLanes;
    } else {
        stage_links(a, S.lk, Vh, se, so, u, half);
        const size_t o = (size_t)half * 9 * Vh;
        Aee = a.A[0] + o + se.h;
        Aoi = a.Aoo_inv + o + so.h;
        Aoo = a.A[1] + o + so.h;
        ds = Vh;
    }
    const float4* psi_e = a.psi;
    const float4* psi_o = a.psi + 6 * (size_t)Vh;
    float2 v[6], r[6], y[6];
    // residual rho = eta - D psi on the block's sites: r (even), rho_o (odd, shared)
    load6_glob(a.eta, Vh, se.h, half, r);
    load6_glob(a.eta + 6 * (size_t)Vh, Vh, so.h, half, y);
    if (!FIRST) {
        float2 w[6];
        load6_glob(psi_e, Vh, se.h, half, v);
        store6_sm(S.sp[0], u, half, v);
        load6_glob(psi_o, Vh, so.h, half, w);
        store6_sm(S.sp[1], u, half, w);
        __syncthreads();
        // even site: A_ee psi_e + H_eo psi_o
        diag6(Aee, ds, v);
        sub6(r, v);
        hop_pair<0, true>(g, a, S, se, u, S.sp[1], psi_o, half, v);
        sub6(r, v);
        // odd site: A_oo psi_o + H_oe psi_e
        diag6(Aoo, ds, w);
        sub6(y, w);
        hop_pair<1, true>(g, a, S, so, u, S.sp[0], psi_e, half, v);
        sub6(y, v);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) S.rho_o[k][threadIdx.x] = y[k];
    // t_o = A_oo^-1 rho_o
    diag6(Aoi, ds, y);
    __syncthreads();  // every lane is done with the psi buffers
    store6_sm(S.sp[1], u, half, y);
    __syncthreads();
    // it = 0: b_e = rho_e - H^B_eo t_o; it = 1 .. nmr: the minimal-residual steps; then the
    // odd sites.  One loop, so that each of the two block hops exists once in the code.
#pragma unroll 1
    for (int it = 0;; ++it) {
        if (it > 0) {
            hop_pair<1, false>(g, a, S, so, u, S.sp[0], nullptr, half, v);
            if (it > a.nmr) break;
            // t_o = A_oo^-1 H^B_oe r_e
            diag6(Aoi, ds, v);
            store6_sm(S.sp[1], u, half, v);
            __syncthreads();
        }
        hop_pair<0, false>(g, a, S, se, u, S.sp[1], nullptr, half, v);
        if (it == 0) {
            sub6(r, v);
#pragma unroll
            for (int k = 0; k < 6; ++k) y[k] = make_float2(0.f, 0.f);
        } else {
            // p = Dhat_B r = A_ee r - H^B_eo t_o
            float2 p[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) p[k] = r[k];
            diag6(Aee, ds, p);
            sub6(p, v);
            // <p, r> = sum conj(p) r and |p|^2, real and imaginary products side by side
            float2 pr = make_float2(0.f, 0.f), px = pr, pp = pr;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                pr = f2_fma(p[k], r[k], pr);
                px = f2_fma(p[k], make_float2(r[k].y, r[k].x), px);
                pp = f2_fma(p[k], p[k], pp);
            }
            float s3[3] = {pr.x + pr.y, px.x - px.y, pp.x + pp.y};
            cta_sum3(s3, S.red);
            const float2 alpha = s3[2] > 0.f ? make_float2(s3[0] / s3[2], s3[1] / s3[2]) : make_float2(0.f, 0.f);
            const float2 ax = f2_dup(alpha.x), ay = make_float2(-alpha.y, alpha.y);
            const float2 nx = f2_dup(-alpha.x), ny = make_float2(alpha.y, -alpha.y);
#pragma unroll
            for (int k = 0; k < 6; ++k) {  // y += alpha r, r -= alpha p
                y[k] = f2_fma(ay, make_float2(r[k].y, r[k].x), f2_fma(ax, r[k], y[k]));
                r[k] = f2_fma(ny, make_float2(p[k].y, p[k].x), f2_fma(nx, p[k], r[k]));
            }
        }
        // the last step hands on y instead of r; the other warps may still read the sums, but
        // not sp[0], which the odd hop of this step read before its barrier
        const bool last = it == a.nmr;
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = last ? y[k] : r[k];
        store6_sm(S.sp[0], u, half, v);
        __syncthreads();
    }
    // d_o = A_oo^-1 (rho_o - H^B_oe y);  psi += d
    float2 w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = S.rho_o[k][threadIdx.x];
    sub6(w, v);
    diag6(Aoi, ds, w);
    if (!FIRST) {
        load6_glob(psi_e, Vh, se.h, half, v);
#pragma unroll
        for (int k = 0; k < 6; ++k) y[k] = f2_add(y[k], v[k]);
        load6_glob(psi_o, Vh, so.h, half, v);
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = f2_add(w[k], v[k]);
    }
    store6_glob(a.psi, Vh, se.h, half, y);
    store6_glob(a.psi + 6 * (size_t)Vh, Vh, so.h, half, w);
}

int sap_check(qxd_ctx* ctx) {
    for (int mu = 0; mu < 4; ++mu)
        if (ctx->g.N[mu] % (2 * kSapB))
            return qxd_fail(ctx, QXD_EARG, "SAP: every simulated extent must be a multiple of 8 (an even number of 4^4 blocks)");
    return QXD_OK;
}

// The blocks' own copies of a flavour (720 bytes per site), built on the first sweep after its
// links or SW term were set, in a buffer that stays for the next ones (qxd_set_clover and one
// application with ncy = nmr = 1: 8^4 0.42 -> 0.26 ms, 32 x 16^3 2.45 -> 2.24 ms); without memory
// for them the sweeps read the fields (for the tests also with QXD_SAP_BLOCKS=0 in the environment).
static int sap_blocks(qxd_ctx* ctx, int fl, SapDev& a, int nblk, cudaStream_t st) {
    QxdFlavour& F = ctx->fl[fl];
    const char* env = std::getenv("QXD_SAP_BLOCKS");
    if (env && env[0] == '0') return QXD_OK;
    // a captured graph may outlive the copies
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return QXD_OK;
    if (!F.sap && !F.sap_off && !dev_alloc(ctx, &F.sap, sizeof(SapBlock) * (size_t)nblk)) F.sap_off = true;
    if (!F.sap) return QXD_OK;
    if (!F.sap_built) {
        {
            ProfScope prof(ctx, "sap_blocks", (double)ctx->g.V * (224 + 432 + 720), st);
            k_sap_blocks<<<nblk, kSapLanes, 0, st>>>(ctx->g, a, static_cast<SapBlock*>(F.sap));
        }
        QXD_CUDA(ctx, cudaGetLastError());
        // other streams may sweep with it as soon as this call returns
        QXD_CUDA(ctx, cudaStreamSynchronize(st));
        F.sap_built = true;
    }
    a.blocks = static_cast<const SapBlock*>(F.sap);
    return QXD_OK;
}

// psi = M eta on full FP32 fields (even half then odd half); psi must not alias eta
int sap_apply_full(qxd_ctx* ctx, int fl, const float4* eta, float4* psi, cudaStream_t st) {
    QXD_TRY(sap_check(ctx));
    const Geo& g = ctx->g;
    const size_t hb = half_bytes(ctx, QXD_FP32);
    const QxdFlavour& F = ctx->fl[fl];
    SapDev a{};
    int nblk = 1;
    for (int mu = 0; mu < 4; ++mu) {
        a.nb[mu] = g.N[mu] / kSapB;
        nblk *= a.nb[mu];
    }
    for (int p = 0; p < 2; ++p) {
        a.U32[p] = ctx->U32 + (size_t)p * 12 * g.Vh;
        a.Z32[p] = F.Z32 + (size_t)p * 2 * g.Vh;
        a.A[p] = F.C32[0] + (size_t)p * 18 * g.Vh;
    }
    a.Aoo_inv = F.C32[1] + (size_t)18 * g.Vh;
    a.eta = eta;
    a.psi = psi;
    a.nmr = ctx->sap_nmr;
    QXD_TRY(sap_blocks(ctx, fl, a, nblk, st));
    const int smem = (int)sizeof(SapShared);
    auto first = a.blocks ? k_sap_sweep<true, true> : k_sap_sweep<true, false>;
    auto next = a.blocks ? k_sap_sweep<false, true> : k_sap_sweep<false, false>;
    QXD_CUDA(ctx, cudaFuncSetAttribute(first, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    QXD_CUDA(ctx, cudaFuncSetAttribute(next, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    QXD_CUDA(ctx, cudaMemsetAsync(psi, 0, 2 * hb, st));
    // algorithmic bytes per site of a sweep's colour: own links 224, eta 96, psi of the
    // block and its halo 192, psi written 96, A 288, A_oo^-1 on odd sites 144, halo links 56
    const double site_bytes = 224 + 96 + 192 + 96 + 288 + 144 + 56;
    for (int cy = 0; cy < ctx->sap_ncy; ++cy) {
        for (int colour = 0; colour < 2; ++colour) {
            ProfScope prof(ctx, "sap_sweep", (double)g.Vh * site_bytes, st);
            if (cy == 0 && colour == 0)
                first<<<nblk / 2, kSapLanes, smem, st>>>(g, a, colour);
            else
                next<<<nblk / 2, kSapLanes, smem, st>>>(g, a, colour);
            QXD_CUDA(ctx, cudaGetLastError());
        }
    }
    return QXD_OK;
}

// z_e = (M (r_e, 0))_e on FP32 even fields
int sap_apply_even(qxd_ctx* ctx, int fl, const void* r_e, void* z_e, cudaStream_t st) {
    const size_t hb = half_bytes(ctx, QXD_FP32);
    void *eta, *psi;
    QXD_TRY(qxd_ws(ctx, WS_SAP + 2, 2 * hb, &eta));
    QXD_TRY(qxd_ws(ctx, WS_SAP + 3, 2 * hb, &psi));
    QXD_CUDA(ctx, cudaMemcpyAsync(eta, r_e, hb, cudaMemcpyDeviceToDevice, st));
    QXD_CUDA(ctx, cudaMemsetAsync(static_cast<char*>(eta) + hb, 0, hb, st));
    QXD_TRY(sap_apply_full(ctx, fl, static_cast<const float4*>(eta), static_cast<float4*>(psi), st));
    QXD_CUDA(ctx, cudaMemcpyAsync(z_e, psi, hb, cudaMemcpyDeviceToDevice, st));
    return QXD_OK;
}

}  // namespace qxd

using namespace qxd;

extern "C" {

int qxd_set_sap(qxd_ctx* ctx, int ncy, int nmr) {
    if (!ctx) return QXD_EARG;
    if (ncy < 1 || ncy > 64 || nmr < 1 || nmr > 64) return qxd_fail(ctx, QXD_EARG, "set_sap: ncy and nmr in 1..64");
    ctx->sap_ncy = ncy;
    ctx->sap_nmr = nmr;
    return QXD_OK;
}

int qxd_sap_apply(qxd_ctx* ctx, int fl, const void* in, void* out, void* stream) {
    if (!ctx) return QXD_EARG;
    if (fl < 0 || fl >= QXD_MAX_FLAVOURS) return qxd_fail(ctx, QXD_EARG, "flavour id out of range 0..7");
    if (!ctx->links_set || !ctx->fl[fl].set) return qxd_fail(ctx, QXD_ESTATE, "sap_apply: links and SW term first");
    if (!in || !out) return qxd_fail(ctx, QXD_EARG, "sap_apply: NULL argument");
    QXD_TRY(sap_check(ctx));
    cudaSetDevice(ctx->device);
    cudaStream_t st = (cudaStream_t)stream;
    const size_t cb = (size_t)ctx->g.V * 12 * 8;
    const size_t hb = half_bytes(ctx, QXD_FP32);
    void *cin, *cout, *fin, *fout;
    QXD_TRY(qxd_ws(ctx, WS_SAP + 4, cb, &cin));
    QXD_TRY(qxd_ws(ctx, WS_SAP + 5, cb, &cout));
    QXD_TRY(qxd_ws(ctx, WS_SAP + 6, 2 * hb, &fin));
    QXD_TRY(qxd_ws(ctx, WS_SAP + 7, 2 * hb, &fout));
    QXD_CUDA(ctx, cudaMemcpyAsync(cin, in, cb, cudaMemcpyDefault, st));
    char* fi = static_cast<char*>(fin);
    char* fo = static_cast<char*>(fout);
    QXD_TRY(launch_pack(ctx, 1, cin, 1, 0, QXD_FP32, fi, 1, st));
    QXD_TRY(launch_pack(ctx, 1, cin, 1, 1, QXD_FP32, fi + hb, 1, st));
    QXD_TRY(sap_apply_full(ctx, fl, reinterpret_cast<const float4*>(fi), reinterpret_cast<float4*>(fo), st));
    QXD_TRY(launch_unpack(ctx, QXD_FP32, fo, 0, 1, cout, 1, 1, st));
    QXD_TRY(launch_unpack(ctx, QXD_FP32, fo + hb, 1, 1, cout, 1, 1, st));
    QXD_CUDA(ctx, cudaMemcpyAsync(out, cout, cb, cudaMemcpyDefault, st));
    QXD_CUDA(ctx, cudaStreamSynchronize(st));
    return QXD_OK;
}

}  // extern "C"
