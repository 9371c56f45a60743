// Field set-up kernels: gauge-field ingest with the C* mirror fill, per-flavour
// hopping phases, and the site-diagonal term 1/(2 kappa) + dD_sw with its
// inverse (Sec. 2.1 eq. cstar-bc-gauge; Sec. 2.3 eqs. frw-covder, sw-term).
#include <algorithm>

#include "blas.h"
#include "qxd_internal.h"

namespace qxd {

using C64 = cplx<double>;

struct M3 {
    C64 a[9];
};

QXD_HD M3 m3_load(const double2* __restrict__ U, int stride, int mu, int h) {
    M3 m;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        double2 v = QXD_LDG(U + (size_t)(mu * 9 + k) * stride + h);
        m.a[k] = {v.x, v.y};
    }
    return m;
}

// product a*b with a or b optionally daggered
template <bool DA, bool DB>
QXD_HD M3 m3_mul(const M3& a, const M3& b) {
    M3 c;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            C64 s = {0.0, 0.0};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                C64 x = DA ? conj(a.a[k * 3 + i]) : a.a[i * 3 + k];
                C64 y = DB ? conj(b.a[j * 3 + k]) : b.a[k * 3 + j];
                cmac(s, x, y);
            }
            c.a[i * 3 + j] = s;
        }
    return c;
}

// link U(y, mu) of the simulated site with coordinates y
QXD_HD M3 link_at(const Geo& g, const double2* __restrict__ U64, const int y[4], int mu) {
    int lex = lex_index(g, y);
    int par = (y[0] + y[1] + y[2] + y[3]) & 1;
    return m3_load(U64 + (size_t)par * 36 * g.Vh, g.Vh, mu, lex >> 1);
}

QXD_HD void step(const Geo& g, const int x[4], int mu, int sign, int y[4]) {
    int lex = neighbour_lex(g, x, mu, sign);
    int n3 = g.N[3], n2 = g.N[2], n1 = g.N[1];
    y[3] = lex % n3;
    lex /= n3;
    y[2] = lex % n2;
    lex /= n2;
    y[1] = lex % n1;
    y[0] = lex / n1;
}

QXD_HD double A_at(const Geo& g, const double* __restrict__ A64, const int y[4], int mu) {
    int lex = lex_index(g, y);
    int par = (y[0] + y[1] + y[2] + y[3]) & 1;
    return QXD_LDG(A64 + (size_t)par * 4 * g.Vh + (size_t)mu * g.Vh + (lex >> 1));
}

// ------------------------------------------------------------------------------
// set_links: physical-lattice input -> internal extended-lattice fields.
__global__ void k_set_links(Geo g, int L1phys, int L2, int L3, const double2* __restrict__ Uin,
                            const double* __restrict__ Ain, double2* __restrict__ U64, double* __restrict__ A64,
                            float4* __restrict__ U32) {
    int h = blockIdx.x * blockDim.x + threadIdx.x;
    int p = blockIdx.y;
    if (h >= g.Vh) return;
    int x[4];
    site_coords(g, p, h, x);
    bool mirror = g.cstar >= 1 && x[1] >= L1phys;
    int x1 = mirror ? x[1] - L1phys : x[1];
    long long phys = (((long long)x[0] * L1phys + x1) * L2 + x[2]) * L3 + x[3];
    const size_t Vh = g.Vh;
    for (int mu = 0; mu < 4; ++mu) {
        // open time boundary: the time link leaving x0 = N0 - 1 would cross it; held
        // as zero, so that no hop and no clover leaf uses it
        const bool cut = g.open0 && mu == 0 && x[0] == g.N[0] - 1;
        double2 u[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            u[k] = cut ? make_double2(0.0, 0.0) : Uin[(phys * 4 + mu) * 9 + k];
            if (mirror) u[k].y = -u[k].y;  // U(x + L1 e1) = U(x)^*
            U64[(size_t)p * 36 * Vh + (size_t)(mu * 9 + k) * Vh + h] = u[k];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
            U32[(size_t)p * 12 * Vh + (size_t)(mu * 3 + c) * Vh + h] =
                make_float4((float)u[2 * c].x, (float)u[2 * c].y, (float)u[2 * c + 1].x, (float)u[2 * c + 1].y);
        double a = Ain[phys * 4 + mu];
        A64[(size_t)p * 4 * Vh + (size_t)mu * Vh + h] = mirror ? -a : a;  // A(x + L1 e1) = -A(x)
    }
}

int launch_set_links(qxd_ctx* ctx, const double2* U, const double* A, cudaStream_t st) {
    const Geo& g = ctx->g;
    dim3 grid(nblocks(g.Vh), 2);
    ProfScope prof(ctx, "set_links", (double)g.V * 4 * (144 + 8 + 144 + 8 + 48), st);
    k_set_links<<<grid, kThreads, 0, st>>>(g, ctx->geom.L[1], ctx->geom.L[2], ctx->geom.L[3], U, A, ctx->U64,
                                           ctx->A64, ctx->U32);
    QXD_CUDA(ctx, cudaGetLastError());
    return QXD_OK;
}

// ------------------------------------------------------------------------------
// Hopping phases z(x,mu)^qhat exp(i theta_mu [x crosses the boundary forward]).
// The fermion phase of eq. periodic-bc-quark sits on the link leaving x at
// x_mu = N_mu - 1; the backward hop reads the same link daggered and so picks
// up exp(-i theta_mu).  C* directions carry no phase (theta = 0 there).
__global__ void k_phases(Geo g, int qhat, double th0, double th1, double th2, double th3,
                         const double2* __restrict__ U64, const double* __restrict__ A64,
                         double2* __restrict__ V64, float4* __restrict__ Z32) {
    int h = blockIdx.x * blockDim.x + threadIdx.x;
    int p = blockIdx.y;
    if (h >= g.Vh) return;
    int x[4];
    site_coords(g, p, h, x);
    const double th[4] = {th0, th1, th2, th3};
    const size_t Vh = g.Vh;
    double2 z[4];
    for (int mu = 0; mu < 4; ++mu) {
        double ang = (double)qhat * A64[(size_t)p * 4 * Vh + (size_t)mu * Vh + h];
        bool phase_dir = !(g.cstar >= 1 && mu >= 1 && mu <= g.cstar);
        if (phase_dir && x[mu] == g.N[mu] - 1) ang += th[mu];
        double s, c;
        sincos(ang, &s, &c);
        z[mu] = make_double2(c, s);
        for (int k = 0; k < 9; ++k) {
            double2 u = U64[(size_t)p * 36 * Vh + (size_t)(mu * 9 + k) * Vh + h];
            V64[(size_t)p * 36 * Vh + (size_t)(mu * 9 + k) * Vh + h] =
                make_double2(u.x * c - u.y * s, u.x * s + u.y * c);
        }
    }
    Z32[(size_t)p * 2 * Vh + h] = make_float4((float)z[0].x, (float)z[0].y, (float)z[1].x, (float)z[1].y);
    Z32[(size_t)p * 2 * Vh + Vh + h] = make_float4((float)z[2].x, (float)z[2].y, (float)z[3].x, (float)z[3].y);
}

// ------------------------------------------------------------------------------
// Site-diagonal term.  For each plane mu < nu:
//   Fhat = (Q - Q^+)/8, Q = sum of the four clover leaves at x;
//   G_{mu nu} = su3csw Fhat_{mu nu} + u1csw qhat (i/4) Im{sum of the four U(1)
//               plaquettes} 1   (q Ahat = qhat (i/4) Im{...}, qel cancels).
// In the chiral basis sum_{mu,nu} (i/4) sigma_{mu nu} (x) G_{mu nu} is block diagonal:
//   block(+-) = (i/2) [[E3, E1 - i E2], [E1 + i E2, -E3]],
//   E+_l = G_{0l} - B_l,  E-_l = -G_{0l} - B_l,  B_1 = G_23, B_2 = -G_13, B_3 = G_12.
// Each block gets 1/(2 kappa) on the diagonal and is inverted by Gauss-Jordan
// elimination with partial pivoting.

//
// Two kernels.  k_leaves forms each plaquette's four clover leaves once, from two shared
// two-link products A = U_mu(x) U_nu(x+mu), B = U_nu(x) U_mu(x+nu):
//   at x:        A B^+                     at x+mu+nu:  B^+ A
//   at x+mu:     U_nu(x+mu) (B^+ U_mu(x))  at x+nu:     (U_nu(x)^+ A) U_mu(x+nu)^+
// (8 colour products per plaquette instead of 12) and stores their anti-Hermitian parts
// X - X^+ (9 reals each) and sin of the U(1) plaquette angle.  k_clover gathers the four
// leaves that belong to a site.  With C* boundaries only the physical half is formed: on
// the mirror half U -> U^* and A -> -A, hence G -> G^*, and a block m goes over into
// s2 m^* s2 (s2 the second Pauli matrix on the block's spin index), its inverse alike.
//
// FP64-pipe bound (about 7,600 FP64 instructions per physical site, 1.7 ms at the measured
// FMA rate for the lattice below).  One thread per site with all 24 leaves, and a
// Gauss-Jordan elimination on [m | 1] in local memory, took 7.14 ms on 32 x 32 x 16 x 16
// with C* (V = 262,144); here 2.05 ms.
// The leaves of a slab of x0 slices (and the slice before it) are held at a time, so that
// the workspace stays near 512 MB on any lattice.

// what a leaf slab covers: x0 = base + slot (mod N0), slot in [0, slots)
struct LeafSlab {
    int base, slots;
    int L1;        // x1 extent that is stored (the physical one with C*)
    int slice;     // stored sites of one x0
    double* t;     // [plane 6][37][slots * slice]: 4 leaves x 9 reals, then the sine
};

constexpr int kLeafReals = 37;

QXD_HD void plane_dirs(int plane, int& mu, int& nu) {  // (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)
    mu = plane < 3 ? 0 : plane < 5 ? 1 : 2;
    nu = plane < 3 ? plane + 1 : plane < 5 ? plane - 1 : 3;
}

// X - X^+ : imaginary parts of the diagonal, then entries (0,1), (0,2), (1,2) as (re, im)
QXD_HD void store_antiherm(const M3& X, double* __restrict__ t, size_t stride) {
#pragma unroll
    for (int i = 0; i < 3; ++i) t[i * stride] = 2.0 * X.a[4 * i].im;
    int o = 3;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i + 1; j < 3; ++j) {
            const C64 u = X.a[3 * i + j], l = X.a[3 * j + i];
            t[o * stride] = u.re - l.re;
            t[(o + 1) * stride] = u.im + l.im;
            o += 2;
        }
}

__global__ void __launch_bounds__(128) k_leaves(Geo g, LeafSlab sl, const double2* __restrict__ U64,
                                                const double* __restrict__ A64) {
    const int n = sl.slots * sl.slice;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int x[4], mu, nu;
    plane_dirs(blockIdx.y, mu, nu);
    int r = i;
    x[3] = r % g.N[3];
    r /= g.N[3];
    x[2] = r % g.N[2];
    r /= g.N[2];
    x[1] = r % sl.L1;
    x[0] = (sl.base + r / sl.L1) % g.N[0];
    int xm[4], xn[4];
    step(g, x, mu, +1, xm);
    step(g, x, nu, +1, xn);
    const M3 U1 = link_at(g, U64, x, mu), U2 = link_at(g, U64, xm, nu);
    const M3 U3 = link_at(g, U64, xn, mu), U4 = link_at(g, U64, x, nu);
    const M3 A = m3_mul<false, false>(U1, U2), B = m3_mul<false, false>(U4, U3);
    double* t = sl.t + (size_t)blockIdx.y * kLeafReals * n + i;
    store_antiherm(m3_mul<false, true>(A, B), t, n);
    store_antiherm(m3_mul<false, false>(U2, m3_mul<true, false>(B, U1)), t + (size_t)9 * n, n);
    store_antiherm(m3_mul<true, false>(B, A), t + (size_t)18 * n, n);
    store_antiherm(m3_mul<false, true>(m3_mul<true, false>(U4, A), U3), t + (size_t)27 * n, n);
    // open time boundary: a plaquette of a time plane with corner x0 = N0 - 1 is absent (its
    // SU(3) leaves vanish with the time links held as zero)
    const bool cut = g.open0 && mu == 0 && x[0] == g.N[0] - 1;
    t[(size_t)36 * n] = cut ? 0.0 : sin(A_at(g, A64, x, mu) + A_at(g, A64, xm, nu) - A_at(g, A64, xn, mu) - A_at(g, A64, x, nu));
}

// invert a complex 6x6 matrix in place by Gauss-Jordan elimination with partial (row)
// pivoting, in registers (all loops unrolled, swaps by selection); false if singular
__device__ __forceinline__ bool invert6(C64 m[6][6]) {
    int piv[6];
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        int pc = c;
        double best = norm2(m[c][c]);
#pragma unroll
        for (int r = c + 1; r < 6; ++r) {
            const double v = norm2(m[r][c]);
            if (v > best) {
                best = v;
                pc = r;
            }
        }
        ok = ok && best > 1e-280 && isfinite(best);
        piv[c] = pc;
#pragma unroll
        for (int r = c + 1; r < 6; ++r)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const C64 a = m[c][k], b = m[r][k];
                m[c][k] = pc == r ? b : a;
                m[r][k] = pc == r ? a : b;
            }
        const double s = 1.0 / norm2(m[c][c]);
        const C64 d = {m[c][c].re * s, -m[c][c].im * s};
        m[c][c] = {1.0, 0.0};
#pragma unroll
        for (int k = 0; k < 6; ++k) m[c][k] = m[c][k] * d;
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            if (r == c) continue;
            const C64 f = m[r][c];
            m[r][c] = {0.0, 0.0};
#pragma unroll
            for (int k = 0; k < 6; ++k) cmac(m[r][k], -f, m[c][k]);
        }
    }
#pragma unroll
    for (int c = 5; c >= 0; --c)
#pragma unroll
        for (int r = c + 1; r < 6; ++r)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const C64 a = m[k][c], b = m[k][r];
                m[k][c] = piv[c] == r ? b : a;
                m[k][r] = piv[c] == r ? a : b;
            }
    return ok;
}

__device__ __forceinline__ void store_packed(const double pk[36], int blk, int p, int h, size_t Vh,
                                             double2* __restrict__ D64, float4* __restrict__ D32) {
#pragma unroll
    for (int k = 0; k < 18; ++k)
        D64[(size_t)p * 36 * Vh + (size_t)(blk * 18 + k) * Vh + h] = make_double2(pk[2 * k], pk[2 * k + 1]);
#pragma unroll
    for (int k = 0; k < 9; ++k)
        D32[(size_t)p * 18 * Vh + (size_t)(blk * 9 + k) * Vh + h] =
            make_float4((float)pk[4 * k], (float)pk[4 * k + 1], (float)pk[4 * k + 2], (float)pk[4 * k + 3]);
}

// the packed block s2 m^* s2 of the mirror site: [[a, b], [b^+, d]] -> [[d^*, -(b^+)^*], [.., a^*]]
__device__ __forceinline__ void mirror_packed(const double pk[36], double q[36]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        q[i] = pk[3 + i];
        q[3 + i] = pk[i];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (i < j) {
                const int a = 6 + 2 * herm_off(i, j), d = 6 + 2 * herm_off(3 + i, 3 + j);
                q[a] = pk[d];
                q[a + 1] = -pk[d + 1];
                q[d] = pk[a];
                q[d + 1] = -pk[a + 1];
            }
            // new upper right block: -(b^+)^*_{ij} = -b_{ji}
            const int o = 6 + 2 * herm_off(i, 3 + j), w = 6 + 2 * herm_off(j, 3 + i);
            q[o] = -pk[w];
            q[o + 1] = -pk[w + 1];
        }
}

// site-diagonal block of chirality blockIdx.y and its inverse for the sites x0 in [x0a, x0a + nx0)
__global__ void __launch_bounds__(64) k_clover(Geo g, LeafSlab sl, int x0a, int nx0, int qhat, double kappa,
                                               double su3csw, double u1csw, double cF, double2* __restrict__ A_64,
                                               float4* __restrict__ A_32, double2* __restrict__ Ai_64,
                                               float4* __restrict__ Ai_32, int* __restrict__ flag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nx0 * sl.slice) return;
    const int chi = blockIdx.y;
    int x[4];
    int r = i;
    x[3] = r % g.N[3];
    r /= g.N[3];
    x[2] = r % g.N[2];
    r /= g.N[2];
    x[1] = r % sl.L1;
    x[0] = x0a + r / sl.L1;
    const int n = sl.slots * sl.slice;
    // E_l = +-G_{0l} - B_l (B_1 = G_23, B_2 = -G_13, B_3 = G_12), anti-Hermitian, 9 reals
    double E[3][9];
#pragma unroll
    for (int plane = 0; plane < 6; ++plane) {
        int mu, nu;
        plane_dirs(plane, mu, nu);
        const int l = plane < 3 ? plane : 5 - plane;
        const double sgn = plane < 3 ? (chi == 0 ? 1.0 : -1.0) : (plane == 4 ? 1.0 : -1.0);
        double F[9], im = 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) F[k] = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {  // lower corners x, x - mu, x - mu - nu, x - nu
            int y[4] = {x[0], x[1], x[2], x[3]}, z[4];
            if (c == 1 || c == 2) {
                step(g, y, mu, -1, z);
                for (int d = 0; d < 4; ++d) y[d] = z[d];
            }
            if (c >= 2) {
                step(g, y, nu, -1, z);
                for (int d = 0; d < 4; ++d) y[d] = z[d];
            }
            const bool mirror = y[1] >= sl.L1;  // its fields are the conjugates of the physical site's
            const double cj = mirror ? -1.0 : 1.0;
            int slot = y[0] - sl.base;
            if (slot < 0) slot += g.N[0];
            const int site = ((slot * sl.L1 + (mirror ? y[1] - sl.L1 : y[1])) * g.N[2] + y[2]) * g.N[3] + y[3];
            const double* t = sl.t + (size_t)plane * kLeafReals * n + site;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const double v = QXD_LDG(t + (size_t)(9 * c + k) * n);
                const bool imag = k < 3 || (k & 1) == 0;  // 3: re, 4: im, ...
                F[k] += imag ? cj * v : v;
            }
            im += cj * QXD_LDG(t + (size_t)36 * n);
        }
        const double u1 = u1csw * (double)qhat * 0.25 * im;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double G = (su3csw / 8.0) * F[k] + (k < 3 ? u1 : 0.0);
            E[l][k] = plane < 3 ? sgn * G : E[l][k] + sgn * G;
        }
    }
    // (i/2) [[E3, E1 - i E2], [E1 + i E2, -E3]] + m0; i E of an anti-Hermitian E is Hermitian:
    // diagonal -a, upper entries (-im, re)
    const double m0 = 0.5 / kappa + ((g.open0 && (x[0] == 0 || x[0] == g.N[0] - 1)) ? cF - 1.0 : 0.0);
    double pk[36];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        pk[a] = m0 - 0.5 * E[2][a];
        pk[3 + a] = m0 + 0.5 * E[2][a];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            // entry (a, b) of E1, E2 as complex numbers
            C64 e[2];
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                if (a == b) e[l] = {0.0, E[l][a]};
                else {
                    const int lo = a < b ? a : b, hi = a < b ? b : a;
                    const int o = 3 + 2 * (lo + hi - 1);
                    e[l] = {a < b ? E[l][o] : -E[l][o], E[l][o + 1]};
                }
            }
            const int o = 6 + 2 * herm_off(a, 3 + b);
            pk[o] = 0.5 * (e[1].re - e[0].im);
            pk[o + 1] = 0.5 * (e[0].re + e[1].im);
            if (a < b) {
                const int q = 3 + 2 * (a + b - 1);
                const int u = 6 + 2 * herm_off(a, b), d = 6 + 2 * herm_off(3 + a, 3 + b);
                pk[u] = -0.5 * E[2][q + 1];
                pk[u + 1] = 0.5 * E[2][q];
                pk[d] = 0.5 * E[2][q + 1];
                pk[d + 1] = -0.5 * E[2][q];
            }
        }
    }
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const int h = lex_index(g, x) >> 1;
    const bool twin = sl.L1 != g.N[1];
    int pm = 0, hm = 0;
    if (twin) {
        const int xm[4] = {x[0], x[1] + sl.L1, x[2], x[3]};
        pm = (p + sl.L1) & 1;
        hm = lex_index(g, xm) >> 1;
    }
    store_packed(pk, chi, p, h, g.Vh, A_64, A_32);
    double q[36];
    if (twin) {
        mirror_packed(pk, q);
        store_packed(q, chi, pm, hm, g.Vh, A_64, A_32);
    }
    C64 m[6][6];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        m[a][a] = {pk[a], 0.0};
#pragma unroll
        for (int b = a + 1; b < 6; ++b) {
            const int o = 6 + 2 * herm_off(a, b);
            m[a][b] = {pk[o], pk[o + 1]};
            m[b][a] = {pk[o], -pk[o + 1]};
        }
    }
    const bool ok = invert6(m);
    if (!ok) atomicExch(flag, 1);
    // average the two triangles (Hermitian up to rounding)
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        pk[a] = ok ? m[a][a].re : 0.0;
#pragma unroll
        for (int b = a + 1; b < 6; ++b) {
            const int o = 6 + 2 * herm_off(a, b);
            pk[o] = ok ? 0.5 * (m[a][b].re + m[b][a].re) : 0.0;
            pk[o + 1] = ok ? 0.5 * (m[a][b].im - m[b][a].im) : 0.0;
        }
    }
    store_packed(pk, chi, p, h, g.Vh, Ai_64, Ai_32);
    if (twin) {
        mirror_packed(pk, q);
        store_packed(q, chi, pm, hm, g.Vh, Ai_64, Ai_32);
    }
}

static int launch_clover(qxd_ctx* ctx, int fl, cudaStream_t st) {
    const Geo& g = ctx->g;
    const QxdFlavour& F = ctx->fl[fl];
    LeafSlab sl{};
    sl.L1 = g.cstar ? g.L1 : g.N[1];
    sl.slice = sl.L1 * g.N[2] * g.N[3];
    const size_t per = 6ull * kLeafReals * sizeof(double) * sl.slice;
    const int N0 = g.N[0];
    int S = (int)std::min<size_t>(N0, (512ull << 20) / per);  // slices of a slab
    if (S < N0) S = std::max(S - 1, 1);                       // room for the slice before it
    bool whole = false;
    void* t = nullptr;
    for (;; S = (S + 1) / 2) {  // smaller slabs where there is no memory for them
        whole = S + 1 >= N0;
        sl.slots = whole ? N0 : S + 1;
        const int rc = qxd_ws(ctx, WS_CLOVER, per * sl.slots, &t);
        if (rc == QXD_OK) break;
        if (S == 1) return rc;
    }
    sl.t = static_cast<double*>(t);
    ProfScope prof(ctx, "set_clover", (double)g.V * (4 * 144 + 4 * 8 + 2 * (576 + 288)), st);
    for (int a = 0; a < N0; a += whole ? N0 : S) {
        const int nx0 = whole ? N0 : std::min(S, N0 - a);
        sl.base = whole ? 0 : (a + N0 - 1) % N0;
        k_leaves<<<dim3(nblocks((long long)sl.slots * sl.slice), 6), kThreads, 0, st>>>(g, sl, ctx->U64, ctx->A64);
        QXD_CUDA(ctx, cudaGetLastError());
        k_clover<<<dim3(nblocks((long long)nx0 * sl.slice, 64), 2), 64, 0, st>>>(
            g, sl, a, nx0, F.f.qhat, F.f.kappa, F.f.su3csw, F.f.u1csw, ctx->geom.cF, F.C64[0], F.C32[0], F.C64[1],
            F.C32[1], ctx->dev_flag);
        QXD_CUDA(ctx, cudaGetLastError());
    }
    return QXD_OK;
}

int launch_set_flavour(qxd_ctx* ctx, int fl, cudaStream_t st) {
    const Geo& g = ctx->g;
    QxdFlavour& F = ctx->fl[fl];
    dim3 grid(nblocks(g.Vh), 2);
    const double* th = ctx->geom.theta;
    {
    ProfScope prof(ctx, "set_phases", (double)g.V * 4 * (144 + 8 + 144 + 8), st);
    k_phases<<<grid, kThreads, 0, st>>>(g, F.f.qhat, th[0], th[1], th[2], th[3], ctx->U64, ctx->A64, F.V64, F.Z32);
    }
    QXD_CUDA(ctx, cudaGetLastError());
    QXD_CUDA(ctx, cudaMemsetAsync(ctx->dev_flag, 0, sizeof(int), st));
    QXD_TRY(launch_clover(ctx, fl, st));
    int flag = 0;
    QXD_CUDA(ctx, cudaMemcpyAsync(&flag, ctx->dev_flag, sizeof(int), cudaMemcpyDeviceToHost, st));
    QXD_CUDA(ctx, cudaStreamSynchronize(st));
    if (flag) return qxd_fail(ctx, QXD_ENAN, "set_clover: singular site-diagonal block");
    return QXD_OK;
}

// Double-float copies of the FP64 links and of the site-diagonal term (and, when
// an operator needs it, of its inverse), built on the first double-float
// application of the flavour: each is as large as its FP64 original, so they
// exist only where the mixed solvers or QXD_DF64 are used.
int ensure_df64(qxd_ctx* ctx, int fl, cudaStream_t st, bool inverse) {
    QxdFlavour& F = ctx->fl[fl];
    const size_t n = 2ull * 36 * ctx->g.Vh;
    float4** made[3] = {nullptr, nullptr, nullptr};  // copies allocated by this call
    int nmade = 0;
    auto build = [&](float4** dst, const double2* src) -> int {
        if (*dst) return QXD_OK;
        if (!dev_alloc(ctx, reinterpret_cast<void**>(dst), n * sizeof(float4))) {
            // leave no partial set behind: a caller may go on without the copies
            for (int i = 0; i < nmade; ++i) {
                cudaFree(*made[i]);
                *made[i] = nullptr;
            }
            return qxd_fail(ctx, QXD_ENOMEM, "double-float copy of the links or site-diagonal terms: allocation failed");
        }
        made[nmade++] = dst;
        return blas_split_df64(ctx, src, *dst, n, st);
    };
    QXD_TRY(build(&F.Vdf, F.V64));
    QXD_TRY(build(&F.Cdf[0], F.C64[0]));
    if (inverse) QXD_TRY(build(&F.Cdf[1], F.C64[1]));
    return QXD_OK;
}

}  // namespace qxd
