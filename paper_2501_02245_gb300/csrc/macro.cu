// Macroscopic synthetic solve (Eq. macro with the constitutive relations of
// Eq. full_constitutive and Eq. NSF_constitutive), monatomic gas, on ALL cells.
//
// Flux and relaxation choices (the paper defers them to another work; the
// same choices are made in the CPU reference):
//  * inviscid: kinetic flux-vector splitting (the Euler flux the
//    discrete-velocity upwind scheme carries for Maxwellian states, in closed
//    form) on index-space MUSCL-minmod states of (rho, u, p), first order
//    next to boundaries;
//  * viscous: NSF from the mean of the two cells' least-squares gradients
//    corrected along the line of centres, at the mean cell u and T, plus the
//    mean of the two cells' HoT;
//  * far field: the same splitting against the boundary state plus the
//    cell's HoT;
//    wall: cell pressure, no mass flux, NSF at u = 0 and T = T_w from a
//    one-sided gradient; at the wall of a DVM cell plus the frozen difference
//    between the kinetic wall flux of f^{n+1/2} and that NSF wall flux at
//    W^{n+1/2};
//  * DP-LUR pseudo-time relaxation (Wright, Candler & Bose 1998): scalar
//    diagonal (1/CFL + 1/2) sum lambda |S| (+ V/dt with the time term of
//    Eq. macro), k_sub Jacobi sweeps over Rusanov-split Euler flux changes.
// Every interior face flux is evaluated once, by one thread (face kernel),
// and gathered by both cells in a fixed order (cell kernel), so the scheme is
// exactly conservative and deterministic.
#include <algorithm>
#include <cooperative_groups.h>
#include "special.cuh"

namespace cg = cooperative_groups;

namespace gsis {


static MacroArgs margs(gsis_ctx* c) {
    MacroArgs a;
    a.N = c->m.N;
    a.nbr = c->m.nbr;
    a.side_bc = c->m.side_bc;
    a.Sout = c->m.Sout;
    a.xf = c->m.xf;
    a.cen = c->m.cen;
    a.vol = c->m.vol;
    a.lsq_w = c->m.lsq_w;
    a.bc_state = c->d_bc_state;
    a.fgeo = c->fgeo;
    a.bgeo = c->bgeo;
    a.fst = c->fst;
    a.bside = c->m.bside;
    a.nbside = c->m.nbside;
    a.nd = c->normal_components;
    a.fnd = c->face_nd;
    a.mu0 = c->mu0;
    a.omega = c->p.omega;
    return a;
}

// A flat line of cells (fnd = 1) is solved with the library's functions and divisions,
// meshes of two and three directions with the tables of special.cuh and recip64.  At
// the shocks' settings (cfl = 100, four relaxation sweeps) the pseudo-time iteration of a
// line above Mach 2 or so amplifies a difference in the last bit (1e-15 of the initial
// state becomes 6e-7 in two GSIS iterations at Mach 5, 1e-4 in ten), so any other rounding
// of these operations gives another trajectory; twelve sweeps, or cfl = 10, damp it.
// The bodies' settings do not amplify.  (LINE below: fnd = 1.  50 pseudo-steps of 200
// cells take 1.60 ms, 1.48 with the tables.)
template <bool LINE>
__device__ __forceinline__ double mu_of(double T, double mu0, double omega) {
    return LINE ? viscosity(T, mu0, omega) : mu0 * exp_tab(omega * log_tab(T));
}
__device__ __forceinline__ double mu_of(const MacroArgs& a, double T) {
    return a.fnd == 1 ? mu_of<true>(T, a.mu0, a.omega) : mu_of<false>(T, a.mu0, a.omega);
}
template <bool LINE>
__device__ __forceinline__ double quotient(double a, double b) { return LINE ? a / b : __dmul_rn(a, recip64(b)); }

// ---------------------------------------------------------------------------- gradients
// Least-squares gradient (face neighbours plus boundary face centres with the
// boundary value: far field -> boundary state; wall -> u = 0, |u| = 0, T = T_w,
// rho = cell value).  gu[(3 j + i) N + c] = d u_j / d x_i, gT[i N + c].  ND:
// the LSQ weights have components 0..ND-1 only (MacroArgs::fnd) and the sides
// of the other directions carry nothing; their entries are written as zero.
// The neighbours' values are all loaded before any of them is used (a missing
// neighbour repeats the cell: its difference is zero), so that a thread waits
// for memory twice (indices, values) instead of twice per side.
template <int ND, bool RHO_U>
__device__ __forceinline__ void gradients_nd(const MacroArgs& a, const double* Wp, double* gu, double* gT,
                                             double* grho, double* gU, double* acell, int c) {
    constexpr int NS = 2 * ND, NQ = RHO_U ? 6 : 4;
    const int N = a.N;
    int n[NS];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const int2 v = *reinterpret_cast<const int2*>(a.nbr + c * 6 + 2 * d);
        n[2 * d] = v.x;
        n[2 * d + 1] = v.y;
    }
    double val[NS][6], w[NS][ND], phic[6];   // ux, uy, uz, T, rho, U
    auto state = [](const double* p, double* o) {
        o[0] = p[1]; o[1] = p[2]; o[2] = p[3]; o[3] = p[4];
        if (RHO_U) {
            o[4] = p[0];
            o[5] = sqrt(p[1] * p[1] + p[2] * p[2] + p[3] * p[3]);
        }
    };
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        state(Wp + (n[s] >= 0 ? n[s] : c) * 5, val[s]);
#pragma unroll
        for (int i = 0; i < ND; ++i) w[s][i] = a.lsq_w[((long long)c * 6 + s) * 3 + i];
    }
    state(Wp + c * 5, phic);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        if (n[s] >= 0) continue;
        const int bc = a.side_bc[c * 6 + s];
        const double* st = a.bc_state + s * 5;
        if (bc == GSIS_BC_FARFIELD) {
            state(st, val[s]);
        } else if (bc == GSIS_BC_WALL) {
            val[s][0] = 0.0; val[s][1] = 0.0; val[s][2] = 0.0; val[s][3] = st[4];
            if (RHO_U) val[s][5] = 0.0;   // (rho keeps the cell's value)
        }
    }
    if (acell) acell[c] = sqrt(GAMMA * phic[3]);
    double g[6][3];
    for (int q = 0; q < 6; ++q) g[q][0] = g[q][1] = g[q][2] = 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const double dphi = val[s][q] - phic[q];
#pragma unroll
            for (int i = 0; i < ND; ++i) g[q][i] += w[s][i] * dphi;
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int i = 0; i < 3; ++i) gu[(long long)(j * 3 + i) * N + c] = g[j][i];
#pragma unroll
    for (int i = 0; i < 3; ++i) gT[(long long)i * N + c] = g[3][i];
    if (RHO_U) {
        for (int i = 0; i < 3; ++i) {
            grho[(long long)c * 3 + i] = g[4][i];
            gU[(long long)c * 3 + i] = g[5][i];
        }
    }
}

template <bool RHO_U>
__device__ __forceinline__ void gradients_cell(const MacroArgs& a, const double* Wp, double* gu, double* gT,
                                               double* grho, double* gU, double* acell, int c) {
    switch (a.fnd) {
        case 1: gradients_nd<1, RHO_U>(a, Wp, gu, gT, grho, gU, acell, c); break;
        case 2: gradients_nd<2, RHO_U>(a, Wp, gu, gT, grho, gU, acell, c); break;
        default: gradients_nd<3, RHO_U>(a, Wp, gu, gT, grho, gU, acell, c); break;
    }
}

// The gradients of cell c as the 3 x 3 and 3 arrays of nsf_of.
__device__ __forceinline__ void cell_grad(const double* gu, const double* gT, int N, int c, double* u, double* T) {
#pragma unroll
    for (int i = 0; i < 9; ++i) u[i] = gu[(long long)i * N + c];
#pragma unroll
    for (int i = 0; i < 3; ++i) T[i] = gT[(long long)i * N + c];
}

__global__ void k_gradients(MacroArgs a, const double* __restrict__ Wp, int with_rho_U, double* __restrict__ gu,
                            double* __restrict__ gT, double* __restrict__ grho, double* __restrict__ gU,
                            double* __restrict__ acell) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.N) return;
    if (with_rho_U) gradients_cell<true>(a, Wp, gu, gT, grho, gU, acell, c);
    else gradients_cell<false>(a, Wp, gu, gT, nullptr, nullptr, acell, c);
}

void launch_gradients(gsis_ctx* c, const double* Wprim, bool with_rho_U) {
    const int N = c->m.N;
    k_gradients<<<(N + 63) / 64, 64, 0, c->stream>>>(margs(c), Wprim, with_rho_U ? 1 : 0, c->gu, c->gT, c->grho,
                                                     c->gU, c->acell);
    c->launches++;
}

// ---------------------------------------------------------------------------- NSF
__device__ __forceinline__ void nsf_of(double mu, const double* gu /*[j][i]*/, const double* gT, double* sig,
                                       double* q) {
    // G[i][j] = d u_j / d x_i = gu[j*3 + i]
    const double div = gu[0] + gu[4] + gu[8];
    const double two3 = 2.0 / 3.0;
    sig[0] = -mu * (2.0 * gu[0] - two3 * div);
    sig[1] = -mu * (2.0 * gu[4] - two3 * div);
    sig[2] = -mu * (2.0 * gu[8] - two3 * div);
    sig[3] = -mu * (gu[0 * 3 + 1] + gu[1 * 3 + 0]);   // xy: du_x/dy + du_y/dx
    sig[4] = -mu * (gu[0 * 3 + 2] + gu[2 * 3 + 0]);   // xz
    sig[5] = -mu * (gu[1 * 3 + 2] + gu[2 * 3 + 1]);   // yz
    const double kap = 3.75 * mu;
    q[0] = -kap * gT[0];
    q[1] = -kap * gT[1];
    q[2] = -kap * gT[2];
}

__global__ void k_nsf(int N, const double* __restrict__ Wp, const double* __restrict__ gu,
                      const double* __restrict__ gT, double mu0, double omega, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const double mu = viscosity(Wp[c * 5 + 4], mu0, omega);
    double u[9], t[3];
    cell_grad(gu, gT, N, c, u, t);
    nsf_of(mu, u, t, out + (long long)c * HOTN, out + (long long)c * HOTN + 6);
}

void launch_nsf(gsis_ctx* c, const double* Wprim, double* out) {
    launch_gradients(c, Wprim, false);
    const int N = c->m.N;
    k_nsf<<<(N + 127) / 128, 128, 0, c->stream>>>(N, Wprim, c->gu, c->gT, c->mu0, c->p.omega, out);
    c->launches++;
}

// ---------------------------------------------------------------------------- conversions
__global__ void k_prim_to_cons(int N, const double* __restrict__ Wp, double* __restrict__ U) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const double r = Wp[c * 5], ux = Wp[c * 5 + 1], uy = Wp[c * 5 + 2], uz = Wp[c * 5 + 3], T = Wp[c * 5 + 4];
    U[c * 5] = r;
    U[c * 5 + 1] = r * ux;
    U[c * 5 + 2] = r * uy;
    U[c * 5 + 3] = r * uz;
    U[c * 5 + 4] = r * (1.5 * T + 0.5 * (ux * ux + uy * uy + uz * uz));
}

// (One reciprocal per state, reused: on GB300 an FP64 division costs about ten
// FP64-pipe operations.)
__device__ __forceinline__ void cons_to_prim(const double* U, double* Wp) {
    const double r = U[0], ir = 1.0 / r;
    const double ux = __dmul_rn(U[1], ir), uy = __dmul_rn(U[2], ir), uz = __dmul_rn(U[3], ir);
    Wp[0] = r;
    Wp[1] = ux;
    Wp[2] = uy;
    Wp[3] = uz;
    Wp[4] = fma(2.0 * U[4], ir, -fma(uz, uz, fma(ux, ux, __dmul_rn(uy, uy)))) * (1.0 / 3.0);
}

__global__ void k_cons_to_prim(int N, const double* __restrict__ U, double* __restrict__ Wp) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    cons_to_prim(U + c * 5, Wp + c * 5);
}

// Face geometry of the synthetic solve, computed once per mesh: for the high
// face of each direction |S|, n = S/|S|, the unit vector e between the cell
// centres, their distance and its reciprocal, S, and the cells of the face's
// stencil (MacroArgs::fst); for every side |S|, n and the unit vector from
// the cell centre to the face centre and its length.
__global__ void k_face_geometry(MacroArgs a, double* __restrict__ fgeo, double* __restrict__ bgeo,
                                int4* __restrict__ fst) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.N) return;
    for (int s = 0; s < 6; ++s) {
        const double* So = a.Sout + ((long long)c * 6 + s) * 3;
        const double Sabs = sqrt(So[0] * So[0] + So[1] * So[1] + So[2] * So[2]);
        double eb[3];
        for (int i = 0; i < 3; ++i) eb[i] = a.xf[((long long)c * 6 + s) * 3 + i] - a.cen[c * 3 + i];
        const double bd = sqrt(eb[0] * eb[0] + eb[1] * eb[1] + eb[2] * eb[2]);
        double* B = bgeo + ((long long)c * 6 + s) * 8;
        B[0] = Sabs;
        for (int i = 0; i < 3; ++i) B[1 + i] = Sabs > 0.0 ? So[i] / Sabs : 0.0;
        for (int i = 0; i < 3; ++i) B[4 + i] = bd > 0.0 ? eb[i] / bd : 0.0;
        B[7] = bd;
        if (s & 1) {
            const int d = s >> 1;
            const int R = a.nbr[c * 6 + s];
            double* G = fgeo + ((long long)c * 3 + d) * FGEO_N;
            for (int q = 0; q < FGEO_N; ++q) G[q] = 0.0;
            // cells of the face's stencil: below L, L's neighbour R, beyond R
            fst[(long long)c * 3 + d] = make_int4(a.nbr[c * 6 + s - 1], R, R >= 0 ? a.nbr[R * 6 + s] : -1, 0);
            if (R >= 0) {
                double e[3];
                for (int i = 0; i < 3; ++i) e[i] = a.cen[R * 3 + i] - a.cen[c * 3 + i];
                const double dist = sqrt(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);
                G[0] = Sabs;
                for (int i = 0; i < 3; ++i) G[1 + i] = So[i] / Sabs;
                for (int i = 0; i < 3; ++i) G[4 + i] = e[i] / dist;
                G[7] = dist;
                G[8] = 1.0 / dist;
                for (int i = 0; i < 3; ++i) G[9 + i] = So[i];
            }
        }
    }
}

void launch_face_geometry(gsis_ctx* c) {
    const int N = c->m.N;
    k_face_geometry<<<(N + 127) / 128, 128, 0, c->stream>>>(margs(c), c->fgeo, c->bgeo, c->fst);
    c->launches++;
}

// W <- Wh + w (W - Wh): under-relaxed synthetic correction of the primitives.
__global__ void k_blend(int N, const double* __restrict__ Wh, double w, double* __restrict__ W) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * 5) return;
    const double h = Wh[i];
    W[i] = h + w * (W[i] - h);
}

void launch_blend(gsis_ctx* c, const double* Wh, double w, double* W) {
    const int n = c->m.N * 5;
    k_blend<<<(n + 255) / 256, 256, 0, c->stream>>>(c->m.N, Wh, w, W);
    c->launches++;
}

void launch_prim_to_cons(gsis_ctx* c, const double* Wprim, double* Ucons) {
    const int N = c->m.N;
    k_prim_to_cons<<<(N + 127) / 128, 128, 0, c->stream>>>(N, Wprim, Ucons);
    c->launches++;
}

void launch_cons_to_prim(gsis_ctx* c, const double* Ucons, double* Wprim) {
    const int N = c->m.N;
    k_cons_to_prim<<<(N + 127) / 128, 128, 0, c->stream>>>(N, Ucons, Wprim);
    c->launches++;
}

// ---------------------------------------------------------------------------- fluxes
// a . b over the first ND components.  Every sum of products of the pseudo-steps
// below is written out with its fused and its rounded products (fma, __dmul_rn): left
// to the compiler, the choice depends on the code around it, and the one-lane, the two-lane,
// the fused and the per-phase forms of a step would end in different last bits.
template <int ND>
__device__ __forceinline__ double dot_rn(const double* a, const double* b) {
    if (ND == 1) return __dmul_rn(a[0], b[0]);
    double v = fma(a[0], b[0], __dmul_rn(a[1], b[1]));
    if (ND > 2) v = fma(a[2], b[2], v);
    return v;
}

// Flux carried by the molecules of the Maxwellian (r, u, T) that cross a
// face of unit normal n in the direction sign*n (half-range moments of the
// normal Gaussian N(u.n, T); tangential thermal motion in closed form): c[q] X[q]
// with c = r (mass, momentum) and r/2 (energy).
// (ND: the normal has components 0..ND-1 only; the others are exact zeros,
// so the terms they multiply are left out.)
template <int ND, bool LINE>
__device__ __forceinline__ void half_range(const double* u, double T, const double* n, double sign, double* X) {
    const double un = dot_rn<ND>(u, n);
    // s = un / sqrt(T) and sqrt(T) = T / sqrt(T) from one reciprocal square root
    // (instead of a square root and two FP64 divisions).  P is the share of the
    // Maxwellian that crosses, (1 + sign erf(s/sqrt 2))/2, from its tail
    // q = h(|s|) exp(-s^2/2): q where the gas recedes, 1 - q where it approaches.
    const double ist = rsqrt(T), st = T * ist, s = un * ist;
    double e, P;
    if constexpr (LINE) {
        e = exp(-0.5 * s * s);
        P = 0.5 * (1.0 + sign * erf(s * 0.7071067811865476));   // 1/sqrt(2)
    } else {
        e = exp_tab(-0.5 * s * s);
        const double q = __dmul_rn(mills(__longlong_as_double((long long)mag_bits(s))), e);
        const bool towards = (__double2hiint(s) >= 0) == (sign > 0.0);
        P = towards ? 1.0 - q : q;
    }
    const double D = __dmul_rn(sign * st * e, 0.3989422804014327);   // 1/sqrt(2 pi)
    const double M0 = fma(un, P, D);
    const double u2 = __dmul_rn(un, un);
    const double M1 = fma(u2 + T, P, __dmul_rn(un, D));
    const double M2 = fma(fma(u2, un, __dmul_rn(3.0 * un, T)), P, __dmul_rn(u2 + 2.0 * T, D));
    double ut[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) ut[i] = i < ND ? fma(-un, n[i], u[i]) : u[i];
    X[0] = M0;
#pragma unroll
    for (int i = 0; i < 3; ++i) X[1 + i] = i < ND ? fma(M1, n[i], __dmul_rn(ut[i], M0)) : __dmul_rn(ut[i], M0);
    X[4] = fma(fma(ut[2], ut[2], fma(ut[0], ut[0], __dmul_rn(ut[1], ut[1]))) + 2.0 * T, M0, M2);
}

// Kinetic flux-vector splitting per unit area through the unit normal n: the
// left Maxwellian's molecules moving along +n plus the right one's moving
// along -n -- the Euler flux that the discrete-velocity upwind scheme carries
// for Maxwellian states.  The left half is rounded, the right one added with one
// fused multiply-add: written out, so that kfvs_pair rounds the same way.
template <int ND, bool LINE>
__device__ __forceinline__ void kfvs(double rL, const double* uL, double pL, double rR, const double* uR, double pR,
                     const double* n, double* F) {
    double X[5];
    half_range<ND, LINE>(uL, quotient<LINE>(pL, rL), n, 1.0, X);
    for (int q = 0; q < 5; ++q) F[q] = fma(q < 4 ? rL : 0.5 * rL, X[q], 0.0);
    half_range<ND, LINE>(uR, quotient<LINE>(pR, rR), n, -1.0, X);
    for (int q = 0; q < 5; ++q) F[q] = fma(q < 4 ? rR : 0.5 * rR, X[q], F[q]);
}

// The same sum formed by a pair of lanes (2i, 2i + 1), each with its own side's
// state (odd lanes: the right one): the two half-range chains run side by side.
// The even lane gets the flux, the same bits as kfvs.
template <int ND, bool LINE>
__device__ __forceinline__ void kfvs_pair(double r, const double* u, double p, bool right, const double* n, double* F) {
    double X[5];
    half_range<ND, LINE>(u, quotient<LINE>(p, r), n, right ? -1.0 : 1.0, X);
    const unsigned pair = 3u << (threadIdx.x & 30);
    const double ro = __shfl_xor_sync(pair, r, 1);
#pragma unroll
    for (int q = 0; q < 5; ++q)
        F[q] = fma(q < 4 ? ro : 0.5 * ro, __shfl_xor_sync(pair, X[q], 1), fma(q < 4 ? r : 0.5 * r, X[q], 0.0));
}

// Euler flux tensor of conserved state U: F[q * 3 + i] = flux of component q
// along axis i (so that F.S is euler_flux_dot(U, S)), one division.  Only the
// axes i < ND are formed: on a mesh whose face normals have no component
// along the others (ND = normal_components), F.S never reads them.
// sub: the tensor less this one.
template <int ND>
__device__ __forceinline__ void euler_tensor(const double* U, double* F, const double* sub = nullptr) {
    const double r = U[0], ir = quotient<ND == 1>(1.0, r);
    const double u[3] = {__dmul_rn(U[1], ir), __dmul_rn(U[2], ir), __dmul_rn(U[3], ir)};
    const double e = fma(-(0.5 * r), dot_rn<3>(u, u), U[4]);
    const double h = fma(GAMMA - 1.0, e, U[4]);
#pragma unroll
    for (int i = 0; i < ND; ++i) {
        double Fi[4] = {U[1 + i], __dmul_rn(U[1], u[i]), __dmul_rn(U[2], u[i]), __dmul_rn(U[3], u[i])};
        Fi[1 + i] = fma(GAMMA - 1.0, e, Fi[1 + i]);   // + p
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q * 3 + i] = sub ? Fi[q] - sub[q * 3 + i] : Fi[q];
        F[12 + i] = sub ? fma(h, u[i], -sub[12 + i]) : __dmul_rn(h, u[i]);
    }
}

// Change of the Euler flux tensor of a cell for the relaxation increment
// dU, F(U + dU) - F(U), with F(U) kept in F0 for the pseudo-step: each
// neighbour then reads the values instead of evaluating both fluxes (and their
// divisions) itself.  Arrays of the synthetic solve that neighbours or later
// phases read are component-major ([component][N]): a warp's load of one
// component touches two or three lines instead of one per lane.
template <int ND>
__device__ __forceinline__ void flux_change(const double* U, const double* dU, const double* F0, double* dF, int N,
                                            int c) {
    double Up[5], F1[15];
#pragma unroll
    for (int q = 0; q < 5; ++q) Up[q] = U[q] + dU[q];
    euler_tensor<ND>(Up, F1, F0);
#pragma unroll
    for (int q = 0; q < 5; ++q)
#pragma unroll
        for (int i = 0; i < ND; ++i) dF[(long long)(q * 3 + i) * N + c] = F1[q * 3 + i];
}

__device__ __forceinline__ void prim5(const double* w, double* q) {   // (rho, u, p)
    q[0] = w[0]; q[1] = w[1]; q[2] = w[2]; q[3] = w[3]; q[4] = __dmul_rn(w[0], w[4]);
}

// Face state of a cell (rho, u, p: q, its primitives w) towards its neighbour on the
// other side of the face, to which df are the differences: q +- half the minmod of
// df and the difference to the cell beyond (wo; none: no such cell, zero slope).
__device__ __forceinline__ void face_state(const double* q, const double* w, const double* wo, bool right, bool none,
                                           const double* df, double* f) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const double d = k < 4 ? (right ? wo[k] - q[k] : q[k] - wo[k])
                               : (right ? fma(wo[0], wo[4], -q[4]) : fma(-wo[0], wo[4], q[4]));
        const double h = none ? 0.0 : hmm_t<double>(df[k], d), m = right ? -h : h;
        f[k] = k < 4 ? q[k] + m : fma(w[0], w[4], m);
    }
}

// Interior face between L = cell c and R = its neighbour across side 2d+1
// (area vector S pointing L -> R).  Writes the total face flux (inviscid +
// viscous + HoT) F.S to Ff[(5 d + q) N + c] and lambda |S| to lamf[d N + c];
// faces that do not exist (boundary) get lamf = -1.
// ND: on a mesh whose face normals, cell-to-cell vectors and LSQ weights have
// components 0..ND-1 only (MacroArgs::fnd), the gradient entries along the
// other directions are exact zeros and are not formed or multiplied: the same
// values as the 3D expressions.  (Every velocity component keeps its gradient:
// the out-of-plane velocity of a 2D flow is zero only up to rounding -- and up
// to the storage noise of BF16/FP16 VDFs -- and its viscous stress is what
// damps it.)
// What bounds it: FP64 instructions (a warp's holds the pipe of its SM
// sub-partition for 64 cycles), so reciprocals that depend on the mesh are
// stored, the others come from recip64, and the limiter runs on the integer pipe.
// PAIR: a pair of lanes takes the face (kfvs_pair), each with one side's face state;
// the rest is formed by both and stored by the even one.  The same values.  For
// solves that leave sub-partitions idle: 200 cells 1.72 -> 1.60 ms per block of
// pseudo-steps, 30 cells 0.85 -> 0.75.
template <int ND, bool PAIR>
__device__ __forceinline__ void face_flux_nd(const MacroArgs& a, const double* Wm, const double* gu,
                                             const double* gT, const double* hot, const double* acell,
                                             double* Ff, double* lamf, int t) {
    constexpr bool LINE = ND == 1;
    const int N = a.N, d = t / N, L = t - d * N;
    const int4 st = a.fst[(long long)L * 3 + d];
    const int Rr = st.y;
    if (Rr < 0) {
        lamf[(long long)d * N + L] = -1.0;
        return;
    }
    const double* G = a.fgeo + ((long long)L * 3 + d) * FGEO_N;
    const double Sabs = G[0];
    const double nn[3] = {G[1], G[2], G[3]}, S[3] = {G[9], G[10], G[11]};
    // MUSCL face states: q -/+ 0.5 minmod of the one-sided differences (the
    // halved limiter on the integer pipe), first order where the second
    // neighbour is missing (the cell itself is read in its place)
    const bool right = PAIR && (threadIdx.x & 1);
    double wL[5], wR[5], qL[5], qR[5], Fv[5];
    const double *pl = Wm + (st.x >= 0 ? st.x : L) * 5, *ph = Wm + (st.z >= 0 ? st.z : Rr) * 5;
    {
        const double *pL = Wm + L * 5, *pR = Wm + Rr * 5;
#pragma unroll
        for (int q = 0; q < 5; ++q) { wL[q] = pL[q]; wR[q] = pR[q]; }
    }
    double df[5];
    prim5(wL, qL);
    prim5(wR, qR);
#pragma unroll
    for (int q = 0; q < 4; ++q) df[q] = qR[q] - qL[q];
    const double dfL = fma(wR[0], wR[4], -qL[4]), dfR = qR[4] - qL[4];   // (the two sides' roundings of the pressure's)
    if constexpr (PAIR) {
        double fs[5];   // the face state of this lane's side
        df[4] = right ? dfR : dfL;
        face_state(right ? qR : qL, right ? wR : wL, right ? ph : pl, right, (right ? st.z : st.x) < 0, df, fs);
        kfvs_pair<ND, LINE>(fs[0], fs + 1, fs[4], right, nn, Fv);
    } else {
        double fl[5], fr[5];
        df[4] = dfL;
        face_state(qL, wL, pl, false, st.x < 0, df, fl);
        df[4] = dfR;
        face_state(qR, wR, ph, true, st.z < 0, df, fr);
        kfvs<ND, LINE>(fl[0], fl + 1, fl[4], fr[0], fr + 1, fr[4], nn, Fv);
    }
    // viscous + HoT
    const double uf[3] = {0.5 * (wL[1] + wR[1]), 0.5 * (wL[2] + wR[2]), 0.5 * (wL[3] + wR[3])};
    const double Tf = 0.5 * (wL[4] + wR[4]);
    const double muf = mu_of<LINE>(Tf, a.mu0, a.omega);
    const double e[3] = {G[4], G[5], G[6]};
    const double dist = G[7], idist = G[8];
    // face gradients: cell average corrected along the line of centres, for every
    // velocity component j and the directions i below ND (the others are zero:
    // the LSQ weights and the line of centres have no such component)
    double guf[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, gTf[3] = {0, 0, 0};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        double gav[3];
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            gav[i] = 0.5 * (gu[(long long)(j * 3 + i) * N + L] + gu[(long long)(j * 3 + i) * N + Rr]);
        }
        const double corr = fma(wR[1 + j] - wL[1 + j], idist, -dot_rn<ND>(gav, e));
#pragma unroll
        for (int i = 0; i < ND; ++i) guf[j * 3 + i] = fma(corr, e[i], gav[i]);
    }
    {
        double gav[3];
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            gav[i] = 0.5 * (gT[(long long)i * N + L] + gT[(long long)i * N + Rr]);
        }
        const double corr = fma(wR[4] - wL[4], idist, -dot_rn<ND>(gav, e));
#pragma unroll
        for (int i = 0; i < ND; ++i) gTf[i] = fma(corr, e[i], gav[i]);
    }
    // Eq. NSF_constitutive (nsf_of) with the zero gradient entries (directions
    // i >= ND) not multiplied: the same values
    const double* hL = hot + (long long)L * HOTN;
    const double* hR = hot + (long long)Rr * HOTN;
    double Sg[6], Q[3], hf[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) hf[q] = 0.5 * (hL[q] + hR[q]);
    {
        double div = guf[0];
        if (ND > 1) div += guf[4];
        if (ND > 2) div += guf[8];
        const double two3 = 2.0 / 3.0;
        const double t = __dmul_rn(two3, div);
        auto stress = [&](double g, double h) { return __dmul_rn(-muf, g) + h; };
        Sg[0] = stress(2.0 * guf[0] - t, hf[0]);
        Sg[1] = stress(2.0 * guf[4] - t, hf[1]);
        Sg[2] = stress(2.0 * guf[8] - t, hf[2]);
        Sg[3] = stress(ND > 1 ? guf[1] + guf[3] : guf[3], hf[3]);   // du_x/dy + du_y/dx
        Sg[4] = stress(ND > 2 ? guf[2] + guf[6] : guf[6], hf[4]);   // du_x/dz + du_z/dx
        Sg[5] = ND > 1 ? stress(ND > 2 ? guf[5] + guf[7] : guf[7], hf[5]) : hf[5];   // du_y/dz + du_z/dy
        const double kap = 3.75 * muf;
#pragma unroll
        for (int i = 0; i < 3; ++i) Q[i] = i < ND ? fma(-kap, gTf[i], hf[6 + i]) : hf[6 + i];
    }
    // sigma . S and q . S over the normal's components 0..ND-1
    const double row[3][3] = {{Sg[0], Sg[3], Sg[4]}, {Sg[3], Sg[1], Sg[5]}, {Sg[4], Sg[5], Sg[2]}};
    double SigS[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) SigS[r] = dot_rn<ND>(row[r], S);
    if (!right) {
        double* F = Ff + (long long)(5 * d) * N + L;
        F[0] = __dmul_rn(Fv[0], Sabs);
        F[(long long)N] = fma(Fv[1], Sabs, SigS[0]);
        F[(long long)2 * N] = fma(Fv[2], Sabs, SigS[1]);
        F[(long long)3 * N] = fma(Fv[3], Sabs, SigS[2]);
        const double w = dot_rn<3>(SigS, uf);
        F[(long long)4 * N] = fma(Fv[4], Sabs, ND == 1 ? fma(Q[0], S[0], w) : w + dot_rn<ND>(Q, S));
    }
    const double aL = acell[L], aR = acell[Rr];
    const double lam = fabs(dot_rn<ND>(uf, nn)) + 0.5 * (aL + aR) + quotient<LINE>(5.0 * muf, 0.5 * (wL[0] + wR[0]) * dist);
    if (!right) lamf[(long long)d * N + L] = lam * Sabs;
}

template <bool PAIR = false>
__device__ __forceinline__ void face_flux_one(const MacroArgs& a, const double* Wm, const double* gu,
                                              const double* gT, const double* hot, const double* acell,
                                              double* Ff, double* lamf, int t) {
    switch (a.fnd) {
        case 1: face_flux_nd<1, PAIR>(a, Wm, gu, gT, hot, acell, Ff, lamf, t); break;
        case 2: face_flux_nd<2, PAIR>(a, Wm, gu, gT, hot, acell, Ff, lamf, t); break;
        default: face_flux_nd<3, PAIR>(a, Wm, gu, gT, hot, acell, Ff, lamf, t); break;
    }
}

// NSF flux through wall side s of cell c at state w (prim) with the cells' gradients
// guN, gTN (component-major): no mass flux, cell pressure, NSF stress and heat flux at u = 0,
// T = T_w from the cell gradient corrected along the cell-to-face line.
__device__ void wall_nsf_flux(const MacroArgs& a, const double* w, const double* guN, const double* gTN, int c, int s,
                              double* Fb) {
    double gu[9], gT[3];
    cell_grad(guN, gTN, a.N, c, gu, gT);
    const double* So = a.Sout + ((long long)c * 6 + s) * 3;
    const double Tw = a.bc_state[s * 5 + 4];
    const double* G = a.bgeo + ((long long)c * 6 + s) * 8;
    const double eb[3] = {G[4], G[5], G[6]};
    const double bdist = G[7];
    double guw[9], gTw[3];
    for (int j = 0; j < 3; ++j) {
        const double* gc = gu + j * 3;
        const double corr = (0.0 - w[1 + j]) / bdist - (gc[0] * eb[0] + gc[1] * eb[1] + gc[2] * eb[2]);
        for (int i = 0; i < 3; ++i) guw[j * 3 + i] = gc[i] + corr * eb[i];
    }
    {
        const double corr = (Tw - w[4]) / bdist - (gT[0] * eb[0] + gT[1] * eb[1] + gT[2] * eb[2]);
        for (int i = 0; i < 3; ++i) gTw[i] = gT[i] + corr * eb[i];
    }
    double sig[6], qw[3];
    nsf_of(mu_of(a, Tw), guw, gTw, sig, qw);
    const double p = w[0] * w[4];
    const double SigS[3] = {sig[0] * So[0] + sig[3] * So[1] + sig[4] * So[2],
                            sig[3] * So[0] + sig[1] * So[1] + sig[5] * So[2],
                            sig[4] * So[0] + sig[5] * So[1] + sig[2] * So[2]};
    Fb[0] = 0.0;
    Fb[1] = p * So[0] + SigS[0];
    Fb[2] = p * So[1] + SigS[1];
    Fb[3] = p * So[2] + SigS[2];
    Fb[4] = qw[0] * So[0] + qw[1] * So[1] + qw[2] * So[2];
}

// Wall correction of the synthetic solve: for each wall side of a DVM cell,
// the kinetic wall flux of f^{n+1/2} minus the NSF wall flux at W^{n+1/2}
// (gradients of W^{n+1/2} in gu, gT); zero elsewhere.
__global__ void k_wall_corr(MacroArgs a, const int* __restrict__ cell2dvm, const double* __restrict__ Wh,
                            const double* __restrict__ gu, const double* __restrict__ gT,
                            const double* __restrict__ wall_kin, double* __restrict__ wall_corr) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.N) return;
    for (int s = 0; s < 6; ++s) {
        double* o = wall_corr + ((long long)c * 6 + s) * 5;
        if (a.nbr[c * 6 + s] < 0 && a.side_bc[c * 6 + s] == GSIS_BC_WALL && cell2dvm[c] >= 0) {
            double F[5];
            wall_nsf_flux(a, Wh + c * 5, gu, gT, c, s, F);
            const double* kin = wall_kin + ((long long)c * 6 + s) * 5;
            for (int q = 0; q < 5; ++q) o[q] = kin[q] - F[q];
        } else {
            for (int q = 0; q < 5; ++q) o[q] = 0.0;
        }
    }
}

void launch_wall_corr(gsis_ctx* c) {
    const int N = c->m.N;
    k_wall_corr<<<(N + 63) / 64, 64, 0, c->stream>>>(margs(c), c->cell2dvm, c->Wh, c->gu, c->gT, c->wall_kin,
                                                     c->wall_corr);
    c->launches++;
}

// Wall loads per unit wall area for every cell with wall sides, written to
// out[c * FIELDS_N + FIELD_WALL + (0: heat flux into the wall, 1: pressure,
// 2..4: shear vector)]: the wall fluxes F (kinetic, wall_kin of the current f,
// for DVM cells; the NSF wall flux at the current state for NS cells), with
// pressure F_m.n and shear F_m - (F_m.n) n of the momentum part F_m, summed
// over the wall sides and divided by their area.
__global__ void k_wall_loads(MacroArgs a, const int* __restrict__ cell2dvm, const double* __restrict__ W,
                             const double* __restrict__ gu, const double* __restrict__ gT,
                             const double* __restrict__ wall_kin, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.N) return;
    double num[5] = {0, 0, 0, 0, 0}, area = 0.0;
    for (int s = 0; s < 6; ++s) {
        if (a.nbr[c * 6 + s] >= 0 || a.side_bc[c * 6 + s] != GSIS_BC_WALL) continue;
        double F[5];
        if (cell2dvm[c] >= 0) {
            for (int q = 0; q < 5; ++q) F[q] = wall_kin[((long long)c * 6 + s) * 5 + q];
        } else {
            wall_nsf_flux(a, W + c * 5, gu, gT, c, s, F);
        }
        const double* G = a.bgeo + ((long long)c * 6 + s) * 8;   // |S|, unit normal
        const double Fn = F[1] * G[1] + F[2] * G[2] + F[3] * G[3];
        num[0] += F[4];
        num[1] += Fn;
        for (int i = 0; i < 3; ++i) num[2 + i] += F[1 + i] - Fn * G[1 + i];
        area += G[0];
    }
    double* o = out + (long long)c * FIELDS_N + FIELD_WALL;
    for (int q = 0; q < 5; ++q) o[q] = area > 0.0 ? num[q] / area : 0.0;
}

// Eq. full_constitutive at the current state, out[c * FIELDS_N + 0..8]:
// sigma = sigma_NSF(W) + HoT_sigma (xx, yy, zz, xy, xz, yz), q = q_NSF(W) +
// HoT_q, with the HoT of the last kinetic step (zero in NS cells); and the
// pressure rho T at index 9.
__global__ void k_constitutive(int N, const double* __restrict__ W, const double* __restrict__ gu,
                               const double* __restrict__ gT, const double* __restrict__ hot, double mu0,
                               double omega, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    double sig[6], q[3];
    double u[9], t[3];
    cell_grad(gu, gT, N, c, u, t);
    nsf_of(viscosity(W[c * 5 + 4], mu0, omega), u, t, sig, q);
    double* o = out + (long long)c * FIELDS_N;
    const double* h = hot + (long long)c * HOTN;
    for (int k = 0; k < 6; ++k) o[k] = sig[k] + h[k];
    for (int k = 0; k < 3; ++k) o[6 + k] = q[k] + h[6 + k];
    o[9] = W[c * 5] * W[c * 5 + 4];
}

void launch_fields(gsis_ctx* c, bool wall, bool cons) {
    const int N = c->m.N;
    if (wall && c->has_wall) launch_wall_flux(c);   // kinetic wall fluxes of the current f
    launch_gradients(c, c->W, false);               // gradients of the current state
    if (wall) {
        k_wall_loads<<<(N + 127) / 128, 128, 0, c->stream>>>(margs(c), c->cell2dvm, c->W, c->gu, c->gT,
                                                            c->wall_kin, c->fields);
        c->launches++;
    }
    if (cons) {
        k_constitutive<<<(N + 127) / 128, 128, 0, c->stream>>>(N, c->W, c->gu, c->gT, c->hot, c->mu0, c->p.omega,
                                                               c->fields);
        c->launches++;
    }
}

// Flux F.S_out through boundary side s of cell c and lambda |S| of the side,
// into Fbnd[c][s][0..5]: far field, the kinetic flux-vector splitting against
// the far-field state with the cell's HoT; wall, the NSF wall flux plus the
// wall correction.  Formed in the face phase (boundary side j of a.bside), so
// that the residual phase only gathers.
template <bool PAIR = false>
__device__ __forceinline__ void boundary_flux_one(const MacroArgs& a, const double* Wm, const double* gu,
                                                  const double* gT, const double* hot, const double* wall_corr,
                                                  double* Fbnd, int j) {
    const int cs = a.bside[j], c = cs / 6, s = cs - 6 * c;
    const int bc = a.side_bc[cs];
    const double* wc = Wm + c * 5;
    const double rho_c = wc[0], T_c = wc[4], p_c = rho_c * T_c;
    const double u_c[3] = {wc[1], wc[2], wc[3]};
    const double* So = a.Sout + (long long)cs * 3;
    const double* st = a.bc_state + s * 5;
    const double* G = a.bgeo + (long long)cs * 8;
    const double Sabs = G[0];
    const double nn[3] = {G[1], G[2], G[3]};
    const double* h = hot + (long long)c * HOTN;
    double Fb[5];
    const double bdist = G[7];
    if (bc == GSIS_BC_FARFIELD) {
        if constexpr (PAIR) {
            const bool right = threadIdx.x & 1;
            const double u[3] = {right ? st[1] : u_c[0], right ? st[2] : u_c[1], right ? st[3] : u_c[2]};
            if (a.fnd == 1) kfvs_pair<3, true>(right ? st[0] : rho_c, u, right ? st[0] * st[4] : p_c, right, nn, Fb);
            else kfvs_pair<3, false>(right ? st[0] : rho_c, u, right ? st[0] * st[4] : p_c, right, nn, Fb);
        } else {
            if (a.fnd == 1) kfvs<3, true>(rho_c, u_c, p_c, st[0], st + 1, st[0] * st[4], nn, Fb);
            else kfvs<3, false>(rho_c, u_c, p_c, st[0], st + 1, st[0] * st[4], nn, Fb);
        }
        const double row[3][3] = {{h[0], h[3], h[4]}, {h[3], h[1], h[5]}, {h[4], h[5], h[2]}};
        const double SigS[3] = {dot_rn<3>(row[0], So), dot_rn<3>(row[1], So), dot_rn<3>(row[2], So)};
        const double ufb[3] = {0.5 * (u_c[0] + st[1]), 0.5 * (u_c[1] + st[2]), 0.5 * (u_c[2] + st[3])};
        Fb[0] = __dmul_rn(Fb[0], Sabs);
        for (int q = 1; q < 4; ++q) Fb[q] = fma(Fb[q], Sabs, SigS[q - 1]);
        Fb[4] = fma(Fb[4], Sabs, dot_rn<3>(SigS, ufb) + dot_rn<3>(h + 6, So));
    } else {
        wall_nsf_flux(a, wc, gu, gT, c, s, Fb);
        const double* wcr = wall_corr + (long long)cs * 5;
        for (int q = 0; q < 5; ++q) Fb[q] += wcr[q];
    }
    if (PAIR && (threadIdx.x & 1)) return;   // (the even lane has the flux)
    const double a_c = sqrt(GAMMA * p_c / rho_c);
    const double mu_c = mu_of(a, T_c);
    const double lam = fabs(dot_rn<3>(u_c, nn)) + a_c +
                       5.0 * mu_c / (rho_c * 2.0 * bdist);
    double* o = Fbnd + (long long)cs * 6;
    for (int q = 0; q < 5; ++q) o[q] = Fb[q];
    o[5] = lam * Sabs;
}

// Faces, rounded up to whole warps so that no warp mixes interior faces and
// boundary sides (it would run both).
__host__ __device__ __forceinline__ int face_items(int N, int ndir) { return (N * ndir + 31) / 32 * 32; }

// Faces of the two-lane form, rounded up to whole warps of 16.
__device__ __forceinline__ int pair_items(int nf) { return (nf + 15) / 16 * 16; }

// Face phase of the per-phase kernels: interior faces (N * ndir threads), then
// the far-field and wall sides.
__global__ void k_face_flux(MacroArgs a, const double* __restrict__ Wm, const double* __restrict__ gu,
                            const double* __restrict__ gT, const double* __restrict__ hot,
                            const double* __restrict__ acell, int ndir, double* __restrict__ Ff,
                            double* __restrict__ lamf, const double* __restrict__ wall_corr,
                            double* __restrict__ Fbnd) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, nf = a.N * ndir, nfp = face_items(a.N, ndir);
    if (t < nf) face_flux_one(a, Wm, gu, gT, hot, acell, Ff, lamf, t);
    else if (t >= nfp && t < nfp + a.nbside) boundary_flux_one(a, Wm, gu, gT, hot, wall_corr, Fbnd, t - nfp);
}

// Cell residual R_c = -sum_F F.S_out (gathering the face fluxes in side
// order: interior faces from Ff, far-field and wall sides from Fbnd), lambda|S|
// per side, the reciprocal 1/D of the diagonal (in D) and dU0 = R/D.
// (ND index directions carry flux; every load is issued before the sums.)
template <int ND>
__device__ __forceinline__ void cell_residual_nd(const MacroArgs& a, const double* U, const double* Un,
                                                 const double* Ff, const double* lamf, const double* Fbnd, double cfl,
                                                 double dt, double* R, double* D, double* lamS, double* dU, double* F0,
                                                 double* dF, int c) {
    constexpr int NS = 2 * ND;
    const int N = a.N;
    int n[NS];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const int2 v = *reinterpret_cast<const int2*>(a.nbr + c * 6 + 2 * d);
        n[2 * d] = v.x;
        n[2 * d + 1] = v.y;
    }
    double F[NS][5], ls[NS], Uc[5];
#pragma unroll
    for (int s = 0; s < NS; ++s) {   // the face's low cell: this one for high sides, the neighbour for low sides
        const int d = s >> 1, L = (s & 1) || n[s] < 0 ? c : n[s];
#pragma unroll
        for (int q = 0; q < 5; ++q) F[s][q] = Ff[(long long)(5 * d + q) * N + L];
        ls[s] = lamf[(long long)d * N + L];
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) Uc[q] = U[c * 5 + q];
    double Rc[5] = {0, 0, 0, 0, 0};
    double lam_sum = 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        if (n[s] >= 0) {
#pragma unroll
            for (int q = 0; q < 5; ++q) Rc[q] = (s & 1) ? Rc[q] - F[s][q] : Rc[q] + F[s][q];
        } else {
            const int bc = a.side_bc[c * 6 + s];
            ls[s] = 0.0;
            if (bc == GSIS_BC_FARFIELD || bc == GSIS_BC_WALL) {   // formed in the face phase
                const double* Fb = Fbnd + ((long long)c * 6 + s) * 6;
                for (int q = 0; q < 5; ++q) Rc[q] -= Fb[q];
                ls[s] = Fb[5];
            }
        }
        lamS[(long long)s * N + c] = ls[s];
        lam_sum += ls[s];
    }
    double Dc = __dmul_rn(1.0 / cfl + 0.5, lam_sum);
    if (dt > 0.0) {
        const double Vdt = a.vol[c] / dt;
#pragma unroll
        for (int q = 0; q < 5; ++q) Rc[q] = fma(-Vdt, Uc[q] - Un[c * 5 + q], Rc[q]);
        Dc += Vdt;
    }
    const double iD = 1.0 / Dc;
    D[c] = iD;   // the relaxation sweeps multiply by the reciprocal
    double dUc[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        dUc[q] = __dmul_rn(Rc[q], iD);
        R[(long long)q * N + c] = Rc[q];
        dU[(long long)q * N + c] = dUc[q];
    }
    if (dF) {   // relaxation sweeps follow: the flux tensor of U_c and its change for dU_c
        double T[15];
        euler_tensor<ND>(Uc, T);
#pragma unroll
        for (int q = 0; q < 5; ++q)
#pragma unroll
            for (int i = 0; i < ND; ++i) F0[(long long)(q * 3 + i) * N + c] = T[q * 3 + i];
        flux_change<ND>(Uc, dUc, T, dF, N, c);
    }
}

__device__ __forceinline__ void cell_residual_one(const MacroArgs& a, const double* U, const double* Un,
                                                  const double* Ff, const double* lamf, const double* Fbnd, double cfl,
                                                  double dt, double* R, double* D, double* lamS, double* dU, double* F0,
                                                  double* dF, int c) {
    switch (a.nd) {
        case 1: cell_residual_nd<1>(a, U, Un, Ff, lamf, Fbnd, cfl, dt, R, D, lamS, dU, F0, dF, c); break;
        case 2: cell_residual_nd<2>(a, U, Un, Ff, lamf, Fbnd, cfl, dt, R, D, lamS, dU, F0, dF, c); break;
        default: cell_residual_nd<3>(a, U, Un, Ff, lamf, Fbnd, cfl, dt, R, D, lamS, dU, F0, dF, c); break;
    }
}

__global__ void k_cell_residual(MacroArgs a, const double* __restrict__ U, const double* __restrict__ Un,
                                const double* __restrict__ Ff, const double* __restrict__ lamf,
                                const double* __restrict__ Fbnd, double cfl, double dt,
                                double* __restrict__ R, double* __restrict__ D, double* __restrict__ lamS,
                                double* __restrict__ dU, double* __restrict__ F0, double* __restrict__ dF) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < a.N) cell_residual_one(a, U, Un, Ff, lamf, Fbnd, cfl, dt, R, D, lamS, dU, F0, dF, c);
}

// One Jacobi sweep: dU_new = (R - 1/2 sum_j [dF_j . S_out - lambda|S| dU_j]) / D,
// dF_j = F(U_j + dU_j) - F(U_j) read from the neighbour's flux-change tensor
// (dFin); with dFout the cell's own tensor for dU_new follows for the next sweep.
// The two sums are accumulated apart (FMA chains over the normal components
// that can be nonzero) and combined once.
// The loads of both sides are issued before the sums.  The new increment is
// left in dUc (registers) and, with dUout, stored.
template <int ND>
__device__ __forceinline__ void relax_nd(const MacroArgs& a, const double* U, const double* R, const double* D,
                                         const double* lamS, const double* dUin, double* dUout, const double* dFin,
                                         double* dFout, const double* F0, int c, double* dUc) {
    const int N = a.N;
    double Rc[5], fs[5] = {0, 0, 0, 0, 0}, ld[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 5; ++q) Rc[q] = R[(long long)q * N + c];
    const double iD = D[c];   // 1 / D
    // the two sides of a direction at a time in 3D (all four at once in 2D: in 3D
    // the six sides' values would not fit the registers)
#pragma unroll(ND < 3 ? ND : 1)
    for (int d = 0; d < ND; ++d) {
        const int2 nb = *reinterpret_cast<const int2*>(a.nbr + c * 6 + 2 * d);
        double dF[2][5][ND], dn[2][5], So[2][ND], ls[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int s = 2 * d + h, nn = h ? nb.y : nb.x, m = nn >= 0 ? nn : c;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
#pragma unroll
                for (int i = 0; i < ND; ++i) dF[h][q][i] = dFin[(long long)(q * 3 + i) * N + m];
                dn[h][q] = dUin[(long long)q * N + m];
            }
#pragma unroll
            for (int i = 0; i < ND; ++i) So[h][i] = a.Sout[((long long)c * 6 + s) * 3 + i];
            ls[h] = lamS[(long long)s * N + c];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if ((h ? nb.y : nb.x) < 0) continue;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
#pragma unroll
                for (int i = 0; i < ND; ++i) fs[q] = fma(dF[h][q][i], So[h][i], fs[q]);
                ld[q] = fma(ls[h], dn[h][q], ld[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        dUc[q] = __dmul_rn(fma(-0.5, fs[q] - ld[q], Rc[q]), iD);
        if (dUout) dUout[(long long)q * N + c] = dUc[q];
    }
    if (dFout) {
        double Uc[5], T[15];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            Uc[q] = U[c * 5 + q];
#pragma unroll
            for (int i = 0; i < ND; ++i) T[q * 3 + i] = F0[(long long)(q * 3 + i) * N + c];
        }
        flux_change<ND>(Uc, dUc, T, dFout, N, c);
    }
}

__device__ __forceinline__ void relax_one(const MacroArgs& a, const double* U, const double* R, const double* D,
                                          const double* lamS, const double* dUin, double* dUout, const double* dFin,
                                          double* dFout, const double* F0, int c, double* dUc) {
    switch (a.nd) {
        case 1: relax_nd<1>(a, U, R, D, lamS, dUin, dUout, dFin, dFout, F0, c, dUc); break;
        case 2: relax_nd<2>(a, U, R, D, lamS, dUin, dUout, dFin, dFout, F0, c, dUc); break;
        default: relax_nd<3>(a, U, R, D, lamS, dUin, dUout, dFin, dFout, F0, c, dUc); break;
    }
}

__global__ void k_relax(MacroArgs a, const double* __restrict__ U, const double* __restrict__ R,
                        const double* __restrict__ D, const double* __restrict__ lamS, const double* __restrict__ dUin,
                        double* __restrict__ dUout, const double* __restrict__ dFin, double* __restrict__ dFout,
                        const double* __restrict__ F0) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    double dUc[5];
    if (c < a.N) relax_one(a, U, R, D, lamS, dUin, dUout, dFin, dFout, F0, c, dUc);
}

// U += dU (dU of this cell), primitive state Wm.
__device__ __forceinline__ void update_one(double* U, const double* dUc, double* Wm, int c) {
    double Uc[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        Uc[q] = U[c * 5 + q] + dUc[q];
        U[c * 5 + q] = Uc[q];
    }
    cons_to_prim(Uc, Wm + c * 5);
}

__global__ void k_update(int N, double* __restrict__ U, const double* __restrict__ dU, double* __restrict__ Wm) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    double dUc[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) dUc[q] = dU[(long long)q * N + c];
    update_one(U, dUc, Wm, c);
}

// The last Jacobi sweep of a pseudo-step followed by the update of the
// cell's own state (U += dU, primitive Wm): the sweep reads U only through the
// flux change, which the last sweep does not form, so each cell may update
// its state in place (one phase instead of two, the same values).
__device__ __forceinline__ void relax_update_one(const MacroArgs& a, double* U, const double* R, const double* D,
                                                 const double* lamS, const double* dUin, const double* dFin, double* Wm,
                                                 int c) {
    double dUc[5];
    relax_one(a, U, R, D, lamS, dUin, nullptr, dFin, nullptr, nullptr, c, dUc);
    update_one(U, dUc, Wm, c);
}

__global__ void k_relax_update(MacroArgs a, double* __restrict__ U, const double* __restrict__ R,
                               const double* __restrict__ D, const double* __restrict__ lamS,
                               const double* __restrict__ dUin, const double* __restrict__ dFin,
                               double* __restrict__ Wm) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < a.N) relax_update_one(a, U, R, D, lamS, dUin, dFin, Wm, c);
}

// The whole pseudo-time block of one solve in one thread-block cluster of
// `cs` CTAs (meshes up to a few thousand cells: the 1D shocks, solve
// batches).  The same per-cell and per-face functions as the multi-block
// kernels, separated by cluster barriers (release/acquire at cluster scope,
// so every CTA of the cluster sees the others' global-memory writes of the
// previous phase), so the result is identical.  Jobs are clusters 0, 1, ...
// of the grid.
// What bounds it: a warp's FP64 instruction holds the FP64 pipe of its SM
// sub-partition for 64 cycles, so a phase lasts (FP64 instructions per item) x
// 64 cycles x the chunks of 32 items on the busiest sub-partition.  Chunk g goes
// to warp g / cs of CTA g mod cs: the chunks spread over all 4 cs
// sub-partitions of the cluster (a CTA-major order put every cell of a solve
// of up to 512 cells on one SM).
__device__ __forceinline__ void fused_sync(int cs) {
    if (cs > 1)
        cg::this_cluster().sync();
    else
        __syncthreads();
}

__global__ void __launch_bounds__(MACRO_FUSED_THREADS, 1) k_macro_fused(const MacroJob* __restrict__ jobs, int cs) {
    const MacroJob& J = jobs[blockIdx.x / cs];
    const int first = (((threadIdx.x >> 5) * cs + blockIdx.x % cs) << 5) + (threadIdx.x & 31), stride = cs * blockDim.x;
    const MacroArgs a = J.a;
    const int N = a.N, nf = N * J.ndir, nfp = face_items(N, J.ndir);
    // two lanes per face while every chunk of 16 faces still has a sub-partition of its own
    const bool paired = (pair_items(nf) + a.nbside + 15) / 16 <= 4 * cs;
    for (int it = 0; it < J.steps; ++it) {
        for (int c = first; c < N; c += stride)
            gradients_cell<false>(a, J.Wm, J.gu, J.gT, nullptr, nullptr, J.acell, c);
        fused_sync(cs);
        for (int t = first; !paired && t < nfp + a.nbside; t += stride) {
            if (t < nf) face_flux_one(a, J.Wm, J.gu, J.gT, J.hot, J.acell, J.Ff, J.lamf, t);
            else if (t >= nfp) boundary_flux_one(a, J.Wm, J.gu, J.gT, J.hot, J.wall_corr, J.Fbnd, t - nfp);
        }
        if (paired) {   // (one chunk of 16 per warp: items 0.., first is a multiple of 32 plus the lane)
            const int t = first >> 1, nfq = pair_items(nf);
            if (t < nf) face_flux_one<true>(a, J.Wm, J.gu, J.gT, J.hot, J.acell, J.Ff, J.lamf, t);
            else if (t >= nfq && t < nfq + a.nbside)
                boundary_flux_one<true>(a, J.Wm, J.gu, J.gT, J.hot, J.wall_corr, J.Fbnd, t - nfq);
        }
        fused_sync(cs);
        for (int c = first; c < N; c += stride)
            cell_residual_one(a, J.U, J.Un, J.Ff, J.lamf, J.Fbnd, J.cfl, J.dt, J.R, J.D, J.lamS, J.dU, J.F0,
                              J.k_sub > 0 ? J.dFa : nullptr, c);
        fused_sync(cs);
        double* din = J.dU;
        double* dout = J.dU2;
        for (int s = 0; s + 1 < J.k_sub; ++s) {
            double* fin = (s & 1) ? J.dFb : J.dFa;
            double* fout = (s & 1) ? J.dFa : J.dFb;
            double dUc[5];
            for (int c = first; c < N; c += stride)
                relax_one(a, J.U, J.R, J.D, J.lamS, din, dout, fin, fout, J.F0, c, dUc);
            fused_sync(cs);
            double* t = din; din = dout; dout = t;
        }
        if (J.k_sub > 0) {
            for (int c = first; c < N; c += stride)
                relax_update_one(a, J.U, J.R, J.D, J.lamS, din, (J.k_sub - 1) & 1 ? J.dFb : J.dFa, J.Wm, c);
        } else {
            for (int c = first; c < N; c += stride) {
                double dUc[5];
                for (int q = 0; q < 5; ++q) dUc[q] = din[(long long)q * N + c];
                update_one(J.U, dUc, J.Wm, c);
            }
        }
        fused_sync(cs);
    }
}

// Largest usable cluster size <= want (a power of two, at most 8) for the
// fused kernel on the current device; 1 if clusters cannot be resident.
int fused_cluster_size(int want) {
    static int cached[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    int cs = 1;
    while (cs * 2 <= want && cs * 2 <= 8) cs *= 2;
    for (; cs > 1; cs /= 2) {
        if (cached[cs] == 0) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(cs);
            cfg.blockDim = dim3(MACRO_FUSED_THREADS);
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = cs;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, k_macro_fused, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            cached[cs] = n > 0 ? 1 : -1;
        }
        if (cached[cs] > 0) return cs;
    }
    return 1;
}

MacroJob macro_job(gsis_ctx* c, int steps, bool time_term) {
    MacroJob J;
    J.a = margs(c);
    J.steps = steps;
    J.ndir = c->normal_components;
    J.k_sub = c->p.k_sub;
    J.cfl = c->p.cfl;
    J.dt = time_term ? c->p.dt : 0.0;
    J.Wm = c->Wm; J.U = c->U; J.Un = c->Un; J.gu = c->gu; J.gT = c->gT; J.hot = c->hot; J.Ff = c->Ff;
    J.lamf = c->lamf; J.wall_corr = c->wall_corr; J.R = c->R; J.D = c->D; J.lamS = c->lamS; J.dU = c->dU;
    J.dU2 = c->dU2;
    J.acell = c->acell;
    J.F0 = c->F0;
    J.dFa = c->dFa;
    J.dFb = c->dFb;
    J.Fbnd = c->Fbnd;
    return J;
}

// cs: cluster size from fused_cluster_size (called before any stream capture).
void launch_macro_fused(const MacroJob* d_jobs, int njobs, cudaStream_t stream, int cs) {
    if (cs > 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(njobs * cs);
        cfg.blockDim = dim3(MACRO_FUSED_THREADS);
        cfg.stream = stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cs;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, k_macro_fused, d_jobs, cs);
        return;
    }
    k_macro_fused<<<njobs, MACRO_FUSED_THREADS, 0, stream>>>(d_jobs, 1);
}

// Cluster size of one fused solve alone: the fewest CTAs (a power of two, at
// most 8) that give every chunk of 16 faces (two lanes per face) a sub-partition
// of its own, or of 32 faces if eight CTAs are too few for that.
int fused_cluster_for(int N, int ndir, int nbside) {
    for (int per : {16, 32}) {
        const int chunks = ((N * ndir + per - 1) / per * per + nbside + per - 1) / per;
        int want = 1;
        while (want < 8 && 4 * want < chunks) want *= 2;
        if (4 * want >= chunks || per == 32) return fused_cluster_size(want);
    }
    return 1;
}

// ---------------------------------------------------------------------------- persistent kernel
// The whole block of pseudo-steps of one solve in ONE cooperative launch
// over all SMs (meshes above MACRO_FUSED_MAX_CELLS cells: the cylinder, the
// sphere).  The same per-cell and per-face functions as the per-phase
// kernels, separated by a grid-wide barrier, so the result is identical;
// what goes away is the launch latency of the ~(4 + k_sub) kernels per
// pseudo-step.  Every wait of the barrier is bounded by spin_limit polls:
// a block that runs out records the error and returns, and every other
// block returns at its next barrier (the host reports GSIS_ERR_TIMEOUT).
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_relaxed_gpu(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Returns false when the barrier failed (this block's wait ran out, or
// another block's did): the caller returns at once.
__device__ __forceinline__ bool grid_barrier(GridBarrier* bar, unsigned expected, unsigned long long spin_limit) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned g = ld_acquire_gpu(&bar->gen);   // read before arriving: gen cannot move before we arrive
        __threadfence();                                // this block's writes before its arrival
        const unsigned arrived = atomicAdd(&bar->count, 1u);
        if (arrived == expected - 1) {
            bar->count = 0;                             // reset for the next barrier before releasing
            __threadfence();
            atomicAdd(&bar->gen, 1u);
        } else {
            unsigned long long polls = 0;
            while (ld_acquire_gpu(&bar->gen) == g) {
                if (++polls > spin_limit || ld_relaxed_gpu(&bar->err) != 0) {
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        if (!ok) atomicExch(&bar->err, 1);
        __threadfence();                                // the other blocks' writes before ours
        s_ok = ok && ld_relaxed_gpu(&bar->err) == 0;
    }
    __syncthreads();
    return s_ok != 0;
}

__global__ void __launch_bounds__(MACRO_PERSISTENT_THREADS, 2)
    k_macro_persistent(MacroJob J, GridBarrier* bar, unsigned long long spin_limit, int stall) {
    const MacroArgs a = J.a;
    const int N = a.N, nf = N * J.ndir, nfp = face_items(N, J.ndir);
    const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    // stall (test hook): the barrier waits for one block more than the grid
    // holds, so its wait can only end by running out of spin_limit polls
    const unsigned expected = gridDim.x + (stall ? 1u : 0u);
    for (int it = 0; it < J.steps; ++it) {
        for (int c = first; c < N; c += stride)
            gradients_cell<false>(a, J.Wm, J.gu, J.gT, nullptr, nullptr, J.acell, c);
        if (!grid_barrier(bar, expected, spin_limit)) return;
        for (int t = first; t < nfp + a.nbside; t += stride) {
            if (t < nf) face_flux_one(a, J.Wm, J.gu, J.gT, J.hot, J.acell, J.Ff, J.lamf, t);
            else if (t >= nfp) boundary_flux_one(a, J.Wm, J.gu, J.gT, J.hot, J.wall_corr, J.Fbnd, t - nfp);
        }
        if (!grid_barrier(bar, expected, spin_limit)) return;
        for (int c = first; c < N; c += stride)
            cell_residual_one(a, J.U, J.Un, J.Ff, J.lamf, J.Fbnd, J.cfl, J.dt, J.R, J.D, J.lamS, J.dU, J.F0, J.k_sub > 0 ? J.dFa : nullptr, c);
        if (!grid_barrier(bar, expected, spin_limit)) return;
        double* din = J.dU;
        double* dout = J.dU2;
        for (int s = 0; s + 1 < J.k_sub; ++s) {
            double* fin = (s & 1) ? J.dFb : J.dFa;
            double* fout = (s & 1) ? J.dFa : J.dFb;
            double dUc[5];
            for (int c = first; c < N; c += stride)
                relax_one(a, J.U, J.R, J.D, J.lamS, din, dout, fin, fout, J.F0, c, dUc);
            if (!grid_barrier(bar, expected, spin_limit)) return;
            double* t = din; din = dout; dout = t;
        }
        if (J.k_sub > 0) {
            for (int c = first; c < N; c += stride)
                relax_update_one(a, J.U, J.R, J.D, J.lamS, din, (J.k_sub - 1) & 1 ? J.dFb : J.dFa, J.Wm, c);
        } else {
            for (int c = first; c < N; c += stride) {
                double dUc[5];
                for (int q = 0; q < 5; ++q) dUc[q] = din[(long long)q * N + c];
                update_one(J.U, dUc, J.Wm, c);
            }
        }
        if (!grid_barrier(bar, expected, spin_limit)) return;
    }
}

// Co-resident CTAs of the persistent kernel on this device (0 if a
// cooperative launch is not possible).
static int persistent_capacity(gsis_ctx* c) {
    if (c->pers_grid != 0) return c->pers_grid;
    int dev = 0, sms = 0, coop = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_macro_persistent, MACRO_PERSISTENT_THREADS, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        per_sm = 0;
    }
    c->pers_grid = (coop && per_sm > 0) ? per_sm * sms : -1;
    return c->pers_grid;
}

// One cooperative launch for `steps` pseudo-steps; the barrier's error word
// is copied to c->h_err (read by the host after its next synchronisation).
static bool launch_macro_persistent(gsis_ctx* c, const MacroJob& J, bool stall) {
    const int cap = persistent_capacity(c);
    if (cap <= 0) return false;
    // every co-resident CTA: the phases are bound by the FP64 pipes of all SMs (a grid sized to the work
    // alone left SMs idle), capped where some CTAs would find no item in any phase
    const long long work = std::max<long long>((long long)J.a.N * J.ndir, J.a.N);
    const int grid = (int)std::min<long long>(cap, std::max<long long>(1, work / 32));
    cudaMemsetAsync(c->d_bar, 0, sizeof(GridBarrier), c->stream);
    MacroJob Jc = J;
    GridBarrier* bar = c->d_bar;
    unsigned long long spin = c->p.spin_limit;
    int st = stall ? 1 : 0;
    void* args[] = {&Jc, &bar, &spin, &st};
    if (cudaLaunchCooperativeKernel((const void*)k_macro_persistent, dim3(grid), dim3(MACRO_PERSISTENT_THREADS), args,
                                    0, c->stream) != cudaSuccess)
        return false;
    cudaMemcpyAsync(c->h_err, &c->d_bar->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    c->launches++;
    return true;
}

// `steps` DP-LUR pseudo-steps on c->U / c->Wm (prim kept in step), HoT from
// c->hot, time term against c->Un when time_term.  Small meshes run the fused
// one-CTA kernel (one launch per block of steps), larger ones the persistent
// cooperative kernel (one launch per block of steps); inside a graph capture
// and where a cooperative launch is not available the per-phase kernels run
// over the whole grid.  Every path computes the same result.
void macro_block(gsis_ctx* c, int steps, bool with_hot, bool time_term, bool capturing) {
    (void)with_hot;
    const int N = c->m.N;
    if (steps <= 0) return;
    // automatic choice: the per-phase kernels above the fused kernel's limit (measured on the 16,384-cell
    // cylinder, 100 pseudo-steps, when the phases took 11.1 ms (5.95 now): persistent kernel 13.0 ms with
    // one CTA on each of 128 SMs and 23.8 ms with every co-resident CTA -- its 600 grid barriers cost more
    // than the launches they replace)
    int path = c->macro_path;
    if (path == MACRO_AUTO) path = N <= MACRO_FUSED_MAX_CELLS ? MACRO_FUSED : MACRO_MULTI;
    if (capturing && (path == MACRO_PERSISTENT || path == MACRO_PERSISTENT_STALL)) path = MACRO_MULTI;
    if (path == MACRO_FUSED) {
        MacroJob J = macro_job(c, steps, time_term);
        cudaMemcpyAsync(c->d_job, &J, sizeof(MacroJob), cudaMemcpyHostToDevice, c->stream);
        launch_macro_fused(c->d_job, 1, c->stream, fused_cluster_for(N, c->normal_components, c->m.nbside));
        c->launches++;
        return;
    }
    if (path == MACRO_PERSISTENT || path == MACRO_PERSISTENT_STALL) {
        if (launch_macro_persistent(c, macro_job(c, steps, time_term), path == MACRO_PERSISTENT_STALL)) return;
        cudaGetLastError();   // no cooperative launch here: fall through to the per-phase kernels
    }
    const int TB = 64;
    const int nb = (N + TB - 1) / TB;
    const int ndir = c->normal_components;   // index directions that carry flux
    const int nf = (face_items(N, ndir) + c->m.nbside + TB - 1) / TB;   // faces, then the boundary sides
    MacroArgs a = margs(c);
    const double dt = time_term ? c->p.dt : 0.0;
    for (int it = 0; it < steps; ++it) {
        launch_gradients(c, c->Wm, false);
        k_face_flux<<<nf, TB, 0, c->stream>>>(a, c->Wm, c->gu, c->gT, c->hot, c->acell, ndir, c->Ff, c->lamf,
                                               c->wall_corr, c->Fbnd);
        k_cell_residual<<<nb, TB, 0, c->stream>>>(a, c->U, c->Un, c->Ff, c->lamf, c->Fbnd, c->p.cfl, dt, c->R, c->D,
                                                  c->lamS, c->dU, c->F0, c->p.k_sub > 0 ? c->dFa : nullptr);
        c->launches += 2;
        double* din = c->dU;
        double* dout = c->dU2;
        for (int s = 0; s < c->p.k_sub; ++s) {
            double* fin = (s & 1) ? c->dFb : c->dFa;
            if (s + 1 < c->p.k_sub) {
                double* fout = (s & 1) ? c->dFa : c->dFb;
                k_relax<<<nb, TB, 0, c->stream>>>(a, c->U, c->R, c->D, c->lamS, din, dout, fin, fout, c->F0);
            } else {
                k_relax_update<<<nb, TB, 0, c->stream>>>(a, c->U, c->R, c->D, c->lamS, din, fin, c->Wm);
            }
            c->launches++;
            double* t = din; din = dout; dout = t;
        }
        if (c->p.k_sub == 0) {
            k_update<<<nb, TB, 0, c->stream>>>(N, c->U, din, c->Wm);
            c->launches++;
        }
    }
}

// ---------------------------------------------------------------------------- residual epsilon
// Convergence criterion of Sec. 4: max over {rho, u (as a vector), T} of
// sqrt(sum (Wn - Wp)^2 vol / sum Wp^2 vol), quantities with a zero denominator
// left out.  out[0] = epsilon, out[1] = number of cells with non-finite or
// non-positive rho / T in Wn.
__device__ __forceinline__ void eps_sums(int first, int stride, int N, const double* __restrict__ Wn,
                                         const double* __restrict__ Wp, const double* __restrict__ vol, double* acc) {
    for (int c = first; c < N; c += stride) {
        const double V = vol[c];
        const double* a = Wn + c * 5;
        const double* b = Wp + c * 5;
        const double dr = a[0] - b[0];
        acc[0] += dr * dr * V;
        acc[1] += b[0] * b[0] * V;
        double du = 0.0, uu = 0.0;
        for (int i = 1; i < 4; ++i) { du += (a[i] - b[i]) * (a[i] - b[i]); uu += b[i] * b[i]; }
        acc[2] += du * V;
        acc[3] += uu * V;
        const double dT = a[4] - b[4];
        acc[4] += dT * dT * V;
        acc[5] += b[4] * b[4] * V;
        bool bad = !(a[0] > 0.0) || !(a[4] > 0.0) || !isfinite(a[0]) || !isfinite(a[4]);
        for (int i = 1; i < 4; ++i) bad = bad || !isfinite(a[i]);
        acc[6] += bad ? 1.0 : 0.0;
    }
}

__device__ __forceinline__ void eps_result(const double* acc, double* out) {
    double e = 0.0;
    for (int q = 0; q < 3; ++q)
        if (acc[2 * q + 1] > 0.0) e = fmax(e, sqrt(acc[2 * q] / acc[2 * q + 1]));
    out[0] = e;
    out[1] = acc[6];
}

// One block (small meshes).
__global__ void k_eps(int N, const double* __restrict__ Wn, const double* __restrict__ Wp,
                      const double* __restrict__ vol, double* __restrict__ out) {
    __shared__ double sm[32 * 7];
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    eps_sums(threadIdx.x, blockDim.x, N, Wn, Wp, vol, acc);
    block_sum<7>(acc, sm);
    if (threadIdx.x == 0) eps_result(acc, out);
}

// Larger meshes in two launches: the sums of each block into part[block][7],
// then their totals, one warp per sum (fixed order).  One block alone is bound
// by its SM's FP64 pipes: 136 us on 16,384 cells.
__global__ void __launch_bounds__(128) k_eps_part(int N, const double* __restrict__ Wn, const double* __restrict__ Wp,
                                                  const double* __restrict__ vol, double* __restrict__ part) {
    __shared__ double sm[32 * 7];
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    eps_sums(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, N, Wn, Wp, vol, acc);
    block_sum<7>(acc, sm);
    if (threadIdx.x == 0)
        for (int q = 0; q < 7; ++q) part[blockIdx.x * 7 + q] = acc[q];
}

__global__ void __launch_bounds__(224) k_eps_final(int nb, const double* __restrict__ part, double* __restrict__ out) {
    __shared__ double tot[7];
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
    for (int b = lane; b < nb; b += 32) t += part[b * 7 + q];
    t = warp_sum(t);
    if (lane == 0) tot[q] = t;
    __syncthreads();
    if (threadIdx.x == 0) eps_result(tot, out);
}

void launch_eps(gsis_ctx* c, const double* Wn, const double* Wp) {
    const int N = c->m.N;
    if (N <= 1024) {
        k_eps<<<1, 256, 0, c->stream>>>(N, Wn, Wp, c->m.vol, c->eps_buf);
        c->launches++;
        return;
    }
    const int nb = std::min(EPS_BLOCKS, (N + 127) / 128);
    k_eps_part<<<nb, 128, 0, c->stream>>>(N, Wn, Wp, c->m.vol, c->eps_buf + 4);
    k_eps_final<<<1, 224, 0, c->stream>>>(nb, c->eps_buf + 4, c->eps_buf);
    c->launches += 2;
}

}  // namespace gsis
