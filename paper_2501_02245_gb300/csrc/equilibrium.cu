// Distribution records: reference distributions of the kinetic model, their
// conservation correction, Grad-13 interface distributions and boundary
// Maxwellians, all in the separable form
//     D(xi) = A e_x(ix) e_y(iy) e_z(iz) * P(c),   c = xi - u,
//     e_d = exp(-c_d^2 / (2T)),  P = p0 + p.c + c.P2.c + (r.c) c^2,
// so that one exp per 1D node (not per 3D node) is evaluated.
//
//  * Shakhov reference g_0t of Sec. 2 (Eq. general_model with d_r = 0):
//      p0 = 1, p = -5T s q, r = s q, s = 1/(15 p T^2)
//  * Grad-13 distribution of Eq. G13_VDF:
//      p0 = 1, p = -q/(rho T^2), P2 = sigma/(2 rho T^2), r = q/(5 rho T^3)
//  * conservation correction (the Lagrange-multiplier form of Gamba and
//    Tharkabhushanam, J. Comput. Phys. 228 (2009), Maxwellian weighted):
//      D <- D + M (a0 + a.xi + a4 |xi|^2) with the 5x5 system
//      sum_v w psi phi^T M a = U - sum_v w psi D,  psi = (1, xi, |xi|^2/2),
//      phi = (1, xi, |xi|^2),
//    whose sums are assembled exactly from 1D sums C_d[k] = sum_i e_d c_d^k.
#include <algorithm>
#include <type_traits>
#include "gsis_device.cuh"

namespace gsis {

// Conservation correction of one record.  C[d][k] = sum_i e_d c_d^k over the
// axis nodes; every moment sum of the correction system is a sum of products
// C[0][a] C[1][b] C[2][c].  Written in powers of c (the polynomials 1, c, c^2
// span the same space as 1, xi, |xi|^2, and about u the target is (rho, 0, 0,
// 0, 3 rho T)), the system is the Gram matrix of (1, c_x, c_y, c_z, c^2) under
// the Maxwellian weight: symmetric positive definite, solved by an L D L^T
// factorisation without pivoting.  On return a[5] are the coefficients of
// (1, c, c^2) to be added to the base polynomial.
// (The generic form -- all products of the terms of psi and phi in xi, a pivoted
// elimination -- cost up to 250 FP64 operations per matrix entry, serially: 50 us
// for one record.)
__device__ __forceinline__ void correction_coefs(const RecSpec& s, const double (&C)[3][6], double wA, double* a) {
    const double* X[3] = {C[0], C[1], C[2]};
    double G[5][5], b[5];   // lower triangle
    double p2[3];           // products of the other two axes: (0,0) and (2,0) + (0,2)
    double w2[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int e = (d + 1) % 3, f = (d + 2) % 3;
        p2[d] = X[e][0] * X[f][0];
        w2[d] = fma(X[e][2], X[f][0], X[e][0] * X[f][2]);
    }
    G[0][0] = X[0][0] * p2[0];
    double t22 = 0.0, t4 = 0.0;   // <c_d^2 c_e^2> and <c_d^4> summed
    G[4][0] = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        G[1 + d][0] = X[d][1] * p2[d];
        G[1 + d][1 + d] = X[d][2] * p2[d];
        G[4][0] += G[1 + d][1 + d];
        G[4][1 + d] = fma(X[d][3], p2[d], X[d][1] * w2[d]);
        t4 = fma(X[d][4], p2[d], t4);
        t22 = fma(X[d][2], w2[d], t22);   // each pair twice
    }
    G[2][1] = X[0][1] * X[1][1] * X[2][0];
    G[3][1] = X[0][1] * X[1][0] * X[2][1];
    G[3][2] = X[0][0] * X[1][1] * X[2][1];
    G[4][4] = t4 + t22;
    // right-hand side: target minus the moments of the base polynomial
    const double target = s.rho / wA;
    b[0] = fma(-s.p0, G[0][0], target);
    b[4] = fma(-s.p0, G[4][0], 3.0 * s.T * target);
#pragma unroll
    for (int d = 0; d < 3; ++d) b[1 + d] = -s.p0 * G[1 + d][0];
    const bool odd = s.r[0] != 0.0 || s.r[1] != 0.0 || s.r[2] != 0.0 || s.p[0] != 0.0 || s.p[1] != 0.0 || s.p[2] != 0.0;
    const bool stress = s.P2[0] != 0.0 || s.P2[1] != 0.0 || s.P2[2] != 0.0 || s.P2[3] != 0.0 || s.P2[4] != 0.0 ||
                        s.P2[5] != 0.0;
    if (odd || stress) {
        // S_de = <c_d c_e c^2>
        double S[3][3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            S[d][d] = fma(X[d][4], p2[d], X[d][2] * w2[d]);
            const int e = (d + 1) % 3, f = (d + 2) % 3;
            const double v = fma(fma(X[d][3], X[e][1], X[d][1] * X[e][3]), X[f][0], X[d][1] * X[e][1] * X[f][2]);
            S[d][e] = v;
            S[e][d] = v;
        }
        if (odd) {   // p.c + (r.c) c^2
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int e = (d + 1) % 3, f = (d + 2) % 3;
                const double q4 = fma(X[e][4], X[f][0], fma(X[e][0], X[f][4], 2.0 * X[e][2] * X[f][2]));
                const double Q = fma(X[d][5], p2[d], fma(2.0 * X[d][3], w2[d], X[d][1] * q4));   // <c_d c^4>
                b[0] -= fma(s.p[d], G[1 + d][0], s.r[d] * G[4][1 + d]);
                b[4] -= fma(s.p[d], G[4][1 + d], s.r[d] * Q);
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    b[1 + k] -= fma(s.p[d], k >= d ? G[1 + k][1 + d] : G[1 + d][1 + k], s.r[d] * S[k][d]);
            }
        }
        if (stress) {   // c.P2.c, with P2 = (xx, yy, zz, xy, xz, yz)
            const double P[3][3] = {{s.P2[0], s.P2[3], s.P2[4]}, {s.P2[3], s.P2[1], s.P2[5]}, {s.P2[4], s.P2[5], s.P2[2]}};
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    b[0] = fma(-P[d][e], d >= e ? G[1 + d][1 + e] : G[1 + e][1 + d], b[0]);
                    b[4] = fma(-P[d][e], S[d][e], b[4]);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {   // <c_k c_d c_e>
                        double m = 1.0;
#pragma unroll
                        for (int x = 0; x < 3; ++x) m *= X[x][(k == x) + (d == x) + (e == x)];
                        b[1 + k] = fma(-P[d][e], m, b[1 + k]);
                    }
                }
        }
    }
    // L D L^T
    double L[5][5], iD[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        double V[5];
#pragma unroll
        for (int k = 0; k < j; ++k) V[k] = L[j][k];   // holds L[j][k] D[k] until scaled
        double dj = G[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) {
            L[j][k] = V[k] * iD[k];
            dj = fma(-L[j][k], V[k], dj);
        }
        iD[j] = recip64(dj);
#pragma unroll
        for (int i = j + 1; i < 5; ++i) {   // column j of the rows below: G_ij - sum_k L_ik D_k L_jk
            double v = G[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) v = fma(-L[i][k], L[j][k], v);
            L[i][j] = v;
        }
    }
#pragma unroll
    for (int j = 0; j < 5; ++j)
#pragma unroll
        for (int k = 0; k < j; ++k) b[j] = fma(-L[j][k], b[k], b[j]);
#pragma unroll
    for (int j = 4; j >= 0; --j) {
        a[j] = b[j] * iD[j];
#pragma unroll
        for (int i = j + 1; i < 5; ++i) a[j] = fma(-L[i][j], a[i], a[j]);
    }
}

// LPR lanes (a "group") per record: the FP64 operations of a warp instruction
// cost the same whatever the number of active lanes, so with many records four
// share a warp (LPR = 8) and the serial correction runs for all four at once;
// with few, a record has the whole warp (LPR = 32: fewer nodes per lane).  The
// records [0, n0) go to out0, [n0, nrec) to out1.
template <int LPR>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, LPR);
    return v;
}

template <int LPR>
__global__ void k_build_records(const RecSpec* __restrict__ specs, int nrec, int n0, Records out0, Records out1,
                                VGridDev vg) {
    constexpr int PER_WARP = 32 / LPR;
    const int lane = threadIdx.x & 31, sl = lane & (LPR - 1);
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp * PER_WARP >= nrec) return;       // the whole warp is past the last record
    const int r0 = warp * PER_WARP + (lane / LPR);
    const bool valid = r0 < nrec;              // groups past the end compute a copy and store nothing
    const int rr = valid ? r0 : nrec - 1;
    const RecSpec s = specs[rr];
    const Records& out = rr < n0 ? out0 : out1;
    const long long r = rr < n0 ? rr : rr - n0;
    const int NT = vg.NT, nx = vg.nx, ny = vg.ny;
    double* tab = out.tab + r * NTAB * NT;
    double* scal = out.scal + r * RS;
    const double T = s.T;
    const double ist = rsqrt(2.0 * PI * T), A = s.rho * (ist * ist * ist);   // rho (2 pi T)^(-3/2)
    double C[3][6];
    for (int d = 0; d < 3; ++d)
        for (int k = 0; k < 6; ++k) C[d][k] = 0.0;
    // reduced grid: the z "nodes" are the planes G (p = 0) and H (p = 1); integrating the separable form
    // over xi_z (u_z = r_z = 0 and no xz / yz stress in a flow without z dependence) leaves the same form
    // with the plane values E_z = int xi_z^{2p} e_z dxi_z = sqrt(2 pi T) (1, T), C_z = 0 and
    // C2_z = (2p + 1) T, the ratio of the Gaussian moments 3T^2 / T and T / 1
    const double sq2piT = 2.0 * PI * T * ist;
    const double i2T = 0.5 / T;   // exp(-c^2 / (2T)) as exp(-c^2 * i2T): one division per record, not per node
#pragma unroll
    for (int d = 0; d < 3; ++d) {   // the axes' node ranges in turn (static axis index for the sums)
        const int lo = d == 0 ? 0 : (d == 1 ? nx : nx + ny), hi = d == 0 ? nx : (d == 1 ? nx + ny : NT);
        if (vg.reduced && d == 2) continue;
        for (int idx = lo + sl; idx < hi; idx += LPR) {
            const double c = vg.xi[idx] - s.u[d], c2 = c * c;
            const double e = exp(-c2 * i2T);
            if (valid) tab[idx] = e;
            // e c^k for k = 0..5
            const double e1 = e * c, e2 = e * c2, e3 = e1 * c2;
            C[d][0] += e;
            C[d][1] += e1;
            C[d][2] += e2;
            C[d][3] += e3;
            C[d][4] = fma(e2, c2, C[d][4]);
            C[d][5] = fma(e3, c2, C[d][5]);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < 6; ++k) C[d][k] = group_sum<LPR>(C[d][k]);
    if (vg.reduced) {   // exact xi_z integrals int c_z^k e_z dxi_z of the Gaussian (k = 0..5)
        const double zk[6] = {1.0, 0.0, T, 0.0, 3.0 * T * T, 0.0};
        for (int k = 0; k < 6; ++k) C[2][k] = sq2piT * zk[k];
    }
    double alpha[5] = {0, 0, 0, 0, 0};
    if (s.correct) correction_coefs(s, C, vg.w * A, alpha);
    const double p0 = s.p0 + alpha[0];
    double pp[3], p2d[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        pp[d] = s.p[d] + alpha[1 + d];
        p2d[d] = s.P2[d] + alpha[4];
    }
    if (valid && sl == 0) {
        scal[RS_P0] = p0;
        scal[RS_P2XY] = s.P2[3];
        scal[RS_P2XZ] = s.P2[4];
        scal[RS_P2YZ] = s.P2[5];
        scal[RS_OFFD] = (s.P2[3] != 0.0 || s.P2[4] != 0.0 || s.P2[5] != 0.0) ? 1.0 : 0.0;
        scal[RS_AMP] = A;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            scal[RS_U + d] = s.u[d];
            scal[RS_P + d] = pp[d];
            scal[RS_P2D + d] = p2d[d];
            scal[RS_R + d] = s.r[d];
#pragma unroll
            for (int k = 0; k < 6; ++k) scal[RS_SUMS + 6 * d + k] = C[d][k];
        }
    }
    __syncwarp();   // the record's values written by other lanes of the group are read below
    if (valid) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int lo = d == 0 ? 0 : (d == 1 ? nx : nx + ny), hi = d == 0 ? nx : (d == 1 ? nx + ny : NT);
            for (int idx = lo + sl; idx < hi; idx += LPR) {
                double E, c, c2;
                if (vg.reduced && d == 2) {
                    const int p = idx - nx - ny;
                    E = p ? sq2piT * T : sq2piT;
                    c = 0.0;
                    c2 = p ? 3.0 * T : T;
                } else {
                    E = tab[idx];
                    c = vg.xi[idx] - s.u[d];
                    c2 = c * c;
                }
                if (d == 0) E *= A;
                const double v[NTAB] = {E, fma(pp[d], c, p2d[d] * c2), c, c2, s.r[d] * c};
#pragma unroll
                for (int t = 0; t < NTAB; ++t) tab[t * NT + idx] = v[t];
                if (out.tabf) {   // FP32 copies in stored units: E_x carries the VDF storage scale once
                    float* tf = out.tabf + r * NTAB * NT;
#pragma unroll
                    for (int t = 0; t < NTAB; ++t) tf[t * NT + idx] = (float)(t == 0 && d == 0 ? v[t] * vg.vscale : v[t]);
                }
            }
        }
        if (out.scalf)
            for (int q = sl; q <= RS_OFFD; q += LPR) out.scalf[r * RS + q] = (float)scal[q];
    }
}

// ---------------------------------------------------------------------------- records of lines
// The records of a flat line of cells (face_nd = 1): the correction system in the
// conserved quantities, entry by entry from the terms of its polynomials, and a pivoted
// elimination.  The line's synthetic solve amplifies a difference in the last bit
// (mu_of in macro.cu), so its records keep these operations and their order, where other
// meshes take the shorter form above.  LPR lanes build one record.  The axis sums are
// eight partial sums per axis, over the nodes i, i + 8, ..., whatever LPR: with 32 lanes
// those 8 d + i have axis d and each lane one of the 30 entries of the system, with 8 every
// lane its share of each axis and four entries.  50 to 87 us a launch with 8; 25 for
// the short form.
struct Term { double c; int a, b, d; };

__device__ static int psi_terms(int row, const double* u, Term* t, double scale) {
    // psi_row in powers of c (c = xi - u); scale = 1 for psi, 2 for phi_4 only
    switch (row) {
        case 0: t[0] = {1.0, 0, 0, 0}; return 1;
        case 1: t[0] = {1.0, 1, 0, 0}; t[1] = {u[0], 0, 0, 0}; return 2;
        case 2: t[0] = {1.0, 0, 1, 0}; t[1] = {u[1], 0, 0, 0}; return 2;
        case 3: t[0] = {1.0, 0, 0, 1}; t[1] = {u[2], 0, 0, 0}; return 2;
        default: {
            double h = 0.5 * scale;
            t[0] = {h, 2, 0, 0}; t[1] = {h, 0, 2, 0}; t[2] = {h, 0, 0, 2};
            t[3] = {scale * u[0], 1, 0, 0}; t[4] = {scale * u[1], 0, 1, 0}; t[5] = {scale * u[2], 0, 0, 1};
            t[6] = {h * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), 0, 0, 0};
            return 7;
        }
    }
}

// Terms of the base polynomial with a nonzero coefficient.
__device__ static int base_terms(const RecSpec& s, Term* t) {
    const Term all[19] = {
        {s.p0, 0, 0, 0},
        {s.p[0], 1, 0, 0}, {s.p[1], 0, 1, 0}, {s.p[2], 0, 0, 1},
        {s.P2[0], 2, 0, 0}, {s.P2[1], 0, 2, 0}, {s.P2[2], 0, 0, 2},
        {2.0 * s.P2[3], 1, 1, 0}, {2.0 * s.P2[4], 1, 0, 1}, {2.0 * s.P2[5], 0, 1, 1},
        {s.r[0], 3, 0, 0}, {s.r[0], 1, 2, 0}, {s.r[0], 1, 0, 2},
        {s.r[1], 2, 1, 0}, {s.r[1], 0, 3, 0}, {s.r[1], 0, 1, 2},
        {s.r[2], 2, 0, 1}, {s.r[2], 0, 2, 1}, {s.r[2], 0, 0, 3}};
    int n = 0;
    for (int i = 0; i < 19; ++i)
        if (all[i].c != 0.0) t[n++] = all[i];
    return n;
}

__device__ static double poly_moment(const Term* t1, int n1, const Term* t2, int n2, const double (*Cs)[6]) {
    double s = 0.0;
    for (int i = 0; i < n1; ++i)
        for (int j = 0; j < n2; ++j)
            s += t1[i].c * t2[j].c * (Cs[0][t1[i].a + t2[j].a] * Cs[1][t1[i].b + t2[j].b] * Cs[2][t1[i].d + t2[j].d]);
    return s;
}

// Solve A x = b (5x5) by Gaussian elimination with partial pivoting.
__device__ static void solve5(double A[5][5], double b[5], double x[5]) {
    for (int col = 0; col < 5; ++col) {
        int piv = col;
        double best = fabs(A[col][col]);
        for (int r = col + 1; r < 5; ++r)
            if (fabs(A[r][col]) > best) { best = fabs(A[r][col]); piv = r; }
        if (piv != col) {
            for (int k = 0; k < 5; ++k) { double t = A[col][k]; A[col][k] = A[piv][k]; A[piv][k] = t; }
            double t = b[col]; b[col] = b[piv]; b[piv] = t;
        }
        for (int r = col + 1; r < 5; ++r) {
            double m = A[r][col] / A[col][col];
            for (int k = col; k < 5; ++k) A[r][k] -= m * A[col][k];
            b[r] -= m * b[col];
        }
    }
    for (int r = 4; r >= 0; --r) {
        double s = b[r];
        for (int k = r + 1; k < 5; ++k) s -= A[r][k] * x[k];
        x[r] = s / A[r][r];
    }
}

// Conserved moments (rho, rho u, rho E) of a state.
__device__ static void cons_of(double rho, const double* u, double T, double* U) {
    U[0] = rho;
    U[1] = rho * u[0]; U[2] = rho * u[1]; U[3] = rho * u[2];
    U[4] = rho * (1.5 * T + 0.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
}

template <int LPR>
__global__ void k_build_records_line(const RecSpec* __restrict__ specs, int nrec, int n0, Records out0, Records out1,
                                     VGridDev vg) {
    constexpr int AXES = LPR == 32 ? 1 : 3, SLOTS = LPR == 32 ? 1 : 4;   // axes and entries of the system per lane
    const int lane = threadIdx.x & (LPR - 1);
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp * (32 / LPR) >= nrec) return;   // (whole warps)
    const int r0 = warp * (32 / LPR) + (threadIdx.x & 31) / LPR;
    const bool valid = r0 < nrec;   // groups past the end compute a copy and store nothing
    const int rr = valid ? r0 : nrec - 1;
    const RecSpec s = specs[rr];
    const Records& out = rr < n0 ? out0 : out1;
    const long long r = rr < n0 ? rr : rr - n0;
    const int NT = vg.NT, nx = vg.nx, ny = vg.ny;
    double* tab = out.tab + r * NTAB * NT;
    double* scal = out.scal + r * RS;
    const double T = s.T;
    const double A = s.rho * pow(2.0 * PI * T, -1.5);
    const double sq2piT = sqrt(2.0 * PI * T);   // (the reduced grid's planes: see k_build_records)
    const double i2T = 0.5 / T;
    double part[AXES][6];
#pragma unroll
    for (int q = 0; q < AXES; ++q) {
        const int d = LPR == 32 ? lane >> 3 : q;
#pragma unroll
        for (int k = 0; k < 6; ++k) part[q][k] = 0.0;
        if (d > 2) continue;
        const int lo = d == 0 ? 0 : (d == 1 ? nx : nx + ny), hi = d == 0 ? nx : (d == 1 ? nx + ny : NT);
        for (int idx = lo + (lane & 7); idx < hi; idx += 8) {
            if (vg.reduced && d == 2) {
                const int p = idx - nx - ny;
                if (valid) {
                    tab[idx] = p ? sq2piT * T : sq2piT;
                    tab[2 * NT + idx] = 0.0;
                    tab[3 * NT + idx] = p ? 3.0 * T : T;
                }
                continue;
            }
            const double c = vg.xi[idx] - s.u[d];
            const double e = exp(-(c * c) * i2T);
            if (valid) {
                tab[idx] = e;
                tab[2 * NT + idx] = c;
                tab[3 * NT + idx] = c * c;
            }
            double pw = e;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                part[q][k] += pw;
                pw *= c;
            }
        }
    }
    double Cs[3][6];
#pragma unroll
    for (int q = 0; q < AXES; ++q)
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            double v = part[q][k];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, 8);
            if (LPR == 32) {
#pragma unroll
                for (int d = 0; d < 3; ++d) Cs[d][k] = __shfl_sync(0xffffffffu, v, 8 * d);
            } else {
                Cs[q][k] = v;
            }
        }
    if (vg.reduced) {   // exact xi_z integrals int c_z^k e_z dxi_z of the Gaussian (k = 0..5)
        const double zk[6] = {1.0, 0.0, T, 0.0, 3.0 * T * T, 0.0};
        for (int k = 0; k < 6; ++k) Cs[2][k] = sq2piT * zk[k];
    }
    double alpha[5] = {0, 0, 0, 0, 0};
    if (s.correct) {
        Term tp[7], tq[19];
        const double wa = vg.w * A;
        double U[5];
        cons_of(s.rho, s.u, T, U);
        double mine[SLOTS];   // entries 0-4: right-hand side, 5-29: the matrix by rows
#pragma unroll
        for (int m = 0; m < SLOTS; ++m) {
            const int e = lane + LPR * m;
            mine[m] = 0.0;
            if (e < 5) {
                const int na = psi_terms(e, s.u, tp, 1.0);
                const int nb = base_terms(s, tq);
                mine[m] = U[e] - wa * poly_moment(tp, na, tq, nb, Cs);
            } else if (e < 30) {
                const int ra = (e - 5) / 5, rb = (e - 5) % 5;
                const int na = psi_terms(ra, s.u, tp, 1.0);
                const int nbb = psi_terms(rb, s.u, tq, rb == 4 ? 2.0 : 1.0);
                mine[m] = wa * poly_moment(tp, na, tq, nbb, Cs);
            }
        }
        __syncwarp();
        double Am[5][5], rhs[5];
#pragma unroll
        for (int e = 0; e < 30; ++e) {
            const double v = __shfl_sync(0xffffffffu, mine[e / LPR], e % LPR, LPR);
            if (e < 5) rhs[e] = v;
            else Am[(e - 5) / 5][(e - 5) % 5] = v;
        }
        solve5(Am, rhs, alpha);
    }
    double pp[3] = {s.p[0], s.p[1], s.p[2]};
    double p2d[3] = {s.P2[0], s.P2[1], s.P2[2]};
    double p0 = s.p0;
    if (s.correct) {
        const double ua = alpha[1] * s.u[0] + alpha[2] * s.u[1] + alpha[3] * s.u[2];
        const double u2 = s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2];
        p0 = s.p0 + alpha[0] + ua + alpha[4] * u2;
        for (int q = 0; q < 3; ++q) {
            pp[q] = s.p[q] + alpha[1 + q] + 2.0 * alpha[4] * s.u[q];
            p2d[q] = s.P2[q] + alpha[4];
        }
    }
    if (valid && lane == 0) {
        scal[RS_P0] = p0;
        scal[RS_P2XY] = s.P2[3];
        scal[RS_P2XZ] = s.P2[4];
        scal[RS_P2YZ] = s.P2[5];
        scal[RS_OFFD] = (s.P2[3] != 0.0 || s.P2[4] != 0.0 || s.P2[5] != 0.0) ? 1.0 : 0.0;
    }
    __syncwarp();   // the record's values written by other lanes are read below
    if (!valid) return;
    for (int idx = lane; idx < NT; idx += LPR) {
        const int q = idx < nx ? 0 : (idx < nx + ny ? 1 : 2);
        const double pq = q == 0 ? pp[0] : (q == 1 ? pp[1] : pp[2]), p2q = q == 0 ? p2d[0] : (q == 1 ? p2d[1] : p2d[2]);
        const double c = tab[2 * NT + idx];
        tab[NT + idx] = pq * c + p2q * tab[3 * NT + idx];   // C2 = c^2 (plane value if reduced)
        tab[4 * NT + idx] = s.r[q] * c;
        if (q == 0) tab[idx] *= A;
        if (out.tabf) {   // FP32 copies in stored units: E_x carries the VDF storage scale once
            float* tf = out.tabf + r * NTAB * NT;
            for (int t = 0; t < NTAB; ++t)
                tf[t * NT + idx] = (float)(t == 0 && q == 0 ? tab[idx] * vg.vscale : tab[t * NT + idx]);
        }
    }
    if (out.scalf && lane <= RS_OFFD) out.scalf[r * RS + lane] = (float)scal[lane];
}

// Records [0, n0) into out0 and the rest into out1.  A record per warp while the
// warps leave sub-partitions idle (2,048 records: about three warps each), four
// above.
static void build_records(const RecSpec* d_specs, int nrec, int n0, const Records& out0, const Records& out1,
                          const VGridDev& vg, cudaStream_t st) {
    if (nrec <= 0) return;
    const int threads = 64;
    if (nrec <= 2048) {
        const int blocks = (nrec * 32 + threads - 1) / threads;
        k_build_records<32><<<blocks, threads, 0, st>>>(d_specs, nrec, n0, out0, out1, vg);
    } else {
        const int blocks = ((nrec + 3) / 4 * 32 + threads - 1) / threads;
        k_build_records<8><<<blocks, threads, 0, st>>>(d_specs, nrec, n0, out0, out1, vg);
    }
}

// Context-free launcher of the record builder (caller supplies every buffer).
void build_records_raw(const RecSpec* d_specs, int nrec, const Records& out, const VGridDev& vg, cudaStream_t st) {
    build_records(d_specs, nrec, nrec, out, out, vg, st);
}

// Records up to which a line's have a warp each: a few leave SMs idle (30 cells 2.27 ms a
// case, 2.33 with four to a warp); more fill the FP64 pipes, which four to a warp
// share (64 shocks of 100 to 800 cells 126 ms, 134 with a warp each).
constexpr int LINE_WARP_RECORDS = 304;
// Records of a context's own solve (records [0, n0) into out0, the rest into out1).
static void solve_records(gsis_ctx* c, int nrec, int n0, const Records& out0, const Records& out1, const RecSpec* d_specs) {
    if (nrec <= 0) return;
    if (c->face_nd == 1 && nrec <= LINE_WARP_RECORDS)
        k_build_records_line<32><<<(nrec + 1) / 2, 64, 0, c->stream>>>(d_specs, nrec, n0, out0, out1, c->vg);
    else if (c->face_nd == 1)
        k_build_records_line<8><<<(nrec + 7) / 8, 64, 0, c->stream>>>(d_specs, nrec, n0, out0, out1, c->vg);
    else build_records(d_specs, nrec, n0, out0, out1, c->vg, c->stream);
    c->launches++;
}

void launch_build_records(gsis_ctx* c, const Records& out, int nrec, const RecSpec* d_specs) {
    solve_records(c, nrec, nrec, out, out, d_specs);
}

// ---------------------------------------------------------------------------- spec builders
__device__ static void spec_maxwellian(RecSpec& s, double rho, const double* u, double T, int correct) {
    s.rho = rho; s.T = T;
    for (int d = 0; d < 3; ++d) { s.u[d] = u[d]; s.p[d] = 0.0; s.r[d] = 0.0; }
    for (int k = 0; k < 6; ++k) s.P2[k] = 0.0;
    s.p0 = 1.0;
    s.correct = correct;
}

// Shakhov reference state of each DVM cell from W^n and the heat flux of f^n
// about u^n (third moment stored by the moments pass), tau = mu(T)/p, and the
// diffuse-wall densities from the lagged outgoing half-range fluxes.
__global__ void k_cell_eq(int Nd, const int* __restrict__ dvm_cell, const double* __restrict__ W,
                          const double* __restrict__ mom, const int* __restrict__ side_bc,
                          const double* __restrict__ wall_den, double mu0, double omega,
                          RecSpec* specs, double* itau, double* rho_w, float* itauf, float* rho_wf) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Nd) return;
    const int c = dvm_cell[k];
    const double rho = W[c * 5], T = W[c * 5 + 4];
    const double u[3] = {W[c * 5 + 1], W[c * 5 + 2], W[c * 5 + 3]};
    const double* m = mom + (long long)k * MOMN;
    const double q[3] = {0.5 * m[10], 0.5 * m[11], 0.5 * m[12]};
    const double p = rho * T;
    const double sc = 1.0 / (15.0 * p * T * T);
    RecSpec s;
    spec_maxwellian(s, rho, u, T, 1);
    for (int d = 0; d < 3; ++d) { s.p[d] = -5.0 * T * sc * q[d]; s.r[d] = sc * q[d]; }
    specs[k] = s;
    itau[k] = p / viscosity(T, mu0, omega);   // 1/tau, tau = mu(T)/p
    if (itauf) itauf[k] = (float)itau[k];
    for (int sd = 0; sd < 6; ++sd) {
        double v = 0.0;
        if (side_bc[c * 6 + sd] == GSIS_BC_WALL) v = m[13 + sd] / wall_den[c * 6 + sd];
        rho_w[(long long)k * 6 + sd] = v;
        if (rho_wf) rho_wf[(long long)k * 6 + sd] = (float)v;
    }
}

// Factor vectors of g~/tau for the sweep (eval_g in sweep_device.cuh), one
// block per DVM cell, from the cell's record (Eq. updatef's corrected
// Maxwellian tables) and 1/tau; formed in FP64 and stored in the sweep's
// arithmetic type T:
//   x(ix) = (E, E (B + R C2), E R, E C2)             [gx4]
//   y(q)  = E_yz/tau (D + R_yz C2_yz, 1, C2_yz, R_yz)   [gy4]
// so that g~/tau = sum of the four products x_i y_i (the Shakhov record has no
// stress terms, see eval_g).
template <typename T>
__global__ void k_build_gtab(int Nd, Records rec, VGridDev vg, const double* __restrict__ itau,
                             const float* __restrict__ itauf, T* __restrict__ gx4, T* __restrict__ gy4) {
    const int k = blockIdx.x;
    if (k >= Nd) return;
    const int NT = vg.NT, nx = vg.nx, ny = vg.ny, nyz = vg.ny * vg.nz;
    if constexpr (std::is_same<T, float>::value) {
        // FP32 arithmetic for FP32 factor vectors, from the FP32 record copies
        // (whose E_x carries the storage scale; the FP64 form below puts it on
        // the y-z part): the same products rounded once to FP32 become a few
        // rounding steps in FP32, far under the storage rounding, and the FP64
        // pipe (the bound of the FP64 form) is left alone.
        const float* tf = rec.tabf + (long long)k * NTAB * NT;
        const float* sf = rec.scalf + (long long)k * RS;
        const float p0 = sf[RS_P0];
        const float it = itauf[k];
        for (int ix = threadIdx.x; ix < nx; ix += blockDim.x) {
            const float E = tf[ix], B = tf[NT + ix], C2 = tf[3 * NT + ix], R = tf[4 * NT + ix];
            *reinterpret_cast<float4*>(gx4 + ((long long)k * nx + ix) * 4) =
                make_float4(E, E * (B + R * C2), E * R, E * C2);
        }
        for (int q = threadIdx.x; q < nyz; q += blockDim.x) {
            const int iz = q / ny, jy = nx + q - iz * ny, jz = nx + ny + iz;
            const float Eyz = tf[jy] * tf[jz] * it;
            const float D = p0 + (tf[NT + jy] + tf[NT + jz]);
            const float Ryz = tf[4 * NT + jy] + tf[4 * NT + jz];
            const float C2yz = tf[3 * NT + jy] + tf[3 * NT + jz];
            *reinterpret_cast<float4*>(gy4 + ((long long)k * nyz + q) * 4) =
                make_float4(Eyz * (D + Ryz * C2yz), Eyz, Eyz * C2yz, Eyz * Ryz);
        }
        return;
    }
    const double* tab = rec.tab + (long long)k * NTAB * NT;
    const double* sc = rec.scal + (long long)k * RS;
    const double p0 = sc[RS_P0];
    const double it = itau[k];
    for (int ix = threadIdx.x; ix < nx; ix += blockDim.x) {
        const double E = tab[ix], B = tab[NT + ix], C2 = tab[3 * NT + ix], R = tab[4 * NT + ix];
        T* o = gx4 + ((long long)k * nx + ix) * 4;
        o[0] = (T)E;
        o[1] = (T)(E * (B + R * C2));
        o[2] = (T)(E * R);
        o[3] = (T)(E * C2);
    }
    for (int q = threadIdx.x; q < nyz; q += blockDim.x) {
        const int jy = nx + q % ny, jz = nx + ny + q / ny;
        const double Eyz = tab[jy] * tab[jz] * it * vg.vscale;   // g~/tau in stored units
        const double D = p0 + (tab[NT + jy] + tab[NT + jz]);
        const double Ryz = tab[4 * NT + jy] + tab[4 * NT + jz];
        const double C2yz = tab[3 * NT + jy] + tab[3 * NT + jz];
        T* o = gy4 + ((long long)k * nyz + q) * 4;
        o[0] = (T)(Eyz * (D + Ryz * C2yz));
        o[1] = (T)Eyz;
        o[2] = (T)(Eyz * C2yz);
        o[3] = (T)(Eyz * Ryz);
    }
}

void launch_cell_eq(gsis_ctx* c) {
    const int Nd = (int)c->Nd;
    if (Nd == 0) return;
    k_cell_eq<<<(Nd + 127) / 128, 128, 0, c->stream>>>(Nd, c->dvm_cell, c->W, c->mom, c->m.side_bc, c->wall_den,
                                                        c->mu0, c->p.omega, c->specs, c->itau, c->rho_w, c->itauf,
                                                        c->rho_wf);
    c->launches++;
    launch_build_records(c, c->recG, Nd, c->specs);
    if (c->p.vdf_dtype == GSIS_F64)
        k_build_gtab<double><<<Nd, 128, 0, c->stream>>>(Nd, c->recG, c->vg, c->itau, c->itauf, (double*)c->gx4,
                                                        (double*)c->gy4);
    else
        k_build_gtab<float><<<Nd, 128, 0, c->stream>>>(Nd, c->recG, c->vg, c->itau, c->itauf, (float*)c->gx4,
                                                       (float*)c->gy4);
    c->launches++;
}

// Boundary records: far field -> conservation-corrected Maxwellian of the
// boundary state; wall -> unit-density Maxwellian at rest at T_w (emission
// shape, scaled by rho_w in the sweep).
__global__ void k_bc_specs(RecSpec* specs, const int* bc_type, const double* bc_state) {
    const int s = threadIdx.x;
    if (s >= 6) return;
    const double* st = bc_state + s * 5;
    RecSpec r;
    if (bc_type[s] == GSIS_BC_FARFIELD) {
        spec_maxwellian(r, st[0], st + 1, st[4], 1);
    } else if (bc_type[s] == GSIS_BC_WALL) {
        const double z[3] = {0.0, 0.0, 0.0};
        spec_maxwellian(r, 1.0, z, st[4], 0);
    } else {
        const double z[3] = {0.0, 0.0, 0.0};
        spec_maxwellian(r, 1.0, z, 1.0, 0);
    }
    specs[s] = r;
}

void launch_bc_records(gsis_ctx* c) {
    k_bc_specs<<<1, 32, 0, c->stream>>>(c->specs, c->d_bc_type, c->d_bc_state);
    c->launches++;
    launch_build_records(c, c->recBC, 6, c->specs);
}

// Denominator of the diffuse-wall density: sum over incoming velocities
// (xi . S_out <= 0) of w |xi . S_out| M_w, one block per (cell, wall side).
// Also the incoming half-range moments of the wall Maxwellian,
// wall_in[c][s] = sum_{xi.S <= 0} w (xi.S) (1, xi, |xi|^2/2) M_w, so that the
// kinetic wall flux of a face is (outgoing moments) + rho_w * wall_in.
__global__ void k_wall_den(int N, const int* __restrict__ side_bc, const double* __restrict__ Sout,
                           Records bc, VGridDev vg, double* wall_den, double* wall_in) {
    const int c = blockIdx.x;
    __shared__ double sm[32 * 6];
    for (int s = 0; s < 6; ++s) {
        if (side_bc[c * 6 + s] != GSIS_BC_WALL) continue;
        const double* S = Sout + ((long long)c * 6 + s) * 3;
        const double* sc = rec_scal(bc, s);
        const double* tb = rec_tab(bc, s, vg.NT);
        double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (long long v = threadIdx.x; v < vg.Nv; v += blockDim.x) {
            int ix, iy, iz;
            vsplit(v, vg.nx, vg.ny, ix, iy, iz);
            const double x0 = vg.xi[ix], x1 = vg.xi[vg.nx + iy], x2 = vg.xi[vg.nx + vg.ny + iz];
            const double xn = x0 * S[0] + x1 * S[1] + x2 * S[2];
            if (!(xn > 0.0)) {
                const double m = eval_rec(sc, tb, vg.NT, vg.nx, vg.ny, ix, iy, iz);
                const double g = xn * m;
                double psi[5];
                psi_node(vg, x0, x1, x2, iz, psi);
                acc[0] += -g * psi[0];
                acc[1] += g * psi[0];
                acc[2] += g * psi[1];
                acc[3] += g * psi[2];
                acc[4] += g * psi[3];
                acc[5] += g * psi[4];
            }
        }
        block_sum<6>(acc, sm);
        if (threadIdx.x == 0) {
            wall_den[c * 6 + s] = acc[0] * vg.w;
            for (int q = 0; q < 5; ++q) wall_in[((long long)c * 6 + s) * 5 + q] = acc[1 + q] * vg.w;
        }
    }
}

void launch_wall_den(gsis_ctx* c) {
    k_wall_den<<<c->m.N, 256, 0, c->stream>>>(c->m.N, c->m.side_bc, c->m.Sout, c->recBC, c->vg, c->wall_den,
                                              c->wall_in);
    c->launches++;
}

// Grad-13 interface distributions (Eq. G13_VDF) of NS cells next to DVM
// cells, from W^n and the NSF stress / heat flux at W^n, conservation-corrected.
__device__ static void spec_grad13(RecSpec& s, const double* Wc, const double* nsf9) {
    const double rho = Wc[0], T = Wc[4];
    const double u[3] = {Wc[1], Wc[2], Wc[3]};
    spec_maxwellian(s, rho, u, T, 1);
    const double rT2 = rho * T * T;
    for (int d = 0; d < 3; ++d) {
        const double q = nsf9[6 + d];
        s.p[d] = -q / rT2;
        s.r[d] = q / (5.0 * rT2 * T);
    }
    for (int k = 0; k < 6; ++k) s.P2[k] = nsf9[k] / (2.0 * rT2);
}

__global__ void k_ghost_specs(int ng, const int* __restrict__ ghost_cell, const double* __restrict__ W,
                              const double* __restrict__ nsf, RecSpec* specs) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    const int c = ghost_cell[g];
    RecSpec s;
    spec_grad13(s, W + c * 5, nsf + (long long)c * HOTN);
    specs[g] = s;
}

void launch_ghost_records(gsis_ctx* c) {
    if (c->n_ghost == 0) return;
    k_ghost_specs<<<(c->n_ghost + 127) / 128, 128, 0, c->stream>>>(c->n_ghost, c->ghost_cell, c->W, c->nsf, c->specs);
    c->launches++;
    launch_build_records(c, c->recGhost, c->n_ghost, c->specs);
}

// M~(W^{n+1}) and M~(W^{n+1/2}) for Eq. updatef: specs [0, Nd) and [Nd, 2 Nd).
__global__ void k_corr_specs(int Nd, const int* __restrict__ dvm_cell, const double* __restrict__ Wnew,
                             const double* __restrict__ Whalf, RecSpec* specs) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 2 * Nd) return;
    const double* w = k < Nd ? Wnew + dvm_cell[k] * 5 : Whalf + dvm_cell[k - Nd] * 5;
    const double u[3] = {w[1], w[2], w[3]};
    RecSpec s;
    spec_maxwellian(s, w[0], u, w[4], 1);
    specs[k] = s;
}

void launch_correction_records(gsis_ctx* c) {
    const int Nd = (int)c->Nd;
    if (Nd == 0) return;
    k_corr_specs<<<(2 * Nd + 127) / 128, 128, 0, c->stream>>>(Nd, c->dvm_cell, c->W, c->Wh, c->specs);
    c->launches++;
    solve_records(c, 2 * Nd, Nd, c->recNew, c->recHalf, c->specs);
}

// Seed distributions for cells entering the DVM region: Grad-13 from W and
// its NSF stress / heat flux (adaptive start, Sec. 3.2) or the corrected
// Maxwellian M~(W) (all-kinetic start), into recNew slots of the new list.
__global__ void k_seed_specs(int ne, const int* __restrict__ enter, const int* __restrict__ dvm_cell,
                             const double* __restrict__ W, const double* __restrict__ nsf, int grad13,
                             RecSpec* specs) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ne) return;
    const int c = dvm_cell[enter[e]];
    RecSpec s;
    if (grad13) {
        spec_grad13(s, W + c * 5, nsf + (long long)c * HOTN);
    } else {
        const double u[3] = {W[c * 5 + 1], W[c * 5 + 2], W[c * 5 + 3]};
        spec_maxwellian(s, W[c * 5], u, W[c * 5 + 4], 1);
    }
    specs[e] = s;
}

void launch_seed_records(gsis_ctx* c, int ne, int grad13) {
    if (ne == 0) return;
    k_seed_specs<<<(ne + 127) / 128, 128, 0, c->stream>>>(ne, c->enter_list, c->dvm_cell, c->W, c->nsf, grad13,
                                                           c->specs);
    c->launches++;
    launch_build_records(c, c->recNew, ne, c->specs);
}


// ---------------------------------------------------------------------------- two-VDF reference pair
// Reference pair of Eq. general_model, g = (1 - 1/Z_r) g_t + g_r / Z_r for
// f0 and f1, for states S[n][12] = (rho, u (3), T_t, T_r, q_t (3), q_r (3)) on
// a full 3D grid.  Four conservation-corrected records per state: the
// Shakhov forms g_0t at (T_t, q_t) and g_0r at (T, q0), each corrected to its
// own translational energy, and the Maxwellians M~ at T_t and at T; per node
//   g0 = a g_0t + b g_0r,
//   g1 = a [(d_r/2) T_r g_0t + M~_t (q_r.c)/(rho T_t)] + b [(d_r/2) T g_0r + M~_T (q1.c)/(rho T)],
// a = 1 - 1/Z_r, b = 1/Z_r, T = (3 T_t + d_r T_r)/(3 + d_r) and (q0, q1) the
// mixing of (q_t, q_r) of Sec. 2 (g_1t and g_1r with R = 1: their
// Maxwellian factor is rho^-1 times that of g_0t, g_0r).
__device__ static void two_vdf_mix(const TwoVdfGas& g, const double* qt, const double* qr, double* q0, double* q1) {
    const double m00 = (2.0 - 3.0 * g.A[0]) * g.Zr + 1.0, m01 = -3.0 * g.A[1] * g.Zr;
    const double m10 = -g.A[2] * g.Zr, m11 = -g.A[3] * g.Zr + 1.0;
    for (int d = 0; d < 3; ++d) {
        q0[d] = m00 * qt[d] + m01 * qr[d];
        q1[d] = m10 * qt[d] + m11 * qr[d];
    }
}

__device__ static RecSpec spec_shakhov(double rho, const double* u, double T, const double* q) {
    RecSpec s;
    spec_maxwellian(s, rho, u, T, 1);
    const double sc = 1.0 / (15.0 * rho * T * T * T);   // 1/(15 p T^2), p = rho T
    for (int d = 0; d < 3; ++d) { s.p[d] = -5.0 * T * sc * q[d]; s.r[d] = sc * q[d]; }
    return s;
}

__global__ void k_two_vdf_specs(int n, const double* __restrict__ S, TwoVdfGas g, RecSpec* __restrict__ specs) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double* s = S + (long long)k * 12;
    const double rho = s[0], Tt = s[4], Tr = s[5];
    const double T = (3.0 * Tt + g.d_r * Tr) / (3.0 + g.d_r);
    double q0[3], q1[3];
    two_vdf_mix(g, s + 6, s + 9, q0, q1);
    RecSpec m;
    specs[4 * k + 0] = spec_shakhov(rho, s + 1, Tt, s + 6);
    specs[4 * k + 1] = spec_shakhov(rho, s + 1, T, q0);
    spec_maxwellian(m, rho, s + 1, Tt, 1);
    specs[4 * k + 2] = m;
    spec_maxwellian(m, rho, s + 1, T, 1);
    specs[4 * k + 3] = m;
}

// out[k][0][v] = g0, out[k][1][v] = g1.  grid (x: row blocks, y: state).
// On one x-row (fixed c_y, c_z) all four records are cubic polynomials of c_x
// times one of two Gaussians of c_x (T_t and T; the Maxwellian and Shakhov
// records of one temperature share it), so
//   g0 = e_t(x) (a0 + a1 c_x + a2 c_x^2 + a3 c_x^3) + e_r(x) (b0 + ...),  g1 likewise,
// with 16 coefficients per row, formed once per block in shared memory (everything
// that depends on y and z, the factors of the mixing and E_y E_z included).  A
// thread keeps one ix and walks the rows: 16 FP64 operations per node (Horner's
// rule) for both outputs, against 43 for the four records evaluated apart.  FP64
// bound: 1,110 us before, for 96 states of 48 x 48 x 24 nodes.
constexpr int TV_THREADS = 256;

__global__ void __launch_bounds__(TV_THREADS) k_two_vdf_eval(int n, const double* __restrict__ S, TwoVdfGas g,
                                                             Records rec, VGridDev vg, int rows_per_block,
                                                             double* __restrict__ out) {
    extern __shared__ double2 sh_coef[];   // [rows_per_block][8]: (g0_t, g0_r, g1_t, g1_r) of c_x^0..3 in pairs
    const int k = blockIdx.y;
    if (k >= n) return;
    const int nx = vg.nx, ny = vg.ny, NT = vg.NT, rows = ny * vg.nz;
    const int row0 = blockIdx.x * rows_per_block, nr = min(rows_per_block, rows - row0);
    const double* s = S + (long long)k * 12;
    const double rho = s[0], Tt = s[4], Tr = s[5];
    const double T = (3.0 * Tt + g.d_r * Tr) / (3.0 + g.d_r);
    double q0[3], q1[3];
    two_vdf_mix(g, s + 6, s + 9, q0, q1);
    const double wt = 1.0 - 1.0 / g.Zr, wr = 1.0 / g.Zr;
    const double* sc = rec.scal + (long long)4 * k * RS;
    const double* tb = rec.tab + (long long)4 * k * NTAB * NT;
    const long long TS = (long long)NTAB * NT;
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
        const int q = row0 + r, iz = q / ny, jy = nx + q - iz * ny, jz = nx + ny + iz;
        double co[16];
#pragma unroll
        for (int t = 0; t < 2; ++t) {   // temperature T_t, then T: Shakhov record t, Maxwellian record 2 + t
            const double *cs = sc + t * RS, *cm = sc + (2 + t) * RS, *ts = tb + t * TS, *tm = tb + (2 + t) * TS;
            const double w = t == 0 ? wt : wr, Th = t == 0 ? Tt : T, iRT = w / (rho * Th);
            const double h = 0.5 * g.d_r * (t == 0 ? Tr : T);
            const double e = ts[jy] * ts[jz], cy = ts[2 * NT + jy], cz = ts[2 * NT + jz];
            const double c2 = ts[3 * NT + jy] + ts[3 * NT + jz], ry = ts[4 * NT + jy] + ts[4 * NT + jz];
            const double G[4] = {w * e * (cs[RS_P0] + (ts[NT + jy] + ts[NT + jz]) + ry * c2),
                                 w * e * fma(cs[RS_R], c2, cs[RS_P]), w * e * (cs[RS_P2D] + ry), w * e * cs[RS_R]};
            const double m0 = e * (cm[RS_P0] + (tm[NT + jy] + tm[NT + jz])), m1 = e * cm[RS_P], m2 = e * cm[RS_P2D];
            const double* qv = t == 0 ? s + 9 : q1;
            const double qx = iRT * qv[0], qyz = iRT * fma(qv[1], cy, qv[2] * cz);
            const double Q[4] = {m0 * qyz, fma(m0, qx, m1 * qyz), fma(m1, qx, m2 * qyz), m2 * qx};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                co[4 * t + i] = G[i];
                co[8 + 4 * t + i] = fma(h, G[i], Q[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) sh_coef[r * 8 + i] = make_double2(co[2 * i], co[2 * i + 1]);
    }
    __syncthreads();
    // thread: one ix, rows r0, r0 + G, ... (consecutive threads write consecutive values)
    const int xt = min(nx, TV_THREADS), G = TV_THREADS / xt, r0 = threadIdx.x / xt;
    if (r0 >= G) return;
    double* o0 = out + (long long)k * 2 * vg.Nv + (long long)row0 * nx;
    double* o1 = o0 + vg.Nv;
    for (int ix = threadIdx.x % xt; ix < nx; ix += xt) {
        const double c = tb[2 * NT + ix], et = tb[ix], er = tb[TS + ix];
        for (int r = r0; r < nr; r += G) {
            double co[16];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const double2 v = sh_coef[r * 8 + i];
                co[2 * i] = v.x;
                co[2 * i + 1] = v.y;
            }
            double p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                p[i] = fma(fma(fma(co[4 * i + 3], c, co[4 * i + 2]), c, co[4 * i + 1]), c, co[4 * i]);
            o0[(long long)r * nx + ix] = fma(et, p[0], er * p[1]);
            o1[(long long)r * nx + ix] = fma(et, p[2], er * p[3]);
        }
    }
}

void launch_two_vdf_reference(gsis_ctx* c, const double* S, int n, const TwoVdfGas& g, RecSpec* specs,
                              const Records& rec, double* out) {
    if (n <= 0) return;
    k_two_vdf_specs<<<(n + 127) / 128, 128, 0, c->stream>>>(n, S, g, specs);
    c->launches++;
    build_records_raw(specs, 4 * n, rec, c->vg, c->stream);
    c->launches++;
    const int rows = c->vg.ny * c->vg.nz;
    // row blocks: enough for eight blocks per SM, at most 256 rows (32 KB of coefficients), whole thread groups
    const int G = std::max(1, TV_THREADS / c->vg.nx);
    long long per = ((long long)rows * n + 1215) / 1216;
    per = std::min<long long>(256, std::max<long long>(per, 4 * G));
    k_two_vdf_eval<<<dim3((unsigned)((rows + per - 1) / per), n), TV_THREADS, (size_t)per * 16 * sizeof(double), c->stream>>>(
        n, S, g, rec, c->vg, (int)per, out);
    c->launches++;
}

}  // namespace gsis
