// The FP64 kinetic sweep of 2D meshes on velocity columns.
//
// A face of a 2D mesh has no z component, so xi.S -- and with it the outflow
// decisions, the upwind sides, the denominator 1/tau + sum max(xi.S, 0)/V and
// its reciprocal -- depends on (xi_x, xi_y) only.  A thread therefore owns one
// (ix, iy) and ZP consecutive planes iz (a column): all of that is formed
// once per cell and column, and the planes only pay for the limited
// differences.  In an index direction with one inflow and one outflow face
// (every radial pair of an O-grid, nearly every other one), with s1 / s0 the
// neighbour on the inflow / outflow side, s2 the second neighbour on the
// inflow side and x_i, x_o the two faces' xi.S/V, the update is
//   num -= x_o (1/2) minmod(c - s1, s0 - c) + x_i (s1 + (1/2) minmod(s1 - s2, c - s1))
// whichever side is the inflow one: the lane loads s1, s0, s2 from rows picked
// by its own outflow test (7 loads per point instead of 9, no selects).  The
// halves go into x (xi is halved once per thread, exactly), so minmod needs no
// scaling: num -= x'_o mm + x'_i (2 s1 + mm), the low side's term first.  Both faces
// outflow or both inflow (a warp vote): the second one takes the place of the term
// that is missing.  Operations, order and roundings are those of k_sweep, so the results are
// the same to the last bit whichever tile the autotuner picks.
//
// What bounds it: the FP64 pipe (a warp instruction holds it for 64 cycles on
// GB300).  A point costs 17 FP64 operations plus 12 / ZP shared ones; a lane
// per velocity (k_sweep) costs 30.  Measured on the 128 x 128 cylinder, 48 x
// 48 x 24 velocities, 10,482 DVM cells, ms per pass pair: lane per velocity
// 81.8 (97.9 before the limiter's absolute values left the FP64 pipe, see
// mag_bits), columns of two planes 70.2, of three 57.6, of four 52.6 at three
// blocks per SM (at two, 432 blocks take two waves); 51.6 with the outflow
// term first whichever side is low, which rounds differently.
// FP32 arithmetic gains nothing here (7.1 ms against 6.9 for the velocity
// pairs: it waits for loads, not for arithmetic) and keeps its own tiles.
#include "sweep_device.cuh"

namespace gsis {

// max(x, 0) on the integer pipe
__device__ __forceinline__ double pos_part(double x) { return pos_t<double>(x) ? x : 0.0; }

// A lane's column: (ix, iy) and the planes iz0 .. iz0 + ZP - 1.  Past the end
// of the grid the position and the planes are clamped (loads stay in bounds)
// and nothing is stored.
template <int ZP>
struct Column {
    char* fz[ZP];        // address of the column's values in row 0 of the VDF
    int ix, iy, iz0, q[ZP];   // q = iy + ny iz
    double x0, x1;            // half of xi_x, xi_y
    int nact;            // planes to store (0: clamped position)
    unsigned mask;       // the lanes that share this lane's cell
};

template <int ZP, int P>
__device__ __forceinline__ void make_column(const VGridDev& vg, double* f, int ptile, int ztile, int lane, Column<ZP>& C) {
    const int nxy = vg.nx * vg.ny;
    C.mask = P == 32 ? 0xffffffffu : ((1u << (P & 31)) - 1u) << (lane & ~(P - 1));
    const int pp = ptile * P + (lane & (P - 1)), p = min(pp, nxy - 1), iz0 = ztile * ZP;
    C.iz0 = iz0;
    C.iy = p / vg.nx;
    C.ix = p - C.iy * vg.nx;
    C.nact = pp < nxy ? min(ZP, vg.nz - iz0) : 0;
    C.x0 = 0.5 * vg.xi[C.ix];
    C.x1 = 0.5 * vg.xi[vg.nx + C.iy];
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        const int iz = min(iz0 + u, vg.nz - 1);
        C.q[u] = C.iy + vg.ny * iz;
        C.fz[u] = reinterpret_cast<char*>(f + (p + (long long)nxy * iz));
    }
}

// Value of a boundary or interface record on the column's planes.
template <int ZP>
__device__ __forceinline__ void column_record(const SweepArgs& a, const Records& R, int r, double scale,
                                              const Column<ZP>& C, double* out) {
    const double* sc = RecT<double>::scal(R, r);
    const double* tab = RecT<double>::tab(R, r, a.vg.NT);
#pragma unroll
    for (int u = 0; u < ZP; ++u)
        out[u] = scale * eval_recT<double>(sc, tab, a.vg.NT, a.vg.nx, a.vg.ny, C.ix, C.iy, min(C.iz0 + u, a.vg.nz - 1));
}

// One cell's stencil on a column, and the column's coefficients.
template <int ZP>
struct Stencil {
    double c0[ZP], s1[2][ZP], s0[2][ZP], s2[2][ZP];
    // halved coefficients: outflow, inflow face, a second face (both outflow: the high one, > 0; both inflow: the
    // high one, < 0; else 0); the denominator
    double xo[2], xi[2], xe[2], den;
    bool oL[2];                   // the low side is the outflow side
};

// base + row * row_bytes in one instruction
__device__ __forceinline__ const char* row_at(const char* base, int row, unsigned row_bytes) {
    const char* r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(row), "r"(row_bytes), "l"(base));
    return r;
}

// Coefficients and loads of cell k (rows picked by the outflow test; a side
// that is not a DVM side repeats the cell).
template <int ZP>
__device__ __forceinline__ void column_load(int k, const CellMeta<double, 2>& m, const Column<ZP>& C,
                                            unsigned row_bytes, Stencil<ZP>& q) {
    auto at = [&](int row, int u) { return *reinterpret_cast<const double*>(row_at(C.fz[u], row, row_bytes)); };
    const bool interior = m.kinds < 0;
    double den = m.it;
#pragma unroll
    for (int u = 0; u < ZP; ++u) q.c0[u] = at(k, u);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        double xL = fma(C.x1, m.S[2 * d][1], C.x0 * m.S[2 * d][0]);
        double xH = fma(C.x1, m.S[2 * d + 1][1], C.x0 * m.S[2 * d + 1][0]);
        int rL = m.rf[2 * d], rH = m.rf[2 * d + 1], nL = m.n2[2 * d], nH = m.n2[2 * d + 1];
        if (!interior) {
            const int kl = side_kind(m.kinds, 2 * d), kh = side_kind(m.kinds, 2 * d + 1);
            if (kl == SK_NONE) xL = 0.0;
            if (kh == SK_NONE) xH = 0.0;
            if (kl != SK_DVM) rL = nL = k;
            if (kh != SK_DVM) rH = nH = k;
        }
        const bool oL = pos_t<double>(xL);
        const double mH = pos_part(xH), iH = pos_t<double>(xH) ? 0.0 : xH;
        const double xo = oL ? xL : mH, xe = oL ? mH : iH;
        den = fma(2.0, xo, den);
        if (__any_sync(C.mask, oL && xe != 0.0)) {   // (the low face first, as the general update)
            if (oL) den = fma(2.0, xe, den);
        }
        q.oL[d] = oL;
        q.xo[d] = xo;
        q.xi[d] = oL ? iH : xL;
        q.xe[d] = xe;
        const int r1 = oL ? rH : rL, r0 = oL ? rL : rH, r2 = oL ? nH : nL;
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            q.s1[d][u] = at(r1, u);
            q.s0[d][u] = at(r0, u);
            q.s2[d][u] = at(r2, u);
        }
    }
    q.den = den;
}

// The update of cell k from its stencil, stored.
template <int ZP>
__device__ __forceinline__ void column_apply(const SweepArgs& a, int k, const CellMeta<double, 2>& m,
                                             const Column<ZP>& C, unsigned row_bytes, const Stencil<ZP>& q) {
    const bool interior = m.kinds < 0;
    double num[ZP];
    {   // g~ / tau: four products of the x and y-z factor vectors (eval_g)
        const int kx = k * a.vg.nx + C.ix, ky = k * (a.vg.ny * a.vg.nz);
        const V4<double> x = ld4(static_cast<const double*>(a.gx4) + 4 * (long long)kx);
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            const V4<double> y = ld4(static_cast<const double*>(a.gy4) + 4 * (long long)(ky + C.q[u]));
            num[u] = fma(x.w, y.w, fma(x.z, y.z, fma(x.y, y.y, x.x * y.x)));
        }
    }
    const double rden = recip_t<double>(q.den);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        // the own limited slope towards the outflow face (zero where a side repeats the cell) and the inflow face
        // value (a boundary or interface side has its distribution instead)
        double dn[ZP], dq[ZP], own[ZP], fin[ZP];
        double co = q.xo[d], ci = q.xi[d];
        const bool oL = q.oL[d];
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            dn[u] = q.c0[u] - q.s1[d][u];
            dq[u] = q.s0[d][u] - q.c0[u];
            own[u] = mm_t<double>(dn[u], dq[u]);
            fin[u] = fma(2.0, q.s1[d][u], mm_t<double>(q.s1[d][u] - q.s2[d][u], dn[u]));
        }
        // a second outflow face takes the inflow term's place with the own slope the other way, a second inflow
        // face the own term's place with its face value
        if (__any_sync(C.mask, q.xe[d] != 0.0)) {
            const bool both = q.xe[d] != 0.0, dvm_h = interior || side_kind(m.kinds, 2 * d + 1) == SK_DVM;
            const int r2 = dvm_h ? m.n2[2 * d + 1] : k;
            double e2[ZP];
#pragma unroll
            for (int u = 0; u < ZP; ++u)
                e2[u] = *reinterpret_cast<const double*>(row_at(C.fz[u], r2, row_bytes));
#pragma unroll
            for (int u = 0; u < ZP; ++u) {
                const double high = fma(2.0, q.s0[d][u], mm_t<double>(q.s0[d][u] - e2[u], neg_if<double>(dq[u], true)));
                if (both && oL) fin[u] = neg_if<double>(own[u], true);
                if (both && !oL) own[u] = high;
            }
            if (both && oL) ci = q.xe[d];
            if (both && !oL) co = q.xe[d];
        }
        if (!interior) {
#pragma unroll
            for (int hs = 0; hs < 2; ++hs) {   // (the side kinds are the same for every lane of the cell)
                const int s = 2 * d + hs, kd = side_kind(m.kinds, s);
                if (kd == SK_NONE || kd == SK_DVM) continue;
                // this side's inflow, and the term that carries it
                const bool in_i = hs ? oL : !oL;
                const double x = in_i ? q.xi[d] : (hs && !oL ? q.xe[d] : 0.0);
                const bool in = __double_as_longlong(x) < 0 && x != 0.0;
                if (!__any_sync(C.mask, in)) continue;
                const double scale = kd == SK_WALL ? __ldg(a.rho_w + (long long)k * 6 + s) : 1.0;
                double v[ZP];
                column_record<ZP>(a, kd == SK_GHOST ? a.recGhost : a.recBC, m.rf[s], 2.0 * scale, C, v);
#pragma unroll
                for (int u = 0; u < ZP; ++u) {
                    if (in && in_i) fin[u] = v[u];
                    if (in && !in_i) own[u] = v[u];
                }
            }
        }
        // the low side first, as the general update: the same roundings
        const double c_low = oL ? co : ci, c_high = oL ? ci : co;
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            num[u] = fma(-c_low, oL ? own[u] : fin[u], num[u]);
            num[u] = fma(-c_high, oL ? fin[u] : own[u], num[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        const double v = rden * num[u];
        if (u < C.nact) *reinterpret_cast<double*>(const_cast<char*>(row_at(C.fz[u], k, row_bytes))) = v;
    }
}

// A block owns P (ix, iy) positions x ZP planes; its G warps split the cells
// of each hyperplane, 32 / P cells to a warp.  P = 16 serves small velocity grids,
// whose blocks of 32 positions would leave SMs idle: the reduced grid of 48 x 48 x 2
// on the same cylinder takes 7.25 ms with 144 blocks of 12 warps, 11.7 with 72 blocks
// of 32 positions, 7.46 with a lane per velocity in 144 blocks of 16 warps (32 x 32 x 2:
// 6.9, 11.7, 7.4).  The sweep data of a warp's next cell (also across the
// barrier: it does not change during the pass) is loaded before the current
// cell is updated.  MINB: blocks per SM the registers are capped for.
template <int ZP, int G, int MINB, int P>
__global__ void __launch_bounds__(32 * G, MINB) k_sweep_col(SweepArgs a, double* __restrict__ f, int pass, int nptile,
                                                            unsigned row_bytes) {
    constexpr int CG = G * (32 / P);   // cells of a hyperplane taken together
    const int lane = threadIdx.x & 31, w = threadIdx.x / P;
    Column<ZP> C;
    make_column<ZP, P>(a.vg, f, blockIdx.x % nptile, blockIdx.x / nptile, lane, C);
    const int h0 = pass ? a.H - 1 : 0;
    const int kb = __ldg(a.hp_off + h0);
    int n = __ldg(a.hp_off + h0 + 1) - kb;
    int k = pass ? kb + n - 1 - w : kb + w;
    CellMeta<double, 2> m;
    if (w < n) load_meta<double, 2>(a, k, m);
    for (int hh = 0; hh < a.H; ++hh) {
        int kbn = 0, nn = 0;   // the next hyperplane
        if (hh + 1 < a.H) {
            const int h = pass ? a.H - 2 - hh : hh + 1;
            kbn = __ldg(a.hp_off + h);
            nn = __ldg(a.hp_off + h + 1) - kbn;
        }
        const int kfirst = pass ? kbn + nn - 1 - w : kbn + w;
        for (int i = w; i < n; i += CG) {
            const bool last = i + CG >= n;
            const int kn = last ? kfirst : (pass ? k - CG : k + CG);
            CellMeta<double, 2> mn;
            if (!last || w < nn) load_meta<double, 2>(a, kn, mn);
            Stencil<ZP> q;
            column_load<ZP>(k, m, C, row_bytes, q);
            column_apply<ZP>(a, k, m, C, row_bytes, q);
            k = kn;
            m = mn;
        }
        if (w >= n) {
            k = kfirst;
            if (w < nn) load_meta<double, 2>(a, k, m);
        }
        n = nn;
        __syncthreads();
    }
}

template <int ZP, int G, int MINB, int P = 32>
static void launch_col(gsis_ctx* c, const SweepArgs& a, int pass) {
    const int nptile = (c->vg.nx * c->vg.ny + P - 1) / P, nztile = (c->vg.nz + ZP - 1) / ZP;
    k_sweep_col<ZP, G, MINB, P><<<nptile * nztile, 32 * G, 0, c->stream>>>(a, (double*)c->f, pass, nptile,
                                                                        (unsigned)(c->vg.Nv * sizeof(double)));
}

// Column shapes: planes, warps per block, positions per block if not 32 (names and order: kColNames in sweep.cu).
void launch_sweep_col(gsis_ctx* c, const SweepArgs& a, int pass, int shape) {
    switch (shape) {
        case 1: launch_col<4, 8, 1>(c, a, pass); break;
        case 2: launch_col<3, 4, 2>(c, a, pass); break;
        case 3: launch_col<2, 8, 1>(c, a, pass); break;
        case 4: launch_col<2, 12, 1, 16>(c, a, pass); break;
        default: launch_col<4, 4, 3>(c, a, pass); break;
    }
}

}  // namespace gsis
