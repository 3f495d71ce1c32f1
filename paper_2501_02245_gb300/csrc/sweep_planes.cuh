// The FP32-arithmetic sweep of 2D and 3D meshes (FP32 / BF16 / FP16 storage) on
// velocity pairs of two planes.  Needs an even nx.
//
// A thread owns two consecutive velocities of an x-row (one word of storage, one
// packed f32x2 operand) on ZP = 2 consecutive planes iz.  The sweep is bound by
// instructions issued and by the latency of its loads with 12 (3D) or 15 (2D) warps per SM:
// - the update is written without selects: with m_s = max(x_s, 0) and n_s = m_s -
//   x_s for the halved face speeds x_s = xi.S_s/(2V),
//     num = g~/tau + sum_d m_L mm(c - l, h - c) + n_L (2 l + mm(l - l2, c - l))
//                        - m_H mm(c - l, h - c) + n_H (2 h + mm(h - h2, c - h)),
//     den = 1/tau + 2 sum (m_L + m_H),
//   mm the minmod (a face is an outflow or an inflow face: one of its m, n is
//   zero), instead of picking each side's upwind rows per velocity; the sums run in
//   the order of compute_cells, and the products of finite values with zero change
//   nothing, so the results are those of the other tiles (to FP32 subnormals, which
//   halving rounds); a pair whose sum is not a number, as where a value downstream has
//   overflowed its storage to an infinity, is formed again by compute_cells;
// - on 2D meshes m, n, den and the reciprocal do not depend on the plane and are
//   formed once per cell;
// - a row's address is one mad.wide from its byte pitch;
// - the row numbers of a warp's next cell are loaded while it updates the current
//   one (across the barrier too), so a cell costs one exposed round trip.  Holding
//   the next cell's stencil or factors as well needs registers that cost more
//   warps than it hides (2D FP32 cylinder 8.5 to 10 ms, 7.9 with the factors).
// Per pass pair, best of sweep_pair.cuh's tiles against this one:
//   10,499 kinetic cells, 48 x 48 x 24 velocities (cylinder): FP32 7.25 -> 5.7 ms, BF16 6.84 ->
//   6.05, FP16 6.72 -> 5.8;
//   11,643 kinetic cells, 48 x 48 x 48 (sphere): BF16 31.4 -> 21.4 ms, FP32 31.2 -> 21.0.
#pragma once
#include "sweep_pair.cuh"

namespace gsis {

__device__ __forceinline__ float2 mm2(float2 a, float2 b) {
    return make_float2(mm_t<float>(a.x, b.x), mm_t<float>(a.y, b.y));
}
__device__ __forceinline__ float2 pos2(float2 a) { return make_float2(fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f)); }

// Pairs (ix, ix + 1) on the planes iz0 .. iz0 + ZP - 1; clamped past the end of
// the grid (loads stay in bounds), nothing stored there.
template <typename S, int NC, int ZP>
struct PairColumn {
    char* fz[ZP];
    int ix, iy, iz0, q[ZP];
    float2 x0;            // half of xi_x of both velocities
    float x1, x2[ZP];     // half of xi_y; of xi_z (3D meshes)
    int nact;
};

template <typename S, int NC, int ZP>
__device__ __forceinline__ void make_pairs(const VGridDev& vg, S* f, int ptile, int ztile, int lane,
                                           PairColumn<S, NC, ZP>& C) {
    const int nxy = vg.nx * vg.ny;
    const int pp = ptile * 64 + 2 * lane, p = min(pp, nxy - 2);
    C.iz0 = ztile * ZP;
    C.iy = p / vg.nx;
    C.ix = p - C.iy * vg.nx;
    C.nact = pp < nxy ? min(ZP, vg.nz - C.iz0) : 0;
    C.x0 = make_float2(0.5f * (float)vg.xi[C.ix], 0.5f * (float)vg.xi[C.ix + 1]);
    C.x1 = 0.5f * (float)vg.xi[vg.nx + C.iy];
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        const int iz = min(C.iz0 + u, vg.nz - 1);
        C.q[u] = C.iy + vg.ny * iz;
        C.x2[u] = NC >= 3 ? 0.5f * (float)vg.xi[vg.nx + vg.ny + iz] : 0.0f;
        C.fz[u] = reinterpret_cast<char*>(f + (p + (long long)nxy * iz));
    }
}

// Stencil of a cell (raw storage words) and its g~/tau factors.
template <typename S> struct PairWord { using W = float2; };
template <> struct PairWord<__nv_bfloat16> { using W = unsigned; };
template <> struct PairWord<__half> { using W = unsigned; };
__device__ __forceinline__ float2 unpack(const float*, float2 w) { return w; }
__device__ __forceinline__ float2 unpack(const __nv_bfloat16*, unsigned w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ float2 unpack(const __half*, unsigned w) {
    return __half22float2(*reinterpret_cast<const __half2*>(&w));
}

template <typename S, int NC, int ZP>
struct PairStencil {
    using W = typename PairWord<S>::W;
    W c0[ZP], l[NC][ZP], h[NC][ZP], l2[NC][ZP], h2[NC][ZP];
};
// g~/tau factors and face data of a cell, and its rows (loaded one cell ahead).
template <int NC, int ZP>
struct PairFactors {
    float4 xa, xb, y[ZP];
    float S[2 * NC][NC], it;
};
template <int NC>
struct PairRows {
    int rf[2 * NC], n2[2 * NC], kinds;
};

template <int NC>
__device__ __forceinline__ void load_rows(const SweepArgs& a, int k, PairRows<NC>& m) {
    const int* p = a.sdi + (long long)k * SD_INTS;
    const int4 r = __ldg(reinterpret_cast<const int4*>(p)), r2 = __ldg(reinterpret_cast<const int4*>(p) + 1);
    m.kinds = __ldg(p + 12);
    m.rf[0] = r.x; m.rf[1] = r.y; m.n2[0] = r2.x; m.n2[1] = r2.y;
    m.rf[2] = r.z; m.rf[3] = r.w; m.n2[2] = r2.z; m.n2[3] = r2.w;
    if constexpr (NC >= 3) {
        const int4 r3 = __ldg(reinterpret_cast<const int4*>(p) + 2);
        m.rf[4] = r3.x; m.rf[5] = r3.y; m.n2[4] = r3.z; m.n2[5] = r3.w;
    }
}

// Rows of a side that is not a DVM side repeat the cell (its differences vanish).
template <typename S, int NC, int ZP>
__device__ __forceinline__ void load_stencil(int k, const PairRows<NC>& m, const PairColumn<S, NC, ZP>& C,
                                             unsigned row_bytes, PairStencil<S, NC, ZP>& q) {
    using W = typename PairWord<S>::W;
    auto at = [&](int row, int u) {
        return *reinterpret_cast<const W*>(row_at(C.fz[u], row, row_bytes));
    };
#pragma unroll
    for (int u = 0; u < ZP; ++u) q.c0[u] = at(k, u);
#pragma unroll
    for (int d = 0; d < NC; ++d) {
        int rl = m.rf[2 * d], rh = m.rf[2 * d + 1], nl = m.n2[2 * d], nh = m.n2[2 * d + 1];
        if (m.kinds >= 0) {   // not every side is a DVM side
            if (side_kind(m.kinds, 2 * d) != SK_DVM) rl = nl = k;
            if (side_kind(m.kinds, 2 * d + 1) != SK_DVM) rh = nh = k;
        }
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            q.l[d][u] = at(rl, u);
            q.h[d][u] = at(rh, u);
            q.l2[d][u] = at(nl, u);
            q.h2[d][u] = at(nh, u);
        }
    }
}

template <typename S, int NC, int ZP>
__device__ __forceinline__ void load_factors(const SweepArgs& a, int k, const PairColumn<S, NC, ZP>& C,
                                             PairFactors<NC, ZP>& g) {
    const float4* x = reinterpret_cast<const float4*>(a.gx4) + ((long long)k * a.vg.nx + C.ix);
    g.xa = __ldg(x);
    g.xb = __ldg(x + 1);
    const float4* y = reinterpret_cast<const float4*>(a.gy4) + (long long)k * (a.vg.ny * a.vg.nz);
#pragma unroll
    for (int u = 0; u < ZP; ++u) g.y[u] = __ldg(y + C.q[u]);
    const float* sv = static_cast<const float*>(a.sdv) + (long long)k * SD_VALS;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(sv + 8 * c));
        g.S[0][c] = v.x; g.S[1][c] = v.y; g.S[2][c] = v.z; g.S[3][c] = v.w;
        if constexpr (NC >= 3) {
            const float2 t = __ldg(reinterpret_cast<const float2*>(sv + 8 * c + 4));
            g.S[4][c] = t.x; g.S[5][c] = t.y;
        }
    }
    g.it = __ldg(a.itauf + k);
}

// Side sd of a boundary or interface cell, if it is no DVM side: its distribution's
// share of the sum (n: its inflow, per plane on 3D meshes).
template <typename S, int NC, int ZP>
__device__ __forceinline__ void add_record(const SweepArgs& a, int k, int kinds, int sd, const PairColumn<S, NC, ZP>& C,
                                           const float2* n, float2* num) {
    const int kd = side_kind(kinds, sd);
    if (kd == SK_NONE || kd == SK_DVM) return;
    const int NT = a.vg.NT, rec = __ldg(a.sdi + (long long)k * SD_INTS + (sd < 4 ? sd : 4 + sd));
    const Records& R = kd == SK_GHOST ? a.recGhost : a.recBC;
    const float* sc = RecT<float>::scal(R, rec);
    const float* tb = RecT<float>::tab(R, rec, NT);
    const float w = kd == SK_WALL ? __ldg(a.rho_wf + (long long)k * 6 + sd) : 1.0f;
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        const float2 x = n[NC == 3 ? u : 0];
        if (!__any_sync(0xffffffffu, x.x > 0.0f || x.y > 0.0f)) continue;
        const int iz = min(C.iz0 + u, a.vg.nz - 1);
        num[u].x = fmaf(x.x, 2.0f * w * eval_recT<float>(sc, tb, NT, a.vg.nx, a.vg.ny, C.ix, C.iy, iz), num[u].x);
        num[u].y = fmaf(x.y, 2.0f * w * eval_recT<float>(sc, tb, NT, a.vg.nx, a.vg.ny, C.ix + 1, C.iy, iz), num[u].y);
    }
}

// The general update of one cell at the velocities v and v + 1 (a pair whose product
// form met an infinity; out of line).
template <typename S, int NC>
__device__ __noinline__ void redo_pair(const SweepArgs& a, S* f, int k, int v) {
    const bool on = true;
    CellMeta<float, NC> m;
    load_meta<float, NC>(a, k, m);
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
        Vel<float, 1> V;
        make_vel<float, 1, false>(a.vg, v + j, 0, V);
        update_cells_k<S, float, NC, 1, 1, false>(a, f, &k, &on, V, &m);
    }
}

template <typename S, int NC, int ZP>
__device__ __forceinline__ void apply_pairs(const SweepArgs& a, S* f, int k, int kinds, const PairFactors<NC, ZP>& m,
                                            const PairColumn<S, NC, ZP>& C, unsigned row_bytes,
                                            const PairStencil<S, NC, ZP>& q) {
    constexpr int DZ = NC == 3 ? ZP : 1;   // coefficients per plane on 3D meshes
    const S* tag = nullptr;
    float2 num[ZP], out[DZ];
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        const float4 y = m.y[u];
        num[u].x = fmaf(m.xa.w, y.w, fmaf(m.xa.z, y.z, fmaf(m.xa.y, y.y, m.xa.x * y.x)));
        num[u].y = fmaf(m.xb.w, y.w, fmaf(m.xb.z, y.z, fmaf(m.xb.y, y.y, m.xb.x * y.x)));
    }
#pragma unroll
    for (int z = 0; z < DZ; ++z) out[z] = bc2(0.5f * m.it);   // half the denominator
    const bool interior = kinds < 0;   // every side a DVM side
#pragma unroll
    for (int d = 0; d < NC; ++d) {
        const float* SL = m.S[2 * d];
        const float* SH = m.S[2 * d + 1];
        const float2 bl = f2fma(bc2(C.x1), bc2(SL[1]), f2mul(C.x0, bc2(SL[0])));
        const float2 bh = f2fma(bc2(C.x1), bc2(SH[1]), f2mul(C.x0, bc2(SH[0])));
        float2 ml[DZ], mh[DZ], nl[DZ], nh[DZ];
#pragma unroll
        for (int z = 0; z < DZ; ++z) {
            float2 xl = bl, xh = bh;
            if constexpr (NC >= 3) {
                xl = f2fma(bc2(C.x2[z]), bc2(SL[NC >= 3 ? 2 : 0]), bl);
                xh = f2fma(bc2(C.x2[z]), bc2(SH[NC >= 3 ? 2 : 0]), bh);
            }
            if (!interior) {   // sides without flux
                if (side_kind(kinds, 2 * d) == SK_NONE) xl = make_float2(0.0f, 0.0f);
                if (side_kind(kinds, 2 * d + 1) == SK_NONE) xh = make_float2(0.0f, 0.0f);
            }
            ml[z] = pos2(xl);
            mh[z] = pos2(xh);
            nl[z] = f2sub(ml[z], xl);
            nh[z] = f2sub(mh[z], xh);
            out[z] = f2add(f2add(out[z], ml[z]), mh[z]);
        }
        const bool rl = !interior && side_kind(kinds, 2 * d) != SK_DVM, rh = !interior && side_kind(kinds, 2 * d + 1) != SK_DVM;
        float2 own[ZP], fl[ZP], fh[ZP];
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            const float2 c = unpack(tag, q.c0[u]), l = unpack(tag, q.l[d][u]), h = unpack(tag, q.h[d][u]);
            const float2 dl = f2sub(c, l), dh = f2sub(h, c), two = make_float2(2.0f, 2.0f);
            own[u] = mm2(dl, dh);
            fl[u] = f2fma(two, l, mm2(f2sub(l, unpack(tag, q.l2[d][u])), dl));
            fh[u] = f2fma(two, h, mm2(f2sub(h, unpack(tag, q.h2[d][u])), make_float2(-dh.x, -dh.y)));
        }
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            const int z = NC == 3 ? u : 0;
            num[u] = f2fma(ml[z], own[u], num[u]);
            if (!rl) num[u] = f2fma(nl[z], fl[u], num[u]);
        }
        if (rl) add_record<S, NC, ZP>(a, k, kinds, 2 * d, C, nl, num);
#pragma unroll
        for (int u = 0; u < ZP; ++u) {
            const int z = NC == 3 ? u : 0;
            num[u] = f2fma(mh[z], make_float2(-own[u].x, -own[u].y), num[u]);
            if (!rh) num[u] = f2fma(nh[z], fh[u], num[u]);
        }
        if (rh) add_record<S, NC, ZP>(a, k, kinds, 2 * d + 1, C, nh, num);
    }
    float2 r[DZ];
#pragma unroll
    for (int z = 0; z < DZ; ++z) {
        r[z].x = recip_t<float>(2.0f * out[z].x);
        r[z].y = recip_t<float>(2.0f * out[z].y);
    }
    float2 v[ZP];
    float t = 0.0f;   // NaN if any value is
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        v[u] = f2mul(num[u], r[NC == 3 ? u : 0]);
        t += v[u].x + v[u].y;
    }
    if (t != t) {
#pragma unroll 1
        for (int u = 0; u < C.nact; ++u) redo_pair<S, NC>(a, f, k, C.ix + a.vg.nx * (u == 0 ? C.q[0] : C.q[ZP - 1]));
        return;
    }
#pragma unroll
    for (int u = 0; u < ZP; ++u)
        if (u < C.nact) st2<S>(reinterpret_cast<S*>(row_at(C.fz[u], k, row_bytes)), v[u]);
}

template <typename S, int NC, int ZP, int G, int MINB>
__global__ void __launch_bounds__(32 * G, MINB) k_sweep_planes(const __grid_constant__ SweepArgs a, S* __restrict__ f,
                                                               int pass, int nptile) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned row_bytes = (unsigned)(a.vg.Nv * sizeof(S));
    PairColumn<S, NC, ZP> C;
    make_pairs<S, NC, ZP>(a.vg, f, blockIdx.x % nptile, blockIdx.x / nptile, lane, C);
    const int dk = pass ? -G : G;
    const int h0 = pass ? a.H - 1 : 0;
    const int kb = __ldg(a.hp_off + h0);
    int n = __ldg(a.hp_off + h0 + 1) - kb;
    int k = pass ? kb + n - 1 - w : kb + w;   // this warp's current cell
    PairRows<NC> r;                           // its rows
    if (w < n) load_rows<NC>(a, k, r);
    for (int hh = 0; hh < a.H; ++hh) {
        int kbn = 0, nn = 0;   // the next hyperplane
        if (hh + 1 < a.H) {
            const int h = pass ? a.H - 2 - hh : hh + 1;
            kbn = __ldg(a.hp_off + h);
            nn = __ldg(a.hp_off + h + 1) - kbn;
        }
        const int kfirst = pass ? kbn + nn - 1 - w : kbn + w;
        for (int i = w; i < n; i += G) {
            const bool more = i + G < n;
            const int kn = more ? k + dk : kfirst, kinds = r.kinds;
            PairStencil<S, NC, ZP> q;
            PairFactors<NC, ZP> g;
            load_stencil(k, r, C, row_bytes, q);
            load_factors(a, k, C, g);
            if (more || w < nn) load_rows<NC>(a, kn, r);
            apply_pairs<S, NC, ZP>(a, f, k, kinds, g, C, row_bytes, q);
            k = kn;
        }
        if (w >= n && w < nn) {
            k = kfirst;
            load_rows<NC>(a, k, r);
        }
        n = nn;
        __syncthreads();
    }
}

template <typename S, int NC, int G, int MINB>
static void launch_planes_t(gsis_ctx* c, const SweepArgs& a, int pass) {
    constexpr int ZP = 2;
    const int nptile = (c->vg.nx * c->vg.ny + 63) / 64, nztile = (c->vg.nz + ZP - 1) / ZP;
    k_sweep_planes<S, NC, ZP, G, MINB><<<nptile * nztile, 32 * G, 0, c->stream>>>(a, (S*)c->f, pass, nptile);
}

// 2D: 128 registers, 15 warps per SM (four warps of 168 registers, 12 per SM, were 3 %
// slower on the FP32 cylinder); 3D: 168 registers, 12 warps per SM (five warps, 10 per
// SM: 17 % slower on the BF16 sphere).  Shape 1 has wider blocks for velocity grids with
// few tiles: 36 x 38 x 17 on 4,335 cells FP32 1.74 ms (2.09 with shape 0, 2.26 with the best
// pair tile), 32^3 on the sphere BF16 7.1 (8.9, 10.3).
template <typename S>
static void launch_planes(gsis_ctx* c, const SweepArgs& a, int pass, int shape) {
    if (shape == 1) {
        if (c->normal_components == 2) launch_planes_t<S, 2, 8, 2>(c, a, pass);
        else launch_planes_t<S, 3, 6, 2>(c, a, pass);
        return;
    }
    if (c->normal_components == 2) launch_planes_t<S, 2, 5, 3>(c, a, pass);
    else launch_planes_t<S, 3, 4, 3>(c, a, pass);
}

}  // namespace gsis
