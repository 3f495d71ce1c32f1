// The kinetic sweep of a 1D line of cells (all cells kinetic, row k = cell k),
// shared by the single-solve launch and the batched persistent one.
//
// On a 1D mesh every hyperplane is one cell, so a warp can take a tile of
// velocities and walk the line alone, without a barrier.  A lane owns one
// (ix, iy) and ZP consecutive planes iz: xi.S, the upwind side, the
// denominator and its reciprocal depend on ix only and are formed once per cell
// and column.  The stencil is a window of registers: the two updated values
// behind, the cell and two old values ahead, and three more in flight, so a point
// costs one load and one store per pass (the general sweep loads five values
// through the L1/L2) and no step waits for its load (a window without that
// distance measured slower than reloading).  Ends of the line: rows are clamped,
// and a repeated value gives the zero slope the scheme prescribes there.
// Operations and roundings are those of the general sweep (long shocks amplify a
// difference in the last bit to 1e-4 of the state in a few iterations), so the results
// are the same: FP64 to the last bit; FP32 too, except values below 2^-100, where
// halving the face speeds meets the subnormals.  FP32: planes in pairs for the f32x2
// instructions (they share every coefficient); FP64: bound by the FP64 pipe, 11
// operations per point plus 6 / ZP shared ones against 23.
// Per iteration: a batch of 64 shocks of 100 to 800 cells, 24^3 to 64^3 velocities,
// FP32 and BF16: 20.0 ms with the general sweep's best tile, 15.2 with this one; 30
// FP64 cells of 1,800 velocities alone 85 us -> 75.
#pragma once
#include <type_traits>
#include "sweep_pair.cuh"

namespace gsis {

// planes in groups: two (f32x2) or one
template <typename T> struct Grp;
template <> struct Grp<double> {
    using P = double;
    static constexpr int W = 1;
};
template <> struct Grp<float> {
    using P = float2;
    static constexpr int W = 2;
};
__device__ __forceinline__ double gsub(double a, double b) { return a - b; }
__device__ __forceinline__ float2 gsub(float2 a, float2 b) { return f2sub(a, b); }
__device__ __forceinline__ double gfma(double a, double b, double c) { return fma(a, b, c); }   // a: coefficient of the column
__device__ __forceinline__ float2 gfma(float a, float2 b, float2 c) { return f2fma(bc2(a), b, c); }
__device__ __forceinline__ double gmm(double a, double b) { return mm_t<double>(a, b); }
__device__ __forceinline__ float2 gmm(float2 a, float2 b) {
    return make_float2(mm_line<float>(a.x, b.x), mm_line<float>(a.y, b.y));
}
__device__ __forceinline__ double gsel(bool c, double a, double b) { return c ? a : b; }
__device__ __forceinline__ float2 gsel(bool c, float2 a, float2 b) { return make_float2(c ? a.x : b.x, c ? a.y : b.y); }
__device__ __forceinline__ double gneg(double a) { return neg_if<double>(a, true); }
__device__ __forceinline__ float2 gneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ void gput(double& g, int, double v) { g = v; }
__device__ __forceinline__ void gput(float2& g, int i, float v) {
    if (i == 0) g.x = v;
    else g.y = v;
}
__device__ __forceinline__ double gget(double g, int) { return g; }
__device__ __forceinline__ float gget(float2 g, int i) { return i == 0 ? g.x : g.y; }

// A lane's column.  Past the end of the grid the position and the planes are
// clamped (loads stay in bounds) and nothing is stored.
template <typename S, typename T, int ZP>
struct LineColumn {
    char* fz[ZP];             // the column's values in row 0
    int ix, iy, iz0, q[ZP];   // q = iy + ny iz
    T x0;                     // half of xi_x
    int nact;                 // planes to store (0: clamped position)
};

template <typename S, typename T, int ZP>
__device__ __forceinline__ void make_line(const VGridDev& vg, S* f, int ptile, int ztile, int lane,
                                          LineColumn<S, T, ZP>& C) {
    const int nxy = vg.nx * vg.ny;
    const int pp = ptile * 32 + lane, p = min(pp, nxy - 1);
    C.iz0 = ztile * ZP;
    C.iy = p / vg.nx;
    C.ix = p - C.iy * vg.nx;
    C.nact = pp < nxy ? min(ZP, vg.nz - C.iz0) : 0;
    C.x0 = T(0.5) * (T)vg.xi[C.ix];
#pragma unroll
    for (int u = 0; u < ZP; ++u) {
        const int iz = min(C.iz0 + u, vg.nz - 1);
        C.q[u] = C.iy + vg.ny * iz;
        C.fz[u] = reinterpret_cast<char*>(f + (p + (long long)nxy * iz));
    }
}

// What a cell's update reads besides f and the factors of g~/tau.
template <typename T>
struct LineFaces {
    T Sl, Sh, it;   // S/V of the low and high side, 1/tau
};

template <typename T>
__device__ __forceinline__ LineFaces<T> load_faces(const SweepArgs& a, int k) {
    const T* sv = static_cast<const T*>(a.sdv) + (long long)k * SD_VALS;
    return {__ldg(sv), __ldg(sv + 1), __ldg(pick<T>(a.itau, a.itauf) + k)};
}

// g~/tau of one cell on a column from its factor vectors
template <typename T, int ZP>
__device__ __forceinline__ void line_source(const V4<T>& x, const V4<T>* y, typename Grp<T>::P* num) {
    constexpr int W = Grp<T>::W;
#pragma unroll
    for (int u = 0; u < ZP; ++u)
        gput(num[u / W], u % W, fma(x.w, y[u].w, fma(x.z, y[u].z, fma(x.y, y[u].y, x.x * y[u].x))));
}

// FP32: the factor vectors of the next LINE_STAGES - 1 cells are on their way
// into shared memory (cp.async), one copy per warp of the tile's x entries and of
// the y-z entries of its few rows: they come from far (the table is larger than
// the L2), and in registers one cell ahead was both too late and too many.
constexpr int LINE_STAGES = 4;
constexpr int LINE_ZP32 = 4;   // planes per FP32 column (FP64: one or two)
// A warp's shared memory: the end cells' boundary inflow (formed before the walk, so
// that the loop body stays short), and the stages (FP32).
template <typename T, int ZP>
struct LineEnds {
    T v[2][ZP][32];
};
struct LineStage {
    float4 x[LINE_STAGES][32];
    float4 y[LINE_STAGES][32 * LINE_ZP32];   // [row of the tile][plane]
};

__device__ __forceinline__ void copy16(float4* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// A boundary record at one node (out of line: the two ends of the line only).
template <typename T>
__device__ __noinline__ T line_record(const T* scal, const T* tab, int NT, int nx, int ny, int ix, int iy, int iz) {
    return eval_recT<T>(scal, tab, NT, nx, ny, ix, iy, iz);
}

// One Gauss-Seidel pass over the N cells (back: decreasing index).  The window is
// three values (the cell and two ahead) and three in flight; the loop body is
// three steps, so that their roles rotate without moves, and serves both
// directions (the instruction cache was the limit of longer bodies).
template <typename S, typename T, int ZP>
__device__ __forceinline__ void line_pass(const SweepArgs& a, const LineColumn<S, T, ZP>& C, int N, bool back,
                                          LineStage* stage, LineEnds<T, ZP>& ends) {
    using P = typename Grp<T>::P;
    constexpr int W = Grp<T>::W, NG = ZP / W;
    constexpr bool F64 = std::is_same<T, double>::value;
    static_assert(ZP % W == 0, "whole groups of planes");
    const unsigned row_bytes = (unsigned)(a.vg.Nv * sizeof(S));
    const int lane = threadIdx.x & 31, nx = a.vg.nx, nyz = a.vg.ny * a.vg.nz;
    const int first = back ? N - 1 : 0, dir = back ? -1 : 1;
    auto cell = [&](int j) { return max(0, min(N - 1, first + dir * j)); };   // j-th cell of the pass, clamped
    auto load = [&](int j, P* o) {
        const int k = cell(j);
#pragma unroll
        for (int u = 0; u < ZP; ++u)
            gput(o[u / W], u % W, ldT<T, S>(reinterpret_cast<const S*>(row_at(C.fz[u], k, row_bytes))));
    };
    // FP32: entries of the tile's y-z rows, copied by the warp together
    const int iy0 = __shfl_sync(0xffffffffu, C.iy, 0), nrow = __shfl_sync(0xffffffffu, C.iy, 31) - iy0 + 1;
    const int slot = (C.iy - iy0) * ZP;
    // (x entry of this lane and, for the lanes below nrow ZP, one y entry: byte offsets within a cell's entries)
    const char* gx = static_cast<const char*>(a.gx4) + (long long)C.ix * (4 * (int)sizeof(T));
    const char* gy = static_cast<const char*>(a.gy4) +
                     (long long)(iy0 + lane / ZP + a.vg.ny * min(C.iz0 + lane % ZP, a.vg.nz - 1)) * (4 * (int)sizeof(T));
    const bool copies_y = lane < nrow * ZP;
    auto fetch = [&](int j) {
        if constexpr (!F64) {
            const int k = cell(j), st = j % LINE_STAGES;
            copy16(&stage->x[st][lane], row_at(const_cast<char*>(gx), k, 16u * nx));
            if (copies_y) copy16(&stage->y[st][lane], row_at(const_cast<char*>(gy), k, 16u * nyz));
            for (int e = lane + 32; e < nrow * ZP; e += 32) {   // (rows of the tile beyond eight: short axes)
                const int r = e / ZP, iz = min(C.iz0 + (e - r * ZP), a.vg.nz - 1);
                copy16(&stage->y[st][e],
                       reinterpret_cast<const float4*>(a.gy4) + ((long long)k * nyz + (iy0 + r + a.vg.ny * iz)));
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        }
    };
    auto source = [&](int j, P* num) {   // g~/tau of the j-th cell
        V4<T> x, y[ZP];
        if constexpr (F64) {
            const int k = cell(j);
            x = ld4(static_cast<const T*>(a.gx4) + 4 * ((long long)k * nx + C.ix));
#pragma unroll
            for (int u = 0; u < ZP; ++u) y[u] = ld4(static_cast<const T*>(a.gy4) + 4 * ((long long)k * nyz + C.q[u]));
        } else {
            const int st = j % LINE_STAGES;
            const float4 v = stage->x[st][lane];
            x = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < ZP; ++u) {
                const float4 w = stage->y[st][slot + u];
                y[u] = {w.x, w.y, w.z, w.w};
            }
        }
        line_source<T, ZP>(x, y, num);
    };
    __syncwarp();   // the stages' last readers (the previous pass or item)
#pragma unroll
    for (int j = 0; j < LINE_STAGES - 1; ++j) fetch(j);
    bool none[2];   // an end without flux
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {   // twice the boundary distributions at the ends
        const int k = s ? N - 1 : 0, kd = side_kind(__ldg(a.sdi + (long long)k * SD_INTS + 12), s);
        if (s) none[1] = kd == SK_NONE;
        else none[0] = kd == SK_NONE;
        const bool given = kd == SK_FAR || kd == SK_WALL;
        const T sc = kd == SK_WALL ? __ldg(pick<T>(a.rho_w, a.rho_wf) + (long long)k * 6 + s) : T(1);
        const T *rs = RecT<T>::scal(a.recBC, s), *rt = RecT<T>::tab(a.recBC, s, a.vg.NT);
#pragma unroll 1
        for (int u = 0; u < ZP; ++u) {
            T v = T(0);
            if (given)
                v = T(2) * (sc * line_record<T>(rs, rt, a.vg.NT, nx, a.vg.ny, C.ix, C.iy, min(C.iz0 + u, a.vg.nz - 1)));
            ends.v[s][u][lane] = v;
        }
    }
    auto faces = [&](int j) {
        const int k = cell(j);
        LineFaces<T> o = load_faces<T>(a, k);
        if (k == 0 && none[0]) o.Sl = T(0);
        if (k == N - 1 && none[1]) o.Sh = T(0);
        return o;
    };
    P win[3][NG], fly[3][NG], b1[NG], b2[NG];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        load(j, win[j]);
        load(j + 3, fly[j]);
    }
#pragma unroll
    for (int g = 0; g < NG; ++g) b1[g] = b2[g] = win[0][g];
    LineFaces<T> fa = faces(0), fb = faces(1);
    P nxt[NG];   // FP64: g~/tau of the next cell
    if constexpr (F64) source(0, nxt);
    for (int j0 = 0; j0 < N; j0 += 3) {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const int j = j0 + v;
            if (j >= N) break;
            const int k = first + dir * j;
            P in[NG], num[NG];
            load(j + 6, in);
            const LineFaces<T> fc = faces(j + 2);
            if constexpr (F64) {
#pragma unroll
                for (int g = 0; g < NG; ++g) num[g] = nxt[g];
                source(j + 1, nxt);
            } else {
                __syncwarp();   // the slot's readers (step j - 1)
                fetch(j + LINE_STAGES - 1);
                asm volatile("cp.async.wait_group %0;\n" ::"n"(LINE_STAGES - 1) : "memory");
                __syncwarp();
                source(j, num);
            }
            const P* c0 = win[v];
            const P* a1 = win[(v + 1) % 3];
            const P* a2 = win[(v + 2) % 3];
            // upwind side of this lane (halved face speeds, outward)
            const T xl = C.x0 * fa.Sl, xh = C.x0 * fa.Sh;
            const bool end_l = k == 0, end_h = k == N - 1;
            const T xb = back ? xh : xl, xa = back ? xl : xh;   // behind, ahead
            const bool ob = pos_t<T>(xb), oa = pos_t<T>(xa);
            const bool from_b = !ob && xb != T(0);              // inflow face behind
            const T xbp = ob ? xb : T(0), xap = oa ? xa : T(0);
            T den = fma(T(2), xbp + xap, fa.it);
            // s1, s2: the neighbours on the inflow side (behind if that face is an inflow face, else ahead),
            // s0 the other one; x_o weights the own limited slope towards s0, at the outflow face there; x_i the
            // inflow face value
            T xo = from_b ? xap : xbp, xi = from_b ? xb : xa;
            // Faces that do not oppose each other (rare): the second outflow face takes the inflow term's place with
            // the own slope the other way, the second inflow face the own term's place with its face value
            const bool both_in = from_b && !oa && xa != T(0), both_out = !from_b && oa;
            const bool rare = __any_sync(0xffffffffu, both_in || both_out);
            if (rare && both_out) den = fma(T(2), back ? xb : xa, fma(T(2), back ? xa : xb, fa.it));   // (the low face first)
            if (rare && both_in) xo = xa;
            const bool end_b = back ? end_h : end_l, end_a = back ? end_l : end_h;
            const bool in_l = from_b != back;   // the inflow side is the low one
            const bool given = from_b ? end_b : end_a;   // ... and a boundary: its distribution instead
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const P s1 = gsel(from_b, b1[g], a1[g]), s2 = gsel(from_b, b2[g], a2[g]), s0 = gsel(from_b, a1[g], b1[g]);
                const P dn = gsub(c0[g], s1);
                P own = gmm(dn, gsub(s0, c0[g]));
                P fin = gfma(T(2), s1, gmm(gsub(s1, s2), dn));
                if (end_l || end_h) {
#pragma unroll
                    for (int i = 0; i < W; ++i)
                        if (given) gput(fin, i, ends.v[in_l ? 0 : 1][g * W + i][lane]);
                }
                if (rare) {
                    P fa2 = gfma(T(2), a1[g], gmm(gsub(a1[g], a2[g]), gsub(c0[g], a1[g])));   // the face value ahead
#pragma unroll
                    for (int i = 0; i < W; ++i)
                        if (end_a) gput(fa2, i, ends.v[back ? 0 : 1][g * W + i][lane]);
                    fin = gsel(both_out, gneg(own), fin);
                    own = gsel(both_in, fa2, own);
                }
                // the low side first, as the general sweep: the same roundings
                num[g] = gfma(in_l ? -xi : -xo, gsel(in_l, fin, own), num[g]);
                num[g] = gfma(in_l ? -xo : -xi, gsel(in_l, own, fin), num[g]);
            }
            const T rden = recip_t<T>(den);
            P fo[NG];
#pragma unroll
            for (int u = 0; u < ZP; ++u) {
                const T w = rden * gget(num[u / W], u % W);
                S st;
                stT<T, S>(&st, w);
                if (u < C.nact) *reinterpret_cast<S*>(row_at(C.fz[u], k, row_bytes)) = st;
                gput(fo[u / W], u % W, ldT<T, S>(&st));   // the stored (rounded) value is what later cells see
            }
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                b2[g] = j == 0 ? fo[g] : b1[g];   // a missing second neighbour repeats the first
                b1[g] = fo[g];
                win[v][g] = fly[v][g];            // the value three cells ahead
                fly[v][g] = in[g];
            }
            fa = fb;
            fb = fc;
        }
    }
    if constexpr (!F64) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Steps pass0 .. pass1 - 1 (0: backward, 1: forward) of one tile.
template <typename S, typename T, int ZP>
__device__ __forceinline__ void line_tile(const SweepArgs& a, S* f, int N, int tile, int lane, int pass0, int pass1,
                                          LineStage* stage, LineEnds<T, ZP>& ends) {
    const int nptile = (a.vg.nx * a.vg.ny + 31) / 32;
    LineColumn<S, T, ZP> C;
    make_line<S, T, ZP>(a.vg, f, tile % nptile, tile / nptile, lane, C);
#pragma unroll 1
    for (int step = pass0; step < pass1; ++step) line_pass<S, T, ZP>(a, C, N, step == 0, stage, ends);
}

}  // namespace gsis
