// qex_dslash_dir.cuh -- the hops of one site along one direction (a run-time
// value that a whole warp shares), for the kernels that split a site's
// directions over threads.
#pragma once

#include "qex_dslash64.cuh"
#include "qex_dslash_site.cuh"
#include "qex_fix64.cuh"

namespace qex {

// Colour a of a half field at index i.
__device__ __forceinline__ double2 load_colour(const double *f, size_t vh, int a, int i) {
    return __ldg(reinterpret_cast<const double2 *>(f) + a * vh + i);
}
__device__ __forceinline__ float2 load_colour(const float *f, size_t vh, int a, int i) {
    return a < 2 ? __ldg(reinterpret_cast<const float2 *>(f) + 2 * (size_t)i + a)
                 : __ldg(reinterpret_cast<const float2 *>(f + 4 * vh) + i);
}
__device__ __forceinline__ void store_colour(double *f, size_t vh, int a, int i, double2 v) {
    reinterpret_cast<double2 *>(f)[a * vh + i] = v;
}
__device__ __forceinline__ void store_colour(float *f, size_t vh, int a, int i, float2 v) {
    if (a < 2)
        reinterpret_cast<float2 *>(f)[2 * (size_t)i + a] = v;
    else
        reinterpret_cast<float2 *>(f + 4 * vh)[i] = v;
}

// Coordinate, neighbours and signs of the k-step hops along mu.
struct DirHop {
    int jf, jb;    // neighbour indices, forward and backward
    bool nf, nb;   // the forward / backward term's factor is -1
};

__device__ __forceinline__ DirHop dir_hop(const Geom &g, const Site &s, int mu, int k) {
    const int c = mu == 0 ? s.c[0] : mu == 1 ? s.c[1] : mu == 2 ? s.c[2] : s.c[3];
    const int eta = (mu > 0 ? s.c[0] : 0) + (mu > 1 ? s.c[1] : 0) + (mu > 2 ? s.c[2] : 0);
    const int step = k * g.stride[mu], wrap = g.L[mu] * g.stride[mu];
    const bool wf = c + k >= g.L[mu], wb = c - k < 0, bc = mu == 3 && g.antiperiodic, odd = eta & 1;
    DirHop h;
    h.jf = (s.lex + step - (wf ? wrap : 0)) >> 1;
    h.jb = (s.lex - step + (wb ? wrap : 0)) >> 1;
    h.nf = odd != (bc && wf);
    h.nb = odd == (bc && wb);
    return h;
}

// acc += sg U v (DAG: U^+ v) for the link at index i of block (p, mu).
template <typename R, int FMT, bool DAG>
__device__ __forceinline__ void dir_mv(Vec3<R> &acc, R sg, const R *links, size_t vh, int p, int mu, int i,
                                       const Vec3<R> &v) {
    if constexpr (FMT == 3) {
        float d;
        const Mat3<R> u = load_link_s16(links, vh, p, mu, i, &d);
        if (DAG)
            acc_mdv(acc, sg * d, u, v);
        else
            acc_mv(acc, sg * d, u, v);
    } else {
        const Mat3<R> u = load_fat<R, FMT>(links, vh, p, mu, i);
        if constexpr (FMT == 2) {
            if (DAG)
                acc_mdv_fix16(acc, sg, u, v);
            else
                acc_mv_fix16(acc, sg, u, v);
        } else {
            if (DAG)
                acc_mdv(acc, sg, u, v);
            else
                acc_mv(acc, sg, u, v);
        }
    }
}

// The terms of (D in)(x) along mu, FP32.
template <typename R, int FMT, bool NAIK, typename In>
__device__ __forceinline__ Vec3<R> dslash_dir(const Geom &g, const R *fat, const R *lng, R c3, int p, int i,
                                              const Site &s, int mu, const In &in) {
    const size_t vh = (size_t)g.vh;
    Vec3<R> acc;
#pragma unroll
    for (int a = 0; a < 3; ++a) acc.c[a].re = acc.c[a].im = R(0);
    const DirHop h = dir_hop(g, s, mu, 1);
    dir_mv<R, FMT, false>(acc, h.nf ? R(-1) : R(1), fat, vh, p, mu, i, in(h.jf));
    dir_mv<R, FMT, true>(acc, h.nb ? R(-1) : R(1), fat, vh, 1 - p, mu, h.jb, in(h.jb));
    if constexpr (NAIK) {
        const DirHop h3 = dir_hop(g, s, mu, 3);
        constexpr int LF = FMT >= 2 ? 3 : 0;  // long links: FP32, or 16-bit with a per-link step
        dir_mv<R, LF, false>(acc, h3.nf ? -c3 : c3, lng, vh, p, mu, i, in(h3.jf));
        dir_mv<R, LF, true>(acc, h3.nb ? -c3 : c3, lng, vh, 1 - p, mu, h3.jb, in(h3.jb));
    }
    return acc;
}

template <typename R> struct Pair;
template <> struct Pair<float> { typedef float2 type; };
template <> struct Pair<double> { typedef double2 type; };

// The four directions' sums at SITES sites, in shared memory: warp mu puts its
// direction's, and after a barrier each colour's total is read.  FP64 hops all
// run on the integer pipe (a t hop in FP64 FMAs would be the longest of the
// four), one set of sums for the one-hop and one for the three-hop terms; the
// fixed-point sums are aligned and added as integers.
template <typename R, int FMT, bool NAIK, int SITES>
struct DirSums {
    float v[4][6][SITES];

    template <typename In>
    __device__ __forceinline__ void put(const Geom &g, const float *fat, const float *lng, float c3, int p, int i,
                                        int mu, int slot, const In &in) {
        const Vec3<float> acc = dslash_dir<float, FMT, NAIK>(g, fat, lng, c3, p, i, site_of(g, p, i), mu, in);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            v[mu][2 * a][slot] = acc.c[a].re;
            v[mu][2 * a + 1][slot] = acc.c[a].im;
        }
    }
    template <typename In>
    __device__ __forceinline__ float2 get(const Geom &, const float *, const float *, float, int, int, int a, int slot,
                                          const In &) const {
        return make_float2((v[0][2 * a][slot] + v[1][2 * a][slot]) + (v[2][2 * a][slot] + v[3][2 * a][slot]),
                           (v[0][2 * a + 1][slot] + v[1][2 * a + 1][slot]) +
                               (v[2][2 * a + 1][slot] + v[3][2 * a + 1][slot]));
    }
};

// As kFixTerms, for sums whose alignment drops up to a unit a direction more: 20 x
// 2^-53 of the terms' sum.
constexpr float kDirTerms = 0x1.8p-11f;

template <int FMT, bool NAIK, int SITES>
struct DirSums<double, FMT, NAIK, SITES> {
    static constexpr int N = NAIK ? 2 : 1;
    int64_t v[N][4][6][SITES];
    int e[N][4][SITES];
    FixMag terms[N][4][3][SITES];  // negative: the direction's hops are all zeros
    int bad[4][SITES];

    template <typename In>
    __device__ __forceinline__ void put(const Geom &g, const double *fat, const double *lng, double, int p, int i,
                                        int mu, int slot, const In &in) {
        const size_t vh = (size_t)g.vh;
        const Site s = site_of(g, p, i);
        FixSum f;
        bool out = false;
#pragma unroll 1
        for (int n = 0; n < N; ++n) {
            const double *links = n ? lng : fat;
            const DirHop h = dir_hop(g, s, mu, 2 * n + 1);
            fix_clear(f);
            fix_hop<false>(f, load_link(links, vh, p, mu, i), in(h.jf), h.nf);
            fix_hop<true>(f, load_link(links, vh, 1 - p, mu, h.jb), in(h.jb), h.nb);
#pragma unroll
            for (int c = 0; c < 6; ++c) v[n][mu][c][slot] = f.a[c];
            e[n][mu][slot] = f.e;
#pragma unroll
            for (int c = 0; c < 3; ++c) terms[n][mu][c][slot] = f.some ? f.terms[c] : fix_const2(-1.f);
            out |= f.bad;
        }
        bad[mu][slot] = out;
    }
    template <typename In>
    __device__ __forceinline__ double2 get(const Geom &g, const double *fat, const double *lng, double c3, int p, int i,
                                           int a, int slot, const In &in) const {
        bool redo = bad[0][slot] | bad[1][slot] | bad[2][slot] | bad[3][slot];  // fixed point does not serve
        bool ample = false;  // the one-hop terms serve for the three-hop ones as well
        int top1 = 0;
        double2 out = make_double2(0.0, 0.0);
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const int top = max(max(e[n][0][slot], e[n][1][slot]), max(e[n][2][slot], e[n][3][slot]));
            int64_t re = 0, im = 0;
            FixMag sum = fix_const2(0.f);
            bool some = false;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const uint32_t sh = (uint32_t)(top - e[n][d][slot]);
                re += fix_sar(v[n][d][2 * a][slot], sh);
                im += fix_sar(v[n][d][2 * a + 1][slot], sh);
                const FixMag t = terms[n][d][a][slot];
                const bool none = fix_least(t) < 0.f;
                some |= !none;
                sum = fix_add2(sum, none ? fix_const2(0.f) : fix_lower(t, sh));
            }
            if (n == 0) {
                ample = some && !fix_few(sum, 2.f * kDirTerms);
                top1 = top;
            }
            redo |= some && fix_few(sum, kDirTerms) && !(n == 1 && ample && fix_below(c3, top, top1));
            const double unit = n ? c3 * fix_unit(top) : fix_unit(top);
            out.x = fma(unit, (double)re, out.x);
            out.y = fma(unit, (double)im, out.y);
        }
        if (redo) return dslash_colour_call<NAIK>(g, fat, lng, c3, p, i, a, in);
        return out;
    }
};

}  // namespace qex
