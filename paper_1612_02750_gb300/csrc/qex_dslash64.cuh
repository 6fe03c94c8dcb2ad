// qex_dslash64.cuh -- the FP64 operator's sum at one output site.
//
// FP64 FMAs alone need 288 x 64 clocks a warp and SM quarter (32^4: 250 us,
// the FP64 pipe's limit, against 96 us of HBM traffic).  Here the x, y and z
// hops run in fixed point on the integer pipe (qex_fix64.cuh: 72 % of the
// work, about 1180 clocks a warp and hop) and the t hops as FP64 FMAs that are
// issued between them, so both pipes work at once: 141 us at 32^4 (651 against
// 1264 at 48^4; with the Naik term 288-304 against 502).  Before the hops kept the
// bound on their terms it was 131 us; at that time, all hops on the integer pipe took
// 136 us, the t hops as a part of their own after or before the others 135-136 us.
// What bounds it now is the integer issue (two clocks an instruction, 4750 a site)
// next to the HBM traffic.
//
// The t hops' links and vectors wait in shared memory (cp.async, 384 bytes a
// thread, read back by the thread that copied them, so no barrier): loaded
// where they are used they cost 160 us, in registers they spill.  128
// registers, 16 warps an SM; 96 registers and 20 warps spilt (140-165 us).  Without
// the Naik term 20 to 40 bytes spill, with it 180 to 310, in L1.  The fallback stands
// inline, two hops a trip: 139 us, as a call 148 to 158, fully unrolled 155.
#pragma once

#include "qex_dslash_site.cuh"
#include "qex_fix64.cuh"

namespace qex {

constexpr int kStageWords = 12;                                         // 16-byte words of a hop: 9 link, 3 vector
constexpr size_t kStageBytes = 2 * kStageWords * sizeof(double2);       // dynamic shared memory a thread

__device__ __forceinline__ void copy_async16(double2 *smem, const double2 *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void copy_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// Input fields of dslash_site64: stored ...
struct Field64 {
    const double *f;
    size_t vh;
    __device__ __forceinline__ Vec3<double> operator()(int j) const { return load_vec(f, vh, j); }
    __device__ __forceinline__ void stage(double2 *slot, int stride, int j) const {
#pragma unroll
        for (int a = 0; a < 3; ++a) copy_async16(slot + a * stride, reinterpret_cast<const double2 *>(f) + a * vh + j);
    }
};
// ... or r + beta p, formed where it is read.
struct Direction64 {
    const double *r, *p;
    double beta;
    size_t vh;
    __device__ __forceinline__ Vec3<double> operator()(int j) const { return axpy_vec(r, p, beta, vh, j); }
    __device__ __forceinline__ void stage(double2 *slot, int stride, int j) const {
        const Vec3<double> v = (*this)(j);
#pragma unroll
        for (int a = 0; a < 3; ++a) slot[a * stride] = make_double2(v.c[a].re, v.c[a].im);
    }
};

// Colour a of (D in)(x) with FP64 FMAs alone, for what fixed point does not serve.
template <bool NAIK, typename In>
__device__ __forceinline__ double2 dslash_colour_fma(const Geom &g, const double *fat, const double *lng, double c3,
                                                     int p, int i, int a, const In &in) {
    const size_t vh = (size_t)g.vh;
    const Site s = site_of(g, p, i);
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 2
    for (int h = 0; h < (NAIK ? 16 : 8); ++h) {
        const int mu = NAIK ? h >> 2 : h >> 1, k = NAIK && (h & 2) ? 3 : 1;
        const bool back = h & 1;
        const int j = hop_index(g, s, mu, back ? -k : k);
        const bool minus = ((eta_bit(s, mu) ^ (back ? bc_bit_bwd(g, s, mu, k) : bc_bit_fwd(g, s, mu, k))) != 0) != back;
        const double2 *u = reinterpret_cast<const double2 *>(k == 1 ? fat : lng) +
                           (size_t)((back ? 1 - p : p) * 4 + mu) * 9 * vh + (back ? j : i);
        const Vec3<double> v = in(j);
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double2 e = __ldg(u + (back ? 3 * b + a : 3 * a + b) * vh);
            const double ui = back ? -e.y : e.y;
            re = fma(e.x, v.c[b].re, re);
            re = fma(-ui, v.c[b].im, re);
            im = fma(e.x, v.c[b].im, im);
            im = fma(ui, v.c[b].re, im);
        }
        const double c = k == 3 ? c3 : 1.0;
        acc.x = fma(minus ? -c : c, re, acc.x);
        acc.y = fma(minus ? -c : c, im, acc.y);
    }
    return acc;
}

// ... as a call of its own, where its registers would cost the caller.
template <bool NAIK, typename In>
__device__ __noinline__ double2 dslash_colour_call(const Geom &g, const double *fat, const double *lng, double c3,
                                                   int p, int i, int a, const In in) {
    return dslash_colour_fma<NAIK>(g, fat, lng, c3, p, i, a, in);
}

// (D in)(x) for the i-th site x (= s) of parity p.  slot: the thread's words
// of the block's dynamic shared memory, `stride` (the block size) apart.
template <bool NAIK, typename In>
__device__ __forceinline__ Vec3<double> dslash_site64(const Geom &g, const double *fat, const double *lng, double c3,
                                                      int p, int i, const Site &s, const In &in, double2 *slot,
                                                      int stride) {
    const size_t vh = (size_t)g.vh;
    Vec3<double> sum;
#pragma unroll
    for (int a = 0; a < 3; ++a) sum.c[a].re = sum.c[a].im = 0.0;
    bool bad = false, few[3] = {false, false, false}, ample[3];
    int e1 = 0;
#pragma unroll 1
    for (int k = 1; k <= (NAIK ? 3 : 1); k += 2) {
        const double *links = !NAIK || k == 1 ? fat : lng;
#pragma unroll
        for (int back = 0; back < 2; ++back) {
            const int j = hop_index(g, s, 3, back ? -k : k);
            const double2 *u = reinterpret_cast<const double2 *>(links) +
                               (size_t)((back ? 1 - p : p) * 4 + 3) * 9 * vh + (back ? j : i);
            double2 *d = slot + back * kStageWords * stride;
#pragma unroll
            for (int w = 0; w < 9; ++w) copy_async16(d + w * stride, u + w * vh);
            in.stage(d + 9 * stride, stride, j);
        }
        const bool eta3 = eta_bit(s, 3) != 0;
        const bool nf3 = eta3 != (bc_bit_fwd(g, s, 3, k) != 0), nb3 = eta3 == (bc_bit_bwd(g, s, 3, k) != 0);
        FixSum f;
        fix_clear(f);
        Cplx<double> t[3];  // the t hops' sum, colour by colour
        int eta = 0;
        // not unrolled: a hop is some 520 instructions
#pragma unroll 1
        for (int mu = 0; mu < 3; ++mu) {
            const int c = mu == 0 ? s.c[0] : mu == 1 ? s.c[1] : s.c[2];
            const int step = k * g.stride[mu], wrap = g.L[mu] * g.stride[mu];
            const int jf = (s.lex + step - (c + k >= g.L[mu] ? wrap : 0)) >> 1;
            const int jb = (s.lex - step + (c - k < 0 ? wrap : 0)) >> 1;
            Cplx<double> tf = {0.0, 0.0}, tb = {0.0, 0.0};  // colour mu of the two t hops
            const Mat3<double> uf = load_link(links, vh, p, mu, i);
            const Vec3<double> vf = in(jf);
            if (mu == 0) copy_wait_all();
            fix_hop<false>(f, uf, vf, eta != 0, [&](int b) {
                const double2 u = slot[(3 * mu + b) * stride], v = slot[(9 + b) * stride];
                tf.re = fma(u.x, v.x, tf.re);
                tf.im = fma(u.x, v.y, tf.im);
                tf.re = fma(-u.y, v.y, tf.re);
                tf.im = fma(u.y, v.x, tf.im);
            });
            fix_hop<true>(f, load_link(links, vh, 1 - p, mu, jb), in(jb), eta == 0, [&](int b) {
                const double2 u = slot[(kStageWords + 3 * b + mu) * stride], v = slot[(kStageWords + 9 + b) * stride];
                tb.re = fma(u.x, v.x, tb.re);
                tb.im = fma(u.x, v.y, tb.im);
                tb.re = fma(u.y, v.y, tb.re);
                tb.im = fma(-u.y, v.x, tb.im);
            });
            eta ^= c & 1;
            t[0] = t[1];
            t[1] = t[2];
            t[2].re = (nf3 ? -tf.re : tf.re) + (nb3 ? -tb.re : tb.re);
            t[2].im = (nf3 ? -tf.im : tf.im) + (nb3 ? -tb.im : tb.im);
        }
        bad |= f.bad;
        const double unit = fix_unit(f.e);
        if (k == 1) e1 = f.e;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double re = fma(unit, (double)f.a[2 * a], t[a].re), im = fma(unit, (double)f.a[2 * a + 1], t[a].im);
            sum.c[a].re = k == 1 ? re : fma(c3, re, sum.c[a].re);
            sum.c[a].im = k == 1 ? im : fma(c3, im, sum.c[a].im);
            if (k == 1)
                ample[a] = f.some && !fix_few(f.terms[a], 2.f * kFixTerms);
            else if (ample[a] && fix_below(c3, f.e, e1))
                continue;  // the one-hop terms alone serve for both
            few[a] |= f.some && fix_few(f.terms[a]);
        }
    }
    if (bad || few[0] || few[1] || few[2])
#pragma unroll 1
        for (int a = 0; a < 3; ++a) {
            if (!(bad || (a == 0 ? few[0] : a == 1 ? few[1] : few[2]))) continue;
            const double2 w = dslash_colour_fma<NAIK>(g, fat, lng, c3, p, i, a, in);
            if (a == 0) sum.c[0] = {w.x, w.y};
            if (a == 1) sum.c[1] = {w.x, w.y};
            if (a == 2) sum.c[2] = {w.x, w.y};
        }
    return sum;
}

// Lets a kernel take a block's dynamic shared memory: past 48 KB, its few
// hundred static bytes included, it has to be told.  Set at each launch, since
// it belongs to the device's context; a failure shows at the launch's check.
template <typename K>
void allow_stage(K kernel, int block) {
    const size_t bytes = block * kStageBytes;
    if (bytes > 40 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace qex
