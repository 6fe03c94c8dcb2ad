// force.cu -- fermion force of S = phi^+ A^{-1} phi, A = m^2 - D_eo D_oe.
//
// With X = A^{-1} phi (even sites) and Y = D_oe X (odd sites),
// dS = 2 Re sum_{x,mu} tr(dU_mu(x) G_mu(x)) where
//   G_mu(x) =  s_mu(x) Y(x+mu) X(x)^+   on even x,
//   G_mu(x) = -s_mu(x) X(x+mu) Y(x)^+   on odd x,
// s_mu the staggered phase times the link's antiperiodic sign; the long
// links take c3 and the x+3mu neighbours.  For every link it writes
// either F = 2 TA(U G) (traceless anti-Hermitian part, the force
// along U -> exp(i e w) U) or 2 G^+ (the gradient with respect to the complex
// link entries) in the internal FP64 link layout.  One thread per link:
// blockIdx.y = parity * 4 + mu.
#include "qex_fix64.cuh"
#include "qex_kernels.cuh"

namespace qex {

// G has rank one, so U G = (U a) b^+ with a the vector at the hop's end and b
// the one at x.  2 TA(U G) is then a mat-vec, w = U a, and 30 real products (72 FP64
// operations a link; forming G and multiplying it by U took about 200, 916 us on
// 24^4 with long links).  All of it runs on the integer pipe (qex_fix64.cuh), where a
// link takes about 1800 instructions, and leaves nothing to the FP64 pipe, whose
// instructions cost 64 clocks each and hardly overlap with the integer ones: 224 us
// against 115 us of HBM traffic.  w is summed under one exponent, like the
// operator's hops, and where a real of it has only terms far below the largest the
// link takes FP64 FMAs.  The products of w and b would meet such reals too often
// (sums of four products, not of 36), so there every real has its own exponent,
// and a sum takes the largest of its four.  With w and b under one exponent each it
// took 165 us but lost the small reals; the products as FP64 FMAs 266 us, 328 with
// w converted to FP64 by the FP64 pipe.

// The vectors a and b of link (x, mu) and the sign of its G.
struct ForceEnds {
    Vec3<double> a, b;
    bool neg;
};

__device__ __forceinline__ ForceEnds force_ends(const Geom &g, int hop, const double *X, const double *Y, int i) {
    const int p = blockIdx.y >> 2, mu = blockIdx.y & 3;
    const size_t vh = (size_t)g.vh;
    const Site s = site_of(g, p, i);
    const int j = hop_index(g, s, mu, hop);
    ForceEnds e;
    // even x: a = Y(x+hop mu), b = X(x); odd x: a = X(x+hop mu), b = Y(x), sign flipped
    e.a = load_vec(p == 0 ? Y : X, vh, j);
    e.b = load_vec(p == 0 ? X : Y, vh, i);
    e.neg = ((eta_bit(s, mu) ^ bc_bit_fwd(g, s, mu, hop)) != 0) != (p == 1);
    return e;
}

// Writes F from its off-diagonal elements (0,1), (0,2), (1,2) and its diagonal.
__device__ __forceinline__ void store_force(double2 *o, size_t vh, const Cplx<double> (&off)[3],
                                            const Cplx<double> (&d)[3]) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        o[4 * r * vh] = make_double2(d[r].re, d[r].im);
#pragma unroll
        for (int c = r + 1; c < 3; ++c) {
            const Cplx<double> f = off[r + c - 1];
            o[(3 * r + c) * vh] = make_double2(f.re, f.im);
            o[(3 * c + r) * vh] = make_double2(-f.re, f.im);
        }
    }
}

// F_rc = w_r conj(b_c) - conj(w_c) b_r, less a third of its trace, w = coef U a,
// in FP64 FMAs (a call of its own: it reads its inputs again).
__device__ __noinline__ void force_fma(const Geom &g, const double *links, double coef, int hop, const double *X,
                                       const double *Y, double2 *o, int i) {
    const size_t vh = (size_t)g.vh;
    const ForceEnds e = force_ends(g, hop, X, Y, i);
    const Vec3<double> &b = e.b;
    Vec3<double> w;
#pragma unroll
    for (int r = 0; r < 3; ++r) w.c[r].re = w.c[r].im = 0.0;
    acc_mv(w, e.neg ? -coef : coef, load_link(links, vh, blockIdx.y >> 2, blockIdx.y & 3, i), e.a);
    Cplx<double> off[3], d[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const double re = fma(w.c[r].re, b.c[r].re, w.c[r].im * b.c[r].im);
        d[r].re = re - re;  // 0, or the NaN of a value that is not finite
        d[r].im = fma(w.c[r].im, b.c[r].re, -(w.c[r].re * b.c[r].im));
#pragma unroll
        for (int c = r + 1; c < 3; ++c) {
            Cplx<double> &f = off[r + c - 1];
            f.re = fma(w.c[r].re, b.c[c].re, w.c[r].im * b.c[c].im);
            f.re = fma(-w.c[c].re, b.c[r].re, fma(-w.c[c].im, b.c[r].im, f.re));
            f.im = fma(w.c[r].im, b.c[c].re, -(w.c[r].re * b.c[c].im));
            f.im = fma(-w.c[c].re, b.c[r].im, fma(w.c[c].im, b.c[r].re, f.im));
        }
    }
    const double third = (d[0].im + d[1].im + d[2].im) / 3.0;
#pragma unroll
    for (int r = 0; r < 3; ++r) d[r].im = 2.0 * (d[r].im - third);
    store_force(o, vh, off, d);
}

// +-a b summed over n products, their units brought to the largest's; F's elements.
struct ForceSum {
    int64_t x;
    int e;  // as fix_to_double's
};

__device__ __forceinline__ int force_exp(int a, int b) { return a > b ? a : b; }

// p0 + p1 - p2 - p3, p_k = a_k b_k.
__device__ __forceinline__ ForceSum force_sum4(const FixNum &a0, const FixNum &b0, const FixNum &a1, const FixNum &b1,
                                               const FixNum &a2, const FixNum &b2, const FixNum &a3,
                                               const FixNum &b3) {
    const int e0 = a0.e + b0.e, e1 = a1.e + b1.e, e2 = a2.e + b2.e, e3 = a3.e + b3.e;
    const int e = force_exp(force_exp(e0, e1), force_exp(e2, e3));
    return {fix_product(a0, b0, e - e0) + fix_product(a1, b1, e - e1) - fix_product(a2, b2, e - e2) -
                fix_product(a3, b3, e - e3),
            e};
}

// Its unit, 2^(e - 2 kFixNum + 64), as fix_to_double takes it.
__device__ __forceinline__ double force_double(int64_t x, int e) {
    return fix_to_double(x, e - 2 * kFixNum + 64 + kFixUnit);
}

// 64 threads, 10 blocks an SM (96 registers): 224 us, as 128 x 5; 264 with 256 x 2
// (a link that takes FMAs holds its block up).
constexpr int kForceBlock = 64;
// What the terms of w's reals have to come to (fix_few), lower than the operator's
// kFixTerms: the roundings of one hop, not of six, stand against them (15 x 2^-53 of
// the terms' sum at most).
constexpr float kForceTerms = 0x1.8p-14f;

__global__ void __launch_bounds__(kForceBlock, 10)
force_kernel(const __grid_constant__ Geom g, const double *__restrict__ links, double coef, int hop,
             const double *__restrict__ X, const double *__restrict__ Y, double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.vh) return;
    const size_t vh = (size_t)g.vh;
    ForceEnds e = force_ends(g, hop, X, Y, i);
    const Mat3<double> u = load_link(links, vh, blockIdx.y >> 2, blockIdx.y & 3, i);
    double2 *o = reinterpret_cast<double2 *>(out) + (size_t)blockIdx.y * 9 * vh + i;
    FixSum f;  // U a
    fix_clear(f);
    fix_hop<false, 0>(f, u, e.a, e.neg);
    if (coef != 1.0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            e.b.c[c].re *= coef;
            e.b.c[c].im *= coef;
        }
    }
    uint32_t most = 0, least = ~0u;  // of b's magnitudes (zeros apart), a low word that is all there is as 1
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const double d = r ? e.b.c[c].im : e.b.c[c].re;
            const uint32_t m = fix_mag(d) | ((uint32_t)fix_bits(d) != 0);
            most = fix_max(most, m);
            least = m - 1 < least ? m - 1 : least;
        }
    }
    // Inf and NaN, and products that may leave the normal range: w's reals reach from
    // 2^(unit) to 2^(unit + 62), the smallest unit of a product is 2^-60 of it
    const int unit = f.e - kFixUnit;
    const bool in_range = most < 0x7FF00000u && unit + (int)(most >> 20) < 1900 &&
                          (least == ~0u || unit + (int)(least >> 20) > 60);
    const bool few = f.some && (fix_few(f.terms[0], kForceTerms) || fix_few(f.terms[1], kForceTerms) ||
                                fix_few(f.terms[2], kForceTerms));
    if (f.bad || few || !in_range) {
        force_fma(g, links, coef, hop, X, Y, o, i);
        return;
    }
    FixNum wr[3], wi[3], br[3], bi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        wr[c] = fix_num(f.a[2 * c], f.e);
        wi[c] = fix_num(f.a[2 * c + 1], f.e);
        br[c] = fix_num(e.b.c[c].re);
        bi[c] = fix_num(e.b.c[c].im);
    }
    Cplx<double> off[3], d[3];
    int de = 2 * kFixNone;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        de = force_exp(de, force_exp(wi[r].e + br[r].e, wr[r].e + bi[r].e));
#pragma unroll
        for (int c = r + 1; c < 3; ++c) {
            const ForceSum re = force_sum4(wr[r], br[c], wi[r], bi[c], wr[c], br[r], wi[c], bi[r]);
            const ForceSum im = force_sum4(wi[r], br[c], wi[c], br[r], wr[r], bi[c], wr[c], bi[r]);
            off[r + c - 1].re = force_double(re.x, re.e);
            off[r + c - 1].im = force_double(im.x, im.e);
        }
    }
    int64_t di[3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
        di[r] = fix_product(wi[r], br[r], de - (wi[r].e + br[r].e)) -
                fix_product(wr[r], bi[r], de - (wr[r].e + bi[r].e));
    const int64_t tr = di[0] + di[1] + di[2];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        // 2 (d_r - tr / 3) = 2/3 (3 d_r - tr), |3 d_r - tr| < 2^60: a third of 4 times it
        const int64_t t = 3 * di[r] - tr;
        d[r].re = 0.0;
        d[r].im = force_double(__mul64hi(t * 4, 0x5555555555555556ll), de - 1);
    }
    store_force(o, vh, off, d);
}

// 2 G^+: element (r, c) is 2 conj(a_c) b_r; 42 FP64 operations, which bound it
// (the links are not read).
__global__ void __launch_bounds__(kBlock)
force_gradient_kernel(const __grid_constant__ Geom g, double coef, int hop, const double *__restrict__ X,
                      const double *__restrict__ Y, double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.vh) return;
    const size_t vh = (size_t)g.vh;
    ForceEnds e = force_ends(g, hop, X, Y, i);
    double2 *o = reinterpret_cast<double2 *>(out) + (size_t)blockIdx.y * 9 * vh + i;
    const double s = e.neg ? -2.0 * coef : 2.0 * coef;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const double re = s * e.b.c[r].re, im = s * e.b.c[r].im;
#pragma unroll
        for (int c = 0; c < 3; ++c)
            o[(3 * r + c) * vh] = make_double2(fma(e.a.c[c].re, re, e.a.c[c].im * im),
                                               fma(e.a.c[c].re, im, -(e.a.c[c].im * re)));
    }
}

}  // namespace qex

using namespace qex;

extern "C" qex_status qex_force(const qex_lattice *lat, const void *fat64, const void *lng64, double c_naik,
                                const void *x_even, const void *y_odd, int kind, void *out_fat, void *out_lng,
                                void *stream) {
    qex_status st;
    if ((st = check_lattice(lat))) return st;
    if (!fat64 || !x_even || !y_odd || !out_fat || (lng64 && !out_lng)) {
        set_error("fat64, x_even, y_odd and out_fat (and out_lng with long links) must not be NULL");
        return QEX_ERR_ARG;
    }
    if (!aligned16(fat64) || !aligned16(x_even) || !aligned16(y_odd) || !aligned16(out_fat) ||
        (lng64 && (!aligned16(lng64) || !aligned16(out_lng)))) {
        set_error("links and fields must be 16-byte aligned");
        return QEX_ERR_ALIGN;
    }
    if (kind != 0 && kind != 1) {
        set_error("kind must be 0 (force 2 TA(U G)) or 1 (gradient 2 G^+)");
        return QEX_ERR_ARG;
    }
    if (lng64)
        for (int mu = 0; mu < 4; ++mu)
            if (lat->dims[mu] < 4) {
                set_error("the Naik term needs every extent >= 4");
                return QEX_ERR_SHAPE;
            }
    const dim3 grid(blocks_for(lat->vh), 8);
    const cudaStream_t s = as_stream(stream);
    for (int set = 0; set < (lng64 ? 2 : 1); ++set) {
        const double coef = set ? c_naik : 1.0;
        const int hop = set ? 3 : 1;
        double *out = (double *)(set ? out_lng : out_fat);
        if (kind == 0)
            force_kernel<<<dim3(blocks_for(lat->vh, kForceBlock), 8), kForceBlock, 0, s>>>(
                lat->geom, (const double *)(set ? lng64 : fat64), coef, hop, (const double *)x_even,
                (const double *)y_odd, out);
        else
            force_gradient_kernel<<<grid, kBlock, 0, s>>>(lat->geom, coef, hop, (const double *)x_even,
                                                          (const double *)y_odd, out);
        QEX_CHECK_LAUNCH("force_kernel");
    }
    return QEX_OK;
}
