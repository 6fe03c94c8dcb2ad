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
// the one at x.  2 TA(U G) is then a mat-vec and 30 real products (72 FP64
// operations a link; forming G and multiplying it by U took about 200).  They
// run in fixed point on the integer pipe (qex_fix64.cuh), which leaves 18 FP64
// operations, the conversions of the nine results: the FP64 pipe bounded the
// kernel (24^4 with long links, 916 us; 32^4, 1.45 ms); now it is HBM (115 us of
// traffic at 24^4) and the integer issue: 158 us, 288 us.  Links out of the
// fixed-point range take FP64 FMAs.

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

__device__ __forceinline__ Digits digits_of(int64_t x) {
    return fix_digits((uint32_t)((uint64_t)x >> 32), (uint32_t)x);
}

// x y added to h 2^32 + m (units of digit products hi lo), as in fix_hop.
__device__ __forceinline__ void add_product(int64_t &h, int64_t &m, const Digits &x, const Digits &y) {
    h = fix_mad(x.hi, y.hi, h);
    m = fix_mad(x.hi, y.lo, m);
    m = fix_mad(x.lo, y.hi, m);
}

// 128 threads, 6 blocks an SM (85 registers): 24^4 with long links 158 us, 162 at
// 5 blocks (96 registers), 182 at 2 blocks of 256.
constexpr int kForceBlock = 128;
constexpr int kForceUnit = kFixUnit + (1023 + 63 - kFixShift) - 64;  // exponent bias of the products' unit

__global__ void __launch_bounds__(kForceBlock, 6)
force_kernel(const __grid_constant__ Geom g, const double *__restrict__ links, double coef, int hop,
             const double *__restrict__ X, const double *__restrict__ Y, double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.vh) return;
    const size_t vh = (size_t)g.vh;
    const ForceEnds e = force_ends(g, hop, X, Y, i);
    const Mat3<double> u = load_link(links, vh, blockIdx.y >> 2, blockIdx.y & 3, i);
    double2 *o = reinterpret_cast<double2 *>(out) + (size_t)blockIdx.y * 9 * vh + i;
    FixSum w;  // U a
    fix_clear(w);
    fix_hop<false, 0>(w, u, e.a, e.neg);
    uint32_t mb = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) mb = fix_max(mb, fix_max(fix_mag(e.b.c[c].re), fix_mag(e.b.c[c].im)));
    bool none = false;
    mb = fix_range(mb, w.bad, none, [&] { return fix_any(e.b); });
    uint32_t top = 0;  // leading bits of the largest |w|
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int h = (int)(w.a[k] >> 32);
        top |= (uint32_t)(h ^ (h >> 31));
    }
    const int up = __clz((int)top) - kFixShift;  // 1 to 28: w's largest high digit to 27 or 28 bits
    const int eb = (int)(mb >> 20), unit_exp = w.e - up + eb - kForceUnit;
    if (w.bad || unit_exp < -900 || unit_exp > 900) {
        force_fma(g, links, coef, hop, X, Y, o, i);
        return;
    }
    const uint32_t kb = ((uint32_t)(eb + kFixShift) << 20) | 0xFFFFFu;
    Digits wr[3], wi[3], nr[3], ni[3], br[3], bi[3];  // w, -w, b
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int64_t re = (int64_t)((uint64_t)w.a[2 * c] << up), im = (int64_t)((uint64_t)w.a[2 * c + 1] << up);
        wr[c] = digits_of(re);
        wi[c] = digits_of(im);
        nr[c] = digits_of(-re);
        ni[c] = digits_of(-im);
        uint32_t lead;
        br[c] = digits_of((int64_t)fix_vec_real(e.b.c[c].re, kb, false, lead));
        bi[c] = digits_of((int64_t)fix_vec_real(e.b.c[c].im, kb, false, lead));
    }
    const double unit = coef * fix_double((uint64_t)(uint32_t)(unit_exp + 1023) << 52);
    Cplx<double> off[3];
    int64_t di[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        int64_t h = 0, m = 0x80000000ll;
        add_product(h, m, wi[r], br[r]);
        add_product(h, m, nr[r], bi[r]);
        di[r] = fix_mad((int)(m >> 32), 1, h);
#pragma unroll
        for (int c = r + 1; c < 3; ++c) {
            h = 0;
            m = 0x80000000ll;
            add_product(h, m, wr[r], br[c]);
            add_product(h, m, wi[r], bi[c]);
            add_product(h, m, nr[c], br[r]);
            add_product(h, m, ni[c], bi[r]);
            off[r + c - 1].re = unit * (double)fix_mad((int)(m >> 32), 1, h);
            h = 0;
            m = 0x80000000ll;
            add_product(h, m, wi[r], br[c]);
            add_product(h, m, nr[r], bi[c]);
            add_product(h, m, nr[c], bi[r]);
            add_product(h, m, wi[c], br[r]);
            off[r + c - 1].im = unit * (double)fix_mad((int)(m >> 32), 1, h);
        }
    }
    const int64_t tr = di[0] + di[1] + di[2];
    // 2 (d_r - tr / 3) = 2/3 (3 d_r - tr), with 2/3 to twice its precision
    const double third2 = unit * (2.0 / 3.0), rest = unit * (0x1p-53 / 3.0);
    Cplx<double> d[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        d[r].re = 0.0;
        const double t = (double)(3 * di[r] - tr);
        d[r].im = fma(third2, t, rest * t);
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
            force_kernel<<<dim3(blocks_for(lat->vh, kForceBlock), 8), kForceBlock, 0, s>>>(lat->geom, (const double *)(set ? lng64 : fat64), coef, hop,
                                                 (const double *)x_even, (const double *)y_odd, out);
        else
            force_gradient_kernel<<<grid, kBlock, 0, s>>>(lat->geom, coef, hop, (const double *)x_even,
                                                          (const double *)y_odd, out);
        QEX_CHECK_LAUNCH("force_kernel");
    }
    return QEX_OK;
}
