// qex_dslash_params.cuh -- what the single-field Dslash kernels share: their
// parameters and the grid reduction that ends the reducing epilogues.
#pragma once

#include "qex_kernels.cuh"

namespace qex {

template <typename R>
struct DsParams {
    Geom g;
    const R *fat;
    const R *lng;
    R c3;
    int p;              // output parity
    const R *in;
    R *out;
    const R *q;
    const double *b;
    R m2;
    CgScalars *S;
    int check_halt;
    const R *r;         // EPI_PUPD
    R *x;               // EPI_PUPD: iterate that takes the pending alpha p_old (NULL: none)
    R *pbuf0, *pbuf1;   // p ping-pong
    int psel;
    int skip_zero_x;
    int reverse;        // walk the sites from the last index down
    int skip_ff;
    double *partials;
    unsigned int *counter;
};

// The grid reduction of EPI_NORMAL and EPI_RESID (part: this thread's sum).
template <typename R, int EPI>
__device__ __forceinline__ void finish_reduction(const DsParams<R> &P, double part, double *smem) {
    CgScalars *S = P.S;
    if (S == nullptr) return;  // uniform over the grid
    const double rr = S->rr;   // before the sum: its latency is hidden there
    double tot;
    if (!grid_sum(part, P.partials, P.counter, smem, &tot)) return;
    if constexpr (EPI == EPI_NORMAL) {
        S->pAp = tot;
        if (!(tot > 0.0) || !isfinite(tot)) {
            S->error = isfinite(tot) ? 2 : 1;
            S->halt = 1;
        } else {
            S->alpha = rr / tot;
        }
    } else {
        // FP64 true residual: accept convergence, or continue with beta from it
        take_true_residual(S, tot, true);
    }
}

// Largest half volume whose Dslash splits each site's directions over four
// threads (dslash_split.cu); fmt: the fat links' format (qex_dslash_site.cuh).
// Split / one thread a site, us: FP64 20^4 25.8/31.1, 20 x 22^3 33.4/34.6, 24^4
// 50.4/49.4; with Naik 24^3 x 48 184/196, 32^4 288/304, 36^4 471/459 (the line lies
// lower: they were 264/258 at 32^4 before the hops kept their bound).  FP32 16^2 x 20^2 4.2/4.3, 16^3 x 32
// 5.0/4.6; with Naik 24^3 x 32 40.8/41.2, 28^4 54.5/51.4.  Two-row FP32 16^4
// 3.4/3.6, 16^2 x 20^2 4.3/4.1; with Naik 32^4 72.8/76.2, 40^4 183/189 (at HBM
// both).  16-bit 10 x 14 x 18 x 22 3.3/3.4, 16^4 3.6/3.4; with Naik 16^4
// 4.9/4.8 (the normal operator 9.7/10.3), 16^3 x 32 7.7/7.1.
inline int64_t split_limit(bool fp64, int fmt, bool naik) {
    if (fp64) return naik ? 340000 : 107000;
    if (fmt >= 2) return naik ? 33000 : 28000;
    if (fmt == 1) return naik ? 600000 : 42000;
    return naik ? 230000 : 52000;
}
inline bool runs_split(const qex_lattice *lat, qex_prec prec, bool naik) {
    const int fmt = prec == QEX_F32_R12 ? 1 : prec == QEX_F32_R12H ? 2 : prec == QEX_F32_S16 ? 3 : 0;
    return lat->vh <= split_limit(prec == QEX_F64, fmt, naik);
}
template <typename R>
void launch_split(const qex_lattice *lat, int fmt, bool naik, int epi, const DsParams<R> &P, bool pdl,
                  cudaStream_t st);

}  // namespace qex
