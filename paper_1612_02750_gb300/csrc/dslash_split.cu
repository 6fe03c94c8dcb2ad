// dslash_split.cu -- the Dslash of a small lattice: the four directions of a
// site on four threads.
//
// A lattice of a few ten thousand even sites gives the one-thread-a-site
// kernel (dslash.cu) fewer warps than the GPU has SM quarters for two each,
// and its time is that of one thread's eight (sixteen) hops in a row.  Here a
// block is 32 sites by four warps, warp mu takes the two (four) hops along mu,
// all of whose loads are in flight at once, and the sums meet in shared memory,
// from which three of the warps run the epilogue, one colour each.  8^4 FP64:
// 10.0 -> 3.4 us (Naik 20.9 -> 5.8), 16-bit 3.0 -> 1.9 us; where it ends:
// split_limit.
#include "qex_dslash_params.cuh"
#include "qex_dslash_dir.cuh"

namespace qex {

constexpr int kSplitSites = 32;
constexpr int kSplitBlock = 4 * kSplitSites;

template <typename R, int FMT, bool NAIK, int EPI>
__global__ void __launch_bounds__(kSplitBlock, (std::is_same<R, double>::value ? 4 : 8))
dslash_split_kernel(const __grid_constant__ DsParams<R> P) {
    typedef typename Pair<R>::type R2;
    __shared__ double smem[32];
    __shared__ DirSums<R, FMT, NAIK, kSplitSites> sums;
    pdl_trigger();
    pdl_wait();  // everything below may read what earlier kernels wrote
    if (P.check_halt && P.S->halt) return;  // uniform over the grid
    if (P.skip_ff && P.S->ru_ff) return;    // uniform: a float-float update
    // first residual from a zero initial guess: D x = 0 (uniform over the grid)
    const bool zero_x = P.skip_zero_x && !P.S->x_nonzero;
    if (EPI == EPI_PLAIN && zero_x) return;
    const Geom &g = P.g;
    const size_t vh = (size_t)g.vh;
    const int p = P.p, mu = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // direction buffers by iteration parity (read before any block can change it)
    const R *in = P.in, *r = P.r, *pold = nullptr;
    R *pnew = nullptr;
    R alpha = R(0), beta = R(0);
    if (P.psel || EPI == EPI_PUPD) {
        const int it = P.S->iters;
        pold = (it & 1) ? P.pbuf1 : P.pbuf0;
        pnew = (it & 1) ? P.pbuf0 : P.pbuf1;
        if (EPI == EPI_PLAIN) in = pnew;
    }
    if (EPI == EPI_PUPD) {
        alpha = (R)P.S->alpha;
        beta = (R)P.S->beta;
    }
    const auto input = [=](int j) {
        if constexpr (EPI == EPI_PUPD)
            return axpy_vec(r, pold, beta, vh, j);
        else
            return load_vec(in, vh, j);
    };
    double part = 0.0;
    for (int base = blockIdx.x * kSplitSites; base < g.vh; base += gridDim.x * kSplitSites) {
        const int i = base + lane;
        const bool mine = i < g.vh;
        if (!(EPI == EPI_RESID && zero_x)) {
            if (mine) sums.put(g, P.fat, P.lng, P.c3, p, i, mu, lane, input);
            __syncthreads();
        }
        const int a = mu;  // this warp's colour
        if (mine && a < 3) {
            R2 acc;
            acc.x = acc.y = R(0);
            if (!(EPI == EPI_RESID && zero_x)) acc = sums.get(g, P.fat, P.lng, P.c3, p, i, a, lane, input);
            if constexpr (EPI == EPI_PLAIN) {
                store_colour(P.out, vh, a, i, acc);
            } else if constexpr (EPI == EPI_PUPD) {
                store_colour(P.out, vh, a, i, acc);
                // index i of the other parity's direction, and of the iterate,
                // which takes the previous iteration's alpha p
                const R2 pv = load_colour(pold, vh, a, i), rv = load_colour(P.r, vh, a, i);
                R2 pn;
                pn.x = fma(beta, pv.x, rv.x);
                pn.y = fma(beta, pv.y, rv.y);
                store_colour(pnew, vh, a, i, pn);
                if (P.x) {
                    R2 xv = load_colour(P.x, vh, a, i);
                    xv.x = fma(alpha, pv.x, xv.x);
                    xv.y = fma(alpha, pv.y, xv.y);
                    store_colour(P.x, vh, a, i, xv);
                }
            } else {
                const R2 qv = load_colour(EPI == EPI_NORMAL && P.psel ? pnew : P.q, vh, a, i);
                R2 o;
                o.x = fma(P.m2, qv.x, -acc.x);
                o.y = fma(P.m2, qv.y, -acc.y);
                if constexpr (EPI == EPI_NORMAL) {  // out = m^2 q - D in;  part = Re <q, out>
                    part += (double)fma(qv.y, o.y, qv.x * o.x);
                } else {  // out = b - m^2 q + D in;  part = ||out||^2   (FP64 only)
                    const double2 bv = load_colour(P.b, vh, a, i);
                    o.x = (R)bv.x - o.x;
                    o.y = (R)bv.y - o.y;
                    part = fma((double)o.x, (double)o.x, part);
                    part = fma((double)o.y, (double)o.y, part);
                }
                store_colour(P.out, vh, a, i, o);
            }
        }
        __syncthreads();  // the sums are read before the next sites' overwrite them
    }
    if constexpr (EPI == EPI_NORMAL || EPI == EPI_RESID) finish_reduction<R, EPI>(P, part, smem);
}

template <typename R, int FMT, bool NAIK>
static void launch_split_t(int grid, bool pdl, int epi, const DsParams<R> &P, cudaStream_t st) {
    auto kernel = epi == EPI_PLAIN ? dslash_split_kernel<R, FMT, NAIK, EPI_PLAIN>
                                   : dslash_split_kernel<R, FMT, NAIK, EPI_NORMAL>;
    if constexpr (std::is_same<R, double>::value) {
        if (epi == EPI_RESID) kernel = dslash_split_kernel<R, FMT, NAIK, EPI_RESID>;
    } else {
        if (epi == EPI_PUPD) kernel = dslash_split_kernel<R, FMT, NAIK, EPI_PUPD>;
    }
    launch_k(kernel, dim3(grid), dim3(kSplitBlock), 0, st, pdl, P);
}

template <typename R, int FMT>
static void launch_split_n(int grid, bool pdl, bool naik, int epi, const DsParams<R> &P, cudaStream_t st) {
    if (naik)
        launch_split_t<R, FMT, true>(grid, pdl, epi, P, st);
    else
        launch_split_t<R, FMT, false>(grid, pdl, epi, P, st);
}

// Blocks: 32 sites each; the launches that end in a grid reduction run a
// persistent grid, so that each block pays the reduction's tail once (normal
// operator, two-row FP32 with Naik, 24^4: 39 us against 55).
constexpr int kSplitMinBlocks64 = 4, kSplitMinBlocks32 = 8;
static int split_grid(const qex_lattice *lat, int epi, bool reduces, int per_sm) {
    const int all = blocks_for(lat->vh, kSplitSites), resident = sm_count() * per_sm;
    return reduces && (epi == EPI_NORMAL || epi == EPI_RESID) && resident < all ? resident : all;
}

template <>
void launch_split<double>(const qex_lattice *lat, int, bool naik, int epi, const DsParams<double> &P, bool pdl,
                          cudaStream_t st) {
    launch_split_n<double, 0>(split_grid(lat, epi, P.S != nullptr, kSplitMinBlocks64), pdl, naik, epi, P, st);
}

template <>
void launch_split<float>(const qex_lattice *lat, int fmt, bool naik, int epi, const DsParams<float> &P, bool pdl,
                         cudaStream_t st) {
    const int grid = split_grid(lat, epi, P.S != nullptr, kSplitMinBlocks32);
    if (fmt == 0)
        launch_split_n<float, 0>(grid, pdl, naik, epi, P, st);
    else if (fmt == 1)
        launch_split_n<float, 1>(grid, pdl, naik, epi, P, st);
    else if (fmt == 2)
        launch_split_n<float, 2>(grid, pdl, naik, epi, P, st);
    else
        launch_split_n<float, 3>(grid, pdl, naik, epi, P, st);
}

}  // namespace qex
