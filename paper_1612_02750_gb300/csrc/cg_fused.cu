// cg_fused.cu -- the CG iteration of a small lattice as one persistent kernel.
//
// On a small lattice (a few thousand even sites) each of the three kernels of
// an iteration does a few microseconds of work and the launch, the drain of
// the grid and the last-block reduction tail cost as much again.  Here one
// cooperative launch (every block resident) runs the inner iterations back to
// back:
//   1. tmp = D_oe (r + beta p_old) with p_new stored        grid barrier
//   2. A p_new = m^2 p_new - D_eo tmp, block sums of <p,Ap>  grid barrier
//      every block sums the block partials in the same fixed order -> alpha
//   3. x += alpha p_new, r -= alpha A p_new, block sums of ||r||^2
//                                                            grid barrier
//      every block sums them -> beta, or the request for a reliable update
// until a reliable update is due (or an error): then the kernel writes the CG
// scalars back and returns, the host runs the FP64 reliable update with the
// ordinary kernels, and launches it again.  The iterations are the ones the
// three-kernel form computes (the reductions sum the same per-site terms in
// another block grouping).
//
// A site's four directions run on four warps, as in dslash_split.cu (a block
// is 32 sites per 128 threads), and its colours on three of them, which keep
// the three phases' vectors of a site at the same thread.
//
// Grid barriers: one 64-bit arrival counter, zeroed by the host before each
// launch and never reset in between; a block adds one (release) and polls until
// all have come (acquire).  Two L2 round trips, against about five for counters
// in two levels with a generation word.  A wait
// that lasts longer than a limit (clock64 cycles, about a second by default;
// the environment variable QEX_BARRIER_TIMEOUT_CYCLES sets another, which the
// tests use to make the limit run out) records a timeout in the error word
// and every block leaves at its next barrier, so a barrier can never hang the
// GPU; each block counts itself out on leaving, and the host then reports
// QEX_ERR_TIMEOUT with the count.
#include <math.h>
#include <stdlib.h>

#include "qex_dslash_dir.cuh"
#include "qex_kernels.cuh"

namespace qex {

template <typename R>
struct FusedArgs {
    Geom g;
    const R *fat, *lng;
    R c3, m2;
    R *x, *r, *p0, *p1, *ap, *tmp;
    CgScalars *S;
    double *partials;            // 2 * gridDim.x: block sums of <p, Ap> and ||r||^2
    unsigned long long *arrived; // blocks that have come to the barriers of this launch; top bit: a wait ran out
    int *bar_err;                // nonzero: a barrier timed out
    unsigned int *exited;        // blocks that have left the kernel
    long long timeout_cycles;    // longest wait at a barrier
};

// Most threads per block (FP64: 25 KB of sums a block of 256 with the Naik term).
template <typename R> struct FusedBlock { static constexpr int value = 512; };
template <> struct FusedBlock<double> { static constexpr int value = 256; };
constexpr long long kBarrierTimeoutCycles = 2000000000ll;  // default limit: about one second at 2 GHz
constexpr unsigned long long kBarrierFailed = 1ull << 63;

// One thread of a block arrives at the grid barrier and waits for `target`
// arrivals; false if some block's wait ran out (then every block leaves at its
// next barrier).  The release and the acquire carry what the block's other
// threads wrote before, and read after, a barrier of the block.
__device__ __forceinline__ bool arrive_and_wait(unsigned long long *arrived, int *err, unsigned long long target,
                                                long long timeout_cycles) {
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(arrived) : "memory");
    const long long t0 = clock64();
    for (;;) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(arrived) : "memory");
        if (v & kBarrierFailed) return false;
        if (v >= target) return true;
        if (clock64() - t0 > timeout_cycles) {
            atomicExch(err, 1);
            atomicOr(arrived, kBarrierFailed);
            return false;
        }
    }
}

// Vectors written by this kernel are read back in later phases of the same
// launch, so they are loaded through L2 (ld.global.cg), never through the
// read-only path that assumes data constant for the kernel's lifetime; only
// the links use that path.
__device__ __forceinline__ Vec3<float> load_vec_cg(const float *base, size_t vh, int i) {
    const float4 t = __ldcg(reinterpret_cast<const float4 *>(base) + i);
    const float2 u = __ldcg(reinterpret_cast<const float2 *>(base + 4 * vh) + i);
    Vec3<float> v;
    v.c[0].re = t.x;
    v.c[0].im = t.y;
    v.c[1].re = t.z;
    v.c[1].im = t.w;
    v.c[2].re = u.x;
    v.c[2].im = u.y;
    return v;
}
__device__ __forceinline__ Vec3<double> load_vec_cg(const double *base, size_t vh, int i) {
    Vec3<double> v;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double2 t = __ldcg(reinterpret_cast<const double2 *>(base) + a * vh + i);
        v.c[a].re = t.x;
        v.c[a].im = t.y;
    }
    return v;
}

__device__ __forceinline__ float2 load_colour_cg(const float *f, size_t vh, int a, int i) {
    return a < 2 ? __ldcg(reinterpret_cast<const float2 *>(f) + 2 * (size_t)i + a)
                 : __ldcg(reinterpret_cast<const float2 *>(f + 4 * vh) + i);
}
__device__ __forceinline__ double2 load_colour_cg(const double *f, size_t vh, int a, int i) {
    return __ldcg(reinterpret_cast<const double2 *>(f) + a * vh + i);
}

template <typename R>
__device__ __forceinline__ Vec3<R> axpy_vec_cg(const R *r, const R *p, R beta, size_t vh, int j) {
    const Vec3<R> rv = load_vec_cg(r, vh, j), pv = load_vec_cg(p, vh, j);
    Vec3<R> v;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        v.c[a].re = fma(beta, pv.c[a].re, rv.c[a].re);
        v.c[a].im = fma(beta, pv.c[a].im, rv.c[a].im);
    }
    return v;
}

// Loop state of the solve, identical in every block, kept in shared memory so
// that it holds no registers during the Dslash phases.
struct FusedState {
    double rr, beta, rmax2, alpha, pAp;
    double rr_ru;
    int iters, trips, need_ru, ru_ff, error;
    int ok;  // the last grid barrier was met
};

// Sum of `part` over the grid, in a fixed order: warps, then the block's warps,
// then the blocks; `then(total)` runs on thread 0.  It is a grid barrier as
// well.  The first warp does all that follows the block's sum, so the others
// wait once.  false: some block's wait ran out.
template <typename Then>
__device__ __forceinline__ bool fused_sum(double part, double *partials, unsigned long long *arrived, int *err,
                                          unsigned long long target, long long timeout_cycles, double *smem,
                                          FusedState &st, const Then &then) {
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if (lane == 0) smem[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = lane < warps ? smem[lane] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        int ok = 1;
        if (lane == 0) {
            partials[blockIdx.x] = v;
            ok = arrive_and_wait(arrived, err, target, timeout_cycles);
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();  // orders the lanes' reads after lane 0's acquire, which a shuffle does not
        if (ok) {
            double t = 0.0;
            for (int k = lane; k < (int)gridDim.x; k += 32) t += __ldcg(partials + k);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) then(t);
        }
        if (lane == 0) st.ok = ok;
    }
    __syncthreads();
    return st.ok != 0;
}

// ONE: every thread has one site at most, and keeps its colour of r, p, x and
// A p in registers from phase to phase.
template <typename R, int FMT, bool NAIK, bool ONE>
__device__ __forceinline__ void cg_fused_body(const FusedArgs<R> &A) {
    __shared__ double smem[32];
    __shared__ FusedState st;
    __shared__ DirSums<R, FMT, NAIK, FusedBlock<R>::value / 4> sums;
    CgScalars *S = A.S;
    if (S->halt) return;  // uniform
    const Geom &g = A.g;
    const size_t vh = (size_t)g.vh;
    const int nb = gridDim.x;
    // warp w: sites of group w / 4 of 32, direction (or colour) w % 4
    const int mu = (threadIdx.x >> 5) & 3, slot = (threadIdx.x >> 7) * 32 + (threadIdx.x & 31);
    const int first = blockIdx.x * (blockDim.x >> 2) + slot, stride = nb * (blockDim.x >> 2);
    const int rounds = ONE ? 1 : (g.vh + stride - 1) / stride;
    if (threadIdx.x == 0) {
        st.rr = S->rr;
        st.beta = S->beta;
        st.rmax2 = S->rmax2;
        st.alpha = S->alpha;
        st.pAp = S->pAp;
        st.iters = S->iters;
        st.trips = S->trips;
        st.need_ru = 0;
        st.ru_ff = 0;
        st.error = 0;
    }
    __syncthreads();
    unsigned long long target = 0;
    const bool keeps = ONE && mu < 3 && first < g.vh;
    typename Pair<R>::type rv, pv, xv, av;  // this thread's r, p, x, A p
    rv.x = rv.y = R(0);
    pv = xv = av = rv;
    if (keeps) {
        rv = load_colour_cg(A.r, vh, mu, first);
        pv = load_colour_cg((st.iters & 1) ? A.p1 : A.p0, vh, mu, first);
        xv = load_colour_cg(A.x, vh, mu, first);
    }
    for (;;) {
        const int it = st.iters;
        const R *pold = (it & 1) ? A.p1 : A.p0;
        R *pnew = (it & 1) ? A.p0 : A.p1;
        {   // 1. tmp = D_oe (r + beta p_old); p_new at the site's own even index
            const R b = (R)st.beta, *const r = A.r;
            const auto direction = [=](int j) { return axpy_vec_cg(r, pold, b, vh, j); };
            for (int n = 0, i = first; n < rounds; ++n, i += stride) {
                const bool mine = i < g.vh;
                if (mine) {
                    if (!ONE && mu < 3) {
                        rv = load_colour_cg(A.r, vh, mu, i);
                        pv = load_colour_cg(pold, vh, mu, i);
                    }
                    sums.put(g, A.fat, A.lng, A.c3, 1, i, mu, slot, direction);
                    if (mu < 3) {
                        pv.x = fma(b, pv.x, rv.x);
                        pv.y = fma(b, pv.y, rv.y);
                        store_colour(pnew, vh, mu, i, pv);
                    }
                }
                __syncthreads();
                if (mine && mu < 3)
                    store_colour(A.tmp, vh, mu, i, sums.get(g, A.fat, A.lng, A.c3, 1, i, mu, slot, direction));
                if (n + 1 < rounds) __syncthreads();
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) st.ok = arrive_and_wait(A.arrived, A.bar_err, target += nb, A.timeout_cycles);
        __syncthreads();
        if (!st.ok) return;
        {   // 2. A p_new = m^2 p_new - D_eo tmp; <p_new, A p_new> -> alpha
            double part = 0.0;
            const R *const tmp = A.tmp;
            const auto field = [=](int j) { return load_vec_cg(tmp, vh, j); };
            for (int n = 0, i = first; n < rounds; ++n, i += stride) {
                const bool mine = i < g.vh;
                if (mine) {
                    if (!ONE && mu < 3) pv = load_colour_cg(pnew, vh, mu, i);
                    sums.put(g, A.fat, A.lng, A.c3, 0, i, mu, slot, field);
                }
                __syncthreads();
                if (mine && mu < 3) {
                    const auto d = sums.get(g, A.fat, A.lng, A.c3, 0, i, mu, slot, field);
                    av.x = fma(A.m2, pv.x, -d.x);
                    av.y = fma(A.m2, pv.y, -d.y);
                    if (!ONE) store_colour(A.ap, vh, mu, i, av);
                    part += (double)fma(pv.y, av.y, pv.x * av.x);
                }
                if (n + 1 < rounds) __syncthreads();
            }
            if (!fused_sum(part, A.partials, A.arrived, A.bar_err, target += nb, A.timeout_cycles, smem, st,
                           [&](double pAp) {
                               st.pAp = pAp;
                               if (!(pAp > 0.0) || !isfinite(pAp))
                                   st.error = isfinite(pAp) ? 2 : 1;
                               else
                                   st.alpha = st.rr / pAp;
                           }))
                return;
            if (st.error) break;
        }
        {   // 3. x += alpha p_new; r -= alpha A p_new; ||r||^2
            const R al = (R)st.alpha;
            double part = 0.0;
            if (mu < 3) {
                for (int n = 0, i = first; n < rounds && i < g.vh; ++n, i += stride) {
                    if (!ONE) {
                        xv = load_colour_cg(A.x, vh, mu, i);
                        rv = load_colour_cg(A.r, vh, mu, i);
                        pv = load_colour_cg(pnew, vh, mu, i);
                        av = load_colour_cg(A.ap, vh, mu, i);
                    }
                    xv.x = fma(al, pv.x, xv.x);
                    xv.y = fma(al, pv.y, xv.y);
                    rv.x = fma(-al, av.x, rv.x);
                    rv.y = fma(-al, av.y, rv.y);
                    if (!ONE) store_colour(A.x, vh, mu, i, xv);
                    store_colour(A.r, vh, mu, i, rv);
                    part += (double)fma(rv.y, rv.y, rv.x * rv.x);
                }
            }
            if (!fused_sum(part, A.partials + nb, A.arrived, A.bar_err, target += nb, A.timeout_cycles, smem, st,
                           [&](double rr_new) {
                               st.iters += 1;
                               st.trips += 1;
                               if (!isfinite(rr_new)) {
                                   st.error = 1;
                                   return;
                               }
                               if (rr_new > st.rmax2) st.rmax2 = rr_new;
                               const bool long_cycle = S->max_cycle > 0 && st.iters - S->ru_iter0 >= S->max_cycle;
                               if (rr_new <= S->stop2 || rr_new < S->delta2 * st.rmax2 || st.iters >= S->maxiter ||
                                   long_cycle) {
                                   // rr keeps its value: beta then comes from the true residual
                                   st.need_ru = 1;
                                   st.ru_ff = (S->ff_ok && rr_new > S->stop2 && st.iters < S->maxiter) ? 1 : 0;
                                   st.rr_ru = rr_new;
                               } else {
                                   st.beta = rr_new / st.rr;
                                   st.rr = rr_new;
                               }
                           }))
                return;
            if (st.error || st.need_ru) break;
        }
    }
    if (keeps) store_colour(A.x, vh, mu, first, xv);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S->rr = st.rr;
        S->beta = st.beta;
        S->rmax2 = st.rmax2;
        S->alpha = st.alpha;
        S->pAp = st.pAp;
        S->iters = st.iters;
        S->trips = st.trips;
        if (st.error) S->error = st.error;
        S->need_ru = st.need_ru;
        if (st.need_ru) {
            S->ru_ff = st.ru_ff;
            S->rr_ru = st.rr_ru;
        }
        S->halt = 1;
    }
}

template <typename R, int FMT, bool NAIK, bool ONE>
__global__ void __launch_bounds__(FusedBlock<R>::value, 512 / FusedBlock<R>::value)
cg_fused_kernel(const __grid_constant__ FusedArgs<R> A) {
    cg_fused_body<R, FMT, NAIK, ONE>(A);
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(A.exited, 1u);  // every way out of the body ends here
}

template <typename R, int FMT, bool NAIK>
static qex_status launch_fused_t(qex_lattice *lat, const FusedArgs<R> &A0, cudaStream_t st) {
    // The smallest block that lets one block an SM cover the lattice: fewer
    // blocks meet sooner at a barrier, smaller ones sum sooner.  12^4 with Naik,
    // us an iteration: 15.1 (128 threads), 14.5 (256), 13.3 (384), 14.7 (512);
    // 8^4: 10.1, 10.7, 11.8, 12.9; 16^4: 20.9, 17.5, 17.6, 16.9.
#ifdef QEX_FUSED_BLOCK
    const int block = QEX_FUSED_BLOCK;
#else
    int block = 128;
    while (block < FusedBlock<R>::value && blocks_for(lat->vh, block / 4) > sm_count()) block += 128;
#endif
    const int want = blocks_for(lat->vh, block / 4);
    auto kernel = cg_fused_kernel<R, FMT, NAIK, true>;
    int nb = want;
    for (int one = 1; one >= 0; --one) {
        if (!one) kernel = cg_fused_kernel<R, FMT, NAIK, false>;
        int per_sm = 0;
        QEX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0));
        if (per_sm < 1) {
            set_error("the fused CG kernel does not fit on an SM");
            return QEX_ERR_CUDA;
        }
        const int cap = per_sm * sm_count();
        nb = want < cap ? want : cap;
        if (want <= cap) break;  // one site a thread at most
    }
    // 2 nb partial sums, then the arrival counter, in the lattice's partials
    // buffer; the error word is counter[3] of the lattice scratch; all fresh for
    // every launch
    if ((size_t)lat->partials_len < 2 * (size_t)nb + 32) {
        set_error("internal: partials buffer too small for the fused CG kernel");
        return QEX_ERR_ARG;
    }
    FusedArgs<R> A = A0;
    A.partials = lat->partials;
    A.arrived = reinterpret_cast<unsigned long long *>(lat->partials + 2 * (size_t)nb + 16);
    QEX_CUDA(cudaMemsetAsync(A.arrived, 0, sizeof(*A.arrived), st));
    QEX_CUDA(cudaMemsetAsync(lat->counter + 3, 0, 2 * sizeof(unsigned int), st));  // error word, exit count
    A.bar_err = reinterpret_cast<int *>(lat->counter + 3);
    A.exited = lat->counter + 4;
    A.timeout_cycles = kBarrierTimeoutCycles;
    if (const char *e = getenv("QEX_BARRIER_TIMEOUT_CYCLES")) {
        const long long v = atoll(e);
        if (v > 0) A.timeout_cycles = v;
    }
    lat->fused_blocks = nb;
    void *args[] = {&A};
    QEX_CUDA(cudaLaunchCooperativeKernel((const void *)kernel, dim3(nb), dim3(block), args, 0, st));
    note_launch();
    return QEX_OK;
}

template <typename R, int FMT>
static qex_status launch_fused_n(qex_lattice *lat, const FusedVectors &v, const void *fat, const void *lng, double c3,
                                 double m2, cudaStream_t st) {
    FusedArgs<R> A = {};
    A.g = lat->geom;
    A.fat = (const R *)fat;
    A.lng = (const R *)lng;
    A.c3 = (R)c3;
    A.m2 = (R)m2;
    A.x = (R *)v.x;
    A.r = (R *)v.r;
    A.p0 = (R *)v.p[0];
    A.p1 = (R *)v.p[1];
    A.ap = (R *)v.ap;
    A.tmp = (R *)v.tmp;
    A.S = lat->scalars;
    return lng ? launch_fused_t<R, FMT, true>(lat, A, st) : launch_fused_t<R, FMT, false>(lat, A, st);
}

// One run of the fused iteration kernel.
qex_status launch_cg_fused(qex_lattice *lat, qex_prec inner, const void *fat, const void *lng, double c3, double m2,
                           const FusedVectors &v, cudaStream_t st) {
    switch (inner) {
        case QEX_F64: return launch_fused_n<double, 0>(lat, v, fat, lng, c3, m2, st);
        case QEX_F32: return launch_fused_n<float, 0>(lat, v, fat, lng, c3, m2, st);
        case QEX_F32_R12: return launch_fused_n<float, 1>(lat, v, fat, lng, c3, m2, st);
        case QEX_F32_R12H: return launch_fused_n<float, 2>(lat, v, fat, lng, c3, m2, st);
        case QEX_F32_S16: return launch_fused_n<float, 3>(lat, v, fat, lng, c3, m2, st);
        default: set_error("unknown inner precision"); return QEX_ERR_ARG;
    }
}

// Whether a barrier of the last fused run timed out (reads the error word),
// and how many of its blocks left the kernel.
qex_status fused_barrier_status(qex_lattice *lat, cudaStream_t st, int *timed_out, int *exited) {
    unsigned int v[2] = {0u, 0u};
    QEX_CUDA(cudaMemcpyAsync(v, lat->counter + 3, sizeof(v), cudaMemcpyDeviceToHost, st));
    QEX_CUDA(cudaStreamSynchronize(st));
    *timed_out = v[0] != 0;
    if (exited) *exited = (int)v[1];
    return QEX_OK;
}

}  // namespace qex
