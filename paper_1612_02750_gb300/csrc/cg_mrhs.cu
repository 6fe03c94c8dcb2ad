// cg_mrhs.cu -- conjugate gradient on A = m^2 - D_eo D_oe for N right-hand
// sides at once (FP64, or FP32 inner with FP64 reliable updates).
//
// The N solves share every operator application (qex_dslash_mrhs reads each
// link once for all of them) and keep their own alpha, beta and residual
// norms.  They iterate in lockstep; a right-hand side whose FP64 true
// residual meets tol is frozen (its `active` flag drops) while the others go
// on.  A reliable update, requested by any active right-hand side, is done
// for all active ones: x += x_hat, r = b - A x in FP64, r_hat = (float) r,
// beta_r = ||r||^2 / rr_r with the previous iterated norm.  An iteration is
// four kernels: direction update (mixed precision: with the iterate's update by
// the previous step, so that p is read once for both), D_oe, normal operator
// with the per-RHS <p, Ap>, residual update with the per-RHS norms.  The host
// enqueues them in batches, one batch ahead of the scalars it reads.
//
// What bounds it (24^4, 16 sources, 16-bit links): the Dslash kernels by the
// L2's bandwidth (about 9 TB/s of neighbour vectors and links), the vector
// kernels by HBM (every field is 64 MB).  Forming p = r + beta p at each of the
// eight neighbour reads instead of in a pass of its own gathered two fields:
// 115 us a D_oe against 66; an iteration took 355 us, now 267.  Small lattices
// are bound by the chain of launches and grid reductions, 2 to 3 us each (8^4, 8
// sources: 32 us an iteration, now 23): each kernel comes up while the one before
// still runs, the sums take one release-acquire atomic a block, and the last
// block has read what it decides on before they are in.  A kernel lets the next
// one up only after its own wait: two kernels waiting at once crowded the running
// one's blocks onto fewer SMs (12^4, 3 sources: 34.5 us an iteration, now 28.5).
#include <math.h>
#include <string.h>

#include "qex_kernels.cuh"

namespace qex {

qex_status check_dslash_args(const qex_lattice *lat, qex_prec prec, const void *fat, const void *lng,
                             const void *in, const void *out);

// blockIdx.y = right-hand side: p = r + beta p and, with x, x += alpha p with
// the p and alpha of the iteration before (0 after a reliable update).
template <typename R>
__global__ void __launch_bounds__(kBlock)
update_p_mrhs_kernel(int vh, R *__restrict__ x, const R *__restrict__ r, R *__restrict__ p, const MrhsScalars *S) {
    pdl_wait();
    pdl_trigger();
    const int rh = blockIdx.y;
    const R beta = (R)S->beta[rh], alpha = x ? (R)S->alpha[rh] : R(0);
    if (S->halt | !S->active[rh]) return;  // uniform
    const size_t off = (size_t)rh * 6 * vh;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < vh; i += gridDim.x * blockDim.x) {
        const Vec3<R> rv = load_vec(r + off, vh, i);
        Vec3<R> pv = load_own(p + off, vh, i);
        if (x) {
            Vec3<R> xv = load_own(x + off, vh, i);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                xv.c[a].re = fma(alpha, pv.c[a].re, xv.c[a].re);
                xv.c[a].im = fma(alpha, pv.c[a].im, xv.c[a].im);
            }
            store_vec(x + off, vh, i, xv);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            pv.c[a].re = fma(beta, pv.c[a].re, rv.c[a].re);
            pv.c[a].im = fma(beta, pv.c[a].im, rv.c[a].im);
        }
        store_vec(p + off, vh, i, pv);
    }
}

// blockIdx.y = right-hand side.  r -= alpha ap; ||r||^2 (with x, also x +=
// alpha p); then, in the last block, the lockstep decision: if any active
// right-hand side asks for a reliable update (or the cap is reached), nobody
// advances rr/beta and the reliable update takes over; otherwise each advances.
template <typename R>
__global__ void __launch_bounds__(kBlock)
update_r_mrhs_kernel(int vh, int nrhs, R *__restrict__ x, R *__restrict__ r, const R *__restrict__ p,
                     const R *__restrict__ ap, MrhsScalars *S, double *partials, unsigned int *counter) {
    __shared__ double smem[32];
    __shared__ bool is_last;
    __shared__ double rr_new[kMaxRhs];
    pdl_wait();
    pdl_trigger();
    // what the last block decides on (a right-hand side a thread), read ahead of
    // the sums: a read after another there costs 0.6 us
    const int q = threadIdx.x, rh = blockIdx.y;
    bool mine = false;
    double rr = 0.0, rmax2 = 0.0, stop2 = 0.0;
    int iters = 0;
    if (q < nrhs) {
        mine = S->active[q] != 0;
        rr = S->rr[q];
        rmax2 = S->rmax2[q];
        stop2 = S->stop2[q];
        iters = S->iters[q];
    }
    const double delta2 = S->delta2;
    const int iter = S->iter + 1, error = S->error;
    const bool capped = iter >= S->maxiter || (S->max_cycle > 0 && iter - S->ru_iter0 >= S->max_cycle);
    const bool on = S->active[rh] != 0;
    const R alpha = (R)S->alpha[rh];
    if (S->halt) return;  // uniform
    const size_t off = (size_t)rh * 6 * vh;
    double part = 0.0;
    if (on) {
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < vh; k += gridDim.x * blockDim.x) {
            const int i = vh - 1 - k;  // against the normal operator's order
            Vec3<R> rv = load_own(r + off, vh, i);
            const Vec3<R> av = load_vec(ap + off, vh, i);
            if (x) {
                Vec3<R> xv = load_own(x + off, vh, i);
                const Vec3<R> pv = load_vec(p + off, vh, i);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    xv.c[a].re = fma(alpha, pv.c[a].re, xv.c[a].re);
                    xv.c[a].im = fma(alpha, pv.c[a].im, xv.c[a].im);
                }
                store_vec(x + off, vh, i, xv);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                rv.c[a].re = fma(-alpha, av.c[a].re, rv.c[a].re);
                rv.c[a].im = fma(-alpha, av.c[a].im, rv.c[a].im);
                part += (double)(rv.c[a].re * rv.c[a].re + rv.c[a].im * rv.c[a].im);
            }
            store_vec(r + off, vh, i, rv);
        }
    }
    const int lane = q & 31, warp = q >> 5, nw = blockDim.x >> 5;
    part = warp_sum(part);
    if (lane == 0) smem[warp] = part;
    __syncthreads();
    if (warp == 0) {
        const double bs = warp_sum(lane < nw ? smem[lane] : 0.0);
        if (lane == 0) {
            partials[(size_t)rh * gridDim.x + blockIdx.x] = bs;
            is_last = arrive_last(counter, gridDim.x * gridDim.y);
        }
    }
    __syncthreads();
    if (!is_last) return;
    // one warp per right-hand side, fixed order over the blocks
    for (int k = warp; k < nrhs; k += nw) {
        double v = 0.0;
#pragma unroll 4
        for (int bx = lane; bx < (int)gridDim.x; bx += 32) v += __ldcg(partials + (size_t)k * gridDim.x + bx);
        v = warp_sum(v);
        if (lane == 0) rr_new[k] = v;
    }
    __syncthreads();
    const double v = mine ? rr_new[q] : 0.0;
    const bool failed = __syncthreads_or(mine && !isfinite(v)) || error;
    if (v > rmax2) rmax2 = v;
    const bool ru = __syncthreads_or(mine && (v <= stop2 || v < delta2 * rmax2)) || capped;
    if (mine) {
        S->iters[q] = iters + 1;
        S->rmax2[q] = rmax2;
        if (!failed && !ru) {
            S->beta[q] = v / rr;
            S->rr[q] = v;
        }
    }
    if (q == 0) {
        S->iter = iter;
        if (failed) S->error = error ? error : 1;
        if (failed || ru) S->halt = 1;
        if (!failed && ru) S->need_ru = 1;
    }
}

// blockIdx.y = right-hand side: x64 += xh32 + alpha p (the step that the next
// direction update would have taken), xh32 = 0 (active ones).
__global__ void __launch_bounds__(kBlock)
accum_x_mrhs_kernel(int vh, double *__restrict__ x, float *__restrict__ xh, const float *__restrict__ p,
                    const MrhsScalars *S) {
    const int rh = blockIdx.y;
    if (!S->active[rh]) return;
    const size_t off = (size_t)rh * 6 * vh;
    const float alpha = (float)S->alpha[rh];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < vh; i += gridDim.x * blockDim.x) {
        Vec3<double> xv = load_own(x + off, vh, i);
        const Vec3<float> hv = load_own(xh + off, vh, i), pv = load_vec(p + off, vh, i);
        Vec3<float> z;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            xv.c[a].re += (double)fmaf(alpha, pv.c[a].re, hv.c[a].re);
            xv.c[a].im += (double)fmaf(alpha, pv.c[a].im, hv.c[a].im);
            z.c[a].re = z.c[a].im = 0.f;
        }
        store_vec(x + off, vh, i, xv);
        store_vec(xh + off, vh, i, z);
    }
}

// blockIdx.y = right-hand side: r32 = (float) r64 (active ones).
__global__ void __launch_bounds__(kBlock)
lower_r_mrhs_kernel(int vh, const double *__restrict__ r64, float *__restrict__ r32, MrhsScalars *S) {
    const int rh = blockIdx.y;
    if (blockIdx.x == 0 && threadIdx.x == 0) S->alpha[rh] = 0.0;  // no step of the iterate is pending
    if (!S->active[rh]) return;
    const size_t off = (size_t)rh * 6 * vh;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < vh; i += gridDim.x * blockDim.x) {
        const Vec3<double> rd = load_vec(r64 + off, vh, i);
        Vec3<float> rv;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            rv.c[a].re = (float)rd.c[a].re;
            rv.c[a].im = (float)rd.c[a].im;
        }
        store_vec(r32 + off, vh, i, rv);
    }
}

// blockIdx.y = right-hand side: ||b_r||^2 -> bb, stop2; zero sources are
// solved at once (x = 0, done).
__global__ void __launch_bounds__(kBlock)
norm2_mrhs_kernel(int vh, int nrhs, const double *__restrict__ b, double *__restrict__ x, MrhsScalars *S,
                  double *partials, unsigned int *counter) {
    __shared__ double smem[32];
    __shared__ unsigned int is_last;
    const int rh = blockIdx.y;
    const size_t off = (size_t)rh * 6 * vh;
    double part = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < vh; i += gridDim.x * blockDim.x) {
        const Vec3<double> v = load_vec(b + off, vh, i);
#pragma unroll
        for (int a = 0; a < 3; ++a) part += v.c[a].re * v.c[a].re + v.c[a].im * v.c[a].im;
    }
    const double bs = block_sum(part, smem);
    if (threadIdx.x == 0) {
        partials[(size_t)rh * gridDim.x + blockIdx.x] = bs;
        __threadfence();
        const unsigned int t = atomicAdd(counter, 1u);
        is_last = (t == gridDim.x * gridDim.y - 1) ? 1u : 0u;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int q = warp; q < nrhs; q += nw) {
        double v = 0.0;
        for (int bx = lane; bx < (int)gridDim.x; bx += 32) v += __ldcg(partials + (size_t)q * gridDim.x + bx);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) {
            S->bb[q] = v;
            S->stop2[q] = S->tol2 * v;
            if (!isfinite(v)) S->error = 1;
            if (v == 0.0) {  // zero source: x = 0 is exact
                S->active[q] = 0;
                S->done[q] = 1;
            }
        }
    }
    if (threadIdx.x == 0) *counter = 0u;
}

// Blocks per SM of the vector kernels over all right-hand sides (24^4, 16
// sources: 297 us an iteration at 4, 302 at 8; at 64, a pass each, the block
// sums' FP64 work took as long as the vectors: 92 us a residual update, now 45).
constexpr int kMrhsBlasPerSm = 4;
static size_t align256m(size_t n) { return (n + 255) & ~size_t(255); }

}  // namespace qex

using namespace qex;

extern "C" qex_status qex_cg_mrhs(const qex_lattice *latc, qex_prec inner, const void *fat64, const void *lng64,
                                  const void *fat32, const void *lng32, double c_naik, double mass, int nrhs,
                                  const void *b64, void *x64, double tol, int maxiter, double delta, void *stream,
                                  qex_cg_stats *stats) {
    qex_status st;
    if ((st = check_lattice(latc)) || (st = check_prec(inner))) return st;
    if ((st = check_dslash_args(latc, QEX_F64, fat64, lng64, b64, x64))) return st;
    if (nrhs < 1 || nrhs > QEX_MRHS_MAX) {
        set_error("nrhs must be in [1, %d] (got %d)", QEX_MRHS_MAX, nrhs);
        return QEX_ERR_ARG;
    }
    const bool mixed = inner != QEX_F64;
    if (mixed && (!fat32 || !aligned16(fat32) || (lng64 && (!lng32 || !aligned16(lng32))))) {
        set_error("mixed precision needs aligned FP32 copies of the fat (and long) links");
        return QEX_ERR_ARG;
    }
    if (!(tol > 0.0) || maxiter < 0 || !(delta >= 0.0 && delta < 1.0)) {
        set_error("need tol > 0, maxiter >= 0 and 0 <= delta < 1");
        return QEX_ERR_ARG;
    }
    qex_lattice *lat = const_cast<qex_lattice *>(latc);
    if ((st = ensure_scratch(lat))) return st;
    const cudaStream_t s = as_stream(stream);
    const int vh = (int)lat->vh;
    // nrhs fields back to back, 6*vh reals apart (16-byte aligned: vh is even)
    const size_t f64 = align256m((size_t)vh * 48 * nrhs), f32 = align256m((size_t)vh * 24 * nrhs);
    // work: r64, tmp64 (+ p64, ap64 in FP64 mode) | xh, r, p, ap, tmp (FP32 mode); scalars
    const size_t need = (mixed ? 2 * f64 + 5 * f32 : 4 * f64) + align256m(sizeof(MrhsScalars));
    if ((st = ensure_work(lat, need))) return st;
    char *w = (char *)lat->work;
    double *r64 = (double *)w;
    w += f64;
    double *tmp64 = (double *)w;
    w += f64;
    void *xi, *ri, *pi, *api, *tmpi;
    const size_t fi = mixed ? f32 : f64;
    if (mixed) {
        xi = w;
        w += fi;
        ri = w;
        w += fi;
    } else {
        xi = x64;
        ri = r64;
    }
    pi = w;
    w += fi;
    api = w;
    w += fi;
    if (mixed) {
        tmpi = w;
        w += fi;
    } else {
        tmpi = tmp64;
    }
    MrhsScalars *S = (MrhsScalars *)w;

    MrhsScalars init;
    memset(&init, 0, sizeof(init));
    init.nrhs = nrhs;
    init.tol2 = tol * tol;
    init.delta2 = mixed ? delta * delta : 0.0;
    init.max_cycle = ru_max_cycle(inner);
    init.maxiter = maxiter;
    for (int q = 0; q < nrhs; ++q) init.active[q] = 1;
    MrhsScalars *host = nullptr;
    QEX_CUDA(cudaMallocHost(&host, 2 * sizeof(MrhsScalars)));  // two readback slots
    *host = init;
    cudaEvent_t t0, t1;
    QEX_CUDA(cudaEventCreate(&t0));
    QEX_CUDA(cudaEventCreate(&t1));
    QEX_CUDA(cudaEventRecord(t0, s));
    QEX_CUDA(cudaMemcpyAsync(S, host, sizeof(MrhsScalars), cudaMemcpyHostToDevice, s));
    const size_t fbytes = (size_t)nrhs * vh * (mixed ? 24 : 48);
    QEX_CUDA(cudaMemsetAsync(pi, 0, fbytes, s));
    if (mixed) QEX_CUDA(cudaMemsetAsync(xi, 0, fbytes, s));
    // about kMrhsBlasPerSm blocks an SM in all, however many right-hand sides
    int nbb = (sm_count() * kMrhsBlasPerSm + nrhs - 1) / nrhs;
    if (nbb > blas_blocks(lat)) nbb = blas_blocks(lat);
    const dim3 bgrid(nbb, nrhs);
    norm2_mrhs_kernel<<<bgrid, kBlock, 0, s>>>(vh, nrhs, (const double *)b64, (double *)x64, S, lat->partials,
                                               lat->counter);
    QEX_CHECK_LAUNCH("norm2_mrhs_kernel");

    MrhsArgs a = {};
    a.nrhs = nrhs;
    a.c3 = c_naik;
    a.m2 = mass * mass;
    a.S = S;
    auto reliable_update = [&]() -> qex_status {
        if (mixed) {
            accum_x_mrhs_kernel<<<bgrid, kBlock, 0, s>>>(vh, (double *)x64, (float *)xi, (const float *)pi, S);
            QEX_CHECK_LAUNCH("accum_x_mrhs_kernel");
        }
        MrhsArgs d = a;
        d.prec = QEX_F64;
        d.fat = fat64;
        d.lng = lng64;
        d.out_parity = 1;
        d.in = x64;
        d.out = tmp64;
        d.epi = EPI_PLAIN;
        MrhsScalars *keep = d.S;
        d.S = nullptr;  // plain application over all fields (frozen ones are harmless)
        qex_status e;
        if ((e = launch_dslash_mrhs(lat, d, s))) return e;
        d.S = keep;
        d.out_parity = 0;
        d.in = tmp64;
        d.out = r64;
        d.epi = EPI_RESID;
        d.q = x64;
        d.b = (const double *)b64;
        if ((e = launch_dslash_mrhs(lat, d, s))) return e;
        if (mixed) {
            lower_r_mrhs_kernel<<<bgrid, kBlock, 0, s>>>(vh, r64, (float *)ri, S);
            QEX_CHECK_LAUNCH("lower_r_mrhs_kernel");
        }
        return QEX_OK;
    };
    auto iteration = [&]() -> qex_status {
        // linked by programmatic launches: the next kernel's blocks come up while
        // this one's last are still running
        if (mixed)
            launch_k(update_p_mrhs_kernel<float>, bgrid, dim3(kBlock), 0, s, true, vh, (float *)xi, (const float *)ri,
                     (float *)pi, (const MrhsScalars *)S);
        else
            launch_k(update_p_mrhs_kernel<double>, bgrid, dim3(kBlock), 0, s, true, vh, (double *)nullptr,
                     (const double *)ri, (double *)pi, (const MrhsScalars *)S);
        QEX_CHECK_LAUNCH("update_p_mrhs_kernel");
        MrhsArgs d = a;
        d.pdl = 1;
        d.prec = inner;
        d.fat = mixed ? fat32 : fat64;
        d.lng = mixed ? lng32 : lng64;
        d.out_parity = 1;
        d.in = pi;
        d.out = tmpi;
        d.epi = EPI_PLAIN;
        // every kernel walks the sites the other way round from the one before,
        // and meets first what that one left in the L2 (2 %)
        d.reverse = 1;
        qex_status e;
        if ((e = launch_dslash_mrhs(lat, d, s))) return e;
        d.out_parity = 0;
        d.in = tmpi;
        d.out = api;
        d.epi = EPI_NORMAL;
        d.q = pi;
        d.reverse = 0;
        if ((e = launch_dslash_mrhs(lat, d, s))) return e;
        if (mixed)
            launch_k(update_r_mrhs_kernel<float>, bgrid, dim3(kBlock), 0, s, true, vh, nrhs, (float *)nullptr,
                     (float *)ri, (const float *)pi, (const float *)api, S, lat->partials, lat->counter);
        else
            launch_k(update_r_mrhs_kernel<double>, bgrid, dim3(kBlock), 0, s, true, vh, nrhs, (double *)xi,
                     (double *)ri, (const double *)pi, (const double *)api, S, lat->partials, lat->counter);
        QEX_CHECK_LAUNCH("update_r_mrhs_kernel");
        return QEX_OK;
    };
    auto fetch = [&](int slot) -> qex_status {
        QEX_CUDA(cudaMemcpyAsync(host + slot, S, sizeof(MrhsScalars), cudaMemcpyDeviceToHost, s));
        QEX_CUDA(cudaEventRecord(slot ? lat->ev1 : lat->ev0, s));
        return QEX_OK;
    };
    auto wait = [&](int slot) -> qex_status {
        QEX_CUDA(cudaEventSynchronize(slot ? lat->ev1 : lat->ev0));
        return QEX_OK;
    };

    qex_status result = QEX_OK;
    if ((st = reliable_update()) || (st = fetch(0)) || (st = wait(0))) {
        cudaFreeHost(host);
        return st;
    }
    // zero sources: x = 0 exactly
    for (int q = 0; q < nrhs; ++q)
        if (host->bb[q] == 0.0) QEX_CUDA(cudaMemsetAsync((double *)x64 + (size_t)q * 6 * vh, 0, (size_t)vh * 48, s));
    // Batches of iterations, the next one enqueued before the scalars of the
    // last are read; the iterations after a halt return at once.
    const int batch = 4;
    int slot = 0;  // the slot of the newest scalars that have arrived
    while (!host[slot].error && !host[slot].halt) {
        int queued = slot ^ 1;
        for (int k = 0; k < batch && !st; ++k) st = iteration();
        if (st || (st = fetch(queued))) break;
        for (;;) {
            const int next = queued ^ 1;
            for (int k = 0; k < batch && !st; ++k) st = iteration();
            if (st || (st = fetch(next)) || (st = wait(queued))) break;
            slot = queued;
            queued = next;
            if (host[slot].halt) break;
        }
        if (st || (st = wait(queued))) break;  // drain the queued batch
        slot = queued;
        if (host[slot].error || !host[slot].need_ru) continue;
        if ((st = reliable_update()) || (st = fetch(0)) || (st = wait(0))) break;
        slot = 0;
    }
    QEX_CUDA(cudaEventRecord(t1, s));
    QEX_CUDA(cudaEventSynchronize(t1));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, t0, t1);
    cudaEventDestroy(t0);
    cudaEventDestroy(t1);
    if (!st) {
        const MrhsScalars &last = host[slot];
        int all = 1;
        for (int q = 0; q < nrhs; ++q) all &= last.done[q];
        if (last.error) {
            set_error("NaN/Inf or CG breakdown in a multi-RHS solve");
            result = QEX_ERR_NAN;
        } else if (!all) {
            set_error("multi-RHS CG did not converge in %d iterations", maxiter);
            result = QEX_ERR_NOT_CONVERGED;
        }
        if (stats) {
            for (int q = 0; q < nrhs; ++q) {
                stats[q].iters = last.iters[q];
                stats[q].reliable_updates = last.reliable_updates > 0 ? last.reliable_updates - 1 : 0;
                stats[q].converged = last.done[q];
                stats[q].ff_updates = 0;
                stats[q].true_rel_resid = last.bb[q] > 0.0 ? sqrt(last.true_rr[q] / last.bb[q]) : 0.0;
                stats[q].time_ms = ms;
            }
        }
    } else {
        result = st;
    }
    cudaFreeHost(host);
    return result;
}
