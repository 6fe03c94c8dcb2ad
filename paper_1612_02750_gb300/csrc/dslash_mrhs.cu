// dslash_mrhs.cu -- the even-odd staggered operator applied to N right-hand
// sides at once, each link read from memory once for all of them, with the
// epilogues of the multi-RHS CG.
//
// Fields: N half fields back to back (field r starts at r * qex_field_bytes).
// Per site the algorithmic traffic is the 8 (16 with Naik) links once plus,
// per right-hand side, the input vector once and the output once.  The
// reducing epilogues run a persistent grid-stride loop and reduce per
// right-hand side in a fixed order (bit-reproducible).
#include "qex_dslash64.cuh"
#include "qex_dslash_site.cuh"
#include "qex_kernels.cuh"

namespace qex {

// Thread mapping: one output site per thread and a group of KR right-hand
// sides per thread (held in registers): each link is loaded and decoded once
// per group and applied to all KR vectors.
// A block is 256 sites of one group; linear block b covers site block
// b / ngroups and group b % ngroups, so the blocks that reuse a link run back
// to back and find it in L2.
constexpr int kMrhsBlock = 256;  // threads (sites) per block
// Right-hand sides per thread (KR) and resident blocks per SM (MINB, the
// register cap).  FP32: 4 at 2 blocks (128 registers), 2 at 3 blocks; FP64: one at
// 2 blocks (dslash_site64).  24^4, two-row links, 16 right-hand sides, KR x MINB:
// 64 us (4 x 2), 70 (4 x 3), 70 (3 x 3), 71 (2 x 3), 73 (2 x 4), 68 (6 x 2).
template <typename R, int KR>
struct MrhsShape {
    static constexpr int minb = KR == 4 ? 2 : 3;
};
template <int KR>
struct MrhsShape<double, KR> {
    static constexpr int minb = 2;
};
// Two fields a thread where their blocks still find an SM each, which halves the
// work in a thread's chain (12^4, 4 right-hand sides: 4.0 us against 5.4); four
// where only theirs do (12 there: 5.4 against 6.1); beyond that two if four would
// leave one or two over among few (24^4, 5 right-hand sides: 27 us against 32).
static bool pairs_are_better(int nrhs, int vh) {
    const int nsb = (vh + kMrhsBlock - 1) / kMrhsBlock;
    if (nsb * ((nrhs + 1) / 2) <= sm_count()) return true;
    if (nsb * ((nrhs + 3) / 4) <= sm_count()) return false;
    return nrhs <= 10 && (nrhs % 4 == 1 || nrhs % 4 == 2);
}
// the largest persistent grid times KR of any reducing variant (partials per launch)
constexpr int kMrhsMaxPartialsPerSm = 8;

// ------------------------------------------------- hops through shared memory
// FP32: the link and the KR vectors of a hop are copied to shared memory one hop
// ahead (cp.async; a thread reads back only its own copies, so no barrier).
// With four vectors and a link in registers only 16 warps fit an SM, too few to
// hide a hop's loads behind the hop before by themselves: the issue slots were
// 55 % in use on 24^4, now 63 %.  What bounds it now is the L2's traffic (links
// and neighbour vectors) and the issue of the copies.  D_oe on 24^4, 16
// right-hand sides: two-row links 72 us, now 64, with Naik 136 and 120, 16-bit
// 77 and 66; 32^4, 8 of them, two-row 123 and 100.
template <int FMT>
struct LinkWords {  // 16-byte words and 8-byte words of a link, as planes
    static constexpr int n16 = FMT == 0 ? 4 : FMT == 1 ? 3 : FMT == 2 ? 1 : 2;
    static constexpr int n8 = FMT == 1 ? 0 : 1;
};

__device__ __forceinline__ void copy_async16_ca(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void copy_async8_ca(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

template <int KR, int N16, int N8>
struct HopStage {
    static constexpr int w16 = N16 + KR, w8 = N8 + KR;  // words a thread: link, then vectors
    static constexpr size_t bytes = (size_t)w16 * 16 + (size_t)w8 * 8;
    uint4 *a;  // [w16][threads]
    uint2 *b;  // [w8][threads]
    __device__ __forceinline__ HopStage(char *base, int stage) {
        char *s = base + stage * bytes * kMrhsBlock;
        a = reinterpret_cast<uint4 *>(s) + threadIdx.x;
        b = reinterpret_cast<uint2 *>(s + (size_t)w16 * 16 * kMrhsBlock) + threadIdx.x;
    }
    template <int FMT>
    __device__ __forceinline__ void issue(const float *links, size_t vh, int p, int mu, int li, const float *in,
                                          const size_t (&off)[KR], int j) const {
        constexpr int n16 = LinkWords<FMT>::n16, n8 = LinkWords<FMT>::n8;
        const char *blk = reinterpret_cast<const char *>(links) + (size_t)(p * 4 + mu) * (16 * n16 + 8 * n8) * vh;
#pragma unroll
        for (int w = 0; w < n16; ++w)
            copy_async16(reinterpret_cast<double2 *>(a + w * kMrhsBlock),
                         reinterpret_cast<const double2 *>(blk + (size_t)w * 16 * vh) + li);
        if (n8) copy_async8_ca(b, reinterpret_cast<const uint2 *>(blk + (size_t)n16 * 16 * vh) + li);
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            copy_async16_ca(a + (N16 + k) * kMrhsBlock, reinterpret_cast<const uint4 *>(in + off[k]) + j);
            copy_async8_ca(b + (N8 + k) * kMrhsBlock, reinterpret_cast<const uint2 *>(in + off[k] + 4 * vh) + j);
        }
    }
    template <int FMT>
    __device__ __forceinline__ Mat3<float> link(float *d) const {
        constexpr int n16 = LinkWords<FMT>::n16, n8 = LinkWords<FMT>::n8;
        uint32_t w[4 * n16 + 2 * n8];
#pragma unroll
        for (int k = 0; k < n16; ++k) {
            const uint4 t = a[k * kMrhsBlock];
            w[4 * k] = t.x;
            w[4 * k + 1] = t.y;
            w[4 * k + 2] = t.z;
            w[4 * k + 3] = t.w;
        }
        if (n8) {
            const uint2 t = b[0];
            w[4 * n16] = t.x;
            w[4 * n16 + 1] = t.y;
        }
        Mat3<float> m;
        if constexpr (FMT >= 2) {
            constexpr int n = FMT == 2 ? 6 : 9;
#pragma unroll
            for (int c = 0; c < n; ++c) {
                m.e[c].re = fix16_lo(w[c]);
                m.e[c].im = fix16_hi(w[c]);
            }
            if (FMT == 3) *d = __uint_as_float(w[9]);
        } else {
            constexpr int n = FMT == 1 ? 6 : 9;
#pragma unroll
            for (int c = 0; c < n; ++c) {
                m.e[c].re = __uint_as_float(w[2 * c]);
                m.e[c].im = __uint_as_float(w[2 * c + 1]);
            }
        }
        if constexpr (FMT == 1 || FMT == 2) reconstruct_row2(m);
        return m;
    }
    __device__ __forceinline__ Vec3<float> vec(int k) const {
        const uint4 t = a[(N16 + k) * kMrhsBlock];
        const uint2 u = b[(N8 + k) * kMrhsBlock];
        Vec3<float> v;
        v.c[0].re = __uint_as_float(t.x);
        v.c[0].im = __uint_as_float(t.y);
        v.c[1].re = __uint_as_float(t.z);
        v.c[1].im = __uint_as_float(t.w);
        v.c[2].re = __uint_as_float(u.x);
        v.c[2].im = __uint_as_float(u.y);
        return v;
    }
};

// The stage of an operator: room for its larger kind of link.
template <int FMT, bool NAIK, int KR>
struct StageOf {
    static constexpr int lf = FMT >= 2 ? 3 : 0;
    static constexpr int n16 = NAIK && LinkWords<lf>::n16 > LinkWords<FMT>::n16 ? LinkWords<lf>::n16
                                                                                 : LinkWords<FMT>::n16;
    static constexpr int n8 = NAIK ? 1 : LinkWords<FMT>::n8;
    typedef HopStage<KR, n16, n8> type;
};

// acc[k] += sg U v_k (DAG: U^+ v_k) from a stage, the arithmetic of dslash_site_n.
template <int FMT, bool DAG, int KR, typename Stage>
__device__ __forceinline__ void stage_mv(const Stage &st, float sg, Vec3<float> (&acc)[KR]) {
    float d = 1.f;
    const Mat3<float> u = st.template link<FMT>(&d);
#pragma unroll
    for (int k = 0; k < KR; ++k) {
        const Vec3<float> v = st.vec(k);
        if constexpr (FMT == 2) {
            if (DAG)
                acc_mdv_fix16(acc[k], sg, u, v);
            else
                acc_mv_fix16(acc[k], sg, u, v);
        } else {
            const float s = FMT == 3 ? sg * d : sg;
            if (DAG)
                acc_mdv(acc[k], s, u, v);
            else
                acc_mv(acc[k], s, u, v);
        }
    }
}

// (D in_k)(x) for the i-th site x (= s) of parity p, KR fields.
template <int FMT, bool NAIK, int KR>
__device__ __forceinline__ void dslash_site_staged(const Geom &g, const float *fat, const float *lng, float c3, int p,
                                                   int i, const Site &s, const float *in, const size_t (&off)[KR],
                                                   char *smem, Vec3<float> (&acc)[KR]) {
    constexpr int H = NAIK ? 16 : 8, LF = FMT >= 2 ? 3 : 0;  // hops in dslash_site_n's order; format of the long links
    typedef typename StageOf<FMT, NAIK, KR>::type Stage;
    const size_t vh = (size_t)g.vh;
#pragma unroll
    for (int k = 0; k < KR; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a) acc[k].c[a].re = acc[k].c[a].im = 0.f;
    auto issue = [&](int h) {
        const int mu = NAIK ? h >> 2 : h >> 1, step = NAIK && (h & 2) ? 3 : 1, back = h & 1;
        const int j = hop_index(g, s, mu, back ? -step : step);
        const Stage st(smem, h & 1);
        if (step == 1)
            st.template issue<FMT>(fat, vh, back ? 1 - p : p, mu, back ? j : i, in, off, j);
        else
            st.template issue<LF>(lng, vh, back ? 1 - p : p, mu, back ? j : i, in, off, j);
    };
    issue(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
    for (int h = 0; h < H; ++h) {
        if (h + 1 < H) issue(h + 1);
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 1;" ::: "memory");
        const int mu = NAIK ? h >> 2 : h >> 1, step = NAIK && (h & 2) ? 3 : 1, back = h & 1;
        const bool minus = ((eta_bit(s, mu) ^ (back ? bc_bit_bwd(g, s, mu, step) : bc_bit_fwd(g, s, mu, step))) != 0) !=
                           (back != 0);
        const Stage st(smem, h & 1);
        if (step == 1) {
            const float sg = minus ? -1.f : 1.f;
            if (back)
                stage_mv<FMT, true, KR>(st, sg, acc);
            else
                stage_mv<FMT, false, KR>(st, sg, acc);
        } else {
            const float sg = minus ? -c3 : c3;
            if (back)
                stage_mv<LF, true, KR>(st, sg, acc);
            else
                stage_mv<LF, false, KR>(st, sg, acc);
        }
    }
}

template <typename R>
struct MParams {
    Geom g;
    const R *fat, *lng;
    R c3;
    int p, nrhs, ngroups;
    const R *in;
    R *out;
    const R *q;
    const double *b;
    R m2;
    MrhsScalars *S;
    int check_halt;
    int reverse;  // walk the site blocks from the last one down
    double *partials;
    unsigned int *counter;
};

template <typename R, int FMT, bool NAIK, int EPI, int KR, bool STAGED = true>
__global__ void __launch_bounds__(kMrhsBlock, (MrhsShape<R, KR>::minb))
dslash_mrhs_kernel(const __grid_constant__ MParams<R> P) {
    __shared__ double wsum[kMrhsBlock / 32][KR], tot[kMaxRhs];
    __shared__ bool is_last;
    extern __shared__ double2 stage[];  // hops on their way (dslash_site64, dslash_site_staged)
    pdl_wait();  // everything below may read what earlier kernels wrote
    pdl_trigger();
    MrhsScalars *S = P.S;
    // what the last block decides on (a right-hand side a thread), read ahead of
    // the sums: a read after another there costs 0.6 us
    bool mine = false;
    double rr = 0.0, stop2 = 0.0;
    if constexpr (EPI != EPI_PLAIN) {
        if ((int)threadIdx.x < P.nrhs) {
            mine = S->active[threadIdx.x] != 0;
            rr = S->rr[threadIdx.x];
            stop2 = S->stop2[threadIdx.x];
        }
    }
    if (P.check_halt && S->halt) return;  // uniform over the grid
    const Geom &g = P.g;
    const size_t vh = (size_t)g.vh;
    const size_t fstride = 6 * vh;  // reals per half field
    const int p = P.p;
    const int nsb = (int)((vh + kMrhsBlock - 1) / kMrhsBlock);
    const int total = nsb * P.ngroups;
    double part[KR];
#pragma unroll
    for (int k = 0; k < KR; ++k) part[k] = 0.0;
    // reducing launches have gridDim.x a multiple of ngroups: the group is fixed per block
    for (int bl = blockIdx.x; bl < total; bl += gridDim.x) {
        const int grp = bl % P.ngroups;
        const int sb = P.reverse ? nsb - 1 - bl / P.ngroups : bl / P.ngroups;
        const int i = sb * kMrhsBlock + threadIdx.x;
        if (i >= g.vh) continue;
        bool act[KR];
        size_t off[KR];
        bool any = false;
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            const int rh = grp * KR + k;  // uniform over the block
            act[k] = rh < P.nrhs && (S == nullptr || S->active[rh]);
            any |= act[k];
            off[k] = (size_t)(act[k] ? rh : 0) * fstride;
        }
        if (!any) continue;
        const Site s = site_of(g, p, i);
        Vec3<R> acc[KR];
        if constexpr (std::is_same<R, double>::value) {
            acc[0] = dslash_site64<NAIK>(g, P.fat, P.lng, P.c3, p, i, s, Field64{P.in + off[0], vh},
                                         stage + threadIdx.x, kMrhsBlock);
        } else if constexpr (!STAGED) {
            dslash_site_n<R, FMT, NAIK, KR>(g, P.fat, P.lng, P.c3, p, i, s,
                                            [&](int j, int k) { return load_vec(P.in + off[k], vh, j); }, acc);
        } else {
            // a field that is not active is read as the first one and not stored
            dslash_site_staged<FMT, NAIK, KR>(g, P.fat, P.lng, P.c3, p, i, s, P.in, off,
                                              reinterpret_cast<char *>(stage), acc);
        }
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            if (!act[k]) continue;
            if constexpr (EPI == EPI_PLAIN) {
                store_vec(P.out + off[k], vh, i, acc[k]);
            } else if constexpr (EPI == EPI_NORMAL) {
                const Vec3<R> qv = load_vec(P.q + off[k], vh, i);
                Vec3<R> o;
                R d = R(0);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    o.c[a].re = fma(P.m2, qv.c[a].re, -acc[k].c[a].re);
                    o.c[a].im = fma(P.m2, qv.c[a].im, -acc[k].c[a].im);
                    d = fma(qv.c[a].re, o.c[a].re, d);
                    d = fma(qv.c[a].im, o.c[a].im, d);
                }
                store_vec(P.out + off[k], vh, i, o);
                part[k] += (double)d;
            } else {  // EPI_RESID, FP64: out = b - m^2 x + D in
                const Vec3<R> qv = load_vec(P.q + off[k], vh, i);
                const Vec3<double> bv = load_vec(P.b + off[k], vh, i);
                Vec3<R> o;
                double d = 0.0;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    o.c[a].re = (R)bv.c[a].re - fma(P.m2, qv.c[a].re, -acc[k].c[a].re);
                    o.c[a].im = (R)bv.c[a].im - fma(P.m2, qv.c[a].im, -acc[k].c[a].im);
                    d = fma((double)o.c[a].re, (double)o.c[a].re, d);
                    d = fma((double)o.c[a].im, (double)o.c[a].im, d);
                }
                store_vec(P.out + off[k], vh, i, o);
                part[k] += d;
            }
        }
    }
    if constexpr (EPI == EPI_PLAIN) {
        return;
    } else {
        // per right-hand side of this block's group: a fixed shuffle tree in
        // each warp, then warps in order -> partials[blockIdx.x * KR + k]
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            const double v = warp_sum(part[k]);
            if (lane == 0) wsum[warp][k] = v;
        }
        __syncthreads();
        if (warp == 0) {
            if (lane < KR) {
                double t = 0.0;
                for (int w = 0; w < kMrhsBlock / 32; ++w) t += wsum[w][lane];
                P.partials[(size_t)blockIdx.x * KR + lane] = t;
            }
            __syncwarp();
            if (lane == 0) is_last = arrive_last(P.counter, gridDim.x);
        }
        __syncthreads();
        if (!is_last) return;
        // right-hand side r = grp * KR + k lives in blocks bx = grp (mod ngroups)
        const int nw = kMrhsBlock / 32;
        for (int r = warp; r < P.nrhs; r += nw) {
            const int grp = r / KR, kk = r % KR;
            double t = 0.0;
#pragma unroll 4
            for (int bx = grp + lane * P.ngroups; bx < (int)gridDim.x; bx += 32 * P.ngroups)
                t += __ldcg(P.partials + (size_t)bx * KR + kk);
            t = warp_sum(t);
            if (lane == 0) tot[r] = t;
        }
        __syncthreads();
        // a right-hand side a thread
        const int r = threadIdx.x;
        const double t = mine ? tot[r] : 0.0;
        const bool finite = isfinite(t);
        if constexpr (EPI == EPI_NORMAL) {
            if (!mine) return;
            S->pAp[r] = t;
            if (!(t > 0.0) || !finite) {
                S->error = finite ? 2 : 1;
                S->halt = 1;
            } else {
                S->alpha[r] = rr / t;
            }
        } else {
            const bool met = finite && t <= stop2;
            if (mine) {
                S->true_rr[r] = t;
                if (finite) {
                    S->beta[r] = rr > 0.0 ? t / rr : 0.0;
                    S->rr[r] = t;
                    S->rmax2[r] = t;
                }
                if (met) {
                    S->done[r] = 1;
                    S->active[r] = 0;
                }
            }
            const int n = __syncthreads_count(mine && !met);
            const bool bad = __syncthreads_or(mine && !finite);
            if (r == 0) {
                if (bad) S->error = 1;
                S->nactive = n;
                S->need_ru = 0;
                S->ru_iter0 = S->iter;
                S->reliable_updates += 1;
                S->halt = (n == 0 || S->iter >= S->maxiter || S->error) ? 1 : 0;
            }
        }
    }
}

template <typename R, int FMT, bool NAIK, int EPI, int KR, bool STAGED = true>
static void launch_m(const qex_lattice *lat, const MrhsArgs &a, cudaStream_t st) {
    MParams<R> P;
    P.g = lat->geom;
    P.fat = (const R *)a.fat;
    P.lng = (const R *)a.lng;
    P.c3 = (R)a.c3;
    P.p = a.out_parity;
    P.nrhs = a.nrhs;
    P.ngroups = (a.nrhs + KR - 1) / KR;
    P.in = (const R *)a.in;
    P.out = (R *)a.out;
    P.q = (const R *)a.q;
    P.b = a.b;
    P.m2 = (R)a.m2;
    P.S = a.S;
    P.check_halt = (a.S && EPI != EPI_RESID) ? 1 : 0;
    P.reverse = a.reverse;
    P.partials = lat->partials;
    P.counter = lat->counter;
    const int nsb = (int)((lat->vh + kMrhsBlock - 1) / kMrhsBlock);
    const int total = nsb * P.ngroups;
    int gx = total;
    if (EPI == EPI_NORMAL || EPI == EPI_RESID) {  // persistent grid, a multiple of ngroups
        int cap = sm_count() * MrhsShape<R, KR>::minb;
        cap -= cap % P.ngroups;
        if (cap < P.ngroups) cap = P.ngroups;
        gx = total < cap ? total : cap;
    }
    size_t smem = kMrhsBlock * kStageBytes;
    if constexpr (!STAGED)
        smem = 0;
    else if constexpr (!std::is_same<R, double>::value)
        smem = kMrhsBlock * 2 * StageOf<FMT, NAIK, KR>::type::bytes;
    auto kernel = dslash_mrhs_kernel<R, FMT, NAIK, EPI, KR, STAGED>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_k(kernel, dim3(gx), dim3(kMrhsBlock), smem, st, a.pdl != 0, P);
}

// Links that stay in the L2 beside the fields come back soon enough without the
// detour, and the copies only cost instructions (16-bit links, 24 right-hand
// sides, D alone: 16^4, 6 MB of links, 22.1 us staged against 20.2; 20^4, 15 MB,
// 49.3 against 48.2; 24^4, 32 MB, 94 both ways, but the CG with 16 takes 268 us
// an iteration against 277); the FP32 formats lose by it only with several blocks
// on an SM (12^4, full links: 12 right-hand sides 5.9 us both ways, 16 of them
// 9.3 against 8.0).
template <int FMT, bool NAIK>
static bool staging_loses(int nrhs, int vh) {
    constexpr int kLink = 16 * LinkWords<FMT>::n16 + 8 * LinkWords<FMT>::n8;
    constexpr int kLong = FMT >= 2 ? 40 : 72;
    if ((long long)vh * 8 * (kLink + (NAIK ? kLong : 0)) > 24000000LL) return false;
    return FMT >= 2 || (vh + kMrhsBlock - 1) / kMrhsBlock * ((nrhs + 3) / 4) > sm_count();
}

template <typename R, int FMT, bool NAIK, int EPI>
static void launch_m_kr(const qex_lattice *lat, const MrhsArgs &a, cudaStream_t st) {
    if constexpr (std::is_same<R, double>::value)
        launch_m<R, FMT, NAIK, EPI, 1>(lat, a, st);
    else if (pairs_are_better(a.nrhs, (int)lat->vh))
        launch_m<R, FMT, NAIK, EPI, 2>(lat, a, st);
    else if (staging_loses<FMT, NAIK>(a.nrhs, (int)lat->vh))
        launch_m<R, FMT, NAIK, EPI, 4, false>(lat, a, st);
    else
        launch_m<R, FMT, NAIK, EPI, 4>(lat, a, st);
}

template <typename R, int FMT, bool NAIK>
static void launch_m_epi(const qex_lattice *lat, const MrhsArgs &a, cudaStream_t st) {
    if (a.epi == EPI_PLAIN)
        launch_m_kr<R, FMT, NAIK, EPI_PLAIN>(lat, a, st);
    else if (a.epi == EPI_NORMAL)
        launch_m_kr<R, FMT, NAIK, EPI_NORMAL>(lat, a, st);
    else if constexpr (std::is_same<R, double>::value)
        launch_m_kr<R, FMT, NAIK, EPI_RESID>(lat, a, st);
}

qex_status launch_dslash_mrhs(qex_lattice *lat, const MrhsArgs &a, cudaStream_t st) {
    if (a.epi == EPI_NORMAL || a.epi == EPI_RESID) {
        qex_status s = ensure_scratch(lat);
        if (s) return s;
        const size_t need = (size_t)(sm_count() + 1) * kMrhsMaxPartialsPerSm;
        if ((size_t)lat->partials_len < need) {
            set_error("internal: partials buffer too small for %d right-hand sides", a.nrhs);
            return QEX_ERR_ARG;
        }
    }
    if (a.prec == QEX_F64) {
        if (a.lng)
            launch_m_epi<double, 0, true>(lat, a, st);
        else
            launch_m_epi<double, 0, false>(lat, a, st);
    } else {
        if (a.epi == EPI_RESID) {
            set_error("the residual epilogue is FP64 only");
            return QEX_ERR_ARG;
        }
        if (a.prec == QEX_F32_R12) {
            if (a.lng)
                launch_m_epi<float, 1, true>(lat, a, st);
            else
                launch_m_epi<float, 1, false>(lat, a, st);
        } else if (a.prec == QEX_F32_R12H) {
            if (a.lng)
                launch_m_epi<float, 2, true>(lat, a, st);
            else
                launch_m_epi<float, 2, false>(lat, a, st);
        } else if (a.prec == QEX_F32_S16) {
            if (a.lng)
                launch_m_epi<float, 3, true>(lat, a, st);
            else
                launch_m_epi<float, 3, false>(lat, a, st);
        } else {
            if (a.lng)
                launch_m_epi<float, 0, true>(lat, a, st);
            else
                launch_m_epi<float, 0, false>(lat, a, st);
        }
    }
    QEX_CHECK_LAUNCH("dslash_mrhs_kernel");
    return QEX_OK;
}

qex_status check_dslash_args(const qex_lattice *lat, qex_prec prec, const void *fat, const void *lng,
                             const void *in, const void *out);

}  // namespace qex

using namespace qex;

extern "C" qex_status qex_dslash_mrhs(const qex_lattice *lat, qex_prec prec, const void *fat, const void *lng,
                                      double c_naik, int out_parity, int nrhs, const void *in, void *out,
                                      void *stream) {
    qex_status st = check_dslash_args(lat, prec, fat, lng, in, out);
    if (st) return st;
    if (out_parity != 0 && out_parity != 1) {
        set_error("out_parity must be 0 or 1");
        return QEX_ERR_ARG;
    }
    if (nrhs < 1 || nrhs > QEX_MRHS_MAX) {
        set_error("nrhs must be in [1, %d] (got %d)", QEX_MRHS_MAX, nrhs);
        return QEX_ERR_ARG;
    }
    MrhsArgs a = {};
    a.prec = prec;
    a.fat = fat;
    a.lng = lng;
    a.c3 = c_naik;
    a.out_parity = out_parity;
    a.nrhs = nrhs;
    a.in = in;
    a.out = out;
    a.epi = EPI_PLAIN;
    return launch_dslash_mrhs(const_cast<qex_lattice *>(lat), a, as_stream(stream));
}
