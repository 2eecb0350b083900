// Whole BiCGStab and IDR(s) cycles in one cooperative launch, for grids small enough that the
// launches and not the points take the time (real operators).
//
// One block per SM keeps its points through the cycle; the blocks meet at a grid barrier (about
// 1.2 us) where a chain of launches needs one launch per reduction (5-7 us each with its block
// reduction, last-block sum and scalar step).  A BiCGStab iteration (two products) on 127^2 points takes
// 10.6 us (21.3 as a chain of launches), an IDR(4) round (five) 56 (93).  Reductions: every block
// writes its partial sums, and after the barrier every block adds all of them in the same order and computes
// the same scalars for itself, so nothing has to be broadcast and results do not depend on timing.
// BiCGStab needs two barriers per iteration instead of four: the new p and r of a neighbour and
// its s are recomputed from the stored vectors where the stencil reads them (bit-identical to
// the owner's values), so x / r / p are updated in the pass that forms v = A p, and s in the pass
// that forms t = A s.  p and v alternate between two buffers, because neighbours still read the
// old ones.
// Data of other blocks is read past the L1 cache (__ldcg).  Every wait ends after a limited number
// of polls; the block that gives up says so in a word of its own, and every block then leaves at its
// next barrier.  The first barrier of a launch comes before anything is written: if it is given up
// (blocks of other streams hold SMs that the launch needs), or the launch is refused (the stream owns
// fewer SMs), the host runs the cycle, or what is left of it, as a chain of launches.  Past it all blocks are
// resident, and a wait that runs out is TG_SYNC_TIMEOUT.
#pragma once

#include "tg_arnoldi.cuh"
#include "tg_idr.cuh"

namespace tg {

constexpr int kPersThreads = 256;
// Blocks of a cycle kernel that fit an SM, so that solves on other streams run beside it: launches
// that each take the SMs' registers run in turn (202 registers a thread where nothing bounds them).
// ms a solve with eight threads that each have an operator and a stream, chain of launches / one block an
// SM / these: IDR(4) 127^2 7.2 / 11.4 / 5.5, float32 + refinement 63^3 2.7 / 3.3 / 2.4, float64 511^2
// 49 / 58 / 41; one thread alone is 0 to 2% slower than with one block.
template <class T> constexpr int kBiPersBlocks = sizeof(T) == 4 ? 3 : 2;
constexpr int kIdrPersBlocks = 3;
constexpr int kPersPart = 16;                 // reduced values per pass at most

// Polls of a wait (half a microsecond each; none: the wait is given up at once): the first barrier
// of a cycle's first launch and of its later launches, and every other barrier.
struct SyncLimits {
    unsigned start = 1u << 16, again = 1u << 16, step = 1u << 20;
};

// The barrier's words, zero at launch.  count: arrivals, and kSyncGaveUp once a block has given up;
// failed: written only by that block, never cleared within a launch.
struct SyncWords {
    unsigned count, failed;
};
constexpr unsigned kSyncGaveUp = 0x80000000u;
constexpr unsigned kFailedStart = 1, kFailedStep = 2;

// The blocks' meeting point: part holds two buffers of kPersPart x blocks partial sums (a block can
// write the next but one reduction only after all have read this one).  Once ok is false (for all
// threads of a block alike) it stays false, and nothing waits or counts any more: sums are
// meaningless then, and their callers leave.
struct GridSync {
    SyncWords *w;
    double *part;
    unsigned first, step;          // limits of the launch's first barrier and of the others
    unsigned round;
    int parity;
    bool ok;
    __device__ GridSync(SyncWords *words, double *p, const SyncLimits &l, bool cycle_start)
        : w(words), part(p), first(cycle_start ? l.start : l.again), step(l.step), round(0), parity(0), ok(true) {}
    __device__ void wait() {
        __shared__ bool ok_s;          // rewritten after the next barrier's first __syncthreads only
        if (!ok) return;
        ++round;
        __syncthreads();
        if (threadIdx.x == 0) {        // the release covers the block's writes (ordered by the barrier above)
            const unsigned target = round * gridDim.x, limit = round == 1 ? first : step;
            unsigned seen = 0, polls = 0;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&w->count) : "memory");
            if (limit == 0) {
                seen = kSyncGaveUp;
                if (!(atomicOr(&w->count, kSyncGaveUp) & kSyncGaveUp)) w->failed = round == 1 ? kFailedStart : kFailedStep;
            }
            while (limit != 0) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&w->count) : "memory");
                if (seen >= target) break;               // complete, or kSyncGaveUp is set
                if (polls++ < limit) continue;
                // give up, unless the barrier is completed or given up first: both are the same word
                const unsigned old = atomicCAS(&w->count, seen, seen | kSyncGaveUp);
                if (old == seen) {
                    w->failed = round == 1 ? kFailedStart : kFailedStep;
                    seen = kSyncGaveUp;
                    break;
                }
            }
            ok_s = seen < kSyncGaveUp;
        }
        __syncthreads();
        ok = ok_s;
    }
    // tot[d] = sum over all threads of the grid of v[d], d < ND (every block gets the same value)
    template <int ND, class P>
    __device__ void sum(P (&v)[ND], double *tot) {
        constexpr int NV = ND <= 1 ? 1 : ND <= 2 ? 2 : ND <= 4 ? 4 : ND <= 8 ? 8 : 16;
        static_assert(ND <= kPersPart, "partial buffers");
        __shared__ double red[(kPersThreads / 32) * NV];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        P w[NV];
#pragma unroll
        for (int d = 0; d < NV; ++d) w[d] = d < ND ? v[d] : P(0);
        const P r = warp_sums<NV>(w);
        if (lane < NV) red[warp * NV + lane] = (double)r;
        __syncthreads();
        double *buf = part + (size_t)parity * kPersPart * gridDim.x;
        parity ^= 1;
        // value d by the eight lanes of its group (lanes 8 d .. 8 d + 7 of the block)
        static_assert(kPersThreads / 32 == 8 && 8 * kPersPart <= kPersThreads, "one lane per warp and value");
        if (threadIdx.x < ((8 * ND + 31) & ~31)) {
            const int d = threadIdx.x >> 3;
            double s = d < ND ? red[(threadIdx.x & 7) * NV + d] : 0.0;
            s += shfl_xor(s, 4);
            s += shfl_xor(s, 2);
            s += shfl_xor(s, 1);
            if (d < ND && !(threadIdx.x & 7)) __stcg(buf + (size_t)d * gridDim.x + blockIdx.x, s);
        }
        wait();
        for (int d = warp; d < ND; d += kPersThreads / 32) {
            const double s = total(buf + (size_t)d * gridDim.x);
            if (lane == 0) tot[d] = s;
        }
        __syncthreads();
    }
    // the sum over the blocks of one value's partials, by a warp (the loads of up to 160 blocks are
    // in flight together: in turn they took 1.5 us)
    __device__ double total(const double *p) const {
        const int lane = threadIdx.x & 31, nb = gridDim.x;
        double v[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) v[u] = lane + 32 * u < nb ? __ldcg(p + lane + 32 * u) : 0.0;
        double s = ((v[0] + v[1]) + (v[2] + v[3])) + v[4];
        for (int b = lane + 160; b < nb; b += 32) s += __ldcg(p + b);
        return warp_sum(s);
    }
};
// comparisons of the scalar steps on the bits: a float64 compare holds its unit for 64 clocks
__device__ __forceinline__ bool bits_le(double a, double b) {      // a <= b for a, b >= 0
    return __double_as_longlong(a) <= __double_as_longlong(b);
}
__device__ __forceinline__ bool bits_tiny(double a) { return bits_le(fabs(a), kTiny); }

constexpr int kPersCols = 64;                 // deflation vectors a cycle's own projection takes

// What a launch reports beside the cycle's state.
struct BiPersOut {
    BiState<double> st;
    double nr, rt;            // residual norm after the projection and the cycle tolerance
    double rr, bb;            // ||b - A x||^2 and ||b||^2 after the cycle
};

// The steps around a cycle that a launch can take with it (whole = 1): the float32 correction
// equation's r / ||r|| and e = 0 (T = float), the projection, the cycle tolerance, and after the
// cycle x += ||r|| e (T = float) and the float64 residual with its norms.
template <class T>
struct BiPersArgs {
    T *x, *r, *rh, *p[2], *v[2], *s, *t;      // x, r: T = float and whole: the correction and its residual
    double *part;
    SyncWords *words;
    SyncLimits limits;
    BiPersOut *out;
    double target2;                           // whole = 0
    int cap, first, max_iters;                // first: the cycle starts here (r_hat = p = r)
    int whole;
    const double *b;
    double *x64, *r64, *xbak;
    const T *W, *B1, *B2;
    const double *Mp;
    int kk, minres, sched;
    double nr, nb, rtol, ex, pw, floor;       // cycle_tol: ex = 1 / (ncyc - cyc + 1), pw = rtol^(cyc / ncyc)
};

// The projection of k_proj_update on a block's own points: c = W^T r, d = M c, x += B1 d,
// r -= B2 e.  The partial sums of c go behind the reductions' buffers.
template <class T>
__device__ __forceinline__ void pers_project(const BiPersArgs<T> &a, GridSync &gs, int n, int lo, int hi) {
    __shared__ double c[kPersCols], d[kPersCols];
    __shared__ T ds[kPersCols], es[kPersCols];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kPersThreads / 32, kk = a.kk, nb = gridDim.x;
    double *buf = a.part + (size_t)2 * kPersPart * nb;
    for (int q = warp; q < kk; q += nw) {
        const T *w = a.W + (size_t)q * n;
        T acc = T(0);
#pragma unroll 4
        for (int i = lo + lane; i < hi; i += 32) acc = ST<T>::fma_cm(w[i], a.r[i], acc);
        acc = warp_sum(acc);
        if (lane == 0) __stcg(buf + (size_t)q * nb + blockIdx.x, (double)acc);
    }
    gs.wait();
    for (int q = warp; q < kk; q += nw) {
        const double s = gs.total(buf + (size_t)q * nb);
        if (lane == 0) c[q] = s;
    }
    __syncthreads();
    // four lanes a row of M c
    for (int i0 = 0; i0 < kk; i0 += kPersThreads / 4) {
        const int i = i0 + (threadIdx.x >> 2);
        double s = 0.0;
        if (i < kk)
            for (int l = threadIdx.x & 3; l < kk; l += 4) s = fma(a.Mp[i + (size_t)l * kk], c[l], s);
        s += shfl_xor(s, 1);
        s += shfl_xor(s, 2);
        if (i < kk && !(threadIdx.x & 3)) d[i] = s;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < kk; q += kPersThreads) {
        ds[q] = (T)d[q];
        es[q] = (T)(a.minres ? c[q] : d[q]);
    }
    __syncthreads();
    for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
        T ax = T(0), ar = T(0);
#pragma unroll 8
        for (int q = 0; q < kk; ++q) {
            ax = axpy(ds[q], a.B1[(size_t)q * n + i], ax);
            ar = axpy(es[q], a.B2[(size_t)q * n + i], ar);
        }
        a.x[i] = a.x[i] + ax;
        a.r[i] = a.r[i] - ar;
    }
}

// A BiCGStab cycle, or the next max_iters iterations of one.  Scalar steps and exits are those of
// k_bi_init, k_bi_v, k_bi_s, k_bi_t and k_bi_x.  On return x, r and (status 0) p[0] are current.
template <class T>
__global__ void __launch_bounds__(kPersThreads, kBiPersBlocks<T>) k_bi_persist(DevOp op, DevOp32 o32, BiPersArgs<T> a) {
    __shared__ BiState<double> S;
    __shared__ double tot[kPersPart];
    GridSync gs(a.words, a.part, a.limits, a.first);
    const int n = op.n, per = (n + gridDim.x - 1) / gridDim.x;
    const int lo = min(n, (int)blockIdx.x * per), hi = min(n, lo + per);
    T *p = a.p[0], *p2 = a.p[1], *v = a.v[0], *v2 = a.v[1];      // the current p and v, and the other buffers
    __shared__ double nr_s, rt_s;
    gs.wait();
    if (!gs.ok) return;                            // nothing is written yet
    if (a.first) {
        if constexpr (std::is_same<T, float>::value) {
            if (a.whole) {
                const double sc = 1.0 / a.nr;
                for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                    a.r[i] = (float)(a.r64[i] * sc);
                    a.x[i] = 0.0f;
                }
                __syncthreads();
            }
        }
        if (a.whole && a.kk > 0) pers_project<T>(a, gs, n, lo, hi);
        T acc[1] = {T(0)};
        for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
            const T ri = a.r[i];
            a.rh[i] = ri;
            a.p[0][i] = ri;
            acc[0] = ST<T>::fma_cm(ri, ri, acc[0]);
        }
        gs.sum<1>(acc, tot);
        if (threadIdx.x == 0) {
            const double rho = tot[0];
            double target2 = a.target2;
            if (a.whole) {
                // float64: nr is the norm of r; float32: r was scaled by 1 / nr
                const bool rel = sizeof(T) == 4;
                const double nrel = a.kk > 0 ? sqrt(rho) : rel ? 1.0 : a.nr, nr = rel ? nrel * a.nr : nrel;
                double rt = a.rtol * a.nb / nr;
                if (a.sched) rt = fmin(pow(rt, a.ex), (a.nb / nr) * a.pw);
                rt = fmax(rt, a.floor);
                nr_s = nr;
                rt_s = rt;
                target2 = (rt * nrel) * (rt * nrel);
            }
            S.rho = S.rr = rho;
            S.ss = 0.0;
            S.target2 = target2;
            S.div2 = sizeof(T) == 4 ? 1e16 * rho : 1.7e308;
            S.mvps = 0; S.cap = a.cap; S.iters = 0; S.half = 0; S.pending = 0;
            S.alpha = S.omega = S.beta = S.rho_next = rho;
            S.status = !isfinite(rho) ? 4 : rho <= target2 ? 1 : fabs(rho) < kTiny ? 2 : 0;
        }
    } else if (threadIdx.x == 0) {
        S = a.out->st;
        nr_s = a.out->nr;
        rt_s = a.out->rt;
    }
    __syncthreads();
    bool pend = false;                             // s, t, v of a full step wait to be applied
    for (int it = 0; S.status == 0 && gs.ok; ++it) {
        const bool flush = it == a.max_iters;      // apply the last step and leave
        if (flush && !pend) break;
        // ---- x, r, p of the last step; v = A p, <r_hat, v>, <r, r>
        {
            const T alpha = (T)S.alpha, omega = (T)S.omega, mom = -omega, beta = (T)S.beta;
            const T *po = p, *vo = v;
            auto r_at = [&](int j) { return axpy(mom, __ldcg(a.t + j), __ldcg(a.s + j)); };
            auto p_at = [&](int j) -> T {
                if (!pend) return __ldcg(po + j);
                return axpy(beta, axpy(mom, __ldcg(vo + j), __ldcg(po + j)), r_at(j));
            };
            T acc[2] = {T(0), T(0)};
            for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                if (pend) {
                    const T si = a.s[i], pi = po[i], ri = r_at(i);
                    a.x[i] = axpy(omega, si, axpy(alpha, pi, a.x[i]));
                    a.r[i] = ri;
                    p2[i] = axpy(beta, axpy(mom, vo[i], pi), ri);
                    acc[1] = ST<T>::fma_cm(ri, ri, acc[1]);
                }
                if (!flush) {
                    const T y = apply_real_all<T>(op, o32, i, p_at);
                    v2[i] = y;
                    acc[0] = ST<T>::fma_cm(a.rh[i], y, acc[0]);
                }
            }
            gs.sum<2>(acc, tot);
            if (threadIdx.x == 0) {
                if (pend) {
                    const double rr = tot[1];
                    S.rr = rr;
                    S.iters += 1;
                    S.rho = S.rho_next;
                    if (!isfinite(rr)) S.status = 4;
                    else if (bits_le(rr, S.target2)) S.status = 1;
                    else if (!bits_le(rr, S.div2)) S.status = 5;
                    else if (bits_tiny(S.omega) || bits_tiny(S.rho_next)) S.status = 2;
                    else if (S.mvps >= S.cap) S.status = 3;
                }
                if (!flush && S.status == 0) {
                    const double sigma = tot[0];
                    S.mvps += 1;
                    if (!isfinite(sigma)) S.status = 4;
                    else if (bits_tiny(sigma)) S.status = 2;
                    else S.alpha = S.rho / sigma;
                }
            }
            __syncthreads();
            T *tmp;
            if (pend) { tmp = p; p = p2; p2 = tmp; }
            if (!flush) { tmp = v; v = v2; v2 = tmp; }
            pend = false;
            if (flush || S.status != 0) break;
        }
        // ---- s = r - alpha v; t = A s; <s, s>, <t, s>, <t, t>, <r_hat, s>, <r_hat, t>
        {
            const T ma = -(T)S.alpha;
            const T *vc = v;
            auto s_at = [&](int j) { return axpy(ma, __ldcg(vc + j), __ldcg(a.r + j)); };
            T acc[5] = {T(0), T(0), T(0), T(0), T(0)};
            for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                const T si = s_at(i), ti = apply_real_all<T>(op, o32, i, s_at), hi_ = a.rh[i];
                a.s[i] = si;
                a.t[i] = ti;
                acc[0] = ST<T>::fma_cm(si, si, acc[0]);
                acc[1] = ST<T>::fma_cm(ti, si, acc[1]);
                acc[2] = ST<T>::fma_cm(ti, ti, acc[2]);
                acc[3] = ST<T>::fma_cm(hi_, si, acc[3]);
                acc[4] = ST<T>::fma_cm(hi_, ti, acc[4]);
            }
            gs.sum<5>(acc, tot);
            if (threadIdx.x < 32) {
                // omega, 1 / omega and alpha / rho by three lanes at once: a division is a chain of
                // seven float64 operations
                const int lane = threadIdx.x;
                const double ts = tot[1], tt = tot[2], rs = tot[3], rt = tot[4];
                const double dv = (lane == 0 ? ts : lane == 1 ? tt : S.alpha) / (lane == 0 ? tt : lane == 1 ? ts : S.rho);
                const double iom = __shfl_sync(0xffffffffu, dv, 1), ar = __shfl_sync(0xffffffffu, dv, 2);
                if (lane == 0) {
                    const double ss = tot[0];
                    S.ss = ss;
                    if (!isfinite(ss)) S.status = 4;
                    else if (bits_le(ss, S.target2)) { S.half = 1; S.pending = 1; }
                    else if (!bits_le(ss, S.div2)) S.status = 5;
                    else if (S.mvps >= S.cap) { S.half = 1; S.pending = 3; }
                    if (S.status == 0 && !S.half) {
                        S.mvps += 1;
                        if (!isfinite(tt) || !isfinite(ts)) S.status = 4;
                        else if (bits_tiny(tt)) { S.half = 1; S.pending = 2; }
                        else {
                            S.omega = dv;
                            S.rho_next = fma(-dv, rt, rs);
                            // (rho_next / rho)(alpha / omega) = (alpha / rho)(rs / omega - rt)
                            if (!bits_tiny(dv)) S.beta = ar * fma(rs, iom, -rt);
                        }
                    }
                }
            }
            __syncthreads();
            if (S.status != 0) break;
            if (S.half) {                          // the half step: x += alpha p, r = s
                const T alpha = (T)S.alpha;
                for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                    a.x[i] = axpy(alpha, p[i], a.x[i]);
                    a.r[i] = a.s[i];
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    S.rr = S.ss;
                    S.status = S.pending;
                    S.iters += 1;
                }
                __syncthreads();
                break;
            }
            pend = true;
        }
    }
    if (S.status == 0 && p != a.p[0])              // hand p over in p[0]
        for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) a.p[0][i] = p[i];
    if (a.whole && S.status != 0 && gs.ok) {
        if constexpr (std::is_same<T, float>::value) {
            for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                const double xi = a.x64[i];
                a.xbak[i] = xi;
                a.x64[i] = fma(a.nr, (double)a.x[i], xi);
            }
        }
        gs.wait();
        double acc[2] = {0.0, 0.0};
        for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
            const double bi = a.b[i], ri = bi - apply_real_all<double>(op, o32, i, [&](int j) { return __ldcg(a.x64 + j); });
            a.r64[i] = ri;
            acc[0] = fma(ri, ri, acc[0]);
            acc[1] = fma(bi, bi, acc[1]);
        }
        gs.sum<2>(acc, tot);
    }
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        a.out->st = S;
        a.out->nr = nr_s;
        a.out->rt = rt_s;
        a.out->rr = tot[0];
        a.out->bb = tot[1];
    }
}

template <class T>
struct IdrPersArgs {
    const T *P;
    T *x, *r, *G, *U, *t;
    size_t ld;
    double *part;
    SyncWords *words;
    SyncLimits limits;
    IdrState<double> *st;
    double target2, kappa;
    int s, cap, first, max_rounds;
};

// An IDR(s) cycle, or the next max_rounds rounds of one, with the scalar steps of tg_idr.cuh.
// Per k two barriers: the update of step k - 1 and U_k touch a block's own points only and share
// a pass, then G_k = A U_k; the dimension reduction takes three.
template <class T>
__global__ void __launch_bounds__(kPersThreads, kIdrPersBlocks) k_idr_persist(DevOp op, DevOp32 o32, IdrPersArgs<T> a) {
    constexpr int M = kIdrMaxS;
    __shared__ IdrState<double> S;
    __shared__ double tot[kPersPart];
    __shared__ T cs[M], al[M];
    __shared__ double inv[M];                      // 1 / M_kk
    GridSync gs(a.words, a.part, a.limits, a.first);
    const int n = op.n, s = a.s, per = (n + gridDim.x - 1) / gridDim.x;
    const int lo = min(n, (int)blockIdx.x * per), hi = min(n, lo + per);
    const size_t ld = a.ld;
    gs.wait();
    if (!gs.ok) return;                            // nothing is written yet
    auto shadow = [&](T ri, int i, T (&acc)[M + 1]) {      // f = P^H r, ||r||^2
#pragma unroll
        for (int q = 0; q < M; ++q)
            if (q < s) acc[q] = ST<T>::fma_cm(a.P[(size_t)q * ld + i], ri, acc[q]);
        acc[M] = ST<T>::fma_cm(ri, ri, acc[M]);
    };
    if (a.first) {
        T acc[M + 1];
#pragma unroll
        for (int q = 0; q <= M; ++q) acc[q] = T(0);
        for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) shadow(a.r[i], i, acc);
        gs.sum<M + 1>(acc, tot);
        if (threadIdx.x == 0) {
            for (int e = 0; e < M * M; ++e) S.M[e] = e % (M + 1) == 0 ? 1.0 : 0.0;
            for (int q = 0; q < M; ++q) {
                S.f[q] = q < s ? tot[q] : 0.0;
                S.alpha[q] = 0.0;
            }
            const double rr = tot[M];
            S.rr = rr; S.target2 = a.target2; S.kappa = a.kappa; S.s = s; S.mvps = 0; S.cap = a.cap; S.rounds = 0;
            S.beta = 0.0; S.omega = 1.0;
            S.status = !isfinite(rr) ? 4 : rr <= a.target2 ? 1 : 0;
        }
    } else if (threadIdx.x == 0) {
        S = *a.st;
    }
    __syncthreads();
    if (threadIdx.x < M) inv[threadIdx.x] = 1.0 / S.M[threadIdx.x * (M + 1)];
    __syncthreads();
    bool fresh = a.first != 0;                     // columns k.. of G and U are not written yet
    auto check_rr = [&](double rr) {               // thread 0
        S.rr = rr;
        if (!isfinite(rr)) S.status = 4;
        else if (rr <= S.target2) S.status = 1;
        else if (S.mvps >= S.cap) S.status = 3;
    };
    for (int round = 0; round < a.max_rounds && S.status == 0 && gs.ok; ++round) {
        for (int k = 0; k <= s; ++k) {
            // ---- update of step k - 1 (own points), then U_k (k < s)
            if (threadIdx.x == 0 && k < s) {       // c = M[k:, k:]^-1 f[k:]
                double c[M];
                for (int q = k; q < s; ++q) {
                    double v = S.f[q];
                    for (int b = k; b < q; ++b) v = fma(-S.M[q + b * M], c[b - k], v);
                    c[q - k] = v * inv[q];
                    cs[q - k] = (T)c[q - k];
                }
            }
            if (threadIdx.x < M) al[threadIdx.x] = (T)S.alpha[threadIdx.x];
            __syncthreads();
            {
                const T om = (T)S.omega, beta = (T)S.beta;
                const int kp = k - 1, nc = s - k;
                T acc[1] = {T(0)};
                for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                    T ri = a.r[i];
                    if (k > 0) {
                        T g = a.G[(size_t)kp * ld + i], u = a.U[(size_t)kp * ld + i];
#pragma unroll 4
                        for (int b = 0; b < kp; ++b) {
                            g = sub(g, dmul(al[b], a.G[(size_t)b * ld + i]));
                            u = sub(u, dmul(al[b], a.U[(size_t)b * ld + i]));
                        }
                        a.G[(size_t)kp * ld + i] = g;
                        a.U[(size_t)kp * ld + i] = u;
                        ri = sub(ri, dmul(beta, g));
                        a.r[i] = ri;
                        a.x[i] = axpy(beta, u, a.x[i]);
                        acc[0] = ST<T>::fma_cm(ri, ri, acc[0]);
                    }
                    if (k < s) {
                        T v = ri, u = T(0);
                        if (!fresh) {
#pragma unroll 4
                            for (int q = 0; q < nc; ++q) {
                                v = sub(v, dmul(cs[q], a.G[(size_t)(k + q) * ld + i]));
                                u = axpy(cs[q], a.U[(size_t)(k + q) * ld + i], u);
                            }
                        }
                        a.U[(size_t)k * ld + i] = axpy(om, v, u);
                    }
                }
                if (k > 0) gs.sum<1>(acc, tot);
                else gs.wait();
            }
            if (k > 0) {
                if (threadIdx.x == 0) check_rr(tot[0]);
                __syncthreads();
                if (S.status != 0) break;
            }
            if (k == s || !gs.ok) break;
            // ---- G_k = A U_k, d = P^H G_k; alpha, M[k:, k], beta, f
            {
                const T *Uk = a.U + (size_t)k * ld;
                T acc[M];
#pragma unroll
                for (int q = 0; q < M; ++q) acc[q] = T(0);
                for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                    const T g = apply_real_all<T>(op, o32, i, [&](int j) { return __ldcg(Uk + j); });
                    a.G[(size_t)k * ld + i] = g;
#pragma unroll
                    for (int q = 0; q < M; ++q)
                        if (q < s) acc[q] = ST<T>::fma_cm(a.P[(size_t)q * ld + i], g, acc[q]);
                }
                gs.sum<M>(acc, tot);
            }
            if (threadIdx.x == 0) {
                S.mvps += 1;
                bool finite = true;
                for (int i = 0; i < k; ++i) {
                    double v = tot[i];
                    for (int b = 0; b < i; ++b) v = fma(-S.M[i + b * M], S.alpha[b], v);
                    S.alpha[i] = v * inv[i];
                }
                for (int j = k; j < s; ++j) {
                    double v = tot[j];
                    for (int b = 0; b < k; ++b) v = fma(-S.alpha[b], S.M[j + b * M], v);
                    S.M[j + k * M] = v;
                    finite = finite && isfinite(v);
                }
                const double mkk = S.M[k + k * M];
                if (!finite) S.status = 4;
                else if (fabs(mkk) < kTiny) S.status = 2;
                else {
                    inv[k] = 1.0 / mkk;
                    const double beta = S.f[k] * inv[k];
                    S.beta = beta;
                    for (int j = k + 1; j < s; ++j) S.f[j] = fma(-beta, S.M[j + k * M], S.f[j]);
                }
            }
            __syncthreads();
            if (S.status != 0) break;
        }
        if (S.status != 0 || !gs.ok) break;
        fresh = false;
        // ---- t = A r; omega
        {
            T acc[3] = {T(0), T(0), T(0)};
            for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                const T ti = apply_real_all<T>(op, o32, i, [&](int j) { return __ldcg(a.r + j); }), ri = a.r[i];
                a.t[i] = ti;
                acc[0] = ST<T>::fma_cm(ti, ri, acc[0]);
                acc[1] = ST<T>::fma_cm(ti, ti, acc[1]);
                acc[2] = ST<T>::fma_cm(ri, ri, acc[2]);
            }
            gs.sum<3>(acc, tot);
            if (threadIdx.x == 0) {
                S.mvps += 1;
                const double tt = tot[1], rr = tot[2];
                if (!isfinite(tt) || !isfinite(tot[0])) S.status = 4;
                else if (tt < kTiny) S.status = 2;
                else {
                    double om = tot[0] / tt;
                    const double rho = fabs(tot[0]) / sqrt(tt * rr);
                    if (rho < S.kappa) om = om * (S.kappa / rho);
                    if (fabs(om) < kTiny) S.status = 2;
                    else S.omega = om;
                }
            }
            __syncthreads();
            if (S.status != 0) break;
        }
        // ---- x += omega r, r -= omega t; f = P^H r, ||r||^2
        {
            const T om = (T)S.omega;
            T acc[M + 1];
#pragma unroll
            for (int q = 0; q <= M; ++q) acc[q] = T(0);
            for (int i = lo + threadIdx.x; i < hi; i += kPersThreads) {
                const T ri = a.r[i];
                a.x[i] = axpy(om, ri, a.x[i]);
                const T rn = sub(ri, dmul(om, a.t[i]));
                a.r[i] = rn;
                shadow(rn, i, acc);
            }
            gs.sum<M + 1>(acc, tot);
            if (threadIdx.x == 0) {
                for (int q = 0; q < s; ++q) S.f[q] = tot[q];
                S.rounds += 1;
                check_rr(tot[M]);
            }
            __syncthreads();
        }
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) *a.st = S;
}

}  // namespace tg
