// Arnoldi steps with two sweeps over the basis: classical Gram-Schmidt twice, the second pass of
// a vector delayed into the sweeps of the next one (DCGS2: Bielich, Langou, Thomas,
// Swirydowicz, Yamazaki and Boman, "Low-synch Gram-Schmidt with delayed reorthogonalization for
// Krylov solvers", Parallel Computing 112, 2022).
//
// When step j starts, columns 0..j-1 of V are orthonormal and column j holds u, the next vector
// after its first pass (A v_{j-1} = V h1 + u).  With w = A u in column j + 1:
//   dots    s = V^H u, z = V^H w (columns 0..j-1), u^H u, u^H w in one sweep;
//           beta^2 = u^H u - ||s||^2, t = (u^H w - s^H z) / beta (= v_j^H w);
//   update  v_j = (u - V s) / beta and the next u = (w - V z - t v_j) / beta in one sweep;
//   Hbar    column j-1 is h1 + s over beta; the next h1 = ([z; t] - Hbar s) / beta, because
//           A v_j = (w - A V s) / beta and A V s = V_{0..j} Hbar s.
// u is kept times a power of two g that brings its norm near 1 (s, beta and w, z, t carry it too and
// lose it in the quotients): without it w = A u grows as ||A||^2 and u^H w as its cube, which left the
// range of a float32 basis at ||A|| = 7e12.
// A last pair of sweeps without w (last = 1) finishes column m.  Against two complete passes per
// step (four sweeps and nine launches) this reads the basis half as often, in three launches;
// the operations on it are the same.  Against that form: the float32 basis of 127^3 rows, bound by
// HBM, 99 -> 62 ms for 300 steps; float64 (bound by the float64 unit) 137 -> 119 ms for 150 steps;
// GMRES(20) on 95^3 88 -> 62 ms; 255^2 rows x 21..61 columns (launches) 70 -> 45 us a step.
#pragma once

#include "tg_kernels.cuh"

namespace tg {

// Device scalars of a run, and where the sweeps find them.
template <class D>
struct ArnState {
    D *s, *z, *h1;        // kMaxCols each
    double *beta;         // beta / g, 1 / beta (0 when u vanished), 1 / g, and the next g
    int j0;               // the run's first column: g = 1 there
    D *t;
    D *part;              // block partials [gridDim.x][2 (j + 1)], then the groups'
    unsigned *ticket;     // ticket 0 and one per group of blocks, zero between launches
    const int *skip;      // when set and nonzero, the sweeps return at once (nullptr: never)
};

constexpr int kArnGroup = 16;       // blocks per group of the two-level reduction
constexpr int kArnTickets = 256;    // ticket words: 1 + gridDim.x / kArnGroup at most
constexpr int kArnCols = 64;        // columns per grid y of the plain dots kernel

// Sums part[b][e] over the grid's x blocks b in a fixed order; true in the one block that then
// holds the totals in tot (shared memory).  Beyond two groups the blocks of a group are summed
// by the last of them, the groups by the last group's block: one block alone would take 2 float64
// additions per clock, 9 us for 304 blocks x 122 entries.
template <class D>
__device__ __forceinline__ bool arn_reduce(D *part, int nent, unsigned *ticket, D *tot) {
    __shared__ bool am_last;
    const int nb = gridDim.x;
    const int gs = nb > 2 * kArnGroup ? kArnGroup : nb, ng = (nb + gs - 1) / gs;
    const int grp = blockIdx.x / gs, b0 = grp * gs, b1 = min(nb, b0 + gs);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned all = (unsigned)(b1 - b0) * gridDim.y;
        am_last = atomicAdd(ticket + 1 + grp, 1u) == all - 1;
        if (am_last) ticket[1 + grp] = 0u;
    }
    __syncthreads();
    if (!am_last) return false;
    __threadfence();
    D *sums = part + (size_t)nb * nent;
    // up to half the threads have an entry each: two threads share one
    const int half = blockDim.x >> 1, two = nent <= half;
    auto add_up = [&](const D *src, int lo, int hi, D *out) {
        const int mid = two ? (lo + hi + 1) >> 1 : hi;
        __shared__ D other[kThreads / 2];
        for (int e = two ? threadIdx.x % half : threadIdx.x; e < nent; e += blockDim.x) {
            const bool second = two && (int)threadIdx.x >= half;
            D a = dzero<D>();
#pragma unroll 8
            for (int b = second ? mid : lo; b < (second ? hi : mid); ++b) a = dadd(a, ldcg(src + (size_t)b * nent + e));
            if (second) other[e] = a;
            else out[e] = a;
        }
        __syncthreads();
        if (two && threadIdx.x < nent) out[threadIdx.x] = dadd(out[threadIdx.x], other[threadIdx.x]);
        __syncthreads();
    };
    add_up(part, b0, b1, ng == 1 ? tot : sums + (size_t)grp * nent);
    if (ng == 1) return true;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        am_last = atomicAdd(ticket, 1u) == (unsigned)ng - 1;
        if (am_last) ticket[0] = 0u;
    }
    __syncthreads();
    if (!am_last) return false;
    __threadfence();
    add_up(sums, 0, ng, tot);
    return true;
}

// Warp sums of NV values per lane (NV a power of two up to 32): returns, in lane l, the sum over
// the lanes of v[l % NV], in a fixed order.  Each exchange halves the values a lane holds, NV - 1
// additions and then plain ones, where NV separate sums take 5 NV: a float64 addition holds its
// unit for 64 clocks, and the separate sums of 32 accumulators took 10 us a launch.
template <int NV, class P>
__device__ __forceinline__ P warp_sums(P (&v)[NV]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = NV / 2; h > 0; h >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const P send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = dadd(keep, shfl_xor(send, h));
        }
    }
    P r = v[0];
#pragma unroll
    for (int o = NV; o < 32; o <<= 1) r = dadd(r, shfl_xor(r, o));
    return r;
}

// high word of the largest part's magnitude
__device__ __forceinline__ int dmag(double a) { return __double2hiint(a) & 0x7fffffff; }
__device__ __forceinline__ int dmag(cplx a) { return max(dmag(a.re), dmag(a.im)); }
__device__ __forceinline__ double cmulc(double a, double b) { return a * b; }
__device__ __forceinline__ cplx cmulc(cplx a, cplx b) { return ST<cplx>::conj_mul(a, b); }
__device__ __forceinline__ double rscale(double s, double a) { return s * a; }
__device__ __forceinline__ cplx rscale(double s, cplx a) { return s * a; }

// beta, t and the coefficient vectors from the totals (tot[2 c] = v_c^H u, tot[2 c + 1] = v_c^H w)
template <class D>
__device__ __forceinline__ void arn_scalars(const D *tot, int j, int nv, const ArnState<D> &a) {
    for (int c = threadIdx.x; c < j; c += blockDim.x) {
        a.s[c] = tot[nv * c];
        if (nv == 2) a.z[c] = tot[2 * c + 1];
    }
    if (threadIdx.x < 32) {
        double ss = 0.0;
        D sz = dzero<D>();
        int mag = 0;                     // high word of the largest part of z, then of t
        for (int c = threadIdx.x; c < j; c += 32) {
            const D s = tot[nv * c];
            ss += dreal(cmulc(s, s));
            if (nv == 2) {
                sz = dadd(sz, cmulc(s, tot[2 * c + 1]));
                mag = max(mag, dmag(tot[2 * c + 1]));
            }
        }
        ss = warp_sum(ss);
        if (nv == 2) sz = warp_sum(sz);
        mag = __reduce_max_sync(0xffffffffu, mag);
        if (threadIdx.x == 0) {
            const double b2 = dreal(tot[nv * j]) - ss;
            const double beta = b2 > 0.0 ? sqrt(b2) : (b2 == b2 ? 0.0 : b2), inv = beta > 0.0 ? 1.0 / beta : (beta == beta ? 0.0 : beta);
            const double ginv = j > a.j0 ? __hiloint2double((2046 << 20) - __double2hiint(a.beta[3]), 0) : 1.0;
            a.beta[0] = beta * ginv;
            a.beta[1] = inv;
            a.beta[2] = ginv;
            if (nv == 2) {
                a.t[0] = rscale(inv, dsub(tot[2 * j + 1], sz));
                // the next u is of the size of A v_j: of its parts in V, z and t over beta, or of the last one
                mag = max(mag, dmag(a.t[0]));
                const int eb = dmag(beta) >> 20;
                int e = mag >= 0x100000 && eb > 0 ? (mag >> 20) - eb : -500;
                if (j > a.j0 && eb > 0) e = max(e, (dmag(a.beta[0]) >> 20) - 1023);
                a.beta[3] = e > -500 && e < 500 ? __hiloint2double((1023 - e) << 20, 0) : 1.0;
            }
        }
    }
}

// The dots for a float64 or float32 basis with 16-byte aligned columns whose leading dimension
// covers whole chunks: the cp.async pipeline of k_gemv_t_pipe with two accumulators per column.
// Columns come in groups of kPipeCols (blockIdx.y); u (column j) and w are staged with each.
template <class E>
__global__ void __launch_bounds__(kThreads, 2) k_arn_dots_pipe(const E *__restrict__ V, size_t ldv, int j, int n,
                                                               int last, ArnState<double> a) {
    pdl_wait();
    if (a.skip && *a.skip) return;
    constexpr int kMaxPerWarp = kPipeCols / 8;
    constexpr int R = PipeRows<E>::value;
    constexpr int PE = 16 / sizeof(E), U = R / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    E *buf = reinterpret_cast<E *>(smem_raw);
    __shared__ double tot[2 * kMaxCols];
    const int nv = last ? 1 : 2;
    const int cbase = blockIdx.y * kPipeCols;
    const int ng = min(j + 1 - cbase, kPipeCols);
    const int cols = ng + nv;                       // the group, u and w
    const size_t stage_elems = (size_t)cols * R;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nchunks = (n + R - 1) / R, G = gridDim.x;
    const int mine = (int)blockIdx.x < nchunks ? (nchunks - 1 - (int)blockIdx.x) / G + 1 : 0;
    auto issue = [&](int it) {
        if (it < mine) {
            const size_t row0 = (size_t)(blockIdx.x + (size_t)it * G) * R;
            E *dst = buf + (size_t)(it % kPipeStages) * stage_elems;
            for (int e = threadIdx.x; e < cols * (R / PE); e += blockDim.x) {
                const int c = e / (R / PE), rp = e % (R / PE);
                const int col = c < ng ? cbase + c : j + (c - ng);
                cp_async16(dst + (size_t)c * R + PE * rp, V + (size_t)col * ldv + row0 + PE * rp);
            }
        }
        cp_async_commit();
    };
    static_assert(kMaxPerWarp == 16, "one accumulator per lane in the final sums");
    E acc[2 * kMaxPerWarp];
#pragma unroll
    for (int q = 0; q < 2 * kMaxPerWarp; ++q) acc[q] = E(0);
#pragma unroll
    for (int s = 0; s < kPipeStages - 1; ++s) issue(s);
    for (int it = 0; it < mine; ++it) {
        cp_async_wait<kPipeStages - 2>();
        __syncthreads();
        issue(it + kPipeStages - 1);                // the buffer of iteration it - 1, read by everyone already
        const E *st = buf + (size_t)(it % kPipeStages) * stage_elems;
        const int left = n - (int)(blockIdx.x + (size_t)it * G) * R;
        E uv[U], wv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = lane + 32 * u < left;
            uv[u] = ok ? st[(size_t)ng * R + lane + 32 * u] : E(0);
            wv[u] = ok && nv == 2 ? st[(size_t)(ng + 1) * R + lane + 32 * u] : E(0);
        }
#pragma unroll
        for (int q = 0; q < kMaxPerWarp; ++q) {
            const int c = warp + 8 * q;
            if (c < ng) {
                const E *sc = st + (size_t)c * R;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const E x = lane + 32 * u < left ? sc[lane + 32 * u] : E(0);
                    acc[2 * q] = fma(x, uv[u], acc[2 * q]);
                    acc[2 * q + 1] = fma(x, wv[u], acc[2 * q + 1]);
                }
            }
        }
    }
    cp_async_wait<0>();
    const int nent = nv * (j + 1);
    {
        const E r = warp_sums<2 * kMaxPerWarp>(acc);         // lane 2 q + v: column warp + 8 q, vector v
        const int c = warp + 8 * (lane >> 1), v = lane & 1;
        if (c < ng && v < nv) a.part[(size_t)blockIdx.x * nent + nv * (cbase + c) + v] = (double)r;
    }
    if (arn_reduce<double>(a.part, nent, a.ticket, tot)) arn_scalars<double>(tot, j, nv, a);
}

// The dots for any basis: columns in groups of kArnCols (blockIdx.y), warp w owns columns
// w, w + 8, ... of its group, 32 kU rows a pass (kU loads per column in flight per lane).
template <class T>
__global__ void __launch_bounds__(kThreads) k_arn_dots(const T *__restrict__ V, size_t ldv, int j, int n, int last,
                                                       ArnState<typename ST<T>::D> a) {
    pdl_wait();
    if (a.skip && *a.skip) return;
    using D = typename ST<T>::D;
    constexpr int kQ = kArnCols / 8, kU = sizeof(T) == 16 ? 2 : 4;
    __shared__ D tot[2 * kMaxCols];
    const int nv = last ? 1 : 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cbase = blockIdx.y * kArnCols;
    const T *u = V + (size_t)j * ldv, *w = u + ldv;
    T acc[2 * kQ];
#pragma unroll
    for (int q = 0; q < 2 * kQ; ++q) acc[q] = ST<T>::zero();
    for (int64_t row0 = (int64_t)blockIdx.x * 32 * kU; row0 < n; row0 += (int64_t)gridDim.x * 32 * kU) {
        T uv[kU], wv[kU];
        bool ok[kU];
#pragma unroll
        for (int r = 0; r < kU; ++r) {
            const int64_t row = row0 + 32 * r + lane;
            ok[r] = row < n;
            uv[r] = ok[r] ? u[row] : ST<T>::zero();
            wv[r] = ok[r] && nv == 2 ? w[row] : ST<T>::zero();
        }
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int c = cbase + warp + 8 * q;
            if (c <= j) {
                const T *vc = V + (size_t)c * ldv + row0 + lane;
                T x[kU];
#pragma unroll
                for (int r = 0; r < kU; ++r) x[r] = ok[r] ? vc[32 * r] : ST<T>::zero();
#pragma unroll
                for (int r = 0; r < kU; ++r) {
                    acc[2 * q] = ST<T>::fma_cm(x[r], uv[r], acc[2 * q]);
                    acc[2 * q + 1] = ST<T>::fma_cm(x[r], wv[r], acc[2 * q + 1]);
                }
            }
        }
    }
    const int nent = nv * (j + 1);
    {
        const T r = warp_sums<2 * kQ>(acc);                  // lane 2 q + v: column warp + 8 q, vector v
        const int c = cbase + warp + 8 * ((lane >> 1) % kQ), v = lane & 1;
        if (lane < 2 * kQ && c <= j && v < nv) a.part[(size_t)blockIdx.x * nent + nv * c + v] = to_d(r);
    }
    if (arn_reduce<D>(a.part, nent, a.ticket, tot)) arn_scalars<D>(tot, j, nv, a);
}

// Column j-1 of Hbar (unless the run starts at j) and the next h1, by one block: four lanes a row
// of Hbar s.  HT is the Hessenberg type: the basis type, or float64 for a float32 basis.
template <class HT, class D>
__device__ __forceinline__ void arn_hessenberg(HT *H, int ldh, int j, int j0, int last, const ArnState<D> &a) {
    const double inv = a.beta[1];
    if (j > j0) {
        HT *col = H + (size_t)(j - 1) * ldh;
        const double ginv = a.beta[2];
        for (int i = threadIdx.x; i < j; i += blockDim.x) col[i] = dadd(a.h1[i], rscale(ginv, a.s[i]));
        if (threadIdx.x == 0) {
            HT b = ST<HT>::zero();
            *reinterpret_cast<double *>(&b) = a.beta[0];
            col[j] = b;
        }
    }
    __syncthreads();
    if (last) return;
    const int sub = threadIdx.x & 3;
    for (int i0 = 0; i0 <= j; i0 += blockDim.x >> 2) {
        const int i = i0 + (threadIdx.x >> 2);
        D acc = dzero<D>();
        if (i <= j)
            for (int l = sub; l < j; l += 4) acc = dadd(acc, dmul(H[i + (size_t)l * ldh], a.s[l]));
        acc = dadd(acc, shfl_xor(acc, 1));
        acc = dadd(acc, shfl_xor(acc, 2));
        if (i <= j && sub == 0) a.h1[i] = rscale(inv, dsub(i < j ? a.z[i] : a.t[0], acc));
    }
}

// Row element of the update sweep: one value, or 4 rows of a float32 basis as float4.
template <class T, bool F4> struct ArnRow { using type = T; };
template <> struct ArnRow<float, true> { using type = float4; };
__device__ __forceinline__ float4 axpy(float a, const float4 &x, const float4 &y) { return f4_axpy(a, x, y); }
__device__ __forceinline__ float4 dadd(const float4 &a, const float4 &b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 sub(const float4 &a, const float4 &b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float4 scal(double s, const float4 &a) {
    const float f = (float)s;
    return make_float4(f * a.x, f * a.y, f * a.z, f * a.w);
}

// The update sweep; the grid's last block does the Hessenberg column instead of rows.  F4: 4
// rows per thread as float4 (float32, 16-byte aligned columns, rows padded to the leading
// dimension).  CS threads share a row and take every CS-th column: with one thread a row, a grid
// of fewer rows than the GPU has threads waits j / 8 times for L2 in turn.
template <class T, class HT, bool F4, int CS, int MC>
__global__ void __launch_bounds__(kThreads) k_arn_update(T *__restrict__ V, size_t ldv, int j, int n, int last,
                                                         HT *H, int ldh, int j0, ArnState<typename ST<T>::D> a) {
    pdl_wait();
    if (a.skip && *a.skip) return;
    using X = typename ArnRow<T, F4>::type;
    constexpr int RB = kThreads / CS, W = F4 ? 4 : 1;
    const int nb = gridDim.x - 1;
    if ((int)blockIdx.x == nb) {
        arn_hessenberg<HT>(H, ldh, j, j0, last, a);
        return;
    }
    __shared__ T ss[MC], zs[MC];         // in the vector type, converted once per block
    __shared__ X red[CS > 1 ? 2 * kThreads : 1];
    for (int c = threadIdx.x; c < j; c += blockDim.x) {
        ss[c] = KS<T>::of(a.s[c]);
        zs[c] = last ? ST<T>::zero() : KS<T>::of(a.z[c]);
    }
    __syncthreads();
    const double inv = a.beta[1], ginv = last ? 0.0 : inv * a.beta[3];
    const T mt = last ? ST<T>::zero() : neg(KS<T>::of(a.t[0]));
    const int rows = (n + W - 1) / W, r = threadIdx.x % RB, q = threadIdx.x / RB;
    const size_t ld = ldv / W;
    X *VX = reinterpret_cast<X *>(V), *u = VX + (size_t)j * ld, *w = u + ld;
    for (int64_t base = (int64_t)blockIdx.x * RB; base < rows; base += (int64_t)nb * RB) {
        const int64_t row = base + r;
        X x{}, y{};
        if (row < rows) {
#pragma unroll 8
            for (int c = q; c < j; c += CS) {
                const X v = VX[(size_t)c * ld + row];
                x = axpy(ss[c], v, x);
                if (!last) y = axpy(zs[c], v, y);
            }
        }
        if constexpr (CS > 1) {
            __syncthreads();             // red is free again
            red[threadIdx.x] = x;
            red[kThreads + threadIdx.x] = y;
            __syncthreads();
            if (q != 0) continue;
#pragma unroll
            for (int p = 1; p < CS; ++p) {
                x = dadd(x, red[p * RB + r]);
                y = dadd(y, red[kThreads + p * RB + r]);
            }
        }
        if (row < rows) {
            const X v = scal(inv, sub(u[row], x));
            u[row] = v;
            if (!last) w[row] = scal(ginv, axpy(mt, v, sub(w[row], y)));
        }
    }
}

}  // namespace tg
