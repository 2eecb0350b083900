// Single-CTA float64 kernels for the small dense problems of the method:
//   - the GMRES-DR restart step (Section 2.1): least squares min ||c - Hbar d||, harmonic
//     Ritz pairs of Hbar (eigenpairs of H_m + |h_{m+1,m}|^2 f e_m^T, H_m^H f = e_m),
//     selection of the k smallest, orthonormal basis P_k of their span, the restart
//     matrices P_{k+1}, Hbar_k = P_{k+1}^H Hbar P_k, c_k = P_{k+1}^H (c - Hbar d);
//   - Cholesky and triangular inverse for CholQR2 (the projection set-up);
//   - Gauss-Jordan inverse of the Galerkin matrix H = V^H A V;
//   - incremental Givens least squares for GMRES(m) cycles;
//   - the k x k solve of each projection.
// The eigenvalue algorithms are the textbook ones (Golub & Van Loan, Matrix Computations,
// Sections 7.4-7.6): Householder reduction to Hessenberg form, Francis double-shift QR
// (real matrices, real Schur form with 2 x 2 blocks for complex pairs) or Wilkinson
// single-shift QR (complex matrices), with accumulated Schur vectors, and eigenvectors
// by back substitution on the (quasi-)triangular factor.  The restart kernel is one block
// of kGdrThreads threads whose work matrices sit in shared memory while they fit (global
// scratch otherwise); the other kernels are one block of kSmallThreads threads on global
// scratch.  On this GPU every float64 warp instruction holds its sub-partition's float64
// unit for tens of cycles whatever the active lanes, and sqrt, division and hypot are
// long sequences of them: the serial chains (QR sweeps, reflectors) are written to keep
// few float64 instructions on the critical path (see the Schur form section).
#include <cfloat>
#include <cmath>
#include "tg_fastmath.cuh"
#include "tg_small.cuh"

namespace tg {

namespace {

constexpr double kEps = DBL_EPSILON;


// ----------------------------------------------------------------------------- generic helpers
template <class T> struct Cx;
template <> struct Cx<double> {
    __device__ static double cj(double a) { return a; }
    __device__ static double ab2(double a) { return a * a; }
    __device__ static double mul(double a, double b) { return a * b; }
    __device__ static double div(double a, double b) { return a / b; }
    __device__ static double re(double a) { return a; }
    __device__ static double zero() { return 0.0; }
    __device__ static double one() { return 1.0; }
    __device__ static double sc(double s, double a) { return s * a; }
    __device__ static double mac(double s, double a, double b) { return fma(a, b, s); }        // s + a b
    __device__ static double macc(double s, double a, double b) { return fma(a, b, s); }       // s + conj(a) b
    __device__ static double nmac(double s, double a, double b) { return fma(-a, b, s); }      // s - a b
};
template <> struct Cx<cplx> {
    __device__ static cplx cj(cplx a) { return conj(a); }
    __device__ static double ab2(cplx a) { return abs2(a); }
    __device__ static cplx mul(cplx a, cplx b) { return a * b; }
    __device__ static cplx div(cplx a, cplx b) { return cdiv(a, b); }
    __device__ static double re(cplx a) { return a.re; }
    __device__ static cplx zero() { return {0.0, 0.0}; }
    __device__ static cplx one() { return {1.0, 0.0}; }
    __device__ static cplx sc(double s, cplx a) { return s * a; }
    // four fused operations; s + a * b takes six (the sum of two products, then s)
    __device__ static cplx mac(cplx s, cplx a, cplx b) {
        return {fma(a.re, b.re, fma(-a.im, b.im, s.re)), fma(a.re, b.im, fma(a.im, b.re, s.im))};
    }
    __device__ static cplx macc(cplx s, cplx a, cplx b) {
        return {fma(a.re, b.re, fma(a.im, b.im, s.re)), fma(a.re, b.im, fma(-a.im, b.re, s.im))};
    }
    __device__ static cplx nmac(cplx s, cplx a, cplx b) {
        return {fma(-a.re, b.re, fma(a.im, b.im, s.re)), fma(-a.re, b.im, fma(-a.im, b.re, s.im))};
    }
};

__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ cplx add(cplx a, cplx b) { return a + b; }
__device__ __forceinline__ double subt(double a, double b) { return a - b; }
__device__ __forceinline__ cplx subt(cplx a, cplx b) { return a - b; }

// ----------------------------------------------------------------------------- Schur form: shared pieces
// Cost model of the QR sweeps on this GPU: every float64 warp instruction occupies its SM
// sub-partition's float64 unit for 64 cycles whatever the number of active lanes, and a dependent
// one waits as long; sqrt and division are sequences of six to seven of them.  So a bulge-chasing
// step takes as long as the chain of operations from one transform to the next, if nothing else
// shares that sub-partition's unit.  One step t of a sweep, between two block barriers:
//   warp 0 (the chain) reads the 3 x 3 (complex 2 x 2) block of transform t and the entry below
//     it, applies transform t to the one column that defines transform t + 1 (lanes in
//     parallel), computes transform t + 1 and stores that column's final values;
//   warp 1 (the window) applies transform t to the few columns and rows next to the diagonal that
//     step t + 1 reads;
//   the far warps (2, 3, 5, 6, 7: none shares the chain's sub-partition) apply it to the other
//     columns, rows and Schur vector rows.
// The three write disjoint entries; the chain and the window share reads at the start of the step,
// which a two-warp barrier separates from the window's writes.  Real m = 60: 22 float64
// operations in the chain, 2750 cycles a step, where row phase, column phase and reflector in turn
// took 3600 (Schur form of a restart 4.6 -> 3.5 ms).
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double shfl_all(double v, int l) { return __shfl_sync(kFull, v, l); }
__device__ __forceinline__ cplx shfl_all(cplx v, int l) { return {shfl_all(v.re, l), shfl_all(v.im, l)}; }
__device__ __forceinline__ void bar_two_warps() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

// lane's place among the far warps' lanes (2, 3, 5, 6, 7), and their number
constexpr int kFarLanes = 5 * 32;
__device__ __forceinline__ int far_index() {
    const int w = threadIdx.x >> 5;
    return w < 2 || w == 4 ? -1 : 32 * (w < 4 ? w - 2 : w - 3) + (threadIdx.x & 31);
}

// Complex Givens rotation G = [conj(a) conj(b); -b a] with G [x; y] = [r; 0], r = ||(x, y)||:
// a = x / r, b = y / r.  Warp-wide call; lanes 0..3 hold x.re, x.im, y.re, y.im in v and
// write a.re, a.im, b.re, b.im to rs[0..3].  (x, y) = 0 gives the identity.  Returns r.
__device__ __forceinline__ double givens_warp(double v, double *rs) {
    const int lane = threadIdx.x & 31;
    auto norm2 = [&](double u) {
        double q = u * u;
        q += __shfl_xor_sync(kFull, q, 1);
        q += __shfl_xor_sync(kFull, q, 2);
        return __shfl_sync(kFull, q, 0);
    };
    double s2 = norm2(v), out, r;
    if (__double_as_longlong(s2) == 0) {
        out = lane == 0 ? 1.0 : 0.0;
        r = 0.0;
    } else {
        double u = v, mx = 1.0;
        if (!mid_range(s2)) {       // scale by the largest component first
            mx = fabs(v);
            mx = fmax(mx, __shfl_xor_sync(kFull, mx, 1));
            mx = fmax(mx, __shfl_xor_sync(kFull, mx, 2));
            mx = __shfl_sync(kFull, mx, 0);
            u = v * (1.0 / mx);
            s2 = norm2(u);
        }
        const double inv = rsqrt_fast(s2);
        out = u * inv;
        r = s2 * inv * mx;
    }
    if (lane < 4) rs[lane] = out;
    return r;
}

// Householder reflector I - g w w^T (g = 2 / w^T w) mapping (x, y, z) to (beta, 0, 0),
// beta = -sign(x) ||(x, y, z)||: w = (x - beta, y, z) and g = 1 / (n2 + ||.|| |x|), n2 the square
// norm.  Warp-wide, every lane with the same x, y, z; writes w and g w to hs[0..5] and returns
// beta.  y = z = 0 gives the identity.
__device__ __forceinline__ double reflect_warp(double x, double y, double z, double *hs) {
    const int lane = threadIdx.x & 31;
    double w0 = 0.0, w1 = 0.0, w2 = 0.0, g = 0.0, beta = x, mx = 1.0;
    double sn = fma(z, z, y * y), n2 = fma(x, x, sn);
    if (!mid_range(n2)) {               // rescale (the reflector does not depend on the scale)
        mx = fmax(fabs(x), fmax(fabs(y), fabs(z)));
        const double r = mx > 0.0 ? 1.0 / mx : 0.0;
        x *= r; y *= r; z *= r;
        sn = fma(z, z, y * y);
        n2 = fma(x, x, sn);
    }
    if (__double_as_longlong(sn) != 0) {       // tests on the bits: a float64 compare is a link of the chain too
        const double alpha = sqrt_fast(n2);
        g = rcp_fast(fma(alpha, fabs(x), n2));
        const double bs = -copysign(alpha, x);
        w0 = x - bs;
        w1 = y;
        w2 = z;
        beta = mx == 1.0 ? bs : bs * mx;
    }
    const int c = lane % 3;
    const double v = c == 0 ? w0 : c == 1 ? w1 : w2, gv = v * g;
    if (lane < 6) hs[lane] = lane < 3 ? v : gv;
    return beta;
}

// ----------------------------------------------------------------------------- reflectors
// One warp: the reflector I - g w w^H (g real) that maps x[0..len-1] to (beta, 0, .., 0): w = x but
// for w_0 = x_0 - beta, beta = -phase(x_0) ||x||, g = 1 / (||x||^2 + ||x|| |x_0|).  w may be x
// itself.  A zero tail gives the identity.  Every lane computes the scalars: no shuffle after the
// norm's, no division of the elements.
template <class T>
__device__ __forceinline__ void reflector_warp(const T *x, int len, T *w, double *gs, T *beta) {
    const int lane = threadIdx.x & 31;
    bool scaled = false;                // tests on bits and flags: a float64 compare is a link of the chain too
    double sc = 1.0, mx = 1.0;
    auto tail = [&]() {
        double s = 0.0;
        for (int i = 1 + lane; i < len; i += 32) s += Cx<T>::ab2(scaled ? Cx<T>::sc(sc, x[i]) : x[i]);
        if (len <= 2) return __shfl_sync(kFull, s, 0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        return s;
    };
    double sn = tail();
    T x0 = x[0];
    double ax2 = Cx<T>::ab2(x0), n2 = ax2 + sn;
    if (!mid_range(n2)) {               // rescale (the reflector does not depend on the scale)
        mx = 0.0;
        for (int i = lane; i < len; i += 32) {
            const double *c = reinterpret_cast<const double *>(x + i);
            mx = fmax(mx, fabs(c[0]));
            if (sizeof(T) == 16) mx = fmax(mx, fabs(c[sizeof(T) / 8 - 1]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(kFull, mx, o));
        if (mx > 1e-300 && mx < 1e300) {
            sc = 1.0 / mx;
            scaled = true;
            sn = tail();
            x0 = Cx<T>::sc(sc, x0);
            ax2 = Cx<T>::ab2(x0);
            n2 = ax2 + sn;
        }
    }
    T w0 = Cx<T>::zero(), bt = x0;
    double g = 0.0;
    if (__double_as_longlong(sn) != 0) {
        const double alpha = mid_range(n2) ? sqrt_fast(n2) : sqrt(n2);
        double a0 = 0.0;
        T ph = Cx<T>::one();
        if constexpr (sizeof(T) == sizeof(double)) {
            a0 = fabs(x0);
            ph = copysign(1.0, x0);
        } else if (__double_as_longlong(ax2) != 0) {
            const double ia = mid_range(ax2) ? rsqrt_fast(ax2) : rsqrt(ax2);
            a0 = ax2 * ia;
            ph = Cx<T>::sc(ia, x0);
        }
        const double d = fma(alpha, a0, n2);
        g = mid_range(d) ? rcp_fast(d) : 1.0 / d;
        bt = Cx<T>::sc(-alpha, ph);
        w0 = subt(x0, bt);
        if (scaled) bt = Cx<T>::sc(mx, bt);
    } else if (scaled) {
        bt = Cx<T>::sc(mx, x0);
    }
    __syncwarp();
    if (scaled || w != x)
        for (int i = 1 + lane; i < len; i += 32) w[i] = scaled ? Cx<T>::sc(sc, x[i]) : x[i];
    if (lane == 0) { w[0] = w0; *gs = g; *beta = bt; }
    __syncwarp();
}

// One warp: x <- (I - g w w^H) x.
template <class T>
__device__ __forceinline__ void reflect_vector(T *x, const T *w, int len, double g) {
    const int lane = threadIdx.x & 31;
    T s = Cx<T>::zero();
    if (len <= 2) {                     // every lane the same sum
        for (int i = 0; i < len; ++i) s = Cx<T>::macc(s, w[i], x[i]);
        __syncwarp();
    } else {
        for (int i = lane; i < len; i += 32) s = Cx<T>::macc(s, w[i], x[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s = add(s, shfl_xor(s, o));
    }
    s = Cx<T>::sc(g, s);
    for (int i = lane; i < len; i += 32) x[i] = Cx<T>::nmac(x[i], s, w[i]);
    __syncwarp();
}

// Warps 0 .. nw-1 of a set: the reflector on `items` vectors of stride `stride` starting at
// base(item): columns x <- (I - g w w^H) x, or rows x <- x (I - g w w^H) (ROWS).  G lanes share an
// item, so that 60 items occupy all four sub-partitions' float64 units and not those of two warps.
template <int G, bool ROWS, class T, class Base>
__device__ __forceinline__ void reflect_items(int items, Base base, size_t stride, const T *w, int len, double g,
                                              int warp, int nw) {
    constexpr int per = 32 / G;
    const int lane = threadIdx.x & 31, part = lane / per, it = lane % per;
    for (int b = warp * per; b < items; b += nw * per) {
        const bool on = b + it < items;
        T *x = base(on ? b + it : b);
        T s = Cx<T>::zero();
        for (int i = part; i < len; i += G) s = ROWS ? Cx<T>::mac(s, x[i * stride], w[i]) : Cx<T>::macc(s, w[i], x[i * stride]);
#pragma unroll
        for (int o = per; o < 32; o <<= 1) s = add(s, shfl_xor(s, o));
        s = Cx<T>::sc(g, s);
        __syncwarp();
        if (on)
            for (int i = part; i < len; i += G)
                x[i * stride] = ROWS ? subt(x[i * stride], Cx<T>::mul(s, Cx<T>::cj(w[i]))) : Cx<T>::nmac(x[i * stride], s, w[i]);
    }
}

// ----------------------------------------------------------------------------- least squares
// Householder QR of the (rows x m) matrix W (copy of Hbar) and of the right-hand side, rows = m + 1;
// d = R^{-1} (Q^H c)[0..m-1], and f = H_m^{-H} e_m, H_m the first m rows of Hbar.  All threads.
// After a restart the reflectors past column k have two rows, so the chain from one to the next
// bounds the factorisation: warp 0 applies reflector j to column j + 1 and computes reflector j + 1
// while the far warps apply j to the other columns (norm, reflector and update in turn by the block,
// four barriers a column, took 212 us at m = 60, k = 20; now 117).
// f comes from the same factorisation.  With Q = [Q_1 q; p^H s] (rows x rows), H_m = Q_1 R, and from
// Q^H Q = I: f = (Q_1 e_m - q (p^H e_m) / s) / conj(r_mm), which needs the last two columns of Q:
// the reflectors applied in reverse to two unit vectors by a warp each, beside the back substitution
// (elimination with pivoting of H_m^H took another 252 us, complex m = 80 1.6 ms).
template <class T>
__device__ void lsq_solve(T *W, int ldw, int rows, int m, T *rhs, T *d, T *f, T *diag, T *q1, T *q2, double *gs) {
    // last row that can be nonzero in column j once columns 0..j-1 are reduced: the running
    // maximum of each column's last nonzero row (a Hessenberg column j ends at j + 1; the
    // full leading block left by a GMRES-DR restart ends at k); the reflector of column j
    // only needs rows j..end_j, which keeps the factorisation exact.
    __shared__ int end_s[kMaxM + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c = threadIdx.x; c < m; c += blockDim.x) {
        int e = 0;
        for (int i = rows - 1; i > 0; --i) {
            const T w = W[i + (size_t)c * ldw];
            const unsigned long long *b = reinterpret_cast<const unsigned long long *>(&w);
            bool nz = (b[0] << 1) != 0ull;                    // nonzero, sign bit ignored
            if (sizeof(T) == 16) nz = nz || (b[sizeof(T) / 8 - 1] << 1) != 0ull;
            if (nz) { e = i; break; }
        }
        end_s[c] = e;
    }
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        q1[i] = i == m - 1 ? Cx<T>::one() : Cx<T>::zero();
        q2[i] = i == m ? Cx<T>::one() : Cx<T>::zero();
    }
    __syncthreads();
    if (warp == 0)
        for (int c = lane, top = 0; c - lane < m; c += 32) {
            int e = c < m ? max(end_s[c], c) : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int below = __shfl_up_sync(kFull, e, o);
                if (lane >= o) e = max(e, below);
            }
            e = max(e, top);
            if (c < m) end_s[c] = e;
            top = __shfl_sync(kFull, e, 31);
        }
    __syncthreads();
    auto col = [&](int j) { return W + j + (size_t)j * ldw; };      // reflector j's rows of column j
    const int fw = far_index() >> 5;
    if (warp == 0) reflector_warp<T>(col(0), end_s[0] + 1, col(0), gs, diag);
    __syncthreads();
    for (int j = 0; j < m; ++j) {
        const int len = end_s[j] - j + 1;
        if (warp == 0) {
            if (j + 1 < m) {
                reflect_vector<T>(col(j) + ldw, col(j), len, gs[j]);
                reflector_warp<T>(col(j + 1), end_s[j + 1] - j, col(j + 1), gs + j + 1, diag + j + 1);
            }
        } else if (fw >= 0) {
            const int nc = max(0, m - j - 2);       // columns j + 2 .. m - 1, then the right-hand side
            auto base = [&](int it) { return it < nc ? col(j) + (size_t)(it + 2) * ldw : rhs + j; };
            if (len <= 4) reflect_items<1, false, T>(nc + 1, base, 1, col(j), len, gs[j], fw, kFarLanes / 32);
            else reflect_items<4, false, T>(nc + 1, base, 1, col(j), len, gs[j], fw, kFarLanes / 32);
        }
        __syncthreads();
    }
    if (warp == 0) {
        // back substitution, a lane per row and 32 rows on: d_i, then all rows above at once
        constexpr int U = kMaxM / 32;
        T r[U], di[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = lane + 32 * u;
            r[u] = di[u] = Cx<T>::zero();
            if (i < m) {
                r[u] = rhs[i];
                if (Cx<T>::ab2(diag[i]) > 0) di[u] = Cx<T>::div(Cx<T>::one(), diag[i]);
            }
        }
#pragma unroll
        for (int u = U - 1; u >= 0; --u) {
            for (int i = min(m - 1, 32 * u + 31); i >= 32 * u; --i) {
                const T v = shfl_all(Cx<T>::mul(r[u], di[u]), i & 31);
                if (lane == 0) d[i] = v;
#pragma unroll
                for (int t = 0; t <= u; ++t)
                    if (lane + 32 * t < i) r[t] = Cx<T>::nmac(r[t], W[lane + 32 * t + (size_t)i * ldw], v);
            }
        }
    } else if (warp <= 2) {
        T *q = warp == 1 ? q1 : q2;
        for (int j = m - 1; j >= 0; --j) reflect_vector<T>(q + j, col(j), end_s[j] - j + 1, gs[j]);
    }
    __syncthreads();
    const T rmm = diag[m - 1], s = q2[m];
    const T a = Cx<T>::ab2(s) > 0 ? Cx<T>::div(q1[m], s) : Cx<T>::zero();
    const T ir = Cx<T>::ab2(rmm) > 0 ? Cx<T>::div(Cx<T>::one(), Cx<T>::cj(rmm)) : Cx<T>::zero();
    for (int i = threadIdx.x; i < m; i += blockDim.x) f[i] = Cx<T>::mul(Cx<T>::nmac(q1[i], q2[i], a), ir);
    __syncthreads();
}

// ----------------------------------------------------------------------------- Hessenberg form
// A (m x m, ld m) <- Q^H A Q upper Hessenberg; Z <- Q (Z must hold I on entry).  w: 2 (m + 1)
// elements.  The float64 units bound it: 8/3 m^3 multiply-adds at 2 a clock.  Warp 0 computes
// a reflector while the other warps apply the one before to Z, which nothing waits for; 4 lanes
// share a row or column (one thread each left half the sub-partitions idle in the column pass):
// 420 -> 278 us at m = 60, 2308 -> 1732 us at complex m = 80.
template <class T>
__device__ void hessenberg(T *A, int m, T *Z, T *w2) {
    __shared__ double g_s[2];
    __shared__ T beta_s;
    const int warp = threadIdx.x >> 5, fw = far_index() >> 5;
    constexpr int nw = kGdrThreads / 32;
    for (int j = 0; j + 1 < m; ++j) {
        const bool last = j + 2 == m;               // no reflector left: only Z
        const int len = m - j - 1, slot = j & 1;
        T *w = w2 + slot * m;
        if (warp == 0 && !last) reflector_warp<T>(A + (j + 1) + (size_t)j * m, len, w, g_s + slot, &beta_s);
        // with long rows of Z all warps take part, else those that leave warp 0's unit alone
        const bool all = last || len * (int)(sizeof(T) / 8) * (int)(sizeof(T) / 8) >= 64;
        if (j > 0 && (all || fw >= 0) && g_s[slot ^ 1] != 0.0)
            reflect_items<4, true, T>(m, [&](int r) { return Z + r + (size_t)j * m; }, m, w2 + (slot ^ 1) * m, len + 1,
                                      g_s[slot ^ 1], all ? warp : fw, all ? nw : kFarLanes / 32);
        __syncthreads();
        if (last) break;
        const double g = g_s[slot];
        if (g == 0.0) continue;
        if (threadIdx.x == 0) A[(j + 1) + (size_t)j * m] = beta_s;
        // left: rows j+1..m-1, columns j+1..m-1
        reflect_items<4, false, T>(len, [&](int c) { return A + (j + 1) + (size_t)(j + 1 + c) * m; }, 1, w, len, g, warp, nw);
        __syncthreads();
        // right: all rows, columns j+1..m-1
        reflect_items<4, true, T>(m, [&](int r) { return A + r + (size_t)(j + 1) * m; }, m, w, len, g, warp, nw);
        __syncthreads();
    }
    // clean below the subdiagonal
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        int i = e % m, j = e / m;
        if (i > j + 1) A[e] = Cx<T>::zero();
    }
    __syncthreads();
}

// ----------------------------------------------------------------------------- real Schur form
// Francis double-shift QR on the real upper Hessenberg H (m x m, ld m), accumulating Z.
// Returns 0 on success, 1 if an eigenvalue failed to converge in 40 m sweeps.
__device__ int real_schur(double *H, int m, double *Z) {
    __shared__ int hi_s, l_s, status_s;
    // what to do next, by turns in two places: after a deflation warp 0 goes on to the next decision
    // at once, and a slower warp may not have read this one yet (every warp has read the one before
    // last: a block barrier lies between)
    __shared__ int act_s[2];
    __shared__ double hs_s[2][6];      // w and g w of the current and the next reflector
    __shared__ double win_s[9];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) { hi_s = m - 1; status_s = 0; }
    __syncthreads();
    int its = 0, total = 0;
    for (int turn = 0;; turn ^= 1) {
        if (tid < 32) {
            // the active block: the largest l <= hi with a negligible H[l, l-1] (0 if none),
            // found by warp 0 with a ballot over the candidates
            const int hi = hi_s;
            __syncwarp();          // every lane has read hi_s before lane 0 may update it
            int l = 0;
            if (hi > 0) {
                for (int base = hi; base > 0 && l == 0; base -= 32) {
                    const int cand = base - lane;
                    bool neg = false;
                    if (cand > 0) {
                        double s = fabs(H[(cand - 1) + (size_t)(cand - 1) * m]) + fabs(H[cand + (size_t)cand * m]);
                        if (s == 0.0) s = 1.0;
                        neg = fabs(H[cand + (size_t)(cand - 1) * m]) <= kEps * s;
                    }
                    const unsigned bal = __ballot_sync(kFull, neg);
                    if (bal) l = base - (__ffs(bal) - 1);     // lowest lane = largest index
                }
            }
            if (lane == 0) {
                if (l > 0) H[l + (size_t)(l - 1) * m] = 0.0;
                int act = 0;
                if (hi < 0) act = -1;
                else {
                    l_s = l;
                    if (l == hi) { hi_s = hi - 1; act = 1; }
                    else if (l == hi - 1) { act = 2; }   // 2x2 block: standardise below
                    else act = 3;                         // QR sweep on l..hi
                }
                act_s[turn] = act;
            }
        }
        __syncthreads();
        const int act = act_s[turn];
        if (act < 0) break;
        if (act == 1) { its = 0; continue; }
        const int hi = hi_s, l = l_s;
        if (act == 2) {
            // 2x2 block [a b; c d] at (hi-1, hi): real eigenvalues -> rotate to triangular form
            __shared__ double cs_s, sn_s;
            __shared__ int rot_s;
            if (tid == 0) {
                double a = H[(hi - 1) + (size_t)(hi - 1) * m], b = H[(hi - 1) + (size_t)hi * m];
                double c = H[hi + (size_t)(hi - 1) * m], d = H[hi + (size_t)hi * m];
                double p = 0.5 * (a - d);
                double disc = p * p + b * c;
                rot_s = 0;
                if (disc >= 0.0 && c != 0.0) {
                    // real eigenvalues: lam - d = p + sign(p) sqrt(disc) (no cancellation);
                    // (lam - d, c) is an eigenvector of the block, and the rotation whose
                    // first column it is makes the block upper triangular
                    double e0 = p + copysign(sqrt(disc), p), e1 = c;
                    double nr = hypot(e0, e1);
                    if (nr > 0) {
                        cs_s = e0 / nr;
                        sn_s = e1 / nr;
                        rot_s = 1;
                    }
                }
            }
            __syncthreads();
            if (rot_s) {
                const double cs = cs_s, sn = sn_s;
                // rows hi-1, hi: H <- G^T H for columns hi-1..m-1
                for (int c = hi - 1 + tid; c < m; c += nt) {
                    double h1 = H[(hi - 1) + (size_t)c * m], h2 = H[hi + (size_t)c * m];
                    H[(hi - 1) + (size_t)c * m] = cs * h1 + sn * h2;
                    H[hi + (size_t)c * m] = -sn * h1 + cs * h2;
                }
                __syncthreads();
                // columns hi-1, hi: H <- H G for rows 0..hi, Z <- Z G
                for (int rr = tid; rr < 2 * m; rr += nt) {
                    double *M = rr < m ? H : Z;
                    const int r = rr < m ? rr : rr - m;
                    if (M == H && r > hi) continue;
                    double h1 = M[r + (size_t)(hi - 1) * m], h2 = M[r + (size_t)hi * m];
                    M[r + (size_t)(hi - 1) * m] = cs * h1 + sn * h2;
                    M[r + (size_t)hi * m] = -sn * h1 + cs * h2;
                }
                __syncthreads();
                if (tid == 0) H[hi + (size_t)(hi - 1) * m] = 0.0;
            }
            if (tid == 0) hi_s = hi - 2;
            __syncthreads();
            its = 0;
            continue;
        }
        // ---- double-shift sweep on rows/cols l..hi
        ++its;
        ++total;
        if (total > 40 * m) {
            if (tid == 0) status_s = 1;
            __syncthreads();
            break;
        }
        if (warp == 0) {
            double sh, t;
            if (its % 10 == 0) {
                // exceptional shift
                double w = fabs(H[hi + (size_t)(hi - 1) * m]) + fabs(H[(hi - 1) + (size_t)(hi - 2 >= 0 ? hi - 2 : 0) * m]);
                sh = 1.5 * w + H[hi + (size_t)hi * m];
                t = w * w;
            } else {
                double a = H[(hi - 1) + (size_t)(hi - 1) * m], b = H[(hi - 1) + (size_t)hi * m];
                double c = H[hi + (size_t)(hi - 1) * m], d = H[hi + (size_t)hi * m];
                sh = a + d;
                t = a * d - b * c;
            }
            // first column of (H - s1 I)(H - s2 I) = H^2 - s H + t I
            const double h00 = H[l + (size_t)l * m], h01 = H[l + (size_t)(l + 1) * m];
            const double h10 = H[(l + 1) + (size_t)l * m], h11 = H[(l + 1) + (size_t)(l + 1) * m];
            reflect_warp(h00 * h00 + h01 * h10 - sh * h00 + t, h10 * (h00 + h11 - sh),
                         (l + 2 <= hi) ? h10 * H[(l + 2) + (size_t)(l + 1) * m] : 0.0, hs_s[l & 1]);
        }
        __syncthreads();
        const int far = far_index();
        for (int k = l; k <= hi - 1; ++k) {
            const double *hb = hs_s[k & 1];
            const bool r3 = k <= hi - 2;               // the last reflector has two rows
            const double w0 = hb[0], w1 = hb[1], w2 = r3 ? hb[2] : 0.0, g0 = hb[3], g1 = hb[4], g2 = r3 ? hb[5] : 0.0;
            if (warp == 0) {
                // rows k+1..k+3 of column k after reflector k: lane 3 (r - 1) + j holds row k + r of
                // column k + j after the row part, then the column part for column k
                const int r = 1 + lane / 3, j = lane % 3;
                const bool ok = lane < 9 && (j < 2 || r3);
                const double *col = H + (size_t)(ok ? k + j : k) * m;
                const double b0 = ok ? col[k] : 0.0, b1 = ok ? col[k + 1] : 0.0, b2 = ok && r3 ? col[k + 2] : 0.0;
                const double b3 = ok && j == 2 && k + 3 <= hi ? col[k + 3] : 0.0;
                bar_two_warps();
                const double c = fma(g2, b2, fma(g1, b1, g0 * b0));
                const double v = fma(r == 1 ? -w1 : r == 2 ? -w2 : 0.0, c, r == 1 ? b1 : r == 2 ? b2 : b3);
                const int base = lane < 9 ? 3 * (lane / 3) : 0;
                const double v0 = __shfl_sync(kFull, v, base), v1 = __shfl_sync(kFull, v, base + 1),
                             v2 = __shfl_sync(kFull, v, base + 2);
                const double xr = fma(-fma(v2, w2, fma(v1, w1, v0 * w0)), g0, v0);
                const double x = __shfl_sync(kFull, xr, 0), y = __shfl_sync(kFull, xr, 3), z = __shfl_sync(kFull, xr, 6);
                double *ck = H + (size_t)k * m;
                if (k < hi - 1) {
                    const double beta = reflect_warp(x, y, k + 3 <= hi ? z : 0.0, hs_s[(k + 1) & 1]);
                    if (lane == 0) {
                        ck[k + 1] = beta;
                        ck[k + 2] = 0.0;
                        if (k + 3 <= hi) ck[k + 3] = 0.0;
                    }
                } else if (lane == 0) {
                    ck[hi] = x;
                }
            } else if (warp == 1) {
                // columns k..k+4 of rows k..k+2, then columns k..k+2 of rows k..k+3 (column k below
                // the diagonal is the chain's)
                const int c = k + lane;
                const bool oc = lane < 5 && c < m;
                double *col = H + (size_t)(oc ? c : k) * m;
                double h0 = 0.0, h1 = 0.0, h2 = 0.0;
                if (oc) {
                    h0 = col[k];
                    h1 = col[k + 1];
                    if (r3) h2 = col[k + 2];
                }
                const double below = k + 3 <= hi ? H[k + 3 + (size_t)(k + 2) * m] : 0.0;
                bar_two_warps();
                const double q = fma(g2, h2, fma(g1, h1, g0 * h0));
                h0 = fma(-q, w0, h0);
                h1 = fma(-q, w1, h1);
                h2 = fma(-q, w2, h2);
                if (lane < (r3 ? 3 : 2)) {
                    win_s[lane] = h0;
                    win_s[3 + lane] = h1;
                    win_s[6 + lane] = h2;
                } else if (oc) {
                    col[k] = h0;
                    col[k + 1] = h1;
                    if (r3) col[k + 2] = h2;
                }
                __syncwarp();
                const int r = lane;                    // row k + r
                if (r < 4 && k + r <= hi) {
                    const double m0 = r < 3 ? win_s[3 * r] : 0.0, m1 = r < 3 ? win_s[3 * r + 1] : 0.0;
                    const double m2 = !r3 ? 0.0 : r < 3 ? win_s[3 * r + 2] : below;
                    const double p = fma(m2, w2, fma(m1, w1, m0 * w0));
                    if (r == 0) H[k + (size_t)k * m] = fma(-p, g0, m0);
                    H[k + r + (size_t)(k + 1) * m] = fma(-p, g1, m1);
                    if (r3) H[k + r + (size_t)(k + 2) * m] = fma(-p, g2, m2);
                }
            } else if (far >= 0) {
                const int na = max(0, m - k - 5), total = na + k + m;
                for (int t = far; t < total; t += kFarLanes) {
                    if (t < na) {                      // row part, columns k+5..
                        double *col = H + (size_t)(k + 5 + t) * m + k;
                        const double h0 = col[0], h1 = col[1], h2 = r3 ? col[2] : 0.0;
                        const double q = fma(g2, h2, fma(g1, h1, g0 * h0));
                        col[0] = fma(-q, w0, h0);
                        col[1] = fma(-q, w1, h1);
                        if (r3) col[2] = fma(-q, w2, h2);
                    } else {                           // column part, rows 0..k-1 and the Schur vectors
                        double *row = (t < na + k ? H + (t - na) : Z + (t - na - k)) + (size_t)k * m;
                        const double h0 = row[0], h1 = row[m], h2 = r3 ? row[2 * (size_t)m] : 0.0;
                        const double q = fma(h2, w2, fma(h1, w1, h0 * w0));
                        row[0] = fma(-q, g0, h0);
                        row[m] = fma(-q, g1, h1);
                        if (r3) row[2 * (size_t)m] = fma(-q, g2, h2);
                    }
                }
            }
            __syncthreads();
        }
    }
    return status_s;
}

// ----------------------------------------------------------------------------- complex Schur form
// Wilkinson single-shift QR on the complex upper Hessenberg H, accumulating Z.  The
// negligibility test uses |re| + |im| (no square roots).
__device__ __forceinline__ double cabs1(cplx a) { return fabs(a.re) + fabs(a.im); }

__device__ int complex_schur(cplx *H, int m, cplx *Z) {
    __shared__ int hi_s, l_s, status_s;
    __shared__ int act_s[2];        // by turns, as in real_schur
    __shared__ double rs_s[2][4];   // a.re, a.im, b.re, b.im of the current and the next rotation
    __shared__ cplx win_s[6];
    __shared__ cplx x_s, y_s;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) { hi_s = m - 1; status_s = 0; }
    __syncthreads();
    int its = 0, total = 0;
    for (int turn = 0;; turn ^= 1) {
        if (tid < 32) {
            const int hi = hi_s;
            __syncwarp();          // every lane has read hi_s before lane 0 may update it
            int l = 0;
            if (hi > 0) {
                for (int base = hi; base > 0 && l == 0; base -= 32) {
                    const int cand = base - lane;
                    bool neg = false;
                    if (cand > 0) {
                        double s = cabs1(H[(cand - 1) + (size_t)(cand - 1) * m]) + cabs1(H[cand + (size_t)cand * m]);
                        if (s == 0.0) s = 1.0;
                        neg = cabs1(H[cand + (size_t)(cand - 1) * m]) <= kEps * s;
                    }
                    const unsigned bal = __ballot_sync(kFull, neg);
                    if (bal) l = base - (__ffs(bal) - 1);
                }
            }
            if (lane == 0) {
                if (l > 0) H[l + (size_t)(l - 1) * m] = {0.0, 0.0};
                int act = 0;
                if (hi <= 0) act = -1;
                else {
                    l_s = l;
                    if (l == hi) { hi_s = hi - 1; act = 1; }
                    else act = 2;
                }
                act_s[turn] = act;
            }
        }
        __syncthreads();
        const int act = act_s[turn];
        if (act < 0) break;
        if (act == 1) { its = 0; continue; }
        ++its;
        ++total;
        if (total > 40 * m) {
            if (tid == 0) status_s = 1;
            __syncthreads();
            break;
        }
        const int hi = hi_s, l = l_s;
        if (tid == 0) {
            cplx a = H[(hi - 1) + (size_t)(hi - 1) * m], b = H[(hi - 1) + (size_t)hi * m];
            cplx c = H[hi + (size_t)(hi - 1) * m], d = H[hi + (size_t)hi * m];
            cplx mu;
            if (its % 10 == 0) {
                mu = d + mkc(1.5 * cabs_(c), 0.0);
            } else {
                // eigenvalue of [a b; c d] closer to d
                cplx p = 0.5 * (a - d);
                cplx disc = p * p + b * c;
                // principal square root
                double r = cabs_(disc);
                double sr = sqrt(fmax(0.0, 0.5 * (r + disc.re)));     // hypot may fall short of |disc.re|
                double si = sqrt(fmax(0.0, 0.5 * (r - disc.re)));
                if (disc.im < 0) si = -si;
                cplx sq_ = mkc(sr, si);
                cplx e1 = p + sq_, e2 = p - sq_;
                mu = d + ((abs2(e1) < abs2(e2)) ? e1 : e2);
            }
            x_s = H[l + (size_t)l * m] - mu;
            y_s = H[(l + 1) + (size_t)l * m];
        }
        __syncthreads();
        if (warp == 0) givens_warp(lane == 0 ? x_s.re : lane == 1 ? x_s.im : lane == 2 ? y_s.re : lane == 3 ? y_s.im : 0.0, rs_s[l & 1]);
        __syncthreads();
        const int far = far_index();
        for (int k = l; k <= hi - 1; ++k) {
            const double *rb = rs_s[k & 1];
            const cplx a = mkc(rb[0], rb[1]), b = mkc(rb[2], rb[3]);
            const int part = lane & 1;                 // real or imaginary part of a lane's value
            // (u p + v q) part, four operations
            auto part_of = [&](cplx u, cplx p, cplx v, cplx q) {
                return fma(part ? v.re : -v.im, q.im,
                           fma(part ? v.im : v.re, q.re, fma(part ? u.re : -u.im, p.im, (part ? u.im : u.re) * p.re)));
            };
            if (warp == 0) {
                // lanes 0..3: row k + 1, columns k and k + 1 after the row part; then column k of
                // rows k + 1 (lanes 0, 1) and k + 2 (lanes 2, 3) after the column part
                const cplx *col = H + (size_t)(k + ((lane >> 1) & 1)) * m + k;
                const cplx hu = col[0], hl = col[1];
                const cplx below = k + 2 <= hi ? H[k + 2 + (size_t)(k + 1) * m] : mkc(0.0, 0.0);
                bar_two_warps();
                const double w = part_of(hl, a, hu, -b);
                const cplx r0 = mkc(__shfl_sync(kFull, w, 0), __shfl_sync(kFull, w, 1)),
                           r1 = mkc(__shfl_sync(kFull, w, 2), __shfl_sync(kFull, w, 3));
                const bool second = lane & 2;
                const double xv = part_of(second ? mkc(0.0, 0.0) : r0, a, second ? below : r1, b);
                cplx *ck = H + (size_t)k * m;
                if (k < hi - 1) {
                    const double r = givens_warp(xv, rs_s[(k + 1) & 1]);
                    if (lane == 0) {
                        ck[k + 1] = mkc(r, 0.0);
                        ck[k + 2] = mkc(0.0, 0.0);
                    }
                } else if (lane < 2) {
                    reinterpret_cast<double *>(ck + hi)[lane] = xv;
                }
            } else if (warp == 1) {
                // rows k, k+1 of columns k..k+2, then columns k, k+1 of rows k..k+2 (column k below
                // the diagonal is the chain's): lane 4 c + 2 o + part
                const int c = lane >> 2, o = (lane >> 1) & 1;
                const bool oc = c < 3 && k + c < m;
                const cplx *col = H + (size_t)(oc ? k + c : k) * m + k;
                const cplx hu = col[0], hl = col[1];
                const cplx below = k + 2 <= hi ? H[k + 2 + (size_t)(k + 1) * m] : mkc(0.0, 0.0);
                bar_two_warps();
                const double v = o == 0 ? part_of(hu, conj(a), hl, conj(b)) : part_of(hl, a, hu, -b);
                if (oc && c < 2) reinterpret_cast<double *>(win_s + 2 * o + c)[part] = v;
                else if (oc) reinterpret_cast<double *>(H + (size_t)(k + c) * m + k + o)[part] = v;
                __syncwarp();
                const int r = c;                       // row k + r, output column k + o
                if (r < 3 && k + r <= hi && !(r > 0 && o == 0)) {
                    const cplx m0 = r < 2 ? win_s[2 * r] : mkc(0.0, 0.0), m1 = r < 2 ? win_s[2 * r + 1] : below;
                    const double u = o == 0 ? part_of(m0, a, m1, b) : part_of(m1, conj(a), m0, -conj(b));
                    reinterpret_cast<double *>(H + (size_t)(k + o) * m + k + r)[part] = u;
                }
            } else if (far >= 0) {
                const int na = max(0, m - k - 3), total = na + k + m;
                for (int t = far; t < total; t += kFarLanes) {
                    if (t < na) {                      // row part (H <- G H), columns k+3..
                        cplx *col = H + (size_t)(k + 3 + t) * m + k;
                        const cplx h1 = col[0], h2 = col[1];
                        col[0] = conj(a) * h1 + conj(b) * h2;
                        col[1] = a * h2 - b * h1;
                    } else {                           // column part (M <- M G^H), rows 0..k-1 and Schur vectors
                        cplx *row = (t < na + k ? H + (t - na) : Z + (t - na - k)) + (size_t)k * m;
                        const cplx h1 = row[0], h2 = row[m];
                        row[0] = h1 * a + h2 * b;
                        row[m] = h2 * conj(a) - h1 * conj(b);
                    }
                }
            }
            __syncthreads();
        }
    }
    return status_s;
}

// ----------------------------------------------------------------------------- eigenvalues
// From the real Schur form T: eigenvalue j as (re, im).  2 x 2 blocks are the complex pairs.
__device__ void real_schur_eigs(const double *T, int m, double *wr, double *wi) {
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
        const bool lower = (j + 1 < m) && T[(j + 1) + (size_t)j * m] != 0.0;   // j is top of a block
        const bool upper = (j > 0) && T[j + (size_t)(j - 1) * m] != 0.0;       // j is bottom of a block
        if (lower || upper) {
            const int t = lower ? j : j - 1;
            double a = T[t + (size_t)t * m], b = T[t + (size_t)(t + 1) * m];
            double c = T[(t + 1) + (size_t)t * m], d = T[(t + 1) + (size_t)(t + 1) * m];
            double p = 0.5 * (a - d);
            double disc = p * p + b * c;
            double im = sqrt(fmax(-disc, 0.0));
            wr[j] = 0.5 * (a + d);
            wi[j] = lower ? im : -im;
        } else {
            wr[j] = T[j + (size_t)j * m];
            wi[j] = 0.0;
        }
    }
    __syncthreads();
}

// a / b by one reciprocal in the middle of the range
__device__ __forceinline__ cplx cdiv_fast(cplx a, cplx b) {
    const double d = abs2(b);
    if (!mid_range(d)) return cdiv(a, b);
    const cplx n = a * conj(b);
    return rcp_fast(d) * n;
}
// |z| < small
__device__ __forceinline__ bool below(cplx z, double small) {
    const double a = abs2(z), b = small * small;
    return mid_range(a) && mid_range(b) ? a < b : cabs_(z) < small;
}
constexpr int kVecLanes = 8;       // lanes that share an eigenvector's back substitution
__device__ __forceinline__ cplx group_sum(cplx s, unsigned gm) {
#pragma unroll
    for (int o = 1; o < kVecLanes; o <<= 1)
        s = {s.re + __shfl_xor_sync(gm, s.re, o), s.im + __shfl_xor_sync(gm, s.im, o)};
    return s;
}

// Back substitution for the eigenvector of eigenvalue (lr, li) at Schur position j of the
// real quasi-triangular T.  Output y (complex, length m, zero below j).
// Eight lanes (mask gm, `part` the lane among them) share a vector: a row's sum is the long serial
// part, the vectors of a warp take different branches, and a thread per vector kept to one warp
// (with the products and residuals 319 us at m = 60, k = 20; now 141).
__device__ void real_schur_vector(const double *T, int m, int j, double lr, double li, cplx *y,
                                  double tnorm, int part, unsigned gm) {
    const double small = fmax(kEps * tnorm, 1e-300);
    const cplx lam = mkc(lr, li);
    for (int i = part; i < m; i += kVecLanes) y[i] = {0.0, 0.0};
    __syncwarp(gm);
    int top;
    if (li == 0.0) {
        if (part == 0) y[j] = {1.0, 0.0};
        top = j - 1;
    } else {
        // 2x2 block at (t, t+1) containing j
        const bool jtop = (j + 1 < m) && T[(j + 1) + (size_t)j * m] != 0.0;
        const int t = jtop ? j : j - 1;
        double a = T[t + (size_t)t * m], b = T[t + (size_t)(t + 1) * m];
        double c = T[(t + 1) + (size_t)t * m], d = T[(t + 1) + (size_t)(t + 1) * m];
        cplx yt = {1.0, 0.0}, yb = {1.0, 0.0};
        if (fabs(b) >= fabs(c)) yb = cdiv(lam - mkc(a, 0.0), mkc(b, 0.0));      // (a - lam) y0 + b y1 = 0
        else yt = cdiv(lam - mkc(d, 0.0), mkc(c, 0.0));                         // c y0 + (d - lam) y1 = 0
        if (part == 0) { y[t] = yt; y[t + 1] = yb; }
        top = t - 1;
        j = t + 1;
    }
    __syncwarp(gm);
    int i = top;
    while (i >= 0) {
        const bool blk = (i > 0) && T[i + (size_t)(i - 1) * m] != 0.0;   // rows (i-1, i) form a block
        if (!blk) {
            cplx s = {0.0, 0.0};
            for (int l = i + 1 + part; l <= j; l += kVecLanes) {
                const double t = T[i + (size_t)l * m];
                s = {fma(t, y[l].re, s.re), fma(t, y[l].im, s.im)};
            }
            s = group_sum(s, gm);
            cplx den = mkc(T[i + (size_t)i * m], 0.0) - lam;
            if (below(den, small)) den = mkc(small, 0.0);
            const cplx v = cdiv_fast(-s, den);
            if (part == 0) y[i] = v;
            i -= 1;
        } else {
            const int t = i - 1;
            cplx s0 = {0.0, 0.0}, s1 = {0.0, 0.0};
            for (int l = i + 1 + part; l <= j; l += kVecLanes) {
                const double t0 = T[t + (size_t)l * m], t1 = T[i + (size_t)l * m];
                s0 = {fma(t0, y[l].re, s0.re), fma(t0, y[l].im, s0.im)};
                s1 = {fma(t1, y[l].re, s1.re), fma(t1, y[l].im, s1.im)};
            }
            s0 = group_sum(s0, gm);
            s1 = group_sum(s1, gm);
            // [a-lam b; c d-lam] [y_t; y_i] = -[s0; s1]
            cplx a = mkc(T[t + (size_t)t * m], 0.0) - lam, b = mkc(T[t + (size_t)i * m], 0.0);
            cplx c = mkc(T[i + (size_t)t * m], 0.0), d = mkc(T[i + (size_t)i * m], 0.0) - lam;
            cplx det = a * d - b * c;
            if (cabs_(det) < small * small) det = mkc(small * small, 0.0);
            const cplx yt = cdiv_fast(-(d * s0) + b * s1, det), yi = cdiv_fast(c * s0 - a * s1, det);
            if (part == 0) { y[t] = yt; y[i] = yi; }
            i -= 2;
        }
        __syncwarp(gm);
    }
}

__device__ void complex_schur_vector(const cplx *T, int m, int j, cplx *y, double tnorm, int part, unsigned gm) {
    const double small = fmax(kEps * tnorm, 1e-300);
    const cplx lam = T[j + (size_t)j * m];
    for (int i = part; i < m; i += kVecLanes) y[i] = {i == j ? 1.0 : 0.0, 0.0};
    __syncwarp(gm);
    for (int i = j - 1; i >= 0; --i) {
        cplx s = {0.0, 0.0};
        for (int l = i + 1 + part; l <= j; l += kVecLanes) s = Cx<cplx>::mac(s, T[i + (size_t)l * m], y[l]);
        s = group_sum(s, gm);
        cplx den = T[i + (size_t)i * m] - lam;
        if (below(den, small)) den = mkc(small, 0.0);
        const cplx v = cdiv_fast(-s, den);
        if (part == 0) y[i] = v;
        __syncwarp(gm);
    }
}

// order: by |theta|, then Re, then Im >= 0 first (one thread, insertion sort; moduli given)
__device__ bool ritz_less_m(double ma, double ar, double ai, double mb, double br, double bi) {
    if (ma != mb) return ma < mb;
    if (ar != br) return ar < br;
    int ka = ai >= 0 ? 0 : 1, kb = bi >= 0 ? 0 : 1;
    return ka < kb;
}

}  // namespace

// ============================================================================= kernels

// Cholesky G = R^H R (G Hermitian positive definite, upper triangle given, k x k) and
// Rinv = R^{-1}.  info[0] = 0 on success, j+1 if the j-th pivot is not positive.
template <class D>
__global__ void k_chol_inv(const D *G, int k, D *R, D *Rinv, int *info) {
    pdl_wait();
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
        int i = e % k, j = e / k;
        R[e] = i <= j ? G[e] : Cx<D>::zero();
        Rinv[e] = Cx<D>::zero();
    }
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        if (threadIdx.x == 0) {
            double djj = Cx<D>::re(R[j + (size_t)j * k]);
            for (int i = 0; i < j; ++i) djj -= Cx<D>::ab2(R[i + (size_t)j * k]);
            if (!(djj > 0.0) && !bad) bad = j + 1;
            R[j + (size_t)j * k] = Cx<D>::sc(sqrt(fmax(djj, 1e-300)), Cx<D>::one());
        }
        __syncthreads();
        const D rjj = R[j + (size_t)j * k];
        for (int c = j + 1 + threadIdx.x; c < k; c += blockDim.x) {
            D s = R[j + (size_t)c * k];
            for (int i = 0; i < j; ++i) s = subt(s, Cx<D>::mul(Cx<D>::cj(R[i + (size_t)j * k]), R[i + (size_t)c * k]));
            R[j + (size_t)c * k] = Cx<D>::div(s, rjj);
        }
        __syncthreads();
    }
    // Rinv: solve R X = I column by column (thread per column)
    for (int c = threadIdx.x; c < k; c += blockDim.x) {
        for (int i = c; i >= 0; --i) {
            D s = (i == c) ? Cx<D>::one() : Cx<D>::zero();
            for (int l = i + 1; l <= c; ++l) s = subt(s, Cx<D>::mul(R[i + (size_t)l * k], Rinv[l + (size_t)c * k]));
            Rinv[i + (size_t)c * k] = Cx<D>::div(s, R[i + (size_t)i * k]);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) info[0] = bad;
}

// Inverse of a general k x k matrix by Gauss-Jordan with partial pivoting (W: scratch
// 2 k^2).  info[0] = 0, or j+1 for a zero pivot.
template <class D>
__global__ void k_inverse(const D *H, int k, D *Hinv, D *W, int *info) {
    pdl_wait();
    __shared__ int p_s, bad;
    D *A = W;
    D *B = W + (size_t)k * k;
    if (threadIdx.x == 0) bad = 0;
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
        A[e] = H[e];
        B[e] = (e % k == e / k) ? Cx<D>::one() : Cx<D>::zero();
    }
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        if (threadIdx.x == 0) {
            int p = j;
            double best = Cx<D>::ab2(A[j + (size_t)j * k]);
            for (int i = j + 1; i < k; ++i)
                if (Cx<D>::ab2(A[i + (size_t)j * k]) > best) { best = Cx<D>::ab2(A[i + (size_t)j * k]); p = i; }
            if (best == 0.0 && !bad) bad = j + 1;
            p_s = p;
        }
        __syncthreads();
        const int p = p_s;
        if (p != j) {
            for (int c = threadIdx.x; c < k; c += blockDim.x) {
                D t = A[j + (size_t)c * k]; A[j + (size_t)c * k] = A[p + (size_t)c * k]; A[p + (size_t)c * k] = t;
                t = B[j + (size_t)c * k]; B[j + (size_t)c * k] = B[p + (size_t)c * k]; B[p + (size_t)c * k] = t;
            }
        }
        __syncthreads();
        const D piv = A[j + (size_t)j * k];
        if (Cx<D>::ab2(piv) == 0.0) { __syncthreads(); continue; }
        // scale row j
        for (int c = threadIdx.x; c < k; c += blockDim.x) {
            A[j + (size_t)c * k] = Cx<D>::div(A[j + (size_t)c * k], piv);
            B[j + (size_t)c * k] = Cx<D>::div(B[j + (size_t)c * k], piv);
        }
        __syncthreads();
        // eliminate column j from the other rows (thread per row)
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
            if (i == j) continue;
            D f = A[i + (size_t)j * k];
            for (int c = 0; c < k; ++c) {
                A[i + (size_t)c * k] = subt(A[i + (size_t)c * k], Cx<D>::mul(f, A[j + (size_t)c * k]));
                B[i + (size_t)c * k] = subt(B[i + (size_t)c * k], Cx<D>::mul(f, B[j + (size_t)c * k]));
            }
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) Hinv[e] = B[e];
    if (threadIdx.x == 0) info[0] = bad;
}

// out = M c (k x k times k), one thread per row.
template <class D>
__global__ void k_small_gemv(const D *M, int k, const D *c, D *out) {
    pdl_wait();
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        D s = Cx<D>::zero();
        for (int j = 0; j < k; ++j) s = add(s, Cx<D>::mul(M[i + (size_t)j * k], c[j]));
        out[i] = s;
    }
}

// ----------------------------------------------------------------------------- GMRES-DR restart
// See tg_small.cuh for the argument layout.
// elements of T before the eigenvector work in shared memory: W and Z, rounded up to an even count
// (the work is complex, 16-byte aligned, and m^2 is odd for odd m)
__host__ __device__ constexpr size_t gdr_y_offset(int m) {
    return ((size_t)(m + 1) * m + (size_t)m * m + 1) & ~(size_t)1;
}

template <class T>
__device__ __forceinline__ void gmresdr_restart_body(const GdrArgs<T> &a) {
    const int m = a.m;
    const int rows = m + 1;
    const int ldh = a.ldh;
    // W: (m+1) x m (least-squares copy), later the m x m eigen matrix / Schur form;
    // Z: m x m Schur vectors, later the basis P.  Both live in shared memory when the launch provided it
    // (the QR sweeps are a long chain of dependent small steps, so their latency rules).
    extern __shared__ __align__(16) unsigned char gdr_smem[];
    T *sm = reinterpret_cast<T *>(gdr_smem);
    T *W = a.smem >= 1 ? sm : a.work;
    T *Z = a.smem >= 2 ? sm + (size_t)rows * m : a.work + (size_t)rows * m;
    T *vtmp = a.work + (size_t)rows * m + (size_t)m * m;       // 2 (m+1) vectors
    T *f = vtmp + 2 * (m + 1);
    cplx *Ysm = a.smem >= 3 ? reinterpret_cast<cplx *>(sm + gdr_y_offset(m)) : a.ywork;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    T *res = a.res;
    // vectors of the least-squares solve, the Hessenberg reduction, the ordering and Gram-Schmidt in
    // turn: with kGdrSmemMax the static shared memory must stay below 17 KB
    __shared__ T vec_s[3 * (kMaxM + 1)];
    __shared__ double gs_s[kMaxM];

    long long t_mark = clock64();
    const bool rr_mode = a.mode == 1;
    if (rr_mode) {
        // Rayleigh-Ritz: the eigen matrix is H itself
        for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
            const int i = e % m, j = e / m;
            W[e] = a.H[i + (size_t)j * ldh];
            Z[e] = (i == j) ? Cx<T>::one() : Cx<T>::zero();
        }
        if (threadIdx.x == 0) a.info->rnorm = 0.0;
        __syncthreads();
    } else {
    // ---- 1. least squares: d = argmin ||c - Hbar d||, res = c - Hbar d
    for (int e = threadIdx.x; e < rows * m; e += blockDim.x) {
        int i = e % rows, j = e / rows;
        W[i + (size_t)j * rows] = a.H[i + (size_t)j * ldh];
    }
    for (int i = threadIdx.x; i < rows; i += blockDim.x) vtmp[m + 1 + i] = a.c[i];
    __syncthreads();
    lsq_solve<T>(W, rows, rows, m, vtmp + (m + 1), a.d, f, vec_s, vec_s + (kMaxM + 1), vec_s + 2 * (kMaxM + 1), gs_s);
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        T s = a.c[i];
        for (int j = 0; j < m; ++j) s = Cx<T>::nmac(s, a.H[i + (size_t)j * ldh], a.d[j]);
        res[i] = s;
    }
    __syncthreads();
    if (warp == 0) {
        double s = 0.0;
        for (int i = lane; i < rows; i += 32) s += Cx<T>::ab2(res[i]);
        s = warp_sum(s);
        if (lane == 0) a.info->rnorm = sqrt(s);
    }

    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[0] = _t - t_mark; t_mark = _t; }
    // ---- 2. the harmonic matrix M = H_m + |h|^2 f e_m^T (in W, ld m), f = H_m^{-H} e_m
    const T hm = a.H[m + (size_t)(m - 1) * ldh];
    const double hm2 = Cx<T>::ab2(hm);
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        int i = e % m, j = e / m;
        T v = a.H[i + (size_t)j * ldh];
        if (j == m - 1) v = add(v, Cx<T>::sc(hm2, f[i]));
        W[e] = v;
        Z[e] = (i == j) ? Cx<T>::one() : Cx<T>::zero();
    }
    __syncthreads();
    // z = [-|h|^2 f; h] (restart direction), kept in a.z
    for (int i = threadIdx.x; i < rows; i += blockDim.x) a.z[i] = (i < m) ? Cx<T>::sc(-hm2, f[i]) : hm;

    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[1] = _t - t_mark; t_mark = _t; }
    }   // steps 1-2: GMRES-DR restart only
    // ---- 3. eigen-decomposition of M: Hessenberg, Schur, eigenvalues
    hessenberg<T>(W, m, Z, vec_s);
    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[2] = _t - t_mark; t_mark = _t; }
    int st;
    double *wr = a.wr, *wi = a.wi;
    if constexpr (sizeof(T) == sizeof(double)) {
        st = real_schur(reinterpret_cast<double *>(W), m, reinterpret_cast<double *>(Z));
        real_schur_eigs(reinterpret_cast<double *>(W), m, wr, wi);
    } else {
        st = complex_schur(reinterpret_cast<cplx *>(W), m, reinterpret_cast<cplx *>(Z));
        for (int j = threadIdx.x; j < m; j += blockDim.x) {
            cplx t = reinterpret_cast<cplx *>(W)[j + (size_t)j * m];
            wr[j] = t.re;
            wi[j] = t.im;
        }
        __syncthreads();
    }
    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[3] = _t - t_mark; t_mark = _t; }
    double tnorm = 0.0;
    {
        __shared__ double tn_s[32];
        double s2 = 0.0;
        for (int e = threadIdx.x; e < m * m; e += blockDim.x) s2 = fmax(s2, Cx<T>::ab2(W[e]));
        for (int o = 16; o > 0; o >>= 1) s2 = fmax(s2, __shfl_down_sync(0xffffffffu, s2, o));
        if (lane == 0) tn_s[warp] = s2;
        __syncthreads();
        if (threadIdx.x == 0) {
            double mx = 0.0;
            for (int w = 0; w < nwarps; ++w) mx = fmax(mx, tn_s[w]);
            tn_s[0] = sqrt(mx);
        }
        __syncthreads();
        tnorm = tn_s[0];
    }

    // ---- 4. order and select
    __shared__ int kk_s;
    int *ord = a.order;
    double *mod_s = reinterpret_cast<double *>(vec_s), *wr_s = mod_s + kMaxM, *wi_s = wr_s + kMaxM;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        mod_s[i] = hypot(wr[i], wi[i]);
        wr_s[i] = wr[i];
        wi_s[i] = wi[i];
    }
    __syncthreads();
    // stable rank sort, one thread per value: the rank of i is the number of values before it
    // in the order plus the equal values of smaller index (the order a stable sort gives)
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        int r = 0;
        for (int j = 0; j < m; ++j) {
            if (j == i) continue;
            const bool jl = ritz_less_m(mod_s[j], wr_s[j], wi_s[j], mod_s[i], wr_s[i], wi_s[i]);
            const bool il = ritz_less_m(mod_s[i], wr_s[i], wi_s[i], mod_s[j], wr_s[j], wi_s[j]);
            if (jl || (j < i && !il)) ++r;
        }
        ord[r] = i;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int kk = a.k;
        if (sizeof(T) == sizeof(double) && kk < m) {
            int t = ord[kk - 1];
            if (wi[t] > 0.0) kk += 1;     // keep both members of the conjugate pair
        }
        kk_s = kk;
        a.info->status = st;
    }
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        a.theta[2 * i] = wr_s[ord[i]];
        a.theta[2 * i + 1] = wi_s[ord[i]];
    }
    __syncthreads();
    const int kk = kk_s;

    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[4] = _t - t_mark; t_mark = _t; }
    // ---- 5. eigenvectors of the kept pairs: g = Z y (complex), unit norm; residuals
    // a.gwork holds the kept eigenvectors as complex columns (m x kk)
    cplx *G = a.gwork;
    cplx *Y = Ysm;
    for (int q = threadIdx.x / kVecLanes; q < kk; q += blockDim.x / kVecLanes) {
        const int j = ord[q], part = lane % kVecLanes;
        const unsigned gm = ((1u << kVecLanes) - 1u) << (lane - part);
        cplx *y = Y + (size_t)q * m;
        if constexpr (sizeof(T) == sizeof(double))
            real_schur_vector(reinterpret_cast<const double *>(W), m, j, wr[j], wi[j], y, tnorm, part, gm);
        else
            complex_schur_vector(reinterpret_cast<const cplx *>(W), m, j, y, tnorm, part, gm);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < m * kk; e += blockDim.x) {
        const int i = e % m, q = e / m;
        const cplx *y = Y + (size_t)q * m;
        cplx s = {0.0, 0.0};
        if constexpr (sizeof(T) == sizeof(double)) {
            // real Schur vectors: two real products per term
            const double *Zd = reinterpret_cast<const double *>(Z);
            for (int l = 0; l < m; ++l) {
                const double zl = Zd[i + (size_t)l * m];
                s.re = fma(zl, y[l].re, s.re);
                s.im = fma(zl, y[l].im, s.im);
            }
        } else {
            for (int l = 0; l < m; ++l) s = Cx<cplx>::mac(s, *reinterpret_cast<const cplx *>(&Z[i + (size_t)l * m]), y[l]);
        }
        G[i + (size_t)q * m] = s;
    }
    __syncthreads();
    __shared__ double znorm_s;
    if (warp == 0 && !rr_mode) {
        double z2 = 0.0;
        for (int i = lane; i < rows; i += 32) z2 += Cx<T>::ab2(a.z[i]);
        z2 = warp_sum(z2);
        if (lane == 0) znorm_s = sqrt(z2);
    }
    __syncthreads();
    const double znorm = rr_mode ? 0.0 : znorm_s;
    for (int q = warp; q < kk; q += nwarps) {
        cplx *g = G + (size_t)q * m;
        double nr = 0.0;
        for (int i = lane; i < m; i += 32) nr += abs2(g[i]);
        nr = sqrt(warp_sum(nr));
        nr = __shfl_sync(0xffffffffu, nr, 0);
        for (int i = lane; i < m; i += 32) g[i] = g[i] * (1.0 / nr);
        __syncwarp();
        // residual ||Hbar g - theta [g; 0]|| = |g_m| ||z||: an eigenpair of
        // H_m + |h|^2 f e_m^T satisfies H_m g - theta g = -|h|^2 f g_m, and the last row of
        // Hbar g is h g_m, so the residual vector is g_m z with z = [-|h|^2 f; h]
        if (!rr_mode) {
            if (lane == 0) a.eres[q] = sqrt(abs2(g[m - 1])) * znorm;
        } else {
            // Rayleigh-Ritz: ||W g - theta Q g||^2 = g^H (W^H W) g - |theta|^2 for Q^H W g = theta g
            double acc = 0.0;
            for (int i = lane; i < m; i += 32) {
                cplx wg = {0.0, 0.0};
                for (int l = 0; l < m; ++l) {
                    const T w = a.WW[i + (size_t)l * m];
                    cplx wc;
                    if constexpr (sizeof(T) == sizeof(double)) wc = mkc(*reinterpret_cast<const double *>(&w), 0.0);
                    else wc = *reinterpret_cast<const cplx *>(&w);
                    wg = wg + wc * g[l];
                }
                acc += (conj(g[i]) * wg).re;
            }
            acc = warp_sum(acc);
            if (lane == 0) {
                const int j = ord[q];
                a.eres[q] = sqrt(fmax(acc - (wr[j] * wr[j] + wi[j] * wi[j]), 0.0));
            }
        }
    }
    __syncthreads();
    if (rr_mode && warp == 0 && a.start_q < kk) {
        // coefficients of the start vector: Ritz vector start_q with its largest entry made
        // real and positive (ties: the smallest index); real problems keep the real part
        const cplx *g = G + (size_t)a.start_q * m;
        double best = -1.0;
        int imax = 0;
        for (int i = lane; i < m; i += 32)
            if (abs2(g[i]) > best) { best = abs2(g[i]); imax = i; }
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_down_sync(0xffffffffu, best, o);
            const int oi = __shfl_down_sync(0xffffffffu, imax, o);
            if (ob > best || (ob == best && oi < imax)) { best = ob; imax = oi; }
        }
        imax = __shfl_sync(0xffffffffu, imax, 0);
        best = __shfl_sync(0xffffffffu, best, 0);
        const cplx ph = conj(g[imax]) * (1.0 / sqrt(best));
        for (int i = lane; i < m; i += 32) {
            const cplx v = g[i] * ph;
            if constexpr (sizeof(T) == sizeof(double)) reinterpret_cast<double *>(a.z)[i] = v.re;
            else reinterpret_cast<cplx *>(a.z)[i] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int nconv = 0;
        for (int q = 0; q < a.nev && q < kk; ++q)
            if (a.eres[q] <= a.rtolev * hypot(a.theta[2 * q], a.theta[2 * q + 1])) ++nconv;
        a.info->nconv = nconv;
        a.info->kk = kk;
    }

    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[5] = _t - t_mark; t_mark = _t; }
    // ---- 6. P_k: orthonormal basis of the kept span (real: Re/Im of pairs), m x kk
    //          then P_{k+1} = orth([[P_k; 0], z]), stored (m+1) x (kk+1) with ld m+1.
    __shared__ int ncol_s;
    int *colof_s = reinterpret_cast<int *>(gs_s);
    if (threadIdx.x == 0) {
        int col = 0;
        for (int q = 0; q < kk; ++q) {
            const double im = a.theta[2 * q + 1];
            if (sizeof(T) == sizeof(double)) {
                if (im == 0.0) { colof_s[q] = col; col += 1; }
                else if (im > 0.0) { colof_s[q] = col; col += 2; }
                else colof_s[q] = -1;      // the partner (Im > 0) supplies both columns
            } else {
                colof_s[q] = col++;
            }
        }
        ncol_s = col;
    }
    __syncthreads();
    // built in the Schur vectors' place (they are not read any more) where it fits
    T *P = rows * (ncol_s + 1) <= m * m ? Z : a.P;
    for (int q = warp; q < kk; q += nwarps) {
        const int c0 = colof_s[q];
        if (c0 < 0) continue;
        const cplx *g = G + (size_t)q * m;
        const double im = a.theta[2 * q + 1];
        if constexpr (sizeof(T) == sizeof(double)) {
            double *Pd = reinterpret_cast<double *>(P);
            if (im == 0.0) {
                // a real eigenvector computed in complex arithmetic carries a common phase:
                // rotate it onto the real axis through its largest entry (ties: smallest index)
                double best = -1.0;
                int imax = 0;
                for (int i = lane; i < m; i += 32)
                    if (abs2(g[i]) > best) { best = abs2(g[i]); imax = i; }
                for (int o = 16; o > 0; o >>= 1) {
                    double ob = __shfl_down_sync(0xffffffffu, best, o);
                    int oi = __shfl_down_sync(0xffffffffu, imax, o);
                    if (ob > best || (ob == best && oi < imax)) { best = ob; imax = oi; }
                }
                imax = __shfl_sync(0xffffffffu, imax, 0);
                best = __shfl_sync(0xffffffffu, best, 0);
                const cplx ph = conj(g[imax]) * (1.0 / sqrt(best));
                for (int i = lane; i < m; i += 32) Pd[i + (size_t)c0 * rows] = (g[i] * ph).re;
                if (lane == 0) Pd[m + (size_t)c0 * rows] = 0.0;
            } else {
                for (int i = lane; i < m; i += 32) {
                    Pd[i + (size_t)c0 * rows] = g[i].re;
                    Pd[i + (size_t)(c0 + 1) * rows] = g[i].im;
                }
                if (lane == 0) {
                    Pd[m + (size_t)c0 * rows] = 0.0;
                    Pd[m + (size_t)(c0 + 1) * rows] = 0.0;
                }
            }
        } else {
            cplx *Pc = reinterpret_cast<cplx *>(P);
            for (int i = lane; i < m; i += 32) Pc[i + (size_t)c0 * rows] = g[i];
            if (lane == 0) Pc[m + (size_t)c0 * rows] = {0.0, 0.0};
        }
    }
    __syncthreads();
    const int nc = ncol_s;     // == kk
    // append z as column kk (GMRES-DR restart only)
    if (!rr_mode)
        for (int i = threadIdx.x; i < rows; i += blockDim.x) P[i + (size_t)nc * rows] = a.z[i];
    __syncthreads();
    // classical Gram-Schmidt applied twice over the nc + 1 columns (length m+1): per column, the
    // projections on the previous columns, then the update, G lanes to a sum (a thread to a sum in
    // global memory took 160 us at m = 60, k = 20, now 90; complex m = 80 1.85 -> 0.57 ms)
    T *proj_s = vec_s;
    __shared__ double inv_s;
    const int clast = rr_mode ? nc - 1 : nc;
    for (int c = 0; c <= clast; ++c) {
        T *pc = P + (size_t)c * rows;
        for (int pass = 0; pass < 2 && c > 0; ++pass) {
            constexpr int G = 8, per = 32 / G;
            const int part = lane / per, it = lane % per;
            for (int b = warp * per; b < c; b += nwarps * per) {
                const T *pq = P + (size_t)min(b + it, c - 1) * rows;
                T s = Cx<T>::zero();
                for (int i = part; i < rows; i += G) s = Cx<T>::macc(s, pq[i], pc[i]);
#pragma unroll
                for (int o = per; o < 32; o <<= 1) s = add(s, shfl_xor(s, o));
                if (part == 0 && b + it < c) proj_s[b + it] = s;
            }
            __syncthreads();
            constexpr int G2 = 4, per2 = 32 / G2;
            const int part2 = lane / per2, it2 = lane % per2;
            for (int b = warp * per2; b < rows; b += nwarps * per2) {
                const int i = min(b + it2, rows - 1);
                T s = Cx<T>::zero();
                for (int q = part2; q < c; q += G2) s = Cx<T>::mac(s, proj_s[q], P[i + (size_t)q * rows]);
#pragma unroll
                for (int o = per2; o < 32; o <<= 1) s = add(s, shfl_xor(s, o));
                if (part2 == 0 && b + it2 < rows) pc[i] = subt(pc[i], s);
            }
            __syncthreads();
        }
        if (warp == 0) {
            double sq2 = 0.0;
            for (int i = lane; i < rows; i += 32) sq2 += Cx<T>::ab2(pc[i]);
            sq2 = warp_sum(sq2);
            if (lane == 0) inv_s = sq2 > 0.0 ? rsqrt(sq2) : 0.0;
        }
        __syncthreads();
        const double inv = inv_s;
        for (int i = threadIdx.x; i < rows; i += blockDim.x) pc[i] = Cx<T>::sc(inv, pc[i]);
        __syncthreads();
    }
    if (P != a.P)
        for (int e = threadIdx.x; e < rows * (clast + 1); e += blockDim.x) a.P[e] = P[e];

    __syncthreads();
    if (threadIdx.x == 0) { long long _t = clock64(); a.info->phase[6] = _t - t_mark; t_mark = _t; }
    if (rr_mode) return;
    // ---- 7. Hnew = P_{k+1}^H Hbar P_k  ((kk+1) x kk, ld m+1 into a.Hnew), cnew = P_{k+1}^H res
    // T1 = Hbar P_k ((m+1) x kk) into W
    for (int e = threadIdx.x; e < rows * nc; e += blockDim.x) {
        const int i = e % rows, q = e / rows;
        T s = Cx<T>::zero();
        for (int j = 0; j < m; ++j) s = Cx<T>::mac(s, a.H[i + (size_t)j * ldh], P[j + (size_t)q * rows]);
        W[i + (size_t)q * rows] = s;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < (nc + 1) * nc; e += blockDim.x) {
        const int i = e % (nc + 1), q = e / (nc + 1);
        T s = Cx<T>::zero();
        for (int l = 0; l < rows; ++l) s = Cx<T>::macc(s, P[l + (size_t)i * rows], W[l + (size_t)q * rows]);
        a.Hnew[i + (size_t)q * ldh] = s;
    }
    for (int i = threadIdx.x; i <= nc; i += blockDim.x) {
        T s = Cx<T>::zero();
        for (int l = 0; l < rows; ++l) s = Cx<T>::macc(s, P[l + (size_t)i * rows], res[l]);
        a.cnew[i] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) a.info->phase[7] = clock64() - t_mark;
}

template <class T>
__global__ void __launch_bounds__(kGdrThreads, 1) k_gmresdr_restart(GdrArgs<T> a) {
    pdl_wait();
    gmresdr_restart_body<T>(a);
}

// many independent restart steps, one block each (the batched coarse phase): block b runs
// args[b] when active[b] is set
template <class T>
__global__ void __launch_bounds__(kGdrThreads, 1) k_gmresdr_restart_batch(const GdrArgs<T> *args, const int *active) {
    pdl_wait();
    if (!active[blockIdx.x]) return;
    const GdrArgs<T> a = args[blockIdx.x];
    gmresdr_restart_body<T>(a);
}

// ----------------------------------------------------------------------------- GMRES(m) Givens step
// Column j of the Arnoldi Hessenberg Hbar (rows 0..j+1, ld = m+1) is copied to H and rotated by
// the previous rotations, a new rotation zeroes h[j+1]; g (the least-squares right-hand side) is
// updated; state->resid = |g[j+1]|; state->done = 1 when resid <= target or h[j,j] = 0.
// One warp: the column and the rotations come in together and lane 0 carries the running entry in
// a register through the rotations (one thread on global memory waited for L2 at every entry:
// 11.3 -> 10.3 us a launch between events, columns of 1 to 20 entries).
template <class D>
__global__ void __launch_bounds__(32) k_givens_step(const D *__restrict__ Hbar, D *H, int ldh, int j, D *cs, D *sn, D *g,
                                                    GivensState *state) {
    pdl_wait();
    if (state->done) return;
    __shared__ D h_s[kMaxM + 1], cs_s[kMaxM], sn_s[kMaxM];
    const int lane = threadIdx.x;
    for (int i = lane; i <= j + 1; i += 32) {
        h_s[i] = Hbar[i + (size_t)j * ldh];
        if (i < j) { cs_s[i] = cs[i]; sn_s[i] = sn[i]; }
    }
    const D gj = g[j];
    const double target = state->target;
    __syncwarp();
    if (lane == 0) {
        D a = h_s[0];
        for (int i = 0; i < j; ++i) {
            const D b = h_s[i + 1];
            h_s[i] = add(Cx<D>::mul(Cx<D>::cj(cs_s[i]), a), Cx<D>::mul(Cx<D>::cj(sn_s[i]), b));
            a = subt(Cx<D>::mul(cs_s[i], b), Cx<D>::mul(sn_s[i], a));
        }
        const D b = h_s[j + 1];
        const double den = sqrt(Cx<D>::ab2(a) + Cx<D>::ab2(b));
        D c = Cx<D>::one(), r = Cx<D>::zero();
        if (den != 0.0) {
            const double inv = 1.0 / den;
            c = Cx<D>::sc(inv, a);
            r = Cx<D>::sc(inv, b);
        }
        cs[j] = c;
        sn[j] = r;
        h_s[j] = Cx<D>::sc(den, Cx<D>::one());
        h_s[j + 1] = Cx<D>::zero();
        const D gn = Cx<D>::sc(-1.0, Cx<D>::mul(r, gj));
        g[j + 1] = gn;
        g[j] = Cx<D>::mul(Cx<D>::cj(c), gj);
        const double resid = sqrt(Cx<D>::ab2(gn));
        state->resid = resid;
        state->steps = j + 1;
        if (!(resid > target) || den == 0.0 || !isfinite(resid)) state->done = 1;
    }
    __syncwarp();
    for (int i = lane; i <= j + 1; i += 32) H[i + (size_t)j * ldh] = h_s[i];
}

// y = R^{-1} g[0..kj-1] for the rotated (upper triangular) Hessenberg.
template <class D>
__global__ void k_givens_solve(const D *H, int ldh, const D *g, D *y, const GivensState *state) {
    pdl_wait();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int kj = state->steps;
    for (int i = kj - 1; i >= 0; --i) {
        D s = g[i];
        for (int c = i + 1; c < kj; ++c) s = subt(s, Cx<D>::mul(H[i + (size_t)c * ldh], y[c]));
        D hii = H[i + (size_t)i * ldh];
        y[i] = Cx<D>::ab2(hii) > 0 ? Cx<D>::div(s, hii) : Cx<D>::zero();
    }
}

// ----------------------------------------------------------------------------- launchers
template <class D>
void launch_chol_inv(const D *G, int k, D *R, D *Rinv, int *info, cudaStream_t s) {
    launch(k_chol_inv<D>, 1, kSmallThreads, 0, s, G, k, R, Rinv, info);
}
template <class D>
void launch_inverse(const D *H, int k, D *Hinv, D *W, int *info, cudaStream_t s) {
    launch(k_inverse<D>, 1, kSmallThreads, 0, s, H, k, Hinv, W, info);
}
template <class D>
void launch_small_gemv(const D *M, int k, const D *c, D *out, cudaStream_t s) {
    launch(k_small_gemv<D>, 1, kSmallThreads, 0, s, M, k, c, out);
}
// W, Z (T) and the eigenvector work Y (complex, m x m) go to shared memory in that order while
// they fit
template <class T>
size_t gmresdr_restart_smem(int m, int *parts) {
    const size_t mm = m;
    const size_t w = (mm + 1) * mm;
    const size_t sizes[3] = {w * sizeof(T), (gdr_y_offset(m) - w) * sizeof(T), mm * mm * sizeof(cplx)};
    size_t smem = 0;
    *parts = 0;
    for (int q = 0; q < 3 && smem + sizes[q] <= kGdrSmemMax; ++q) {
        smem += sizes[q];
        *parts = q + 1;
    }
    return smem;
}
template <class T>
cudaError_t launch_gmresdr_restart(const GdrArgs<T> &a_in, cudaStream_t s) {
    GdrArgs<T> a = a_in;
    const size_t smem = gmresdr_restart_smem<T>(a.m, &a.smem);
    if (smem > 30 * 1024) {         // 48 KB with the static part
        // without the raised limit the launch would fail; report the attribute call instead
        const cudaError_t e = smem_attr_once((const void *)k_gmresdr_restart<T>, (int)kGdrSmemMax);
        if (e != cudaSuccess) return e;
    }
    launch(k_gmresdr_restart<T>, 1, kGdrThreads, smem, s, a);
    return cudaGetLastError();
}
template <class T>
cudaError_t launch_gmresdr_restart_batch(const GdrArgs<T> *args, const int *active, int count, int m, cudaStream_t s) {
    int parts = 0;
    const size_t smem = gmresdr_restart_smem<T>(m, &parts);
    if (smem > 30 * 1024) {         // 48 KB with the static part
        const cudaError_t e = smem_attr_once((const void *)k_gmresdr_restart_batch<T>, (int)kGdrSmemMax);
        if (e != cudaSuccess) return e;
    }
    launch(k_gmresdr_restart_batch<T>, count, kGdrThreads, smem, s, args, active);
    return cudaGetLastError();
}
template <class D>
void launch_givens_step(const D *Hbar, D *H, int ldh, int j, D *cs, D *sn, D *g, GivensState *state, cudaStream_t s) {
    launch(k_givens_step<D>, 1, 32, 0, s, Hbar, H, ldh, j, cs, sn, g, state);
}
template <class D>
void launch_givens_solve(const D *H, int ldh, const D *g, D *y, const GivensState *state, cudaStream_t s) {
    launch(k_givens_solve<D>, 1, 1, 0, s, H, ldh, g, y, state);
}

#define TG_INST(D)                                                                                   \
    template void launch_chol_inv<D>(const D *, int, D *, D *, int *, cudaStream_t);                 \
    template void launch_inverse<D>(const D *, int, D *, D *, int *, cudaStream_t);                  \
    template void launch_small_gemv<D>(const D *, int, const D *, D *, cudaStream_t);                \
    template cudaError_t launch_gmresdr_restart<D>(const GdrArgs<D> &, cudaStream_t);                \
    template size_t gmresdr_restart_smem<D>(int, int *);                                              \
    template cudaError_t launch_gmresdr_restart_batch<D>(const GdrArgs<D> *, const int *, int, int, cudaStream_t); \
    template void launch_givens_step<D>(const D *, D *, int, int, D *, D *, D *, GivensState *, cudaStream_t);  \
    template void launch_givens_solve<D>(const D *, int, const D *, D *, const GivensState *, cudaStream_t);
TG_INST(double)
TG_INST(cplx)
#undef TG_INST

}  // namespace tg
