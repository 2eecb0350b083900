// Float64 contractions on the tensor cores by an exact fixed-point split: the tall-skinny
// product Out = In S and the Gram product A^H B (float64 and complex128).
//
// The float64 unit of this GPU issues 2 multiply-adds per clock and SM; both products need p
// (or k) of them per value read and sat at 0.84-0.93 of that rate, 7 to 30 times above the time
// their bytes take.  The split moves the multiply-adds to mma.sync (1007 f16 multiply-adds per
// clock and SM measured):
//   - a vector along the contraction (a row of In, a column of S, a 128-row piece of a Gram
//     column) is scaled by its largest exponent and each value becomes a 62-bit integer; a
//     value within 2^9 of the largest keeps all its 53 bits, smaller ones are cut at 2^-61 of it;
//   - the integer is written in 8 balanced digits of 8 bits, -128..127, exact in f16
//     (Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication",
//     Numer. Algorithms 59, 2012; on tensor cores Mukunoki, Ozaki, Ogita and Imamura, 2020);
//   - digit products are at most 2^14, so float32 accumulators hold the sum of at most 8 pairs
//     over 128 terms (2^24) exactly; pairs of digits i, j with i + j <= 7 are kept (36 of 64),
//     which leaves an error of about 2^-58 of the largest products;
//   - the eight diagonals i + j are added as integers and rounded to float64 once.
// So a sum of p terms is off by at most p 2^-58 times the product of the two vectors' largest values,
// and is then rounded once.  Where one vector's largest value meets a small one of the other, that is more
// than float64 sums lose.  In the Gram product both vectors are columns, and the bound is below the
// rounding of the columns' norms, however they are scaled.  In Out = In S a row of In may hold a
// large and a small column: Q = A R^-1 multiplies the small one by a large entry of R^-1.  There column
// i of In and row i of S are scaled by opposite powers of two, so that In's columns have norms between 1 and
// 2 (the callers have them from a Gram matrix, or know the columns to be unit vectors): column c of Out is
// then off by no more than p^1.5 2^-56 max_i ||In_i|| |S_ic|, whatever the scales, where float64 sums have
// p 2^-53 sum_i ||In_i|| |S_ic|.  Rows (or pieces) that hold an infinity, a NaN or magnitudes outside
// 2^-823..2^823, and products whose norms are not positive and finite, are computed in plain float64.
#pragma once

#include <cuda_fp16.h>

#include "tg_kernels.cuh"

namespace tg {

constexpr int kSplitDigits = 8;
constexpr int kSplitTerms = 64;         // terms of k_tsm_split's sums (8 pairs x 128 terms x 2^14 = 2^24 is exact)
constexpr int kSplitLo = 200, kSplitHi = 1846;   // biased exponents the split takes (zero too)

__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_f16_new(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}

// exponent field of |x| as the high word (monotone in |x|, so maxima can be taken on it)
__device__ __forceinline__ int split_mag(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ bool split_bad(int mag) {
    const int e = mag >> 20;
    return mag != 0 && (e < kSplitLo || e > kSplitHi);
}

// the scale exponent of a vector with largest magnitude mag (an all-zero vector gets kSplitLo,
// where split_fixed makes every zero a zero)
__device__ __forceinline__ int split_exp(int mag) { return max(mag >> 20, kSplitLo); }

// x as the biased integer Y = X + 0x8080808080808080, X = x 2^(1084 - E) cut towards zero
// (|X| < 2^62); byte 7 - i of Y is digit i plus 128.
__device__ __forceinline__ unsigned long long split_fixed(double x, int E) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)(hi >> 20) & 0x7ff;
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    unsigned long long m = ((unsigned long long)mh << 32 | lo) << 9;
    m >>= min(E - e, 63);
    const long long s = (long long)((int)hi >> 31);
    return (m ^ (unsigned long long)s) + (0x8080808080808080ull - (unsigned long long)s);
}

// the 8 digits of two values as f16 pairs (x0 low, x1 high)
__device__ __forceinline__ void split_pair(unsigned long long y0, unsigned long long y1, unsigned (&d)[kSplitDigits]) {
    const unsigned bias = 0x64806480u;            // 1024 + 128 in f16
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const unsigned a = w == 0 ? (unsigned)(y0 >> 32) : (unsigned)y0, b = w == 0 ? (unsigned)(y1 >> 32) : (unsigned)y1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            // bytes (3, 2) then (1, 0) of both words; 0x64 above a byte makes the f16 1024 + byte
            const unsigned t = __byte_perm(a, b, h == 0 ? 0x7632 : 0x5410);
            const unsigned u = __byte_perm(t, 0x64646464u, 0x4341), v = __byte_perm(t, 0x64646464u, 0x4240);
            const __half2 hu = __hsub2(*reinterpret_cast<const __half2 *>(&u), *reinterpret_cast<const __half2 *>(&bias));
            const __half2 hv = __hsub2(*reinterpret_cast<const __half2 *>(&v), *reinterpret_cast<const __half2 *>(&bias));
            d[4 * w + 2 * h] = *reinterpret_cast<const unsigned *>(&hu);
            d[4 * w + 2 * h + 1] = *reinterpret_cast<const unsigned *>(&hv);
        }
    }
}

// The eight diagonals (integers, |.| <= 8 K 2^14) of a sum of K products scaled by E1 and E2 as
// one float64, (sum_d D_d 2^(8 (7 - d))) 2^(E1 + E2 - 2112), rounded once: integer sums of the
// upper and the lower four diagonals are placed in the mantissas of two float64 constants, two
// float64 additions join them and the scale is added to the exponent.  A float64 instruction
// holds its unit for 64 clocks: conversions and scaling with five of them a result had bounded
// both kernels, and so did, by its 75 instructions, a join in integers alone (n = 191^3,
// p = q = 30: 3.9 and 2.9 ms a product).
// A result whose exponent leaves the normal range comes back unscaled with *far set: the caller
// finishes it with split_rescale (kept out of the joins, whose instructions then interleave).
template <int K>
__device__ __forceinline__ double split_join(const float (&D)[kSplitDigits], int E1, int E2, bool *far) {
    int v[kSplitDigits];
#pragma unroll
    for (int d = 0; d < kSplitDigits; ++d)      // up to 2^22 an addition puts the integer in the low bits
        v[d] = d < 4 && K <= 64 ? __float_as_int(D[d] + 12582912.0f) - 0x4b400000 : __float2int_rn(D[d]);
    const int x = v[6] + (v[7] >> 8);
    const long long h = (long long)(v[0] * 256 + v[1]) * 65536ll + (v[2] * 256 + v[3]);
    const long long l = K <= 64 ? (long long)(v[4] * 256 + v[5]) * 256ll + x
                                : (long long)v[4] * 65536ll + (long long)v[5] * 256ll + x;
    // 1.5 2^52 + h, and 1.5 2^28 + l 2^-24 (l counts 2^-24 of h's unit)
    const double hd = __longlong_as_double(h + 0x4338000000000000ll), ld = __longlong_as_double(l + 0x41b8000000000000ll);
    const double r = (hd - (6755399441055744.0 + 402653184.0)) + ld;
    const int hi = __double2hiint(r), er = (hi >> 20) & 0x7ff, de = E1 + E2 - 2080;
    const bool in = er != 0 && (unsigned)(er + de - 1) < 2046u;
    *far = er != 0 && !in;
    return __hiloint2double(in ? hi + (de << 20) : hi, __double2loint(r));
}
__device__ __forceinline__ double split_rescale(double r, int E1, int E2) { return scalbn(r, E1 + E2 - 2080); }

// ----------------------------------------------------------------------------- Out = In S
// Out (n x q) = In (n x p) S (p x q); complex128 runs as the real product of 2p columns (re, im
// interleaved, as stored) with the 2p x 2q matrix of S.  A block stages tiles of 16 WR rows
// (all p columns, cp.async, nbuf buffers) and holds the digits of its columns of S in shared
// memory in the order of the mma fragments.  Warp (wr, wc) takes 16 rows of the tile and the
// column groups wc, wc + 16 / WR, ... of 2 n-tiles (16 columns): 2 x 8 accumulators of a 16 x 8
// tile, one per diagonal.  Half the n-tiles of a 256-thread form with 4 per warp: its 246
// registers left two warps per scheduler, whose conversion, mma and join phases did not overlap
// (n = 191^3, p = q = 30: 3.0 ms).  gridDim.y splits the columns when the digits of all of S do not fit
// (in place, Out = In, only with gridDim.y = 1: each tile is staged before it is written).
// n = 191^3, p = q = 30: 3.0 ms, with scales 3.4 (the float64 unit: 11.2); complex128, n = 32^4, p = q = 40: 2.0 ms
// (10.9).  The mma take 0.9 ms of the 3.0 and the bytes 0.5; issuing the conversions and joins
// (27 thousand warp instructions a 128-row tile, 2 a clock) bounds it.
// SC: norm2[i nstride] is the square of the norm of In's column i (device), and the scales above are
// taken from it; else the columns are taken to be of unit norm.  Scaling is integer work on the exponents.
constexpr int kTsmThreads = 512, kTsmWarps = 16, kTsmCt = 2;
struct TsmSplitCfg {
    int wr, nbuf, ctb;      // row warps, buffers, n-tiles (8 columns) per block
    size_t smem;
};
__host__ __device__ __forceinline__ int split_kt(int pr) { return (pr + 15) / 16; }
template <class T> __host__ __device__ __forceinline__ int split_pc(int p) {
    return sizeof(T) == 16 ? 8 * split_kt(2 * p) : 16 * split_kt(p);
}

// exponent of the norm whose square is n2 (0 and *ok = false when that is not positive and finite)
__device__ __forceinline__ int split_norm_exp(double n2, bool *ok) {
    *ok = n2 > 0.0 && isfinite(n2);
    return *ok ? ilogb(n2) >> 1 : 0;
}
// x 2^-e by the exponent field; zero when that leaves no normal number
__device__ __forceinline__ double split_scale(double x, int e) {
    const int hi = __double2hiint(x), mag = hi & 0x7fffffff, m = mag < 0x100000 ? 0 : max(mag - (e << 20), 0);
    return __hiloint2double((hi & 0x80000000) | m, __double2loint(x));
}

template <class T, int WR, bool SC>
__global__ void __launch_bounds__(kTsmThreads, 1) k_tsm_split(const T *In, size_t ldi, int p, const T *__restrict__ S,
                                                           int lds, int q, T *Out, size_t ldo, int n, int ctb,
                                                           int nbuf, const T *__restrict__ norm2, int nstride) {
    pdl_wait();
    constexpr bool kC = sizeof(T) == 16;
    constexpr int R = 16 * WR, RS = R + 2, WC = kTsmWarps / WR;
    const int pr = kC ? 2 * p : p, qr = kC ? 2 * q : q;      // real dimensions
    const int KT = split_kt(pr), pc = split_pc<T>(p);        // staged columns: p, then zeros
    const int ct0 = blockIdx.y * ctb, nct = min(ctb, (qr + 7) / 8 - ct0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint2 *sf = reinterpret_cast<uint2 *>(smem_raw);                           // [KT][nct][8][32]
    T *tiles = reinterpret_cast<T *>(smem_raw + (size_t)KT * ctb * kSplitDigits * 256);
    __shared__ int ecol[8 * 32];
    __shared__ short ein[SC ? kMaxCols + 16 : 1];              // exponents of In's columns, 0 past the last
    __shared__ int bad_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, tq = lane & 3;
    const double *Sd = reinterpret_cast<const double *>(S);
    // real entry (k, c) of S, its row scaled
    auto s_at = [&](int k, int c) -> double {
        if (k >= pr || c >= qr) return 0.0;
        double v;
        if constexpr (kC) {
            const double *e = Sd + 2 * ((size_t)(k >> 1) + (size_t)(c >> 1) * lds);
            const int a = k & 1, b = c & 1;
            v = a == b ? e[0] : (a ? -e[1] : e[1]);
        } else {
            v = Sd[(size_t)k + (size_t)c * lds];
        }
        if constexpr (SC) v = scalbn(v, ein[kC ? k >> 1 : k]);
        return v;
    };
    const int ntiles = (n + R - 1) / R;
    const bool vec = kC || !(((uintptr_t)In | (ldi * sizeof(T))) & 15);      // 16-byte aligned columns
    auto issue = [&](int tile, int b) {
        if (tile < ntiles) {
            const int row0 = tile * R, left = n - row0;
            T *dst = tiles + (size_t)b * pc * RS;
            if (vec && left >= R) {
                constexpr int P = 16 / sizeof(T);
                for (int e = tid; e < p * (R / P); e += kTsmThreads) {
                    const int c = e / (R / P), r = P * (e % (R / P));
                    cp_async16(dst + c * RS + r, In + (size_t)c * ldi + row0 + r);
                }
            } else {
                for (int e = tid; e < p * R; e += kTsmThreads) {
                    const int c = e / R, r = e % R;
                    const T *src = In + (size_t)c * ldi + row0 + r;
                    if (r >= left) dst[c * RS + r] = ST<T>::zero();
                    else if constexpr (kC) cp_async16(dst + c * RS + r, src);
                    else cp_async8(dst + c * RS + r, src);
                }
            }
        }
        cp_async_commit();
    };
    for (int e = tid; e < nbuf * (pc - p) * RS; e += kTsmThreads) {
        const int b = e / ((pc - p) * RS), r = e % ((pc - p) * RS);
        tiles[(size_t)b * pc * RS + p * RS + r] = ST<T>::zero();
    }
    int tile = blockIdx.x;
    issue(tile, 0);
    // digits of S: column exponents first, a warp per column
    if (tid == 0) bad_s = 0;
    __syncthreads();
    if constexpr (SC) {
        for (int i = tid; i < pc; i += kTsmThreads) {
            bool ok = true;
            ein[i] = (short)(i < p ? split_norm_exp(*reinterpret_cast<const double *>(norm2 + (size_t)i * nstride), &ok) : 0);
            if (!ok) bad_s = 1;
        }
        __syncthreads();
    }
    for (int c = warp; c < 8 * nct; c += kTsmWarps) {
        int mg = 0;
        for (int k = lane; k < pr; k += 32) mg = max(mg, split_mag(s_at(k, 8 * ct0 + c)));
        mg = __reduce_max_sync(0xffffffffu, mg);
        if (lane == 0) {
            ecol[c] = split_exp(mg);
            if (split_bad(mg)) bad_s = 1;
        }
    }
    __syncthreads();
    for (int e = warp; e < KT * nct; e += kTsmWarps) {
        const int kt = e / nct, ct = e % nct, c = 8 * (ct0 + ct) + g, E = ecol[8 * ct + g];
        unsigned b0[kSplitDigits], b1[kSplitDigits];
        const int k = 16 * kt + 2 * tq;
        split_pair(split_fixed(s_at(k, c), E), split_fixed(s_at(k + 1, c), E), b0);
        split_pair(split_fixed(s_at(k + 8, c), E), split_fixed(s_at(k + 9, c), E), b1);
#pragma unroll
        for (int j = 0; j < kSplitDigits; ++j) sf[((size_t)e * kSplitDigits + j) * 32 + lane] = make_uint2(b0[j], b1[j]);
    }
    const int wr = warp % WR, wc = warp / WR;
    for (int it = 0; tile < ntiles; ++it, tile += gridDim.x) {
        const int buf = nbuf == 2 ? it & 1 : 0;
        if (nbuf == 2) {
            issue(tile + gridDim.x, buf ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const T *tl = tiles + (size_t)buf * pc * RS + 16 * wr + g;
        // the pair (k, k + 1) of row g + 8 h, k even
        auto pair_at = [&](int k, int h, double &x0, double &x1) {
            if constexpr (kC) {
                const cplx v = reinterpret_cast<const cplx *>(tl)[(k >> 1) * RS + 8 * h];
                x0 = v.re;
                x1 = v.im;
            } else {
                const double *td = reinterpret_cast<const double *>(tl);
                x0 = td[k * RS + 8 * h];
                x1 = td[(k + 1) * RS + 8 * h];
            }
            if constexpr (SC) {
                x0 = split_scale(x0, ein[kC ? k >> 1 : k]);
                x1 = split_scale(x1, ein[kC ? k >> 1 : k + 1]);
            }
        };
        int mg[2] = {0, 0};
        for (int kt = 0; kt < KT; ++kt)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                double x0, x1;
                pair_at(16 * kt + 2 * tq + 8 * (u >> 1), u & 1, x0, x1);
                mg[u & 1] = max(mg[u & 1], max(split_mag(x0), split_mag(x1)));
            }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            mg[h] = max(mg[h], __shfl_xor_sync(0xffffffffu, mg[h], 1));
            mg[h] = max(mg[h], __shfl_xor_sync(0xffffffffu, mg[h], 2));
        }
        const int E[2] = {split_exp(mg[0]), split_exp(mg[1])};
        const bool bad = bad_s || split_bad(mg[0]) || split_bad(mg[1]);
        const bool slow = __any_sync(0xffffffffu, bad);
        const int row0 = tile * R, left = n - row0, rg = 16 * wr + g;     // this lane's rows: row0 + rg, + 8
        for (int cg = kTsmCt * wc; cg < nct && !slow; cg += kTsmCt * WC) {
            float acc[kTsmCt][kSplitDigits][4];
            double tot[kTsmCt][4];
            // one k-tile of 16: the first of a sum starts the accumulators
            auto step = [&](int kt, auto first) {
                unsigned a[kSplitDigits][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {       // a0: row g, k lo; a1: row g + 8; a2, a3: k + 8
                    double x0, x1;
                    unsigned dg[kSplitDigits];
                    pair_at(16 * kt + 2 * tq + 8 * (u >> 1), u & 1, x0, x1);
                    split_pair(split_fixed(x0, E[u & 1]), split_fixed(x1, E[u & 1]), dg);
#pragma unroll
                    for (int i = 0; i < kSplitDigits; ++i) a[i][u] = dg[i];
                }
                // n-tiles past the block's last read that one again (and are not stored)
                const uint2 *sk = sf + ((size_t)kt * nct * kSplitDigits) * 32 + lane;
#pragma unroll
                for (int c = 0; c < kTsmCt; ++c) {
                    const uint2 *sc = sk + min(cg + c, nct - 1) * kSplitDigits * 32;
#pragma unroll
                    for (int j = 0; j < kSplitDigits; ++j) {
                        const uint2 b = sc[j * 32];
#pragma unroll
                        for (int i = 0; i + j < kSplitDigits; ++i) {
                            if (decltype(first)::value && j == 0) mma_f16_new(acc[c][i], a[i], b.x, b.y);
                            else mma_f16(acc[c][i + j], a[i], b.x, b.y);
                        }
                    }
                }
            };
            for (int k0 = 0; k0 < KT; k0 += kSplitTerms / 16) {
                step(k0, std::true_type{});
                for (int kt = k0 + 1; kt < min(KT, k0 + kSplitTerms / 16); ++kt) step(kt, std::false_type{});
                // the exact sums of up to kSplitTerms terms
#pragma unroll
                for (int c = 0; c < kTsmCt; ++c) {
                    const int cr = 8 * min(cg + c, nct - 1) + 2 * tq;
                    bool far[4];
                    double v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        float D[kSplitDigits];
#pragma unroll
                        for (int d = 0; d < kSplitDigits; ++d) D[d] = acc[c][d][u];
                        v[u] = split_join<kSplitTerms>(D, E[u >> 1], ecol[cr + (u & 1)], &far[u]);
                    }
                    if (far[0] | far[1] | far[2] | far[3]) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (far[u]) v[u] = split_rescale(v[u], E[u >> 1], ecol[cr + (u & 1)]);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) tot[c][u] = k0 == 0 ? v[u] : tot[c][u] + v[u];
                }
            }
#pragma unroll
            for (int c = 0; c < kTsmCt; ++c) {
                if (cg + c >= nct) continue;
                const int col = 8 * (ct0 + cg + c) + 2 * tq;             // real columns col, col + 1
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (rg + 8 * h >= left) continue;
                    const size_t row = (size_t)row0 + rg + 8 * h;
                    const double v0 = tot[c][2 * h], v1 = tot[c][2 * h + 1];
                    if constexpr (kC) {
                        if (col < qr) reinterpret_cast<cplx *>(Out)[(size_t)(col >> 1) * ldo + row] = mkc(v0, v1);
                    } else {
                        double *Od = reinterpret_cast<double *>(Out) + row;
                        if (col < qr) Od[(size_t)col * ldo] = v0;
                        if (col + 1 < qr) Od[(size_t)(col + 1) * ldo] = v1;
                    }
                }
            }
        }
        if (slow) {        // plain float64 for this warp's 16 rows
            const int c_lo = kC ? 4 * ct0 : 8 * ct0, c_hi = min(q, c_lo + (kC ? 4 : 8) * nct);
            const T *tw = tiles + (size_t)buf * pc * RS + 16 * wr;
            for (int e = lane; e < 16 * (c_hi - c_lo); e += 32) {
                const int r = e & 15, c = c_lo + (e >> 4);
                if ((e >> 4) % WC != wc || 16 * wr + r >= left) continue;
                T sacc = ST<T>::zero();
                for (int i = 0; i < p; ++i) sacc = axpy(S[i + (size_t)c * lds], tw[i * RS + r], sacc);
                Out[(size_t)c * ldo + row0 + 16 * wr + r] = sacc;
            }
        }
        __syncthreads();
        if (nbuf != 2) issue(tile + gridDim.x, 0);
    }
    cp_async_wait<0>();
}

// ----------------------------------------------------------------------------- G = A^H B
// Partial Gram products on the entry list of k_gram_packed.  blockIdx.y selects a pair (I, J) of
// panels of 32 real columns (complex128: 16 columns as re, im); blocks of x take 128-row pieces.
// A warp converts whole columns of a piece (exponent by a warp maximum, digits stored as f16
// planes [digit][column][row]); then warp w owns the 16 x 8 block (w & 1, w >> 1) of the 32 x 32
// products: 36 mma per 16 rows with operands from ldmatrix, joined and added in float64 after
// each piece.  For A = B only panels I <= J and blocks that reach the diagonal run.  30 columns of
// 191^3 rows: 1.2 ms (the float64 unit at 1.05 TFLOP/s: 6.1); 40 complex128 columns of 32^4 rows:
// 2.2 ms (5.9); about half the time is mma.
constexpr int kGramRows = 128, kGramStride = kGramRows + 8, kGramPanel = 32;

__device__ __forceinline__ void ldsm4(unsigned (&r)[4], const void *p) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s));
}
__device__ __forceinline__ void ldsm2(unsigned &r0, unsigned &r1, const void *p) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(s));
}

template <class T>
__global__ void __launch_bounds__(kThreads, 2) k_gram_split(const T *__restrict__ A, const T *__restrict__ B, size_t ld,
                                                            int k, int kb, int n, int sym, int npi, int nent,
                                                            typename ST<T>::D *part) {
    pdl_wait();
    constexpr bool kC = sizeof(T) == 16;
    constexpr int kCw = kC ? 2 : 1;                  // real columns per column
    const int kr = kCw * k, kbr = kCw * kb;
    int I, J;
    if (sym) {                                       // pairs I <= J, J-major
        J = 0;
        while ((J + 1) * (J + 2) / 2 <= (int)blockIdx.y) ++J;
        I = blockIdx.y - J * (J + 1) / 2;
    } else {
        I = blockIdx.y % npi;
        J = blockIdx.y / npi;
    }
    const bool same = A == B && I == J;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned short *pl = reinterpret_cast<unsigned short *>(smem_raw);   // [2][digit][32][kGramStride]
    const size_t side = (size_t)kSplitDigits * kGramPanel * kGramStride;
    unsigned short *plb = same ? pl : pl + side;
    __shared__ int ex[2][kGramPanel];
    __shared__ int bad_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, tq = lane & 3;
    const int mt = warp & 1, nt = warp >> 1;
    // a block entirely below the diagonal of a symmetric panel pair has no entry to produce
    const bool live = !(sym && I == J && 16 * mt >= 8 * nt + 8) && kGramPanel * I + 16 * mt < kr && kGramPanel * J + 8 * nt < kbr;
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t row0 = (int64_t)blockIdx.x * kGramRows; row0 < n; row0 += (int64_t)gridDim.x * kGramRows) {
        const int left = (int)min((int64_t)kGramRows, n - row0);
        __syncthreads();                             // the planes of the last piece are read
        if (tid == 0) bad_s = 0;
        __syncthreads();
        for (int sd = 0; sd < (same ? 1 : 2); ++sd) {
            const T *M = sd == 0 ? A : B;
            const int c0 = (sd == 0 ? I : J) * kGramPanel, cr = sd == 0 ? kr : kbr;
            unsigned short *pp = sd == 0 ? pl : plb;
            // the warp's real columns warp, warp + 8, ...; rows 2 l, 2 l + 1 (+ 64) of lane l
            double x[kGramPanel / 8][4];
#pragma unroll
            for (int e = 0; e < kGramPanel / 8; ++e) {
                const int c = c0 + warp + 8 * e;
                const double *src = reinterpret_cast<const double *>(M + (size_t)(c / kCw) * ld + row0) + c % kCw;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r = 2 * lane + (u & 1) + 64 * (u >> 1);
                    x[e][u] = c < cr && r < left ? src[(size_t)kCw * r] : 0.0;
                }
            }
#pragma unroll
            for (int e = 0; e < kGramPanel / 8; ++e) {
                const int c = warp + 8 * e;
                int mg = max(max(split_mag(x[e][0]), split_mag(x[e][1])), max(split_mag(x[e][2]), split_mag(x[e][3])));
                mg = __reduce_max_sync(0xffffffffu, mg);
                const int E = split_exp(mg);
                if (lane == 0) {
                    ex[sd][c] = E;
                    if (split_bad(mg)) bad_s = 1;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    unsigned d[kSplitDigits];
                    split_pair(split_fixed(x[e][2 * h], E), split_fixed(x[e][2 * h + 1], E), d);
#pragma unroll
                    for (int i = 0; i < kSplitDigits; ++i)
                        *reinterpret_cast<unsigned *>(pp + ((size_t)i * kGramPanel + c) * kGramStride + 2 * lane + 64 * h) = d[i];
                }
            }
        }
        __syncthreads();
        if (!live) continue;
        const int cb0 = kGramPanel * J + 8 * nt + 2 * tq, ca0 = kGramPanel * I + 16 * mt + g;   // real columns
        if (bad_s) {
            // plain float64 sums of this piece for the lane's four entries
            const double *Ad = reinterpret_cast<const double *>(A), *Bd = reinterpret_cast<const double *>(B);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int ca = ca0 + 8 * (u >> 1), cb = cb0 + (u & 1);
                if (ca >= kr || cb >= kbr) continue;
                const double *pa = Ad + kCw * (size_t)(ca / kCw) * ld + ca % kCw, *pb = Bd + kCw * (size_t)(cb / kCw) * ld + cb % kCw;
                double s = 0.0;
                for (int64_t r = row0; r < row0 + left; ++r) s = fma(pa[kCw * r], pb[kCw * r], s);
                tot[u] += s;
            }
            continue;
        }
        float acc[kSplitDigits][4];
#pragma unroll
        for (int d = 0; d < kSplitDigits; ++d)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[d][u] = 0.0f;
        // ldmatrix rows: matrices (columns 0-7, rows k..k+7), (columns 8-15, same), then rows k+8..
        const unsigned short *ap = pl + (size_t)(16 * mt + (lane & 15)) * kGramStride + 8 * (lane >> 4);
        const unsigned short *bp = plb + (size_t)(8 * nt + (lane & 7)) * kGramStride + 8 * ((lane >> 3) & 1);
        for (int ks = 0; ks < kGramRows / 16; ++ks) {
            unsigned a[kSplitDigits][4];
#pragma unroll
            for (int i = 0; i < kSplitDigits; ++i) ldsm4(a[i], ap + (size_t)i * kGramPanel * kGramStride + 16 * ks);
#pragma unroll
            for (int j = 0; j < kSplitDigits; ++j) {
                unsigned b0, b1;
                ldsm2(b0, b1, bp + (size_t)j * kGramPanel * kGramStride + 16 * ks);
#pragma unroll
                for (int i = 0; i + j < kSplitDigits; ++i) mma_f16(acc[i + j], a[i], b0, b1);
            }
        }
        bool far[4];
        double v[4];
        const int ea[2] = {ex[0][16 * mt + g], ex[0][16 * mt + g + 8]};
        const int eb[2] = {ex[same ? 0 : 1][8 * nt + 2 * tq], ex[same ? 0 : 1][8 * nt + 2 * tq + 1]};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float D[kSplitDigits];
#pragma unroll
            for (int d = 0; d < kSplitDigits; ++d) D[d] = acc[d][u];
            v[u] = split_join<kGramRows>(D, ea[u >> 1], eb[u & 1], &far[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) tot[u] += far[u] ? split_rescale(v[u], ea[u >> 1], eb[u & 1]) : v[u];
    }
    if (!live) return;
    const int mcol = kGramPanel * I + 16 * mt + g, ncol = kGramPanel * J + 8 * nt + 2 * tq;     // real columns
    typename ST<T>::D *out = part + (size_t)blockIdx.x * nent;
    auto put = [&](int i, int j, typename ST<T>::D v) {
        if (i < k && j < kb) {
            if (!sym) out[i + (size_t)j * k] = v;
            else if (i <= j) out[(size_t)j * (j + 1) / 2 + i] = v;
        }
    };
    if constexpr (kC) {
        // conj(a) b: re = ar br + ai bi, im = ar bi - ai br; ai is the next row's lane
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const double o0 = __shfl_down_sync(0xffffffffu, tot[2 * h], 4), o1 = __shfl_down_sync(0xffffffffu, tot[2 * h + 1], 4);
            if (!(g & 1)) put((mcol + 8 * h) >> 1, ncol >> 1, mkc(tot[2 * h] + o1, tot[2 * h + 1] - o0));
        }
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) put(mcol + 8 * (u >> 1), ncol + (u & 1), tot[u]);
    }
}

}  // namespace tg
