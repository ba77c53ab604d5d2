// Row-tile building blocks of the CUDA-core kernels: tiles of up to 64 rows in shared memory, register-tiled
// products between them, and sums carried as unevaluated pairs of floats.
//
// What bounds these kernels is arithmetic.  The parameter gradients are sums of terms that cancel by factors
// of hundreds, so the statistics, the row normalisers, the outputs and dphi have to be formed to more than
// fp32 and rounded once.  fp64 does that at 2 multiply-adds per cycle and SM on this part (measured through
// the fp64 form of these kernels: 0.6 T/s); the pair form below does it with five fp32 operations at 128 per
// cycle and SM, and keeps about 46 bits of sum_k |a_k b_k| (pair_base).
#pragma once

#include <algorithm>
#include <type_traits>

#include "luna_simt_dev.cuh"

namespace luna {
namespace simt {
namespace {  // internal linkage in every translation unit that includes this

constexpr int kThr = 512;   // threads per block: with one block per SM the four schedulers hold four warps each
constexpr int kMaxC = 64;   // rows per tile at most
constexpr int kMinC = 8;    // and at least (every tile is a multiple of 8 rows)
constexpr int kSlack = 8;   // floats after the last tile: an 8-column read of its last row may pass its end
constexpr int kSMs = 152;
// Shared memory of a block for the arrays of a tile: 227 KB less what the kernels hold statically (last_arrival's flag,
// the 128 bytes of channel sums of k_causal_bwd_query).  A launch whose static and dynamic parts exceed 227 KB is
// refused, so tiles are chosen, and shapes accepted, by this limit.
constexpr size_t kStaticSmem = 256;
constexpr size_t kSmemLimit = 227 * 1024 - kStaticSmem;

// Row stride in floats of a tile of x columns: whole 16-byte words, an odd number of them, so that eight lanes
// reading 16 bytes each from consecutive rows touch all 32 banks.
__host__ __device__ inline int row_stride(int x) { return 4 * (((x + 3) / 4) | 1); }

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ float at(const float4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// Rows per tile: the most that fit in shared memory (large tiles share each table, state and barrier between
// more rows), but small problems take smaller ones, down to 16, until every SM has a tile.
template <typename Smem>
int pick_cap(int64_t BH, int n, Smem smem) {
    const int caps[] = {64, 48, 32, 24, 16, 8};
    int cap = kMinC;
    for (int c : caps) {
        if (smem(c) > kSmemLimit) continue;
        cap = c;
        if (c == kMinC || c <= 16 || BH * ((n + c - 1) / c) >= kSMs) break;
    }
    return cap;
}

// Calls f(TF, TC) with the register tile of OuterAcc for a D x dv accumulator.
template <typename F>
void outer_dispatch(int D, int dv, F f) {
    auto fits = [&](int tf, int tc) { return ((D + tf - 1) / tf) * ((dv + tc - 1) / tc) <= kThr; };
    if (fits(2, 4)) f(std::integral_constant<int, 2>{}, std::integral_constant<int, 4>{});
    else if (fits(4, 4)) f(std::integral_constant<int, 4>{}, std::integral_constant<int, 4>{});
    else f(std::integral_constant<int, 4>{}, std::integral_constant<int, 8>{});
}

// Parameter gradients of the generic backward kernels, in the partials' buffer of 2 * blocks * gsize doubles
// (`blocks`: of one of the two kernels at most): dW and db of every block of both in a slot of its own, so that
// they are summed in a fixed order, and before the channel normalisation's partials (a.gpart from here on) the
// histograms.  These are the large part and are added to by L2 reductions: the blocks share one per SM, which
// keeps the reductions of concurrent blocks apart and their zeroing and sum at 152 x 70 KB instead of one per block.
inline cudaError_t place_grads(AttnArgs &a, int64_t blocks, cudaStream_t s) {
    const int nw = a.M * a.d + a.M, nh = a.gsize - nw;
    a.gpart64 = 1;
    a.gw = reinterpret_cast<double *>(a.gpart);
    a.gw_n = (int)(2 * blocks);
    a.gh = a.gw + (size_t)a.gw_n * nw;
    a.gh_n = (int)std::min<int64_t>(blocks, kSMs);
    a.gpart = reinterpret_cast<float *>(a.gh + (size_t)a.gh_n * nh);
    return cudaMemsetAsync(a.gh, 0, (size_t)a.gh_n * nh * sizeof(double), s);
}

// ---------------------------------------------------------------------------
// Sums as pairs h + l.

// (h, l) += a b with the rounding error of h's update carried in l.  The product is exact (fma).  The error is
// exact where |h| >= |a b| and the sum does not cancel; elsewhere up to half an ulp of a b is lost.  A start value
// from `pair_base` rules both out.
__device__ __forceinline__ void pair_mac(float &h, float &l, float a, float b) {
    const float t = __fmaf_rn(a, b, h);
    const float q = __fsub_rn(t, h);
    l = __fadd_rn(l, __fmaf_rn(a, b, -q));
    h = t;
}

// h += x with its rounding error returned, whatever the sizes (Knuth's TwoSum).
__device__ __forceinline__ float add_error(float &h, float x) {
    const float t = __fadd_rn(h, x), q = __fsub_rn(t, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, q)), __fsub_rn(x, q));
    h = t;
    return e;
}

// (h, l) += a b, exact in h whatever the sizes (ten operations).
__device__ __forceinline__ void pair_mac_any(float &h, float &l, float a, float b) {
    const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
    l = __fadd_rn(l, __fadd_rn(e, add_error(h, p)));
}

// (h, l) += (h2, l2), exact in the high parts.
__device__ __forceinline__ void pair_add(float &h, float &l, float h2, float l2) {
    const float e = add_error(h, h2);
    l = __fadd_rn(l, __fadd_rn(l2, e));
}

// The pair rounded once.  An infinite or NaN sum has its value in h alone.
__device__ __forceinline__ float pair_value(float h, float l) {
    return fabsf(h) < INFINITY ? __fadd_rn(h, l) : h;
}
__device__ __forceinline__ double pair_double(float h, float l) {
    return fabsf(h) < INFINITY ? (double)h + (double)l : (double)h;
}

// Start value of a sum whose terms' sizes add up to `bound`: 1.5 times a power of two at least twice the bound.
// h then never leaves one binade, so every update of pair_mac is exact to 2^-24 of the start value's ulp, also
// where the terms cancel.  The bound is the sum's own, sum_k |a_k b_k|, formed in a pass of its own before it (one
// operation more per product, and its loads again): with one bound for a whole tile (rows x largest |a| x largest
// |b|) a column of values 1e-4 of the largest was summed no better than in fp32, and an outlier in one row cost
// every other sum of its tile its low half.  0 (an ordinary start) for a bound that is not finite or above 1e37.
__device__ __forceinline__ float pair_base(float bound) {
    if (!(bound < 1e37f)) return 0.0f;
    const int e = (__float_as_int(bound) >> 23) & 0xff;
    return __int_as_float((e + 2) << 23 | 0x400000);
}

// e / n for 0 <= e < 2^20, a shift where n is a power of two (M, and most widths / 4).
struct Div {
    int n, sh;
    __device__ __forceinline__ explicit Div(int n_) {
        n = n_;
        sh = (n_ & (n_ - 1)) == 0 ? 31 - __clz(n_) : -1;
    }
    __device__ __forceinline__ int operator()(int e) const { return sh >= 0 ? e >> sh : e / n; }
};

// ---------------------------------------------------------------------------
// Row tiles.

struct Rows {  // a tile: rows at p + r * ld
    float *p;
    int ld;
    __device__ __forceinline__ float *operator[](int r) const { return p + r * ld; }
};

__device__ Rows take_rows(Carve &cv, int rows, int cols) {
    Rows t{nullptr, row_stride(cols)};
    t.p = cv.take(rows * t.ld);
    return t;
}
void take_rows_host(HostCarve &cv, int rows, int cols) { cv.take(rows * row_stride(cols)); }

// 16-byte loads of whole rows of w elements are possible.
template <typename IO>
__device__ __forceinline__ bool vec_rows(const void *p, int w) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (w * sizeof(IO)) % 16 == 0;
}

__device__ __forceinline__ void put16(float *dst, const float *, const uint4 &v) {
    st4(dst, make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)));
}
__device__ __forceinline__ void put16(float *dst, const __nv_bfloat16 *, const uint4 &v) {
    st4(dst, make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                         __uint_as_float(v.y & 0xffff0000u)));
    st4(dst + 4, make_float4(__uint_as_float(v.z << 16), __uint_as_float(v.z & 0xffff0000u), __uint_as_float(v.w << 16),
                             __uint_as_float(v.w & 0xffff0000u)));
}

// nr contiguous rows of w elements into the tile (cap rows); the pad columns and the rows from nr on are 0.
template <typename IO>
__device__ void load_tile(const Rows &t, const IO *src, int nr, int w, int cap) {
    constexpr int VE = 16 / sizeof(IO);
    if (vec_rows<IO>(src, w)) {
        const Div wv(w / VE);
#pragma unroll 2
        for (int e = threadIdx.x; e < nr * wv.n; e += blockDim.x) {
            const int r = wv(e), c = (e - r * wv.n) * VE;
            put16(t[r] + c, src, *reinterpret_cast<const uint4 *>(src + (size_t)e * VE));
        }
    } else {
        for (int e = threadIdx.x; e < nr * w; e += blockDim.x) {
            const int r = e / w, c = e - r * w;
            t[r][c] = io_load(src + e);
        }
        const int wp = (w + 3) & ~3;
        if (wp != w)
            for (int e = threadIdx.x; e < nr * (wp - w); e += blockDim.x) t[e / (wp - w)][w + e % (wp - w)] = 0.0f;
    }
    for (int e = threadIdx.x; e < (cap - nr) * t.ld; e += blockDim.x) t[nr][e] = 0.0f;
}

// ---------------------------------------------------------------------------
// The feature map over a tile.

// Shared memory of the feature map (the generic SmemPhi, with the projection rows padded and the bucketed
// search block in place of the kinks alone).  cap: the rows that phi_rows is called with, for the gate's and the
// coefficients' factors of each; 0 only where the map has neither.
__device__ SmemPhi carve_phi_tile(Carve &cv, const TableLayout &lay, int cap) {
    SmemPhi s = {};
    if (!lay.act) {
        s.T = cv.take(kEytzinger);
        s.AB = cv.take(lay.nint * ab_stride(lay));
    }
    s.W = cv.take(lay.M * row_stride(lay.d));
    s.b = cv.take(lay.M);
    if (lay.act) {
        s.w1 = cv.take(lay.P); s.b1 = cv.take(lay.P); s.w2 = cv.take(lay.L * lay.hid); s.b2 = cv.take(lay.L);
    }
    if (lay.env) { s.We = cv.take(lay.L * lay.d); s.be = cv.take(lay.L); }
    if (lay.coef) s.coef = cv.take(lay.L);
    if (lay.env || lay.coef) { s.E = cv.take(cap * lay.L); s.H = cv.take(cap * lay.L); s.dE = cv.take(cap * lay.L); }
    return s;
}
void carve_phi_tile_host(HostCarve &cv, const TableLayout &lay, int cap) {
    if (!lay.act) { cv.take(kEytzinger); cv.take(lay.nint * ab_stride(lay)); }
    cv.take(lay.M * row_stride(lay.d)); cv.take(lay.M);
    if (lay.act) { cv.take(lay.P); cv.take(lay.P); cv.take(lay.L * lay.hid); cv.take(lay.L); }
    if (lay.env) { cv.take(lay.L * lay.d); cv.take(lay.L); }
    if (lay.coef) cv.take(lay.L);
    if (lay.env || lay.coef) { cv.take(cap * lay.L); cv.take(cap * lay.L); cv.take(cap * lay.L); }
}

__device__ void load_phi_tile(const SmemPhi &s, const TableLayout &lay, const char *table) {
    auto copy = [&](float *dst, int64_t off, int count) {
        const float *src = reinterpret_cast<const float *>(table + off);
        for (int e = threadIdx.x; e < count; e += blockDim.x) dst[e] = src[e];
    };
    if (!lay.act) {
        const float4 *src = reinterpret_cast<const float4 *>(table + lay.off_Te);
        for (int e = threadIdx.x; e < kEytzinger / 4; e += blockDim.x) st4(s.T + 4 * e, src[e]);
        if (lay.L == 8) {  // an interval's 64 bytes as four 16-byte loads, rows of 18 words in shared memory
            const float4 *ab = reinterpret_cast<const float4 *>(table + lay.off_AB);
            for (int e = threadIdx.x; e < lay.nint * 4; e += blockDim.x) {
                const float4 v = ab[e];
                float2 *d = reinterpret_cast<float2 *>(s.AB + (e >> 2) * 18 + (e & 3) * 4);
                d[0] = make_float2(v.x, v.y);
                d[1] = make_float2(v.z, v.w);
            }
        } else {
            copy_ab(s.AB, lay, table);
        }
    }
    const int ldw = row_stride(lay.d);
    const float *W = reinterpret_cast<const float *>(table + lay.off_W);
    for (int e = threadIdx.x; e < lay.M * ldw; e += blockDim.x) {
        const int i = e / ldw, c = e - i * ldw;
        s.W[e] = c < lay.d ? W[i * lay.d + c] : 0.0f;
    }
    copy(s.b, lay.off_b, lay.M);
    if (lay.act) {
        copy(s.w1, lay.off_w1, lay.P); copy(s.b1, lay.off_b1, lay.P);
        copy(s.w2, lay.off_w2, lay.L * lay.hid); copy(s.b2, lay.off_b2, lay.L);
    }
    if (lay.env) { copy(s.We, lay.off_We, lay.L * lay.d); copy(s.be, lay.off_be, lay.L); }
    if (lay.coef) copy(s.coef, lay.off_coef, lay.L);
}

// phi of rows [0, nr) of X into Phi, zeros in its other rows (cap in all) and pad columns; with sU also the
// projections u[r * M + i] and their intervals.  The projection is one fma chain over the columns in order, as
// in every generic kernel: which side of a kink a row falls on does not depend on the kernel.  Called by every
// thread of the block; synchronises it first if the map has a gate or coefficients.
__device__ void phi_rows(const TableLayout &lay, const SmemPhi &s, const Rows &X, int nr, int cap, const Rows &Phi,
                         float *sU, int *sJ) {
    const int M = lay.M, L = lay.L, d = lay.d, D = lay.D, ldw = row_stride(d), dp = (d + 3) & ~3;
    const float fl = channel_floor(lay);
    const bool ev = lay.env || lay.coef;
    if (ev) {
        __syncthreads();  // the row scratch of an earlier call is no longer read
        gate_rows(lay, s, X.p, X.ld, nr);
        __syncthreads();
    }
    const float sc = phi_scale(lay);
    const unsigned short *sB = reinterpret_cast<const unsigned short *>(s.T + kSearchT);
    const Div byM(M);
    for (int e = threadIdx.x; e < cap * M; e += blockDim.x) {
        const int r = byM(e), i = e - r * M;
        float *out = Phi[r] + i * L;
        if (i == M - 1)
            for (int f = D; f < ((D + 3) & ~3); ++f) Phi[r][f] = 0.0f;
        if (r >= nr) {
            for (int l = 0; l < L; ++l) out[l] = 0.0f;
            continue;
        }
        const float *x = X[r], *w = s.W + i * ldw;
        float u = s.b[i];
#pragma unroll 4
        for (int c = 0; c < dp; c += 4) {
            const float4 a = ld4(w + c), b = ld4(x + c);
            u = fmaf(a.x, b.x, u);
            u = fmaf(a.y, b.y, u);
            u = fmaf(a.z, b.z, u);
            u = fmaf(a.w, b.w, u);
        }
        int j = 0;
        if (!lay.act) {
            j = interval_bucketed(s.T, sB, u);
            const float *ab = s.AB + j * ab_stride(lay);
            if (L == 8) {
                float y[8];
#pragma unroll
                for (int l = 0; l < 8; ++l) {
                    const float2 p = ab_pair(ab, l);
                    y[l] = fmaxf(fmaf(p.x, u, p.y), fl);
                }
                st4(out, make_float4(y[0], y[1], y[2], y[3]));
                st4(out + 4, make_float4(y[4], y[5], y[6], y[7]));
            } else {
                for (int l = 0; l < L; ++l) {
                    const float2 p = ab_pair(ab, l);
                    out[l] = fmaxf(fmaf(p.x, u, p.y), fl);
                }
            }
        } else {
            for (int l = 0; l < L; ++l) out[l] = fmaxf(sc * channel_direct(lay, s, l, u, nullptr), fl);
        }
        if (ev)
            for (int l = 0; l < L; ++l) out[l] *= s.E[r * L + l];
        if (sU) { sU[e] = u; sJ[e] = j; }
    }
}

// ---------------------------------------------------------------------------
// Products.  A unit is 2 rows x 4 columns of the result per thread: six 16-byte shared loads for 32 products
// (160 operations in pair form with the bounds), so the loads take a small part of the issue slots and of the
// shared-memory bandwidth, and the eight chains of a unit hide the fma latency with four warps per scheduler.

__device__ __forceinline__ void abs_mac(float &s, float a, float b) { s = fmaf(fabsf(a), fabsf(b), s); }

// The start values of a unit's sums from their bounds, in place; h starts there.
__device__ __forceinline__ void unit_base(float (&b)[2][4], float (&h)[2][4], float (&l)[2][4]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            b[i][m] = pair_base(b[i][m]);
            h[i][m] = b[i][m];
            l[i][m] = 0.0f;
        }
}
// The sums without their start values (exact).
__device__ __forceinline__ void unit_unbase(float (&h)[2][4], const float (&b)[2][4]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int m = 0; m < 4; ++m) h[i][m] = __fsub_rn(h[i][m], b[i][m]);
}

// One step of a unit's sums over four k: rows x0, x1 of A (k .. k + 3) and the four B rows at b.
__device__ __forceinline__ void unit_nn(float (&h)[2][4], float (&l)[2][4], const float4 &x0, const float4 &x1,
                                        const float *b, int ldb) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const float4 v = ld4(b + kk * ldb);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            pair_mac(h[0][m], l[0][m], at(x0, kk), at(v, m));
            pair_mac(h[1][m], l[1][m], at(x1, kk), at(v, m));
        }
    }
}
// The step's share of the bounds.
__device__ __forceinline__ void unit_abs_nn(float (&s)[2][4], const float4 &x0, const float4 &x1, const float *b, int ldb) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const float4 v = ld4(b + kk * ldb);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            abs_mac(s[0][m], at(x0, kk), at(v, m));
            abs_mac(s[1][m], at(x1, kk), at(v, m));
        }
    }
}
__device__ __forceinline__ void unit_nn(float (&h)[2][4], const float4 &x0, const float4 &x1, const float *b, int ldb) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const float4 v = ld4(b + kk * ldb);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            h[0][m] = fmaf(at(x0, kk), at(v, m), h[0][m]);
            h[1][m] = fmaf(at(x1, kk), at(v, m), h[1][m]);
        }
    }
}

// out(r, c) = sum_{k < K} A[r][k] B[k][c] + sum_{k <= r} T[r][k] B2[k][c] (K rounded up to a multiple of 4; T null:
// the first sum alone): a unit's rows r0, r0 + 1 and columns c0 .. c0 + 3 go to done(r0, c0, h, l) as pairs.  The
// triangle ends exactly at the diagonal: a later row's infinity must not meet a zero of T.
template <typename Done>
__device__ __forceinline__ void prod_nn(const Rows &A, int rows, const Rows &B, int K, int cols, const Rows &T,
                                        const Rows &B2, Done done) {
    const int ng = (cols + 3) / 4, nu = ((rows + 1) / 2) * ng;
    const Div by(ng);
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        const int g = by(u), r0 = 2 * g, c0 = 4 * (u - g * ng);
        float h[2][4], l[2][4], b[2][4] = {};
        for (int k = 0; k < K; k += 4) unit_abs_nn(b, ld4(A[r0] + k), ld4(A[r0 + 1] + k), B[k] + c0, B.ld);
        if (T.p) {
            int k = 0;
            for (; k + 4 <= r0 + 1; k += 4) unit_abs_nn(b, ld4(T[r0] + k), ld4(T[r0 + 1] + k), B2[k] + c0, B2.ld);
            for (; k <= r0 + 1; ++k) {
                const float4 v = ld4(B2[k] + c0);
                const float x0 = T[r0][k], x1 = T[r0 + 1][k];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (k <= r0) abs_mac(b[0][m], x0, at(v, m));
                    abs_mac(b[1][m], x1, at(v, m));
                }
            }
        }
        unit_base(b, h, l);
        for (int k = 0; k < K; k += 4) unit_nn(h, l, ld4(A[r0] + k), ld4(A[r0 + 1] + k), B[k] + c0, B.ld);
        if (T.p) {
            int k = 0;
            for (; k + 4 <= r0 + 1; k += 4) unit_nn(h, l, ld4(T[r0] + k), ld4(T[r0 + 1] + k), B2[k] + c0, B2.ld);
            for (; k <= r0 + 1; ++k) {
                const float4 v = ld4(B2[k] + c0);
                const float x0 = T[r0][k], x1 = T[r0 + 1][k];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (k <= r0) pair_mac(h[0][m], l[0][m], x0, at(v, m));
                    pair_mac(h[1][m], l[1][m], x1, at(v, m));
                }
            }
        }
        unit_unbase(h, b);
        done(r0, c0, h, l);
    }
}

// Plain fp32 sums of the streaming form: fma chains of kChain products, added as pairs.  A tile of 64 rows puts up
// to 64 products behind the 64 of the state in one sum (a former tile of 16 rows: 16), and one chain over all of
// them made dV 1.7 and the outputs 1.2 times as far off as that.  In chains of 8 they are 0.6 and 0.7 times as far
// off (n = 300, d = 64), for 71 of 2372 us of a training step of 8 x 12 heads of 1024 bf16 rows.
constexpr int kChain = 8;

__device__ __forceinline__ void fold_chain(float (&H)[2][4], float (&L)[2][4], float (&h)[2][4]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            L[i][m] = __fadd_rn(L[i][m], add_error(H[i][m], h[i][m]));
            h[i][m] = 0.0f;
        }
}

// out(r, c) = sum_{k < K} A[r][k] B[k][c] in plain fp32, one fma chain per element over k in order.
template <typename Done>
__device__ __forceinline__ void prod_nn_plain(const Rows &A, int rows, const Rows &B, int K, int cols, Done done) {
    const int ng = (cols + 3) / 4, nu = ((rows + 1) / 2) * ng;
    const Div by(ng);
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        const int g = by(u), r0 = 2 * g, c0 = 4 * (u - g * ng);
        float h[2][4] = {};
        for (int k = 0; k < K; k += 4) unit_nn(h, ld4(A[r0] + k), ld4(A[r0 + 1] + k), B[k] + c0, B.ld);
        done(r0, c0, h);
    }
}

// out(r, c) = sum_{k < K} A[r][k] B[k][c] + sum_{r <= k < k2} T[k][r] B2[k][c], T lower triangular, in chains over k.
template <typename Done>
__device__ __forceinline__ void prod_nn_chains(const Rows &A, int rows, const Rows &B, int K, int cols, const Rows &T,
                                               const Rows &B2, int k2, Done done) {
    const int ng = (cols + 3) / 4, nu = ((rows + 1) / 2) * ng;
    const Div by(ng);
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        const int g = by(u), r0 = 2 * g, c0 = 4 * (u - g * ng);
        float H[2][4] = {}, L[2][4] = {}, h[2][4] = {};
        for (int k0 = 0; k0 < K; k0 += kChain) {
            for (int k = k0; k < min(k0 + kChain, K); k += 4)
                unit_nn(h, ld4(A[r0] + k), ld4(A[r0 + 1] + k), B[k] + c0, B.ld);
            fold_chain(H, L, h);
        }
        for (int k0 = r0; k0 < k2; k0 += kChain) {
            for (int k = k0; k < min(k0 + kChain, k2); ++k) {
                const float2 x = *reinterpret_cast<const float2 *>(T[k] + r0);
                const float4 v = ld4(B2[k] + c0);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    h[0][m] = fmaf(x.x, at(v, m), h[0][m]);
                    if (k > r0) h[1][m] = fmaf(x.y, at(v, m), h[1][m]);
                }
            }
            fold_chain(H, L, h);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int m = 0; m < 4; ++m) h[i][m] = pair_value(H[i][m], L[i][m]);
        done(r0, c0, h);
    }
}

// out(r, f) = init(r, f) + sum_{k < K} A[r][k] B[f][k] + (second sum) for f < F: a unit is rows r0, r0 + 1 and the
// four f of f0, f0 + F4, f0 + 2 F4, f0 + 3 F4 (F4 = ceil(F / 4)), so that consecutive lanes read consecutive rows
// of B.  The second sum runs over the rows k of B2: of A2[r][k] B2[k][f] for k <= r (Lower), or of
// A2[k][r] B2[k][f] for r <= k < k2 (Upper), with A2 lower triangular.  init(r, f, h, l) sets a pair (0 before);
// done(r, f, h, l) gets the sums, for f < F.
enum Second { kNone, kLower, kUpper };
template <Second MODE, typename Init, typename Done>
__device__ __forceinline__ void prod_nt(const Rows &A, int rows, const Rows &B, int F, int K, const Rows &A2,
                                        const Rows &B2, int k2, Init init, Done done) {
    const int F4 = (F + 3) / 4, nu = ((rows + 1) / 2) * F4;
    const Div by(F4);
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        const int g = by(u), r0 = 2 * g, f0 = u - g * F4;
        int f[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) f[m] = min(f0 + m * F4, F - 1);
        const float *a0 = A[r0], *a1 = A[r0 + 1];
        float h[2][4], l[2][4], b[2][4] = {};
        for (int k = 0; k < K; k += 4) {
            const float4 x0 = ld4(a0 + k), x1 = ld4(a1 + k);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float4 v = ld4(B[f[m]] + k);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    abs_mac(b[0][m], at(x0, kk), at(v, kk));
                    abs_mac(b[1][m], at(x1, kk), at(v, kk));
                }
            }
        }
        if (MODE == kLower) {
            for (int k = 0; k <= r0 + 1 && k < k2; ++k) {
                const float x0 = A2[r0][k], x1 = A2[r0 + 1][k];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float v = B2[k][f[m]];
                    if (k <= r0) abs_mac(b[0][m], x0, v);
                    abs_mac(b[1][m], x1, v);
                }
            }
        }
        if (MODE == kUpper) {
            for (int k = r0; k < k2; ++k) {
                const float2 x = *reinterpret_cast<const float2 *>(A2[k] + r0);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float v = B2[k][f[m]];
                    abs_mac(b[0][m], x.x, v);
                    if (k > r0) abs_mac(b[1][m], x.y, v);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                float ih = 0.0f, il = 0.0f;
                init(r0 + i, f[m], ih, il);
                b[i][m] = pair_base(b[i][m] + fabsf(ih));
                h[i][m] = b[i][m];
                l[i][m] = il;
                pair_mac(h[i][m], l[i][m], ih, 1.0f);
            }
        for (int k = 0; k < K; k += 4) {
            const float4 x0 = ld4(a0 + k), x1 = ld4(a1 + k);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float4 v = ld4(B[f[m]] + k);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    pair_mac(h[0][m], l[0][m], at(x0, kk), at(v, kk));
                    pair_mac(h[1][m], l[1][m], at(x1, kk), at(v, kk));
                }
            }
        }
        if (MODE == kLower) {
            for (int k = 0; k <= r0 + 1 && k < k2; ++k) {
                const float x0 = A2[r0][k], x1 = A2[r0 + 1][k];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float v = B2[k][f[m]];
                    if (k <= r0) pair_mac(h[0][m], l[0][m], x0, v);
                    pair_mac(h[1][m], l[1][m], x1, v);
                }
            }
        }
        if (MODE == kUpper) {
            for (int k = r0; k < k2; ++k) {
                const float2 x = *reinterpret_cast<const float2 *>(A2[k] + r0);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float v = B2[k][f[m]];
                    pair_mac(h[0][m], l[0][m], x.x, v);
                    if (k > r0) pair_mac(h[1][m], l[1][m], x.y, v);
                }
            }
        }
        unit_unbase(h, b);
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (f0 + m * F4 < F) done(r0 + i, f[m], h[i][m], l[i][m]);
    }
}

// Lower triangle of A B^T for the rows of a tile: S[r][j] for j <= r < rows, 0 above the diagonal, in row `rows`
// of an odd count and in the columns up to a multiple of 4.  PAIR: as pairs from init(r, h, l), rounded once; else
// in chains over k (init is not called).
template <bool PAIR, typename Init>
__device__ __forceinline__ void scores_lower(const Rows &A, const Rows &B, int rows, int K, const Rows &S, Init init) {
    const int F4 = (rows + 3) / 4, nu = ((rows + 1) / 2) * F4;
    const Div by(F4);
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        const int g = by(u), r0 = 2 * g, f0 = u - g * F4;
        float h[2][4] = {}, l[2][4] = {}, b[2][4] = {};
        const int nm = f0 <= r0 + 1 ? min(4, (r0 + 1 - f0) / F4 + 1) : 0;  // columns at or below the diagonal
        const float *a0 = A[r0], *a1 = A[r0 + 1];
        if (PAIR && nm) {
            for (int k = 0; k < K; k += 4) {
                const float4 x0 = ld4(a0 + k), x1 = ld4(a1 + k);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (m < nm) {
                        const float4 v = ld4(B[f0 + m * F4] + k);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            abs_mac(b[0][m], at(x0, kk), at(v, kk));
                            abs_mac(b[1][m], at(x1, kk), at(v, kk));
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float ih = 0.0f, il = 0.0f;
                init(r0 + i, ih, il);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    b[i][m] = pair_base(b[i][m] + fabsf(ih));
                    h[i][m] = b[i][m];
                    l[i][m] = il;
                    pair_mac(h[i][m], l[i][m], ih, 1.0f);
                }
            }
        }
        if (nm) {
            for (int k0 = 0; k0 < K; k0 += PAIR ? K : kChain) {
                for (int k = k0; k < (PAIR ? K : min(k0 + kChain, K)); k += 4) {
                    const float4 x0 = ld4(a0 + k), x1 = ld4(a1 + k);
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        if (m < nm) {
                            const float4 v = ld4(B[f0 + m * F4] + k);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {
                                if (PAIR) {
                                    pair_mac(h[0][m], l[0][m], at(x0, kk), at(v, kk));
                                    pair_mac(h[1][m], l[1][m], at(x1, kk), at(v, kk));
                                } else {
                                    b[0][m] = fmaf(at(x0, kk), at(v, kk), b[0][m]);
                                    b[1][m] = fmaf(at(x1, kk), at(v, kk), b[1][m]);
                                }
                            }
                        }
                    }
                }
                if (!PAIR) fold_chain(h, l, b);  // leaves b at 0
            }
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = f0 + m * F4;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = r0 + i;
                float v = 0.0f;
                if (j <= r && r < rows) v = pair_value(__fsub_rn(h[i][m], b[i][m]), l[i][m]);
                S[r][j] = v;
            }
        }
    }
}

// sum_{r < nr} A[r][f] B[r][c] of two f (values at a, row stride lda) and four c (at b) as pairs.
__device__ __forceinline__ void outer_rows(float (&h)[2][4], float (&l)[2][4], const float *a, int lda, const float *b,
                                           int ldb, int nr) {
    float s[2][4] = {};
#pragma unroll 4
    for (int r = 0; r < nr; ++r) {
        const float2 x = *reinterpret_cast<const float2 *>(a + r * lda);
        const float4 y = ld4(b + r * ldb);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            abs_mac(s[0][m], x.x, at(y, m));
            abs_mac(s[1][m], x.y, at(y, m));
        }
    }
    unit_base(s, h, l);
#pragma unroll 2
    for (int r = 0; r < nr; ++r) {
        const float2 x = *reinterpret_cast<const float2 *>(a + r * lda);
        const float4 y = ld4(b + r * ldb);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            pair_mac(h[0][m], l[0][m], x.x, at(y, m));
            pair_mac(h[1][m], l[1][m], x.y, at(y, m));
        }
    }
    unit_unbase(h, s);
}

// (h, l) = sum_{r < nr} A[r][f] (w, wl)[r] (w null: 1) for the column at a.
__device__ __forceinline__ void column_sum(float &h, float &l, const float *a, int lda, const float *w, const float *wl,
                                           int nr) {
    float s = 0.0f;
#pragma unroll 4
    for (int r = 0; r < nr; ++r) abs_mac(s, a[r * lda], w ? w[r] : 1.0f);
    s = pair_base(s);
    h = s;
    l = 0.0f;
#pragma unroll 4
    for (int r = 0; r < nr; ++r) {
        const float x = a[r * lda];
        pair_mac(h, l, x, w ? w[r] : 1.0f);
        if (w) l = __fmaf_rn(x, wl[r], l);
    }
    h = __fsub_rn(h, s);
}

// Register accumulator of sum_r A[r][f] B[r][c] over every tile of a block: a thread owns TF x TC elements, the
// smallest of 2 x 4, 4 x 4, 4 x 8 that covers D x dv with 512 threads, and forms them 2 x 4 at a time: the tile's
// pairs and start values beside all the running ones.
template <int TF, int TC>
struct OuterAcc {
    float H[TF][TC], L[TF][TC];
    float zh, zl;  // thread f < D: sum_r A[r][f] w[r]
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < TF; ++i)
#pragma unroll
            for (int m = 0; m < TC; ++m) H[i][m] = L[i][m] = 0.0f;
        zh = zl = 0.0f;
    }
    // rows [0, nr); w, wl: weights of z as pairs (null: 1)
    __device__ __forceinline__ void add(const Rows &A, int D, const Rows &B, int dv, const float *w, const float *wl,
                                        int nr) {
        const int nc = (dv + TC - 1) / TC;
        const int tf = threadIdx.x / nc, tc = threadIdx.x - tf * nc;
        if (tf * TF < D) {
#pragma unroll
            for (int i = 0; i < TF; i += 2)
#pragma unroll
                for (int q = 0; q < TC; q += 4) {
                    float h[2][4], l[2][4];
                    outer_rows(h, l, A.p + tf * TF + i, A.ld, B.p + tc * TC + q, B.ld, nr);
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int m = 0; m < 4; ++m) pair_add(H[i + k][q + m], L[i + k][q + m], h[k][m], l[k][m]);
                }
        }
        if ((int)threadIdx.x < D) {
            float h, l;
            column_sum(h, l, A.p + threadIdx.x, A.ld, w, wl, nr);
            pair_add(zh, zl, h, l);
        }
    }
    // The sums of partial `slot` at S [slot][D][dv], z [slot][D], rounded; with `pairs`, high and low parts at
    // [2 slot], [2 slot + 1], so that the partials of a head are rounded once, after their sum.
    __device__ __forceinline__ void store(int D, int dv, float *S, float *z, size_t slot, bool pairs) const {
        const int nc = (dv + TC - 1) / TC;
        const int tf = threadIdx.x / nc, tc = threadIdx.x - tf * nc;
        S += slot * (pairs ? 2 : 1) * D * dv;
        z += slot * (pairs ? 2 : 1) * D;
#pragma unroll
        for (int i = 0; i < TF; ++i)
#pragma unroll
            for (int m = 0; m < TC; ++m) {
                const int f = tf * TF + i, c = tc * TC + m;
                if (f < D && c < dv) store_pair(S + f * dv + c, D * dv, H[i][m], L[i][m], pairs);
            }
        if ((int)threadIdx.x < D) store_pair(z + threadIdx.x, D, zh, zl, pairs);
    }
    static __device__ __forceinline__ void store_pair(float *p, int step, float h, float l, bool pairs) {
        const float v = pair_value(h, l);
        *p = v;
        if (pairs) p[step] = fabsf(h) < INFINITY ? __fadd_rn(__fsub_rn(h, v), l) : 0.0f;
    }
};

// S[f][c] += sum_{r < nr} A[r][f] B[r][c] and z[f] += sum_r A[r][f] (w, wl)[r] (null: 1) in shared memory, each rounded
// once.  The running state loses half an ulp per tile.
__device__ void advance_rows(const Rows &S, float *z, const Rows &A, int D, const Rows &B, int dv, const float *w,
                             const float *wl, int nr) {
    const int ng = (dv + 3) / 4, nu = ((D + 1) / 2) * ng;
    for (int u = threadIdx.x; u < nu; u += blockDim.x) {
        const int g = u / ng, f0 = 2 * g, c0 = 4 * (u - g * ng);
        float h[2][4], l[2][4];
        outer_rows(h, l, A.p + f0, A.ld, B.p + c0, B.ld, nr);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 v = ld4(S[f0 + i] + c0);
            float o[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                float H = at(v, m), L = 0.0f;
                pair_add(H, L, h[i][m], l[i][m]);
                o[m] = pair_value(H, L);
            }
            st4(S[f0 + i] + c0, make_float4(o[0], o[1], o[2], o[3]));
        }
    }
    if ((int)threadIdx.x < D) {
        float h, l, H = z[threadIdx.x], L = 0.0f;
        column_sum(h, l, A.p + threadIdx.x, A.ld, w, wl, nr);
        pair_add(H, L, h, l);
        z[threadIdx.x] = pair_value(H, L);
    }
}

// done(r, h, l) for r < rows, once per row: the pair of sum_{k < K} A[r][k] v(r, k) + sum_{j < K2(r)} A2[r][j], by
// 8 lanes of a warp.
template <typename V, typename K2, typename Done>
__device__ __forceinline__ void row_dots(const Rows &A, int rows, int K, V v, const Rows &A2, K2 k2, Done done) {
    const int lane = threadIdx.x & 7;
    for (int r0 = 0; r0 < rows; r0 += kThr / 8) {
        const int r = r0 + (int)threadIdx.x / 8;
        float h = 0.0f, l = 0.0f;
        if (r < rows) {
            for (int k = lane; k < K; k += 8) pair_mac_any(h, l, A[r][k], v(r, k));
            const int ke = k2(r);
            for (int j = lane; j < ke; j += 8) pair_mac_any(h, l, A2[r][j], 1.0f);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
            pair_add(h, l, h2, l2);
        }
        if (r < rows && lane == 0) done(r, h, l);
    }
}

// The quotient of two pairs as a pair; inv = 1 / dh.
__device__ __forceinline__ void pair_quot(float h, float l, float dh, float dl, float inv, float &qh, float &ql) {
    if (!(fabsf(inv) < INFINITY) || !(fabsf(h) < INFINITY)) {
        qh = h / dh;
        ql = 0.0f;
        return;
    }
    qh = __fmul_rn(h, inv);
    ql = __fmul_rn(__fadd_rn(__fmaf_rn(-qh, dh, h), __fmaf_rn(-qh, dl, l)), inv);
}

// A query row's normaliser and dden as pairs.  The row's terms of dphi, S dnum + z dden, cancel under a common scale
// of phi(q): a rounding of den or dden that is common to the row does not, and in fp32 these were most of the error
// of db1, dw2 and db2.  dnum is rounded element by element, and dden is formed from the rounded dnum, so that the
// cancellation holds for exactly the dnum that S is multiplied with.
struct RowPairs {
    float *dh, *dl, *inv;  // den (and 1 / dh)
    float *gh, *gl;        // dden
    __device__ __forceinline__ void set_den(int r, float h, float l, float eps) const {
        pair_mac_any(h, l, eps, 1.0f);
        const float v = pair_value(h, l);
        dh[r] = v;
        dl[r] = fabsf(h) < INFINITY ? __fadd_rn(__fsub_rn(h, v), l) : 0.0f;
        inv[r] = 1.0f / v;
    }
    // dden = -(sum_c dnum_c num_c) / den from the pair of the sum
    __device__ __forceinline__ void set_dden(int r, float h, float l) const {
        gh[r] = gl[r] = 0.0f;
        if (dh[r] == 0.0f) return;
        float qh, ql;
        pair_quot(-h, -l, dh[r], dl[r], inv[r], qh, ql);
        const float v = pair_value(qh, ql);
        gh[r] = v;
        gl[r] = fabsf(v) < INFINITY ? __fadd_rn(__fsub_rn(qh, v), ql) : 0.0f;
    }
    // rows [0, nr) of dO divided by den, each element rounded once, in place
    __device__ __forceinline__ void divide_rows(const Rows &dO, int nr, int cols) const {
        const Div by((cols + 3) / 4);
#pragma unroll 2
        for (int e = threadIdx.x; e < nr * by.n; e += blockDim.x) {
            const int r = by(e);
            float *p = dO[r] + 4 * (e - r * by.n);
            const float den = dh[r], lo = dl[r], iv = inv[r];
            float4 v = ld4(p);
            float *x = &v.x;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float qh, ql;
                pair_quot(x[k], 0.0f, den, lo, iv, qh, ql);
                x[k] = den != 0.0f ? pair_value(qh, ql) : 0.0f;
            }
            st4(p, v);
        }
    }
};
__device__ RowPairs take_row_pairs(Carve &cv, int cap) {
    RowPairs p;
    p.dh = cv.take(cap); p.dl = cv.take(cap); p.inv = cv.take(cap); p.gh = cv.take(cap); p.gl = cv.take(cap);
    return p;
}
void take_row_pairs_host(HostCarve &cv, int cap) { for (int k = 0; k < 5; ++k) cv.take(cap); }

// A unit's share of sum_c dnum_c num_c of its two rows (num: the sums of prod_nn) as pairs at P[r][2 g],
// P[r][2 g + 1], g the unit's column group; rows < nr.
__device__ __forceinline__ void unit_dots(const Rows &dnum, const Rows &P, int nr, int r0, int c0, const float (&h)[2][4],
                                          const float (&l)[2][4]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (r0 + i >= nr) continue;
        const float4 g = ld4(dnum[r0 + i] + c0);
        float ph = 0.0f, pl = 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            pair_mac_any(ph, pl, at(g, m), h[i][m]);
            pl = __fmaf_rn(at(g, m), l[i][m], pl);
        }
        *reinterpret_cast<float2 *>(P[r0 + i] + c0 / 2) = make_float2(ph, pl);
    }
}

// done(r, h, l): the sum of the ng pairs of row r < rows, by 8 lanes of a warp.
template <typename Done>
__device__ __forceinline__ void sum_unit_dots(const Rows &P, int rows, int ng, Done done) {
    const int lane = threadIdx.x & 7;
    for (int r0 = 0; r0 < rows; r0 += kThr / 8) {
        const int r = r0 + (int)threadIdx.x / 8;
        float h = 0.0f, l = 0.0f;
        if (r < rows)
            for (int g = lane; g < ng; g += 8) pair_add(h, l, P[r][2 * g], P[r][2 * g + 1]);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
            pair_add(h, l, h2, l2);
        }
        if (r < rows && lane == 0) done(r, h, l);
    }
}

// The quotient of a pair by den, rounded once; inv = 1 / den.
__device__ __forceinline__ float pair_div(float h, float l, float den, float inv) {
    if (!(fabsf(inv) < INFINITY) || !(fabsf(h) < INFINITY)) return h / den;
    const float q = __fmul_rn(h, inv);
    return __fmaf_rn(__fadd_rn(__fmaf_rn(-q, den, h), l), inv, q);
}

// Up to four consecutive values to p (vec: all four, p aligned to their size).
__device__ __forceinline__ void store4(float *p, const float (&v)[4], int n, bool vec) {
    if (vec) {
        st4(p, make_float4(v[0], v[1], v[2], v[3]));
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (m < n) p[m] = v[m];
    }
}
__device__ __forceinline__ void store4(__nv_bfloat16 *p, const float (&v)[4], int n, bool vec) {
    if (vec) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
        uint2 w;
        w.x = *reinterpret_cast<unsigned *>(&a);
        w.y = *reinterpret_cast<unsigned *>(&b);
        *reinterpret_cast<uint2 *>(p) = w;
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (m < n) io_store(p + m, v[m]);
    }
}
template <typename IO>
__device__ __forceinline__ bool vec_store(const IO *p, int w) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && w % 4 == 0;
}

// Zeros to rows [r0, r1) of w elements.
template <typename IO>
__device__ void zero_rows(IO *p, int r0, int r1, int w) {
    for (int64_t e = (int64_t)r0 * w + threadIdx.x; e < (int64_t)r1 * w; e += blockDim.x) io_store(p + e, 0.0f);
}

__device__ void zero_words(float *p, int n) {
    for (int e = threadIdx.x; e < n; e += blockDim.x) p[e] = 0.0f;
}

// The fp32 state [D][dv] into rows of shared memory (zeros in the pads), z beside it.
__device__ void load_state(const Rows &S, float *z, const float *gS, const float *gz, int D, int dv) {
    const int Dp = (D + 3) & ~3;
    if (dv % 4 == 0 && (reinterpret_cast<uintptr_t>(gS) & 15) == 0) {
        const Div q(dv / 4);
#pragma unroll 4
        for (int e = threadIdx.x; e < D * q.n; e += blockDim.x) {
            const int f = q(e), c = 4 * (e - f * q.n);
            st4(S[f] + c, ld4(gS + 4 * e));
        }
    } else {
        const int wp = (dv + 3) & ~3;
        for (int e = threadIdx.x; e < D * wp; e += blockDim.x) {
            const int f = e / wp, c = e - f * wp;
            S[f][c] = c < dv ? gS[f * dv + c] : 0.0f;
        }
    }
    for (int e = threadIdx.x; e < (Dp - D) * S.ld; e += blockDim.x) S[D][e] = 0.0f;
    for (int f = threadIdx.x; f < D; f += blockDim.x) z[f] = gz[f];
}

// ---------------------------------------------------------------------------
// Backward through phi for a tile.

// dW of a block: a thread owns rows i0, i0 + 1 and columns c0 .. c0 + 3 of the M x d matrix, over every G-th row
// of the tiles (G = 512 / tiles of 2 x 4).  The sums cancel and run from zero over the whole block, so every
// product is added exactly whatever its size: with pair_mac they kept 40 bits of sum |dU x| and not 46.
struct GradTile {
    float h[2][4], l[2][4];
    float bh, bl;  // thread i < M: db
};

__device__ __forceinline__ void grad_zero(GradTile &g) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int m = 0; m < 4; ++m) g.h[i][m] = g.l[i][m] = 0.0f;
    g.bh = g.bl = 0.0f;
}

__host__ __device__ inline int du_stride(int M) { return (M + 3) & ~3; }

// An fp64 value from a finite fp32 one, by moving bits: the conversion instruction runs at the fp64 rate.
// Zeros and subnormals (no implicit bit to move) take the conversion.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (e == 0u || e == 255u) return (double)x;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// From dLoss/dphi (dPhi) of rows [0, nr): the histogram of the channel-MLP gradients (or those gradients, with
// another activation) and the variants' gradients into the fp64 sums at hist / gvar by L2 reductions, dU
// (stride du_stride(M)), and dU^T X into g.  The caller synchronises before and after.
__device__ void phi_backward_rows(const TableLayout &lay, const SmemPhi &s, const Rows &X, int nr, int cap,
                                  const Rows &Phi, const Rows &dPhi, const float *sU, const int *sJ, float *sdU,
                                  double *hist, double *gvar, GradTile &g) {
    const int M = lay.M, L = lay.L, d = lay.d;
    const float fl = channel_floor(lay);
    const bool ev = lay.env || lay.coef;
    const float sc = phi_scale(lay);
    const int du_ld = du_stride(M);
    if (ev) {
        // phi = e_l phi0 with e_l = h_l(x) c_l per row: dLoss/de_l = sum over the projections of dPhi phi0
        __syncthreads();  // the row scratch of an earlier call is no longer read
        gate_rows(lay, s, X.p, X.ld, nr);
        for (int e = threadIdx.x; e < nr * L; e += blockDim.x) {
            const int r = e / L, l = e - r * L;
            double acc = 0.0;
            for (int i = 0; i < M; ++i)
                acc = fma((double)dPhi[r][i * L + l],
                          (double)channel_value(lay, s, sU[r * M + i], sJ[r * M + i], l, fl), acc);
            s.dE[e] = (float)acc;
        }
        __syncthreads();
    }
    // per sample (row, projection): g_l = dLoss/dphi0_l on an active output; dU = sum_l g_l dphi0_l/du
    const Div byM(M);
    for (int e = threadIdx.x; e < nr * M; e += blockDim.x) {
        const int r = byM(e), i = e - r * M;
        const float u = sU[e];
        float uh = 0.0f, ul = 0.0f;
        float *gp = dPhi[r] + i * L;
        const float *ph = Phi[r] + i * L;
        if (L == 8 && !lay.act && !ev) {
            const int j = sJ[e];
            const float *ab = s.AB + j * ab_stride(lay);
            double *hj = hist + (size_t)j * 16;
            const double u64 = widen(u);
            const float4 g0 = ld4(gp), g1 = ld4(gp + 4), p0 = ld4(ph), p1 = ld4(ph + 4);
#pragma unroll
            for (int l = 0; l < 8; ++l) {
                const float gl = at(l < 4 ? g0 : g1, l & 3);
                if (at(l < 4 ? p0 : p1, l & 3) > fl && gl != 0.0f) {  // outer ReLU on (always, for signed outputs)
                    pair_mac_any(uh, ul, gl, ab_pair(ab, l).x);
                    const double gw = widen(gl);
                    atomicAdd(hj + 2 * l, gw);
                    atomicAdd(hj + 2 * l + 1, gw * u64);  // exact product
                }
            }
        } else if (!lay.act) {
            const int j = sJ[e];
            const float *ab = s.AB + j * ab_stride(lay);
            double *hj = hist + (size_t)j * L * 2;
            const double u64 = widen(u);
            for (int l = 0; l < L; ++l) {
                const float2 p = ab_pair(ab, l);
                const bool on = ev ? fmaf(p.x, u, p.y) > fl : ph[l] > fl;
                if (on) {  // outer ReLU on (always, for signed outputs)
                    if (ev) {
                        const double gl = (double)gp[l] * (double)s.E[r * L + l];
                        const float g1 = (float)gl, g2 = (float)(gl - (double)g1);
                        pair_mac_any(uh, ul, g1, p.x);
                        ul = fmaf(g2, p.x, ul);
                        if (gl != 0.0) {
                            atomicAdd(hj + 2 * l, gl);
                            atomicAdd(hj + 2 * l + 1, gl * u64);
                        }
                    } else if (gp[l] != 0.0f) {
                        pair_mac_any(uh, ul, gp[l], p.x);
                        const double gl = widen(gp[l]);
                        atomicAdd(hj + 2 * l, gl);
                        atomicAdd(hj + 2 * l + 1, gl * u64);  // exact product
                    }
                }
            }
        } else {
            // direct evaluation: G_l = dLoss/dy_l (scale and gate folded in), kept in dPhi for the unit sums
            for (int l = 0; l < L; ++l) {
                float dydu;
                const float y = channel_direct(lay, s, l, u, &dydu);
                float G = 0.0f;
                if (sc * y > fl) G = (ev ? gp[l] * s.E[r * L + l] : gp[l]) * sc;
                pair_mac_any(uh, ul, G, dydu);
                gp[l] = G;
            }
        }
        sdU[r * du_ld + i] = pair_value(uh, ul);
    }
    for (int e = threadIdx.x; e < (cap - nr) * du_ld; e += blockDim.x) sdU[nr * du_ld + e] = 0.0f;
    if (du_ld != M)
        for (int e = threadIdx.x; e < nr * (du_ld - M); e += blockDim.x)
            sdU[(e / (du_ld - M)) * du_ld + M + e % (du_ld - M)] = 0.0f;
    __syncthreads();
    if (lay.act) {
        // MLP gradients unit by unit over the tile's samples, into [dw2 (L*hid) | dw1 (P) | db1 (P) | db2 (L)]
        const int hid = lay.hid, P = lay.P, ns = nr * M;
        double *dw2 = hist, *dw1 = hist + L * hid, *db1 = dw1 + P, *db2 = db1 + P;
        if (!lay.shared) {
            for (int q = threadIdx.x; q < P; q += blockDim.x) {
                const int l = q / hid;
                const float w1 = s.w1[q], b1 = s.b1[q], w2 = s.w2[q];
                double a2 = 0.0, a1 = 0.0, a0 = 0.0;
                for (int e = 0; e < ns; ++e) {
                    const int r = e / M, i = e - r * M;
                    const float G = dPhi[r][i * L + l];
                    if (G == 0.0f) continue;
                    float da;
                    const float av = act_eval(lay.act, fmaf(w1, sU[e], b1), da);
                    a2 = fma((double)G, (double)av, a2);
                    const double dh = (double)G * (double)w2 * (double)da;
                    a0 += dh;
                    a1 = fma(dh, (double)sU[e], a1);
                }
                atomicAdd(dw2 + q, a2); atomicAdd(dw1 + q, a1); atomicAdd(db1 + q, a0);
            }
        } else {
            // the block's threads take every unit as often as they go into it, each group every Gu-th sample: 64 units on
            // 64 threads were a chain of all the tile's samples (backward pass of 24 heads of 300 fp32 rows, d = 64, tanh:
            // 2678 -> 1466 us; 1660 with tiles of 16 rows on three times the blocks)
            const int Gu = kThr / hid, k = threadIdx.x % hid, e0 = threadIdx.x / hid;
            if (e0 < Gu) {
                const float w1 = s.w1[k], b1 = s.b1[k];
                double a2[kMaxL] = {}, a1 = 0.0, a0 = 0.0;
                for (int e = e0; e < ns; e += Gu) {
                    const int r = e / M, i = e - r * M;
                    float da;
                    const float av = act_eval(lay.act, fmaf(w1, sU[e], b1), da);
                    double dsum = 0.0;  // sum over the channels of G_l w2_lk
                    for (int l = 0; l < L; ++l) {
                        const float G = dPhi[r][i * L + l];
                        a2[l] = fma((double)G, (double)av, a2[l]);
                        dsum = fma((double)G, (double)s.w2[l * hid + k], dsum);
                    }
                    const double dh = dsum * (double)da;
                    a0 += dh;
                    a1 = fma(dh, (double)sU[e], a1);
                }
                for (int l = 0; l < L; ++l) atomicAdd(dw2 + l * hid + k, a2[l]);
                atomicAdd(dw1 + k, a1); atomicAdd(db1 + k, a0);
            }
        }
        for (int l = threadIdx.x; l < L; l += blockDim.x) {
            double acc = 0.0;
            for (int e = 0; e < ns; ++e) acc += (double)dPhi[e / M][(e % M) * L + l];
            atomicAdd(db2 + l, acc);
        }
    }
    if (ev) {
        // Bank+Coef: dc_l = sum over rows of dLoss/de_l h_l; the gate: dLoss/d(We_l . x + be_l) = dLoss/de_l c_l h (1 - h)
        // (kept in dE for store_dx_rows' dX term), then dWe = sum_r that x_r^T and dbe = sum_r that
        double *dWe = gvar, *dbe = gvar + L * d, *dcoef = gvar + (lay.env ? L * d + L : 0);
        if (lay.coef)
            for (int l = threadIdx.x; l < L; l += blockDim.x) {
                double acc = 0.0;
                for (int r = 0; r < nr; ++r) acc = fma((double)s.dE[r * L + l], (double)s.H[r * L + l], acc);
                atomicAdd(dcoef + l, acc);
            }
        if (lay.env) {
            __syncthreads();  // dE read above
            for (int e = threadIdx.x; e < nr * L; e += blockDim.x) {
                const float h = s.H[e], c = lay.coef ? s.coef[e % L] : 1.0f;
                s.dE[e] = s.dE[e] * c * h * (1.0f - h);
            }
            __syncthreads();
            for (int q = threadIdx.x; q < L * d; q += blockDim.x) {
                const int l = q / d, c = q - l * d;
                double acc = 0.0;
                for (int r = 0; r < nr; ++r) acc = fma((double)s.dE[r * L + l], (double)X[r][c], acc);
                atomicAdd(dWe + q, acc);
            }
            for (int l = threadIdx.x; l < L; l += blockDim.x) {
                double acc = 0.0;
                for (int r = 0; r < nr; ++r) acc += (double)s.dE[r * L + l];
                atomicAdd(dbe + l, acc);
            }
        }
    }
    const int nc = (d + 3) / 4, nt = ((M + 1) / 2) * nc;  // at most 512
    const int G = kThr / nt, grp = threadIdx.x / nt, t = threadIdx.x - grp * nt;
    if (grp < G) {
        const int i0 = 2 * (t / nc), c0 = 4 * (t % nc);
        for (int r = grp; r < nr; r += G) {
            const float2 a = *reinterpret_cast<const float2 *>(sdU + r * du_ld + i0);
            const float4 x = ld4(X[r] + c0);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                pair_mac_any(g.h[0][m], g.l[0][m], a.x, at(x, m));
                pair_mac_any(g.h[1][m], g.l[1][m], a.y, at(x, m));
            }
        }
    }
    if ((int)threadIdx.x < M)
        for (int r = 0; r < nr; ++r) pair_mac_any(g.bh, g.bl, sdU[r * du_ld + threadIdx.x], 1.0f);
}

// dX = dU W (+ the envelope gate's term sum_l dLoss/d(We_l . x + be_l) We_l, kept in dE by phi_backward_rows).
template <typename IO>
__device__ void store_dx_rows(const TableLayout &lay, const SmemPhi &s, const float *sdU, int nr, IO *dX) {
    const int M = lay.M, d = lay.d, L = lay.L, ldw = row_stride(d), du_ld = du_stride(M), nc = (d + 3) / 4;
    const bool vec = (reinterpret_cast<uintptr_t>(dX) & 15) == 0 && d % 4 == 0;
    const Div by(nc);
    for (int e = threadIdx.x; e < nr * nc; e += blockDim.x) {
        const int r = by(e), c0 = 4 * (e - r * nc);
        float acc[4] = {};
#pragma unroll 4
        for (int i = 0; i < M; ++i) {
            const float4 w = ld4(s.W + i * ldw + c0);
            const float du = sdU[r * du_ld + i];
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[m] = fmaf(du, at(w, m), acc[m]);
        }
        if (lay.env)
            for (int l = 0; l < L; ++l)
                for (int m = 0; m < 4; ++m)
                    if (c0 + m < d) acc[m] = fmaf(s.dE[r * L + l], s.We[l * d + c0 + m], acc[m]);
        store4(dX + (size_t)r * d + c0, acc, vec ? 4 : d - c0 < 4 ? d - c0 : 4, vec);
    }
}

// dW and db of the block into its slot [dW | db]: the groups' pairs, added in a tree of fixed shape in `scratch`
// (kGradScratch floats of shared memory that nothing else uses any more).  Called by every thread.
constexpr int kGradScratch = 2 * 8 * kThr;
__device__ void store_grad_tile(const TableLayout &lay, GradTile &g, float *scratch, double *slot) {
    const int M = lay.M, d = lay.d, nc = (d + 3) / 4, nt = ((M + 1) / 2) * nc;
    const int G = kThr / nt, grp = threadIdx.x / nt, t = threadIdx.x - grp * nt;
    float2 *sc = reinterpret_cast<float2 *>(scratch);
    __syncthreads();
    int s = 1;
    while (s < G) s *= 2;
    for (s /= 2; s >= 1; s /= 2) {  // groups s .. 2 s - 1 hand their pairs to groups 0 .. s - 1
        if (grp >= s && grp < 2 * s)
#pragma unroll
            for (int k = 0; k < 8; ++k) sc[k * kThr + threadIdx.x] = make_float2(g.h[k / 4][k % 4], g.l[k / 4][k % 4]);
        __syncthreads();
        if (grp < s && grp + s < G)
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float2 v = sc[k * kThr + threadIdx.x + s * nt];
                pair_add(g.h[k / 4][k % 4], g.l[k / 4][k % 4], v.x, v.y);
            }
    }
    if (grp == 0) {
        const int i0 = 2 * (t / nc), c0 = 4 * (t % nc);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (i0 + k / 4 < M && c0 + k % 4 < d)
                slot[(i0 + k / 4) * d + c0 + k % 4] = pair_double(g.h[k / 4][k % 4], g.l[k / 4][k % 4]);
    }
    if ((int)threadIdx.x < M) slot[M * d + threadIdx.x] = pair_double(g.bh, g.bl);
}

}  // namespace
}  // namespace simt
}  // namespace luna
