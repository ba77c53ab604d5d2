// Generic CUDA-core kernels of the LUNA attention path.
//
// They serve the fp32 I/O path (the parity bar there is 1e-4 relative, which
// rules out bf16 tensor-core operands) and every shape the tensor-core path
// does not specialise.  A block owns a range of rows of one head and walks it
// in tiles of up to 64 rows (luna_tile.cuh); the statistics, normalisers and
// feature gradients are pairs of floats rounded once.  Every cross-block sum of
// S, z, dS, dz, dW and db runs in a fixed order; the channel MLPs' gradients come
// from fp64 histograms filled by L2 reductions, whose order varies in the last
// bits of the fp64 sums.
//
// Measured at 8 x 12 heads of 512 fp32 rows, d = D = 64 (us; before: fp64 sums in
// tiles of 16 or 32 rows, 64 of 256 threads in the outer products):
//   key statistics 1402 -> 135, queries 161 -> 53, backward queries 3848 -> 336,
//   backward keys 1451 -> 162, gradient sum 30 -> 14.
// The fma pipe is 33 to 38 % busy and the issue slots half: what is left is
// barriers between a tile's phases, the feature map's gathers and the histogram.
#include <math.h>

#include "luna_prof.cuh"
#include "luna_tile.cuh"

namespace luna {
namespace {
using namespace simt;

// ---------------------------------------------------------------------------
// feature map alone

template <typename IO>
__global__ void __launch_bounds__(kThreads) k_featmap(TableLayout lay, const char *table, const IO *X, int64_t rows,
                                                      float *Phi) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    SmemPhi s = carve_phi_tile(cv, lay, 0);
    if (!carve_fits(cv, smem)) return;
    load_phi_tile(s, lay, table);
    __syncthreads();
    const unsigned short *sB = reinterpret_cast<const unsigned short *>(s.T + kSearchT);
    const int M = lay.M, L = lay.L, d = lay.d, D = lay.D, ldw = row_stride(d);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < rows * M; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / M;
        const int i = (int)(e - r * M);
        const IO *x = X + r * d;
        const float *w = s.W + i * ldw;
        float u = s.b[i];
        for (int c = 0; c < d; ++c) u = fmaf(w[c], io_load(x + c), u);
        const int j = interval_bucketed(s.T, sB, u);
        const float *ab = s.AB + j * ab_stride(lay);
        float *out = Phi + r * D + i * L;
        for (int l = 0; l < L; ++l) {
            const float2 p = ab_pair(ab, l);
            out[l] = fmaxf(fmaf(p.x, u, p.y), channel_floor(lay));
        }
    }
}

// The feature map of the variants (a non-ReLU activation, the envelope gate, Bank+Coef): blocks walk tiles of
// kPhiRows rows through the generic tile helper.
template <typename IO>
__global__ void __launch_bounds__(kThreads) k_featmap_var(TableLayout lay, const char *table, const IO *X,
                                                          int64_t rows, float *Phi) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    SmemPhi s = carve_phi_tile(cv, lay, kPhiRows);
    const Rows sX = take_rows(cv, kPhiRows, lay.d), sPhi = take_rows(cv, kPhiRows, lay.D);
    if (!carve_fits(cv, smem)) return;
    load_phi_tile(s, lay, table);
    for (int64_t t0 = (int64_t)blockIdx.x * kPhiRows; t0 < rows; t0 += (int64_t)gridDim.x * kPhiRows) {
        const int nr = (int)(rows - t0 < kPhiRows ? rows - t0 : kPhiRows);
        __syncthreads();
        load_tile(sX, X + t0 * lay.d, nr, lay.d, kPhiRows);
        __syncthreads();
        phi_rows(lay, s, sX, nr, kPhiRows, sPhi, nullptr, nullptr);
        __syncthreads();
        for (int e = threadIdx.x; e < nr * lay.D; e += blockDim.x) Phi[t0 * lay.D + e] = sPhi[e / lay.D][e % lay.D];
    }
}

// ---------------------------------------------------------------------------
// The attention kernels.  Shared memory of each: the same arrays on the device (Carve) and on the host (HostCarve).

// ---------------------------------------------------------------------------
// key statistics S = sum_j phi(k_j) v_j^T, z = sum_j phi(k_j)   (Sec. 4: S_KV, S_K1)

template <typename IO, int TF, int TC>
__global__ void __launch_bounds__(kThr, 1) k_keystats(AttnArgs a, int cap, int pairs, int finish) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    const Rows sK = take_rows(cv, cap, a.d), sV = take_rows(cv, cap, a.dv), sPhi = take_rows(cv, cap, a.D);
    cv.take(kSlack);
    if (!carve_fits(cv, smem)) return;
    load_phi_tile(s, lay, a.table);

    const int bh = blockIdx.y, split = blockIdx.x;
    const int len = head_length(a.lengths, bh / a.H, a.n);
    const int r0 = split * a.rows_per_split;
    const int r1 = min(len, r0 + a.rows_per_split);
    const IO *K = static_cast<const IO *>(a.K) + head_rows(a, bh) * a.d;
    const IO *V = static_cast<const IO *>(a.V) + head_rows(a, bh) * a.dv;
    OuterAcc<TF, TC> acc;
    acc.zero();
    for (int t0 = r0; t0 < r1; t0 += cap) {
        const int nr = min(cap, r1 - t0);
        __syncthreads();
        load_tile(sK, K + (size_t)t0 * a.d, nr, a.d, cap);
        load_tile(sV, V + (size_t)t0 * a.dv, nr, a.dv, cap);
        __syncthreads();
        phi_rows(lay, s, sK, nr, cap, sPhi, nullptr, nullptr);
        __syncthreads();
        acc.add(sPhi, a.D, sV, a.dv, nullptr, nullptr, nr);
    }
    const size_t slot = (size_t)bh * a.nsplit + split;
    acc.store(a.D, a.dv, a.S_part, a.z_part, slot, pairs != 0);
    if (finish && last_arrival(a.counters + bh, a.nsplit)) {
        if (a.seg_S) {  // causal: exclusive prefix at every segment start, total in slot nsplit
            exclusive_scan(a.S_part + (size_t)bh * a.nsplit * a.D * a.dv, a.nsplit, a.D * a.dv,
                           a.seg_S + head_state(a, bh) * (a.nsplit + 1) * a.D * a.dv, false);
            exclusive_scan(a.z_part + (size_t)bh * a.nsplit * a.D, a.nsplit, a.D,
                           a.seg_z + head_state(a, bh) * (a.nsplit + 1) * a.D, false);
        } else {
            const int np = pairs ? 2 * a.nsplit : a.nsplit;
            ordered_sum(a.S_part + (size_t)bh * np * a.D * a.dv, np, a.D * a.dv,
                        a.S_fin + head_state(a, bh) * a.D * a.dv);
            ordered_sum(a.z_part + (size_t)bh * np * a.D, np, a.D, a.z_fin + head_state(a, bh) * a.D);
        }
        if (threadIdx.x == 0) a.counters[bh] = 0;
    }
}

// ---------------------------------------------------------------------------
// query side: O_i = phi(q_i)^T S / (phi(q_i)^T z + eps)   (Eq. kernel-attn)

template <typename IO>
__global__ void __launch_bounds__(kThr, 1) k_query(AttnArgs a, int cap, int rows_per_block) {
    extern __shared__ __align__(16) float smem[];
    const int bh = blockIdx.y;
    const int b0 = blockIdx.x * rows_per_block, b1 = min(a.n, b0 + rows_per_block);
    const int len = head_length(a.lengths, bh / a.H, a.n);
    IO *O = static_cast<IO *>(a.O) + head_rows(a, bh) * a.dv;
    zero_rows(O, max(b0, len), b1, a.dv);  // padded rows
    if (b0 >= len) return;
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, dv = a.dv, Dp = (D + 3) & ~3;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    const Rows sS = take_rows(cv, Dp, dv);
    float *sz = cv.take(D);
    const Rows sQ = take_rows(cv, cap, a.d), sPhi = take_rows(cv, cap, D);
    float *sden = cv.take(cap);
    if (!carve_fits(cv, smem)) return;
    load_phi_tile(s, lay, a.table);
    load_state(sS, sz, a.S_fin + head_state(a, bh) * D * dv, a.z_fin + head_state(a, bh) * D, D, dv);
    const IO *Q = static_cast<const IO *>(a.Q) + head_rows(a, bh) * a.d;
    const Rows none{};
    const bool vec = vec_store(O, dv);
    const int e1 = min(b1, len);
    for (int t0 = b0; t0 < e1; t0 += cap) {
        const int nr = min(cap, e1 - t0);
        __syncthreads();
        load_tile(sQ, Q + (size_t)t0 * a.d, nr, a.d, cap);
        __syncthreads();
        phi_rows(lay, s, sQ, nr, cap, sPhi, nullptr, nullptr);
        __syncthreads();
        row_dots(sPhi, nr, D, [&](int, int f) { return sz[f]; }, none, [](int) { return 0; },
                 [&](int r, float h, float l) {
                     pair_mac_any(h, l, a.eps, 1.0f);
                     sden[r] = pair_value(h, l);
                 });
        __syncthreads();
        prod_nn_plain(sPhi, nr, sS, Dp, dv, [&](int r0, int c0, const float (&h)[2][4]) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (r0 + i >= nr) continue;
                const float den = sden[r0 + i];
                float o[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) o[m] = den != 0.0f ? h[i][m] / den : 0.0f;
                store4(O + (size_t)(t0 + r0 + i) * dv + c0, o, dv - c0, vec);
            }
        });
    }
}

// query side of the backward pass (non-causal):
//   dnum_i = do_i / den_i,  dden_i = -(do_i . o_i) / den_i
//   dphi(q_i) = S dnum_i + z dden_i,  dS += phi(q_i) dnum_i^T,  dz += phi(q_i) dden_i
// den, the sum dnum_i . num_i and dden are pairs (RowPairs), dphi is a pair rounded once.
template <typename IO, int TF, int TC>
__global__ void __launch_bounds__(kThr, 1) k_bwd_query(AttnArgs a, int cap, int pairs, int finish) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, dv = a.dv, d = a.d, M = a.M, Dp = (D + 3) & ~3, dvp = (dv + 3) & ~3;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    float *tiles = cv.p;
    const Rows sS = take_rows(cv, Dp, dv);
    float *sz = cv.take(Dp);
    const Rows sQ = take_rows(cv, cap, d), sdO = take_rows(cv, cap, dv), sPhi = take_rows(cv, cap, D);
    Rows sP{cv.take(cap * max(row_stride(dv), row_stride(D))), row_stride(dv)};  // parts of dnum . num, then dphi(q_i)
    const Rows sdPhi{sP.p, row_stride(D)};
    const RowPairs rp = take_row_pairs(cv, cap);
    float *sU = cv.take(cap * M);
    int *sJ = reinterpret_cast<int *>(cv.take(cap * M));
    float *sdU = cv.take(cap * du_stride(M));
    cv.take(kSlack);
    if (!carve_fits(cv, smem)) return;
    zero_words(tiles, (int)(cv.p - tiles));
    load_phi_tile(s, lay, a.table);
    const int bh = blockIdx.y, split = blockIdx.x;
    const size_t slot = (size_t)bh * a.nsplit_b + split;
    double *hist = a.gh + (slot % a.gh_n) * (a.gsize - M * d - M);
    __syncthreads();
    load_state(sS, sz, a.S_fin + head_state(a, bh) * D * dv, a.z_fin + head_state(a, bh) * D, D, dv);

    const int len = head_length(a.lengths, bh / a.H, a.n);
    const int r0 = split * a.rows_per_split_b;
    const int rend = min(a.n, r0 + a.rows_per_split_b);
    const int r1 = min(len, rend);
    const IO *Q = static_cast<const IO *>(a.Q) + head_rows(a, bh) * d;
    const IO *dO = static_cast<const IO *>(a.dO) + head_rows(a, bh) * dv;
    IO *dQ = static_cast<IO *>(a.dQ) + head_rows(a, bh) * d;
    zero_rows(dQ, max(r0, len), rend, d);  // padded rows of this range receive zero gradients

    const Rows none{};
    OuterAcc<TF, TC> acc;
    acc.zero();
    GradTile g;
    grad_zero(g);
    for (int t0 = r0; t0 < r1; t0 += cap) {
        const int nr = min(cap, r1 - t0);
        __syncthreads();
        load_tile(sQ, Q + (size_t)t0 * d, nr, d, cap);
        load_tile(sdO, dO + (size_t)t0 * dv, nr, dv, cap);
        __syncthreads();
        phi_rows(lay, s, sQ, nr, cap, sPhi, sU, sJ);
        __syncthreads();
        row_dots(sPhi, nr, D, [&](int, int f) { return sz[f]; }, none, [](int) { return 0; },
                 [&](int r, float h, float l) { rp.set_den(r, h, l, a.eps); });
        __syncthreads();
        rp.divide_rows(sdO, nr, dv);  // dnum in place
        __syncthreads();
        prod_nn(sPhi, nr, sS, Dp, dv, none, none, [&](int q0, int c0, const float (&h)[2][4], const float (&l)[2][4]) {
            unit_dots(sdO, sP, nr, q0, c0, h, l);
        });
        __syncthreads();
        sum_unit_dots(sP, nr, dvp / 4, [&](int r, float h, float l) { rp.set_dden(r, h, l); });
        __syncthreads();
        acc.add(sPhi, D, sdO, dv, rp.gh, rp.gl, nr);
        prod_nt<kNone>(sdO, nr, sS, D, dvp, none, none, 0,
                       [&](int r, int f, float &h, float &l) {
                           if (r < nr) {
                               pair_mac(h, l, sz[f], rp.gh[r]);
                               l = __fmaf_rn(sz[f], rp.gl[r], l);
                           }
                       },
                       [&](int r, int f, float h, float l) {
                           if (r < nr) sdPhi[r][f] = pair_value(h, l);
                       });
        __syncthreads();
        phi_backward_rows(lay, s, sQ, nr, cap, sPhi, sdPhi, sU, sJ, sdU, hist, hist + mlp_words(lay), g);
        store_dx_rows(lay, s, sdU, nr, dQ + (size_t)t0 * d);
    }
    acc.store(D, dv, a.dS_part, a.dz_part, slot, pairs != 0);
    store_grad_tile(lay, g, smem, a.gw + slot * (M * d + M));
    if (finish && last_arrival(a.counters + a.B * a.H + bh, a.nsplit_b)) {
        const int np = pairs ? 2 * a.nsplit_b : a.nsplit_b;
        ordered_sum(a.dS_part + (size_t)bh * np * D * dv, np, D * dv, a.dS_fin + (size_t)bh * D * dv);
        ordered_sum(a.dz_part + (size_t)bh * np * D, np, D, a.dz_fin + (size_t)bh * D);
        if (threadIdx.x == 0) a.counters[a.B * a.H + bh] = 0;
    }
}

// key side of the backward pass (non-causal):
//   dv_j = dS^T phi(k_j),  dphi(k_j) = dS v_j + dz
template <typename IO>
__global__ void __launch_bounds__(kThr, 1) k_bwd_key(AttnArgs a, int cap) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, dv = a.dv, d = a.d, M = a.M, Dp = (D + 3) & ~3, dvp = (dv + 3) & ~3;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    float *tiles = cv.p;
    const Rows sdS = take_rows(cv, Dp, dv);
    float *sdz = cv.take(Dp);
    const Rows sK = take_rows(cv, cap, d), sV = take_rows(cv, cap, dv), sPhi = take_rows(cv, cap, D);
    const Rows sdPhi = take_rows(cv, cap, D);
    float *sU = cv.take(cap * M);
    int *sJ = reinterpret_cast<int *>(cv.take(cap * M));
    float *sdU = cv.take(cap * du_stride(M));
    if (!carve_fits(cv, smem)) return;
    zero_words(tiles, (int)(cv.p - tiles));
    load_phi_tile(s, lay, a.table);
    const int bh = blockIdx.y, split = blockIdx.x;
    const size_t slot = (size_t)bh * a.nsplit_b + split;
    double *hist = a.gh + (slot % a.gh_n) * (a.gsize - M * d - M);
    __syncthreads();
    load_state(sdS, sdz, a.dS_fin + (size_t)bh * D * dv, a.dz_fin + (size_t)bh * D, D, dv);

    const int len = head_length(a.lengths, bh / a.H, a.n);
    const int r0 = split * a.rows_per_split_b;
    const int rend = min(a.n, r0 + a.rows_per_split_b);
    const int r1 = min(len, rend);
    const IO *K = static_cast<const IO *>(a.K) + head_rows(a, bh) * d;
    const IO *V = static_cast<const IO *>(a.V) + head_rows(a, bh) * dv;
    IO *dK = static_cast<IO *>(a.dK) + head_rows(a, bh) * d;
    IO *dV = static_cast<IO *>(a.dV) + head_rows(a, bh) * dv;
    zero_rows(dK, max(r0, len), rend, d);
    zero_rows(dV, max(r0, len), rend, dv);

    const Rows none{};
    const bool vec = vec_store(dV, dv);
    GradTile g;
    grad_zero(g);
    for (int t0 = r0; t0 < r1; t0 += cap) {
        const int nr = min(cap, r1 - t0);
        __syncthreads();
        load_tile(sK, K + (size_t)t0 * d, nr, d, cap);
        load_tile(sV, V + (size_t)t0 * dv, nr, dv, cap);
        __syncthreads();
        phi_rows(lay, s, sK, nr, cap, sPhi, sU, sJ);
        __syncthreads();
        prod_nn_plain(sPhi, nr, sdS, Dp, dv, [&](int q0, int c0, const float (&h)[2][4]) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (q0 + i < nr) store4(dV + (size_t)(t0 + q0 + i) * dv + c0, h[i], dv - c0, vec);
        });
        prod_nt<kNone>(sV, nr, sdS, D, dvp, none, none, 0, [&](int, int f, float &h, float &) { h = sdz[f]; },
                       [&](int r, int f, float h, float l) {
                           if (r < nr) sdPhi[r][f] = pair_value(h, l);
                       });
        __syncthreads();
        phi_backward_rows(lay, s, sK, nr, cap, sPhi, sdPhi, sU, sJ, sdU, hist, hist + mlp_words(lay), g);
        store_dx_rows(lay, s, sdU, nr, dK + (size_t)t0 * d);
    }
    store_grad_tile(lay, g, smem, a.gw + (a.gw_n / 2 + slot) * (M * d + M));
}

// ---------------------------------------------------------------------------
// The partials of every head summed (or scanned) in order, one element per thread with eight loads in flight.

__global__ void __launch_bounds__(256) k_part_reduce(PartReduce mode, int np, int nS, int nz, const float *S_part,
                                                     const float *z_part, float *S, float *z, size_t S_step,
                                                     size_t z_step, int hs_mul) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    const bool isz = e >= nS;
    if (isz) e -= nS;
    const int count = isz ? nz : nS;
    if (e >= count) return;
    const float *p = (isz ? z_part : S_part) + (size_t)blockIdx.y * np * count + e;
    float *out = (isz ? z + (size_t)blockIdx.y * hs_mul * z_step : S + (size_t)blockIdx.y * hs_mul * S_step) + e;
    double t = 0.0;
    for (int p0 = 0; p0 < np; p0 += 8) {
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int q = p0 + k;
            v[k] = q < np ? __ldcg(p + (size_t)(mode == kScanDown ? np - 1 - q : q) * count) : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int q = p0 + k;
            if (q >= np) break;
            if (mode != kSum) out[(size_t)(mode == kScanDown ? np - 1 - q : q) * count] = (float)t;
            t += (double)v[k];
        }
    }
    if (mode == kSum) *out = (float)t;
    else if (mode == kScanUp) out[(size_t)np * count] = (float)t;
}

// ---------------------------------------------------------------------------
// parameter gradients: ordered sum of the per-block partials, then the
// channel-MLP gradients from the interval histogram.
//   With g = dLoss/dPhi on active outputs, m0[j][l] = sum g, m1[j][l] = sum g*u
//   over samples falling in interval j; for hidden unit (l,k) active on the
//   intervals A_k:  G0 = sum_{j in A_k} m0, G1 = sum_{j in A_k} m1 and
//     dw2 = (w1 G1 + b1 G0)/sqrt(M), dw1 = w2 G1/sqrt(M), db1 = w2 G0/sqrt(M),
//     db2 = sum_j m0 / sqrt(M).

// Compensated (Neumaier) fp32 summation: s + c carries the running sum with about twice fp32's
// precision (fp64 arithmetic runs at a small fraction of the fp32 rate on this part).
struct CompSum {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        c += fabsf(s) >= fabsf(x) ? (s - t) + x : (x - t) + s;
        s = t;
    }
};

// Sum of the per-block parameter-gradient partials of the tensor-core kernels, in the fixed order p = 0..nparts-1
// per element: 64 elements per block, each summed by 8 threads over consecutive
// eighths of the partials (8 loads in flight, compensated fp32), then the eight parts combined in order in fp64.
constexpr int kSumElems = 64, kSumSplit = 8;
__global__ void __launch_bounds__(kSumElems * kSumSplit) k_grad_sum(const float *gpart, int nparts, int gsize,
                                                                    double *out) {
    __shared__ double part[kSumSplit][kSumElems];
    grid_dependency_sync();
    const int el = threadIdx.x % kSumElems, q = threadIdx.x / kSumElems;
    const int e = blockIdx.x * kSumElems + el;
    const int p0 = (int)((long long)q * nparts / kSumSplit), p1 = (int)((long long)(q + 1) * nparts / kSumSplit);
    CompSum cs;
    if (e < gsize) {
        int p = p0;
        for (; p + 8 <= p1; p += 8) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = __ldcg(gpart + (size_t)(p + k) * gsize + e);
#pragma unroll
            for (int k = 0; k < 8; ++k) cs.add(v[k]);
        }
        for (; p < p1; ++p) cs.add(__ldcg(gpart + (size_t)p * gsize + e));
    }
    part[q][el] = (double)cs.s + (double)cs.c;
    __syncthreads();
    if (q == 0 && e < gsize) {
        double t = part[0][el];
#pragma unroll
        for (int k = 1; k < kSumSplit; ++k) t += part[k][el];
        out[e] = t;
    }
}

// Sums of the generic kernels' fp64 parameter gradients, in a fixed order: element e < nw over the gw_n slots, the
// others over the gh_n histograms, and both over the `np` partials of the channel normalisation.  16 elements per
// block, each by 32 threads over consecutive shares (there are up to 1216 slots, more with more heads).
constexpr int kSum64Elems = 16, kSum64Split = 32;
__global__ void __launch_bounds__(kSum64Elems * kSum64Split)
    k_grad_sum64(const double *gw, int gw_n, const double *gh, int gh_n, const double *gpart, int np, int nw, int gsize,
                 double *out) {
    __shared__ double part[kSum64Split][kSum64Elems];
    grid_dependency_sync();
    const int el = threadIdx.x % kSum64Elems, q = threadIdx.x / kSum64Elems;
    const int e = blockIdx.x * kSum64Elems + el;
    double t = 0.0;
    auto sum = [&](const double *x, int n, int step) {
        const int p1 = (int)((long long)(q + 1) * n / kSum64Split);
        int p = (int)((long long)q * n / kSum64Split);
        for (; p + 8 <= p1; p += 8) {
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = __ldcg(x + (size_t)(p + k) * step);
#pragma unroll
            for (int k = 0; k < 8; ++k) t += v[k];
        }
        for (; p < p1; ++p) t += __ldcg(x + (size_t)p * step);
    };
    if (e < nw) sum(gw + e, gw_n, nw);
    else if (e < gsize) sum(gh + (e - nw), gh_n, gsize - nw);
    if (e < gsize) sum(gpart + e, np, gsize);
    part[q][el] = t;
#pragma unroll
    for (int o = kSum64Split / 2; o >= 1; o /= 2) {
        __syncthreads();
        if (q < o) part[q][el] += part[q + o][el];
    }
    if (q == 0 && e < gsize) out[e] = part[0][el];
}

// Inclusive scan of x[0..n) into y (forward: prefix sums; backward: suffix sums), accumulated in fp64,
// by one warp, in a fixed order: lane c sums a contiguous chunk, the chunk totals
// are scanned across lanes, then every lane writes its chunk.
__device__ void warp_scan(const double *x, double *y, int n, bool backward) {
    const int lane = threadIdx.x & 31;
    const int chunk = (n + 31) / 32;
    const int b = lane * chunk, e = min(n, b + chunk);
    auto at = [&](int i) { return backward ? n - 1 - i : i; };
    double t = 0.0;  // fp64: the sums over intervals cancel
    for (int i = b; i < e; ++i) t += x[at(i)];
    double incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    double run = incl - t;  // exclusive prefix of this chunk
    for (int i = b; i < e; ++i) {
        run += x[at(i)];
        y[at(i)] = run;
    }
}

// Block l < L: hidden units of channel l from prefix and suffix sums of the
// channel's interval histogram.  Block L: dW and db.  With the shared-channel
// MLP every channel reads every hidden unit: block l writes its channel's fc1
// contributions to fc1_part ([dw1 | db1][l][k], fp64), summed by k_mlp_fc1_sum.
// With a non-ReLU activation the partials already hold the MLP gradients
// (summed unit by unit): block l copies channel l's, block 0 the shared fc1's.
// Block L also writes the gate's and the coefficients' gradients.
__global__ void __launch_bounds__(128) k_mlp_grads(TableLayout lay, const char *table, const double *gsum,
                                                   luna_phi_grads grads, double *fc1_part) {
    __shared__ double h[2][kMaxUnits + 1];
    __shared__ double pre[2][kMaxUnits + 1], suf[2][kMaxUnits + 1];  // fp64: dw2 = w1 G1 + b1 G0 cancels
    const int Md = lay.M * lay.d, L = lay.L, hid = lay.hid, nint = lay.nint;
    const float scale = 1.0f / sqrtf((float)lay.M);
    const int *rank = reinterpret_cast<const int *>(table + lay.off_rank);
    const int *utype = reinterpret_cast<const int *>(table + lay.off_utype);
    const float *w1 = reinterpret_cast<const float *>(table + lay.off_w1);
    const float *b1 = reinterpret_cast<const float *>(table + lay.off_b1);
    const float *w2 = reinterpret_cast<const float *>(table + lay.off_w2);
    // The first hidden unit of each thread comes from the parameter table, which no kernel of the
    // backward call writes: it is read before the wait for the histogram.
    const bool hist_block = (int)blockIdx.x < L && !lay.act;
    int r_first = 0, t_first = 0;
    float w1_first = 0.0f, b1_first = 0.0f, w2_first = 0.0f;
    if (hist_block && (int)threadIdx.x < hid) {
        const int u = lay.shared ? threadIdx.x : blockIdx.x * hid + threadIdx.x, uw = blockIdx.x * hid + threadIdx.x;
        r_first = rank[u];
        t_first = utype[u];
        w1_first = w1[u];
        b1_first = b1[u];
        w2_first = w2[uw];
    }
    grid_dependency_sync();
    if ((int)blockIdx.x == L) {
        for (int e = threadIdx.x; e < Md; e += blockDim.x) grads.dW[e] = (float)gsum[e];
        for (int e = threadIdx.x; e < lay.M; e += blockDim.x) grads.db[e] = (float)gsum[Md + e];
        const double *gv = gsum + Md + lay.M + mlp_words(lay);  // [dWe | dbe] [dcoef]
        if (lay.env) {
            for (int e = threadIdx.x; e < L * lay.d; e += blockDim.x) grads.dWe[e] = (float)gv[e];
            for (int e = threadIdx.x; e < L; e += blockDim.x) grads.dbe[e] = (float)gv[L * lay.d + e];
            gv += L * lay.d + L;
        }
        if (lay.coef)
            for (int e = threadIdx.x; e < L; e += blockDim.x) grads.dcoef[e] = (float)gv[e];
        return;
    }
    const int l = blockIdx.x;
    const double *hist = gsum + Md + lay.M;
    if (lay.act) {  // [dw2 (L*hid) | dw1 (P) | db1 (P) | db2 (L)]
        const int P = lay.P;
        for (int k = threadIdx.x; k < hid; k += blockDim.x) grads.dw2[l * hid + k] = (float)hist[l * hid + k];
        if (!lay.shared || l == 0) {
            const int u0 = lay.shared ? 0 : l * hid;
            for (int k = threadIdx.x; k < hid; k += blockDim.x) {
                grads.dw1[u0 + k] = (float)hist[L * hid + u0 + k];
                grads.db1[u0 + k] = (float)hist[L * hid + P + u0 + k];
            }
        }
        if (threadIdx.x == 0) grads.db2[l] = (float)hist[L * hid + 2 * P + l];
        return;
    }
    {  // the channel's histogram: every load issued before the first store
        constexpr int kLd = (kMaxUnits + 1 + 127) / 128;
        double v0[kLd], v1[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const int j = threadIdx.x + 128 * k;
            v0[k] = j < nint ? hist[(j * L + l) * 2] : 0.0;
            v1[k] = j < nint ? hist[(j * L + l) * 2 + 1] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const int j = threadIdx.x + 128 * k;
            if (j < nint) { h[0][j] = v0[k]; h[1][j] = v1[k]; }
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5;  // warps 0, 1: prefix of m0, m1; warps 2, 3: suffix
    warp_scan(h[warp & 1], (warp < 2 ? pre : suf)[warp & 1], nint, warp >= 2);
    __syncthreads();
    for (int k = threadIdx.x; k < hid; k += blockDim.x) {
        const int u = lay.shared ? k : l * hid + k;  // the unit: its kink and fc1
        const int uw = l * hid + k;                  // fc2 weight (l, k)
        const bool first = k == (int)threadIdx.x;
        const int r = first ? r_first : rank[u];
        const bool above = (first ? t_first : utype[u]) > 0;
        const double w1u = first ? w1_first : w1[u], b1u = first ? b1_first : b1[u];
        const double w2u = first ? w2_first : w2[uw];
        double G0, G1;
        if (above) {  // active on intervals j > r
            G0 = r + 1 < nint ? suf[0][r + 1] : 0.0;
            G1 = r + 1 < nint ? suf[1][r + 1] : 0.0;
        } else {      // active on intervals j <= r
            G0 = pre[0][r];
            G1 = pre[1][r];
        }
        grads.dw2[uw] = (float)((w1u * G1 + b1u * G0) * (double)scale);
        const double c1 = w2u * G1 * (double)scale, c0 = w2u * G0 * (double)scale;
        if (lay.shared) {
            fc1_part[(size_t)l * hid + k] = c1;
            fc1_part[(size_t)(L + l) * hid + k] = c0;
        } else {
            grads.dw1[u] = (float)c1;
            grads.db1[u] = (float)c0;
        }
    }
    if (threadIdx.x == 0) grads.db2[l] = (float)(pre[0][nint - 1] * (double)scale);
}

// Shared-channel MLP: dw1[k], db1[k] = sums over the channels (in order) of their contributions.
__global__ void __launch_bounds__(128) k_mlp_fc1_sum(TableLayout lay, const double *fc1_part, luna_phi_grads grads) {
    grid_dependency_sync();
    const int L = lay.L, hid = lay.hid;
    for (int k = threadIdx.x; k < hid; k += blockDim.x) {
        double a = 0.0, b = 0.0;
        for (int l = 0; l < L; ++l) {
            a += fc1_part[(size_t)l * hid + k];
            b += fc1_part[(size_t)(L + l) * hid + k];
        }
        grads.dw1[k] = (float)a;
        grads.db1[k] = (float)b;
    }
}

// ---------------------------------------------------------------------------
// host side

size_t smem_keystats(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.dv); take_rows_host(cv, cap, a.D);
    cv.take(kSlack);
    return cv.bytes();
}
size_t smem_query(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, r4(a.D), a.dv); cv.take(a.D); take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.D);
    cv.take(cap);
    return cv.bytes();
}
size_t smem_bwd_query(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, r4(a.D), a.dv); cv.take(r4(a.D));
    take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.dv); take_rows_host(cv, cap, a.D);
    cv.take(cap * std::max(row_stride(a.dv), row_stride(a.D)));
    take_row_pairs_host(cv, cap); cv.take(cap * a.M); cv.take(cap * a.M); cv.take(cap * du_stride(a.M));
    cv.take(kSlack);
    cv.at_least(kGradScratch);
    return cv.bytes();
}
size_t smem_bwd_key(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, r4(a.D), a.dv); cv.take(r4(a.D));
    take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.dv); take_rows_host(cv, cap, a.D);
    take_rows_host(cv, cap, a.D);
    cv.take(cap * a.M); cv.take(cap * a.M); cv.take(cap * du_stride(a.M));
    cv.at_least(kGradScratch);
    return cv.bytes();
}

// Rows per block of a kernel that walks `n` rows of each of BH heads in tiles of cap rows, in at most max_splits
// ranges per head.  Of the splits that fill one to eight waves of one block per SM, the one with the smallest
// time in tiles: waves x (tiles per block + the half tile that a block's table and state loads take).
struct Range { int splits, rows; };
Range split_rows(int BH, int n, int cap, int max_splits) {
    const int64_t tiles = (n + cap - 1) / cap;
    Range best{1, (int)(tiles * cap)};
    double best_cost = 1e300;
    for (int w = 1; w <= 8; ++w) {
        int64_t ns = std::max<int64_t>(1, (int64_t)w * kSMs / BH);
        ns = std::min<int64_t>(std::min<int64_t>(ns, tiles), max_splits);
        const int64_t tps = (tiles + ns - 1) / ns;
        ns = (tiles + tps - 1) / tps;
        const double cost = (double)((BH * ns + kSMs - 1) / kSMs) * ((double)tps + 0.5);
        if (cost < best_cost * 0.999) {
            best_cost = cost;
            best = Range{(int)ns, (int)(tps * cap)};
        }
    }
    return best;
}

template <typename IO>
cudaError_t stats_impl(const AttnArgs &a0, cudaStream_t s) {
    AttnArgs a = a0;
    const int cap = pick_cap(a.B * a.H, a.n, [&](int c) { return smem_keystats(a, c); });
    int pairs = 0;
    if (!a.seg_S) {  // (the streaming form's ranges are its state segments)
        const Range r = split_rows(a.B * a.H, a.n, cap, a.nsplit);
        pairs = 2 * r.splits <= a.nsplit;  // the partials' buffer has room for high and low parts
        a.nsplit = r.splits;
        a.rows_per_split = r.rows;
    }
    const size_t sm = smem_keystats(a, cap);
    cudaError_t e = cudaSuccess;
    outer_dispatch(a.D, a.dv, [&](auto tf, auto tc) {
        auto k = k_keystats<IO, decltype(tf)::value, decltype(tc)::value>;
        if ((e = set_smem(k, sm)) != cudaSuccess) return;
        LUNA_LAUNCH("keystats", k, dim3(a.nsplit, a.B * a.H), kThr, sm, s, a, cap, pairs, a.nsplit <= kFinishParts);
        e = cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    if (a.nsplit > kFinishParts) {
        const size_t SD = (size_t)a.D * a.dv;
        if (a.seg_S)
            e = launch_part_reduce(kScanUp, a, a.nsplit, a.S_part, a.z_part, a.seg_S, a.seg_z, (a.nsplit + 1) * SD,
                                   (size_t)(a.nsplit + 1) * a.D, s);
        else
            e = launch_part_reduce(kSum, a, pairs ? 2 * a.nsplit : a.nsplit, a.S_part, a.z_part, a.S_fin, a.z_fin, SD,
                                   a.D, s);
        if (e != cudaSuccess) return e;
    }
    return launch_chrms_scale_state(a, s);
}

template <typename IO>
cudaError_t fwd_impl(const AttnArgs &a, cudaStream_t s) {
    cudaError_t e = stats_impl<IO>(a, s);
    if (e != cudaSuccess) return e;
    const int cap = pick_cap(a.B * a.H, a.n, [&](int c) { return smem_query(a, c); });
    const Range r = split_rows(a.B * a.H, a.n, cap, 1 << 24);
    const size_t sm = smem_query(a, cap);
    if ((e = set_smem(k_query<IO>, sm)) != cudaSuccess) return e;
    LUNA_LAUNCH("query", k_query<IO>, dim3(r.splits, a.B * a.H), kThr, sm, s, a, cap, r.rows);
    return cudaGetLastError();
}

template <typename IO>
cudaError_t bwd_impl(const AttnArgs &a0, bool have_stats, cudaStream_t s) {
    AttnArgs a = a0;
    cudaError_t e;
    if (!have_stats && (e = stats_impl<IO>(a, s)) != cudaSuccess) return e;
    const int BH = a.B * a.H;
    const int cap = pick_cap(BH, a.n, [&](int c) { return std::max(smem_bwd_query(a, c), smem_bwd_key(a, c)); });
    const Range r = split_rows(BH, a.n, cap, a.nsplit_b);
    a.nsplit_b = r.splits;
    a.rows_per_split_b = r.rows;
    if ((e = place_grads(a, BH * (int64_t)r.splits, s)) != cudaSuccess) return e;
    size_t sm = smem_bwd_query(a, cap);
    const int pairs = a.nsplit_b > 1;  // a single partial is the sum itself, rounded once either way
    outer_dispatch(a.D, a.dv, [&](auto tf, auto tc) {
        auto k = k_bwd_query<IO, decltype(tf)::value, decltype(tc)::value>;
        if ((e = set_smem(k, sm)) != cudaSuccess) return;
        LUNA_LAUNCH("bwd_query", k, dim3(a.nsplit_b, BH), kThr, sm, s, a, cap, pairs, a.nsplit_b <= kFinishParts);
        e = cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    if (a.nsplit_b > kFinishParts) {
        AttnArgs b = a;
        b.hs_mul = 1;  // dS, dz are indexed by the sub-problem's own heads
        if ((e = launch_part_reduce(kSum, b, 2 * a.nsplit_b, a.dS_part, a.dz_part, a.dS_fin, a.dz_fin,
                                    (size_t)a.D * a.dv, a.D, s)) != cudaSuccess)
            return e;
    }
    if ((e = launch_chrms_dstate(a, s)) != cudaSuccess) return e;
    sm = smem_bwd_key(a, cap);
    if ((e = set_smem(k_bwd_key<IO>, sm)) != cudaSuccess) return e;
    LUNA_LAUNCH("bwd_key", k_bwd_key<IO>, dim3(a.nsplit_b, BH), kThr, sm, s, a, cap);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int nparts = 0;
    if ((e = launch_chrms_backward(a, 0, &nparts, s)) != cudaSuccess) return e;
    return launch_grad_reduce(a, nparts, s);
}

}  // namespace

cudaError_t launch_part_reduce(PartReduce mode, const AttnArgs &a, int np, const float *S_part, const float *z_part,
                               float *S, float *z, size_t S_step, size_t z_step, cudaStream_t s) {
    const int nS = a.D * a.dv;
    LUNA_LAUNCH("part_reduce", k_part_reduce, dim3((nS + a.D + 255) / 256, a.B * a.H), 256, 0, s, mode, np, nS, a.D, S_part,
                z_part, S, z, S_step, z_step, a.hs_mul);
    return cudaGetLastError();
}

size_t simt_max_smem(const AttnArgs &a) {
    size_t m = smem_keystats(a, kMinC);
    m = std::max(m, smem_query(a, kMinC));
    m = std::max(m, smem_bwd_query(a, kMinC));
    return std::max(m, smem_bwd_key(a, kMinC)) + kStaticSmem;
}

cudaError_t launch_grad_reduce(const AttnArgs &a, int nparts, cudaStream_t s) {
    const int nb = (a.gsize + kSumElems - 1) / kSumElems;
    const bool dep = !a.ch_sigma;
    if (a.gpart64)
        LUNA_LAUNCH_DEP("grad_sum", dep, k_grad_sum64, (a.gsize + kSum64Elems - 1) / kSum64Elems,
                        kSum64Elems * kSum64Split, 0, s, static_cast<const double *>(a.gw), a.gw_n,
                        static_cast<const double *>(a.gh), a.gh_n, reinterpret_cast<const double *>(a.gpart), nparts,
                        a.M * a.d + a.M, a.gsize, a.hist);
    else
        LUNA_LAUNCH_DEP("grad_sum", dep, k_grad_sum, nb, kSumElems * kSumSplit, 0, s,
                        static_cast<const float *>(a.gpart), nparts, a.gsize, a.hist);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if ((e = launch_chrms_hist(a, s)) != cudaSuccess) return e;
    // the partials have been summed: their buffer holds the shared MLP's per-channel fc1 terms
    double *fc1_part = a.gpart64 ? a.gw : reinterpret_cast<double *>(a.gpart);
    LUNA_LAUNCH_DEP("mlp_grads", dep, k_mlp_grads, a.lay.L + 1, 128, 0, s, a.lay, a.table,
                    static_cast<const double *>(a.hist), a.grads, fc1_part);
    if ((e = cudaGetLastError()) != cudaSuccess || !a.lay.shared || a.lay.act) return e;
    LUNA_LAUNCH_DEP("mlp_fc1_sum", dep, k_mlp_fc1_sum, 1, 128, 0, s, a.lay, static_cast<const double *>(fc1_part),
                    a.grads);
    return cudaGetLastError();
}

cudaError_t launch_featmap(const TableLayout &lay, const char *table, const void *X, luna_dtype xt, int64_t rows,
                           float *Phi, cudaStream_t s) {
    if (lay_variant(lay)) {
        HostCarve cv; carve_phi_tile_host(cv, lay, kPhiRows);
        take_rows_host(cv, kPhiRows, lay.d); take_rows_host(cv, kPhiRows, lay.D);
        const size_t sm = cv.bytes();
        const int64_t tiles = (rows + kPhiRows - 1) / kPhiRows;
        const int blocks = (int)(tiles < 4096 ? (tiles > 0 ? tiles : 1) : 4096);
        cudaError_t e;
        if (xt == LUNA_F32) {
            if ((e = set_smem(k_featmap_var<float>, sm)) != cudaSuccess) return e;
            k_featmap_var<float><<<blocks, kThreads, sm, s>>>(lay, table, static_cast<const float *>(X), rows, Phi);
        } else {
            if ((e = set_smem(k_featmap_var<__nv_bfloat16>, sm)) != cudaSuccess) return e;
            k_featmap_var<__nv_bfloat16><<<blocks, kThreads, sm, s>>>(lay, table, static_cast<const __nv_bfloat16 *>(X),
                                                                      rows, Phi);
        }
        return cudaGetLastError();
    }
    HostCarve cv; carve_phi_tile_host(cv, lay, 0);
    const size_t sm = cv.bytes();
    int64_t work = rows * lay.M;
    int blocks = (int)((work + kThreads - 1) / kThreads);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    cudaError_t e;
    if (xt == LUNA_F32) {
        if ((e = set_smem(k_featmap<float>, sm)) != cudaSuccess) return e;
        k_featmap<float><<<blocks, kThreads, sm, s>>>(lay, table, static_cast<const float *>(X), rows, Phi);
    } else {
        if ((e = set_smem(k_featmap<__nv_bfloat16>, sm)) != cudaSuccess) return e;
        k_featmap<__nv_bfloat16><<<blocks, kThreads, sm, s>>>(lay, table, static_cast<const __nv_bfloat16 *>(X),
                                                              rows, Phi);
    }
    return cudaGetLastError();
}

cudaError_t launch_simt_stats(const AttnArgs &a, luna_dtype io, cudaStream_t s) {
    return io == LUNA_F32 ? stats_impl<float>(a, s) : stats_impl<__nv_bfloat16>(a, s);
}
cudaError_t launch_simt_fwd(const AttnArgs &a, luna_dtype io, cudaStream_t s) {
    return io == LUNA_F32 ? fwd_impl<float>(a, s) : fwd_impl<__nv_bfloat16>(a, s);
}
cudaError_t launch_simt_bwd(const AttnArgs &a, luna_dtype io, bool have_stats, cudaStream_t s) {
    return io == LUNA_F32 ? bwd_impl<float>(a, have_stats, s) : bwd_impl<__nv_bfloat16>(a, have_stats, s);
}

}  // namespace luna
