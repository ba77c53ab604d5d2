// Streaming (causal) form on CUDA cores (fp32 arithmetic, sums as pairs of floats).
//
// The paper names the associative streaming form of kernel attention (abstract,
// Sec. 3.2, Conclusion) without writing it out; it is the prefix recurrence
//     S_i = S_{i-1} + phi(k_i) v_i^T,  z_i = z_{i-1} + phi(k_i),
//     O_i = phi(q_i)^T S_i / (phi(q_i)^T z_i + eps).
// Rows are cut into state segments.  The prefix statistics at every segment
// start come from an exclusive scan of per-segment sums (key-statistics kernel
// in scan mode); inside a segment the rows are processed in tiles of up to 64
// rows: a masked intra-tile term tril(phi(Q) phi(K)^T) V plus the carried
// state, then the state advances by the tile's phi(K)^T V.
//
// Backward (derived from the same recurrence):
//   dnum_i = do_i / den_i, dden_i = -(do_i . o_i)/den_i
//   dphi(q_i) = S_i dnum_i + z_i dden_i
//   G_j = sum_{i>=j} phi(q_i) dnum_i^T, g_j = sum_{i>=j} phi(q_i) dden_i
//   dv_j = G_j^T phi(k_j),  dphi(k_j) = G_j v_j + g_j
// A forward sweep per segment records (den_i, dden_i), produces dQ and the
// segment sums of G; a reverse exclusive scan gives G after every segment; then
// a reverse sweep produces dK and dV.
#include <math.h>

#include "luna_prof.cuh"
#include "luna_tile.cuh"

namespace luna {
namespace {
using namespace simt;

// Measured at 8 x 12 heads of 1024 bf16 rows, d = D = 64 (us; before: fp64 sums, tiles of 16 rows, and separate
// sweeps for the segment sums and dQ): outputs 5918 -> 389, backward queries 16081 -> 1123, backward keys
// 6861 -> 743, with the key statistics 2715 -> 211.
//
// Each kernel walks its segment in tiles of `cap` rows (luna_tile.cuh).  The running state is held in fp32 in
// shared memory and advances once per tile from pairs of floats, so a tile of 64 rows rounds it a quarter as
// often as one of 16.

// den_r = eps + phi(q_r) . z + sum_{j<=r} A[r][j], rounded once
__device__ __forceinline__ void tile_dens(const Rows &Pq, int nr, int D, const float *z, const Rows &A, float eps,
                                          float *sden, float *sinv) {
    row_dots(Pq, nr, D, [&](int, int f) { return z[f]; }, A, [](int r) { return r + 1; },
             [&](int r, float h, float l) {
                 pair_mac_any(h, l, eps, 1.0f);
                 const float den = pair_value(h, l);
                 sden[r] = den;
                 sinv[r] = 1.0f / den;
             });
}

// ---------------------------------------------------------------------------

template <typename IO>
__global__ void __launch_bounds__(kThr, 1) k_causal_out(AttnArgs a, int cap) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, dv = a.dv, d = a.d, Dp = (D + 3) & ~3;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    float *tiles = cv.p;
    const Rows S = take_rows(cv, Dp, dv);
    float *z = cv.take(Dp);
    const Rows sQ = take_rows(cv, cap, d), sK = take_rows(cv, cap, d), sV = take_rows(cv, cap, dv);
    const Rows sPq = take_rows(cv, cap, D), sPk = take_rows(cv, cap, D), sA = take_rows(cv, cap, cap);
    float *sden = cv.take(cap), *sinv = cv.take(cap);
    if (!carve_fits(cv, smem)) return;
    const int bh = blockIdx.y, seg = blockIdx.x;
    const int len = head_length(a.lengths, bh / a.H, a.n);
    const int r0 = seg * a.seg_len, rend = min(a.n, r0 + a.seg_len), r1 = min(len, rend);
    IO *O = static_cast<IO *>(a.O) + head_rows(a, bh) * dv;
    zero_rows(O, max(r0, len), rend, dv);
    if (r0 >= r1) return;
    zero_words(tiles, (int)(cv.p - tiles));
    load_phi_tile(s, lay, a.table);
    const size_t so = head_state(a, bh) * (a.nseg + 1) + seg;
    __syncthreads();
    load_state(S, z, a.seg_S + so * D * dv, a.seg_z + so * D, D, dv);
    const IO *Q = static_cast<const IO *>(a.Q) + head_rows(a, bh) * d;
    const IO *K = static_cast<const IO *>(a.K) + head_rows(a, bh) * d;
    const IO *V = static_cast<const IO *>(a.V) + head_rows(a, bh) * dv;
    const bool vec = vec_store(O, dv);
    for (int t0 = r0; t0 < r1; t0 += cap) {
        const int nr = min(cap, r1 - t0);
        __syncthreads();
        load_tile(sQ, Q + (size_t)t0 * d, nr, d, cap);
        load_tile(sK, K + (size_t)t0 * d, nr, d, cap);
        load_tile(sV, V + (size_t)t0 * dv, nr, dv, cap);
        __syncthreads();
        phi_rows(lay, s, sQ, nr, cap, sPq, nullptr, nullptr);
        phi_rows(lay, s, sK, nr, cap, sPk, nullptr, nullptr);
        __syncthreads();
        scores_lower<false>(sPq, sPk, nr, Dp, sA, [](int, float &, float &) {});
        __syncthreads();
        tile_dens(sPq, nr, D, z, sA, a.eps, sden, sinv);
        __syncthreads();
        // O_r = (phi(q_r) S + sum_{j<=r} A[r][j] v_j) / den_r from the pair of the numerator
        prod_nn(sPq, nr, S, Dp, dv, sA, sV,
                [&](int q0, int c0, const float (&h)[2][4], const float (&l)[2][4]) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (q0 + i >= nr) continue;
                        const float den = sden[q0 + i], inv = sinv[q0 + i];
                        float o[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m) o[m] = den != 0.0f ? pair_div(h[i][m], l[i][m], den, inv) : 0.0f;
                        store4(O + (size_t)(t0 + q0 + i) * dv + c0, o, dv - c0, vec);
                    }
                });
        if (t0 + cap >= r1) break;
        __syncthreads();
        advance_rows(S, z, sPk, D, sV, dv, nullptr, nullptr, nr);
    }
}

// Query side of the backward pass, one forward sweep per segment: den_i and dden_i of every row as pairs (kept for the
// key side), dQ, and the segment's sums of G and g.
//   dphi(q_i) = S_{before tile} dnum_i + z dden_i + sum_{j<=i in tile} dP_ij phi(k_j),  dP_ij = dnum_i . v_j + dden_i
// den_i, dnum_i . num_i and dden_i are pairs (RowPairs); dP and dphi are pairs rounded once.
template <typename IO, int TF, int TC>
__global__ void __launch_bounds__(kThr, 1) k_causal_bwd_query(AttnArgs a, int cap, int finish) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, dv = a.dv, d = a.d, M = a.M, Dp = (D + 3) & ~3, dvp = (dv + 3) & ~3;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    float *tiles = cv.p;
    const Rows S = take_rows(cv, Dp, dv);
    float *z = cv.take(Dp);
    const Rows sQ = take_rows(cv, cap, d), sV = take_rows(cv, cap, dv), sdO = take_rows(cv, cap, dv);
    const Rows sPq = take_rows(cv, cap, D), sPk = take_rows(cv, cap, D), sA = take_rows(cv, cap, cap);
    // one buffer holds k_j, then the parts of dnum_i . num_i, then dphi(q_i)
    float *shared = cv.take(cap * max(row_stride(d), max(row_stride(dv), row_stride(D))));
    const Rows sK{shared, row_stride(d)}, sR{shared, row_stride(dv)}, sdPhi{shared, row_stride(D)};
    const RowPairs rp = take_row_pairs(cv, cap);
    float *sU = cv.take(cap * M);
    int *sJ = reinterpret_cast<int *>(cv.take(cap * M));
    float *sdU = cv.take(cap * du_stride(M));
    cv.take(kSlack);
    if (!carve_fits(cv, smem)) return;
    const int bh = blockIdx.y, seg = blockIdx.x;
    __shared__ double sT[kMaxL];  // channel normalisation: the block's sums of phi . dphi per channel
    if ((int)threadIdx.x < kMaxL) sT[threadIdx.x] = 0.0;
    const size_t slot = (size_t)bh * a.nseg + seg;
    double *hist = a.gh + (slot % a.gh_n) * (a.gsize - M * d - M);
    const int len = head_length(a.lengths, bh / a.H, a.n);
    const int r0 = seg * a.seg_len, rend = min(a.n, r0 + a.seg_len), r1 = min(len, rend);
    IO *dQ = static_cast<IO *>(a.dQ) + head_rows(a, bh) * d;
    zero_rows(dQ, max(r0, len), rend, d);
    OuterAcc<TF, TC> acc;
    acc.zero();
    GradTile g;
    grad_zero(g);
    if (r0 < r1) {
        zero_words(tiles, (int)(cv.p - tiles));
        load_phi_tile(s, lay, a.table);
        const size_t so = head_state(a, bh) * (a.nseg + 1) + seg;
        __syncthreads();
        load_state(S, z, a.seg_S + so * D * dv, a.seg_z + so * D, D, dv);
    }
    const IO *Q = static_cast<const IO *>(a.Q) + head_rows(a, bh) * d;
    const IO *K = static_cast<const IO *>(a.K) + head_rows(a, bh) * d;
    const IO *V = static_cast<const IO *>(a.V) + head_rows(a, bh) * dv;
    const IO *dO = static_cast<const IO *>(a.dO) + head_rows(a, bh) * dv;
    for (int t0 = r0; t0 < r1; t0 += cap) {
        const int nr = min(cap, r1 - t0);
        __syncthreads();
        load_tile(sQ, Q + (size_t)t0 * d, nr, d, cap);
        load_tile(sK, K + (size_t)t0 * d, nr, d, cap);
        load_tile(sV, V + (size_t)t0 * dv, nr, dv, cap);
        load_tile(sdO, dO + (size_t)t0 * dv, nr, dv, cap);
        __syncthreads();
        phi_rows(lay, s, sQ, nr, cap, sPq, sU, sJ);
        phi_rows(lay, s, sK, nr, cap, sPk, nullptr, nullptr);
        __syncthreads();
        // pairs too: o and den are formed from A, and a common rounding error of theirs does not cancel in dphi
        scores_lower<true>(sPq, sPk, nr, Dp, sA, [](int, float &, float &) {});
        __syncthreads();
        row_dots(sPq, nr, D, [&](int, int f) { return z[f]; }, sA, [](int r) { return r + 1; },
                 [&](int r, float h, float l) { rp.set_den(r, h, l, a.eps); });
        __syncthreads();
        rp.divide_rows(sdO, nr, dv);  // dnum in place
        __syncthreads();
        prod_nn(sPq, nr, S, Dp, dv, sA, sV, [&](int q0, int c0, const float (&h)[2][4], const float (&l)[2][4]) {
            unit_dots(sdO, sR, nr, q0, c0, h, l);
        });
        __syncthreads();
        sum_unit_dots(sR, nr, dvp / 4, [&](int r, float h, float l) {
            rp.set_dden(r, h, l);
            *reinterpret_cast<float4 *>(a.rowstat + ((size_t)bh * a.n + t0 + r) * 4) =
                make_float4(rp.dh[r], rp.dl[r], rp.gh[r], rp.gl[r]);
        });
        __syncthreads();
        scores_lower<true>(sdO, sV, nr, dvp, sA, [&](int r, float &h, float &l) {
            if (r < nr) { h = rp.gh[r]; l = rp.gl[r]; }
        });
        acc.add(sPq, D, sdO, dv, rp.gh, rp.gl, nr);
        __syncthreads();
        prod_nt<kLower>(sdO, nr, S, D, dvp, sA, sPk, nr,
                        [&](int r, int f, float &h, float &l) {
                            if (r < nr) {
                                pair_mac(h, l, z[f], rp.gh[r]);
                                l = __fmaf_rn(z[f], rp.gl[r], l);
                            }
                        },
                        [&](int r, int f, float h, float l) {
                            if (r >= nr) return;
                            sdPhi[r][f] = pair_value(h, l);
                            if (a.ch_T) atomicAdd(sT + f % a.L, (double)sPq[r][f] * ((double)h + (double)l));
                        });
        __syncthreads();
        if (t0 + cap < r1) advance_rows(S, z, sPk, D, sV, dv, nullptr, nullptr, nr);
        phi_backward_rows(lay, s, sQ, nr, cap, sPq, sdPhi, sU, sJ, sdU, hist, hist + mlp_words(lay), g);
        store_dx_rows(lay, s, sdU, nr, dQ + (size_t)t0 * d);
    }
    acc.store(D, dv, a.dS_part, a.dz_part, slot, false);
    store_grad_tile(lay, g, smem, a.gw + slot * (M * d + M));
    if (a.ch_T && (int)threadIdx.x < a.L) a.ch_T[slot * a.L + threadIdx.x] = sT[threadIdx.x];
    if (finish && last_arrival(a.counters + a.B * a.H + bh, a.nseg)) {
        exclusive_scan(a.dS_part + (size_t)bh * a.nseg * D * dv, a.nseg, D * dv, a.seg_dS + (size_t)bh * a.nseg * D * dv,
                       true);
        exclusive_scan(a.dz_part + (size_t)bh * a.nseg * D, a.nseg, D, a.seg_dz + (size_t)bh * a.nseg * D, true);
        if (threadIdx.x == 0) a.counters[a.B * a.H + bh] = 0;
    }
}

// dK, dV: reverse sweep with the suffix state G (after the current tile).
//   dv_j = G^T phi(k_j) + sum_{i>=j in tile} A_ij dnum_i
//   dphi(k_j) = G v_j + g + sum_{i>=j in tile} dP_ij phi(q_i)
template <typename IO>
__global__ void __launch_bounds__(kThr, 1) k_causal_bwd_key(AttnArgs a, int cap) {
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, dv = a.dv, d = a.d, M = a.M, Dp = (D + 3) & ~3, dvp = (dv + 3) & ~3;
    SmemPhi s = carve_phi_tile(cv, lay, cap);
    float *tiles = cv.p;
    const Rows G = take_rows(cv, Dp, dv);
    float *gz = cv.take(Dp);
    const Rows sK = take_rows(cv, cap, d), sV = take_rows(cv, cap, dv), sdO = take_rows(cv, cap, dv);
    const Rows sPq = take_rows(cv, cap, D), sPk = take_rows(cv, cap, D);
    const Rows sA = take_rows(cv, cap, cap), sP = take_rows(cv, cap, cap);
    // one buffer holds q_i, then dphi(k_j)
    float *shared = cv.take(cap * max(row_stride(d), row_stride(D)));
    const Rows sQ{shared, row_stride(d)}, sdPhi{shared, row_stride(D)};
    const RowPairs rp = take_row_pairs(cv, cap);
    float *sU = cv.take(cap * M);
    int *sJ = reinterpret_cast<int *>(cv.take(cap * M));
    float *sdU = cv.take(cap * du_stride(M));
    if (!carve_fits(cv, smem)) return;
    const int bh = blockIdx.y, seg = blockIdx.x;
    const size_t slot = (size_t)bh * a.nseg + seg;
    double *hist = a.gh + (slot % a.gh_n) * (a.gsize - M * d - M), *gw = a.gw + (a.gw_n / 2 + slot) * (M * d + M);
    const int len = head_length(a.lengths, bh / a.H, a.n);
    const int r0 = seg * a.seg_len, rend = min(a.n, r0 + a.seg_len), r1 = min(len, rend);
    IO *dK = static_cast<IO *>(a.dK) + head_rows(a, bh) * d;
    IO *dV = static_cast<IO *>(a.dV) + head_rows(a, bh) * dv;
    zero_rows(dK, max(r0, len), rend, d);
    zero_rows(dV, max(r0, len), rend, dv);
    if (r1 <= r0) {
        for (int e = threadIdx.x; e < M * d + M; e += blockDim.x) gw[e] = 0.0;
        return;
    }
    zero_words(tiles, (int)(cv.p - tiles));
    load_phi_tile(s, lay, a.table);
    __syncthreads();
    load_state(G, gz, a.seg_dS + slot * D * dv, a.seg_dz + slot * D, D, dv);
    const IO *Q = static_cast<const IO *>(a.Q) + head_rows(a, bh) * d;
    const IO *K = static_cast<const IO *>(a.K) + head_rows(a, bh) * d;
    const IO *V = static_cast<const IO *>(a.V) + head_rows(a, bh) * dv;
    const IO *dO = static_cast<const IO *>(a.dO) + head_rows(a, bh) * dv;
    const bool vec = vec_store(dV, dv);
    GradTile g;
    grad_zero(g);
    for (int t0 = r0 + ((r1 - 1 - r0) / cap) * cap; t0 >= r0; t0 -= cap) {
        const int nr = min(cap, r1 - t0);
        __syncthreads();
        load_tile(sQ, Q + (size_t)t0 * d, nr, d, cap);
        load_tile(sK, K + (size_t)t0 * d, nr, d, cap);
        load_tile(sV, V + (size_t)t0 * dv, nr, dv, cap);
        load_tile(sdO, dO + (size_t)t0 * dv, nr, dv, cap);
        for (int r = threadIdx.x; r < cap; r += blockDim.x) {
            const float4 v = r < nr ? ld4(a.rowstat + ((size_t)bh * a.n + t0 + r) * 4) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            rp.dh[r] = v.x; rp.dl[r] = v.y; rp.inv[r] = 1.0f / v.x;
            rp.gh[r] = v.z; rp.gl[r] = v.w;
        }
        __syncthreads();
        rp.divide_rows(sdO, nr, dv);  // dnum in place
        phi_rows(lay, s, sQ, nr, cap, sPq, nullptr, nullptr);
        phi_rows(lay, s, sK, nr, cap, sPk, sU, sJ);
        __syncthreads();
        scores_lower<false>(sPq, sPk, nr, Dp, sA, [](int, float &, float &) {});
        scores_lower<true>(sdO, sV, nr, dvp, sP, [&](int r, float &h, float &l) { h = rp.gh[r]; l = rp.gl[r]; });
        __syncthreads();
        prod_nn_chains(sPk, nr, G, Dp, dv, sA, sdO, nr, [&](int q0, int c0, const float (&h)[2][4]) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (q0 + i < nr) store4(dV + (size_t)(t0 + q0 + i) * dv + c0, h[i], dv - c0, vec);
        });
        prod_nt<kUpper>(sV, nr, G, D, dvp, sP, sPq, nr, [&](int, int f, float &h, float &) { h = gz[f]; },
                        [&](int r, int f, float h, float l) {
                            if (r < nr) sdPhi[r][f] = pair_value(h, l);
                        });
        __syncthreads();
        if (t0 > r0) advance_rows(G, gz, sPq, D, sdO, dv, rp.gh, rp.gl, nr);
        phi_backward_rows(lay, s, sK, nr, cap, sPk, sdPhi, sU, sJ, sdU, hist, hist + mlp_words(lay), g);
        store_dx_rows(lay, s, sdU, nr, dK + (size_t)t0 * d);
    }
    store_grad_tile(lay, g, smem, gw);
}

// ---------------------------------------------------------------------------

size_t smem_out(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, r4(a.D), a.dv); cv.take(r4(a.D));
    take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.dv);
    take_rows_host(cv, cap, a.D); take_rows_host(cv, cap, a.D); take_rows_host(cv, cap, cap);
    cv.take(cap); cv.take(cap);
    return cv.bytes();
}
size_t smem_bwd_query(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, r4(a.D), a.dv); cv.take(r4(a.D));
    take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.dv); take_rows_host(cv, cap, a.dv);
    take_rows_host(cv, cap, a.D); take_rows_host(cv, cap, a.D); take_rows_host(cv, cap, cap);
    cv.take(cap * std::max(row_stride(a.d), std::max(row_stride(a.dv), row_stride(a.D))));
    take_row_pairs_host(cv, cap); cv.take(cap * a.M); cv.take(cap * a.M); cv.take(cap * du_stride(a.M));
    cv.take(kSlack);
    cv.at_least(kGradScratch);
    return cv.bytes();
}
size_t smem_bwd_key(const AttnArgs &a, int cap) {
    HostCarve cv; carve_phi_tile_host(cv, a.lay, cap);
    take_rows_host(cv, r4(a.D), a.dv); cv.take(r4(a.D));
    take_rows_host(cv, cap, a.d); take_rows_host(cv, cap, a.dv); take_rows_host(cv, cap, a.dv);
    take_rows_host(cv, cap, a.D); take_rows_host(cv, cap, a.D);
    take_rows_host(cv, cap, cap); take_rows_host(cv, cap, cap);
    cv.take(cap * std::max(row_stride(a.d), row_stride(a.D)));
    take_row_pairs_host(cv, cap); cv.take(cap * a.M); cv.take(cap * a.M); cv.take(cap * du_stride(a.M));
    cv.at_least(kGradScratch);
    return cv.bytes();
}

// Rows per tile: a segment is walked tile by tile by one block, so the largest that fits.
template <typename Smem>
int seg_cap(const AttnArgs &a, Smem smem) {
    return pick_cap((int64_t)kSMs * kMaxC, std::min(a.n, a.seg_len), smem);
}

template <typename IO>
cudaError_t seg_stats(const AttnArgs &a, cudaStream_t s) {
    AttnArgs b = a;
    b.nsplit = a.nseg;
    b.rows_per_split = a.seg_len;
    return launch_simt_stats(b, IOType<IO>::code, s);
}

template <typename IO>
cudaError_t causal_fwd_impl(const AttnArgs &a, cudaStream_t s) {
    cudaError_t e = seg_stats<IO>(a, s);
    if (e != cudaSuccess) return e;
    const int cap = seg_cap(a, [&](int c) { return smem_out(a, c); });
    const size_t sm = smem_out(a, cap);
    if ((e = set_smem(k_causal_out<IO>, sm)) != cudaSuccess) return e;
    LUNA_LAUNCH("causal_out", k_causal_out<IO>, dim3(a.nseg, a.B * a.H), kThr, sm, s, a, cap);
    return cudaGetLastError();
}

template <typename IO>
cudaError_t causal_bwd_impl(const AttnArgs &a0, bool have_state, cudaStream_t s) {
    AttnArgs a = a0;
    cudaError_t e;
    if (!have_state && (e = seg_stats<IO>(a, s)) != cudaSuccess) return e;
    if ((e = place_grads(a, (int64_t)a.B * a.H * a.nseg, s)) != cudaSuccess) return e;
    const dim3 grid(a.nseg, a.B * a.H);
    int cap = seg_cap(a, [&](int c) { return smem_bwd_query(a, c); });
    size_t sm = smem_bwd_query(a, cap);
    outer_dispatch(a.D, a.dv, [&](auto tf, auto tc) {
        auto k = k_causal_bwd_query<IO, decltype(tf)::value, decltype(tc)::value>;
        if ((e = set_smem(k, sm)) != cudaSuccess) return;
        LUNA_LAUNCH("causal_bwd_query", k, grid, kThr, sm, s, a, cap, a.nseg <= kFinishParts);
        e = cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    if (a.nseg > kFinishParts) {
        AttnArgs b = a;
        b.hs_mul = 1;  // the suffixes are indexed by the sub-problem's own heads
        if ((e = launch_part_reduce(kScanDown, b, a.nseg, a.dS_part, a.dz_part, a.seg_dS, a.seg_dz,
                                    (size_t)a.nseg * a.D * a.dv, (size_t)a.nseg * a.D, s)) != cudaSuccess)
            return e;
    }
    cap = seg_cap(a, [&](int c) { return smem_bwd_key(a, c); });
    sm = smem_bwd_key(a, cap);
    if ((e = set_smem(k_causal_bwd_key<IO>, sm)) != cudaSuccess) return e;
    LUNA_LAUNCH("causal_bwd_key", k_causal_bwd_key<IO>, grid, kThr, sm, s, a, cap);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int nparts = 0;
    if (a.ch_sigma) {  // the scale term of the channel normalisation (kappa from the queries' T rows)
        a.ch_T_rows = a.B * a.H * a.nseg;
        if ((e = launch_chrms_backward(a, nparts, &nparts, s)) != cudaSuccess) return e;
    }
    return launch_grad_reduce(a, nparts, s);
}

}  // namespace

size_t causal_max_smem(const AttnArgs &a) {
    return std::max(smem_out(a, kMinC), std::max(smem_bwd_query(a, kMinC), smem_bwd_key(a, kMinC))) + kStaticSmem;
}

cudaError_t launch_causal_fwd(const AttnArgs &a, luna_dtype io, bool, cudaStream_t s) {
    return io == LUNA_F32 ? causal_fwd_impl<float>(a, s) : causal_fwd_impl<__nv_bfloat16>(a, s);
}

cudaError_t launch_causal_bwd(const AttnArgs &a, luna_dtype io, bool have_state, cudaStream_t s) {
    return io == LUNA_F32 ? causal_bwd_impl<float>(a, have_state, s) : causal_bwd_impl<__nv_bfloat16>(a, have_state, s);
}

}  // namespace luna
