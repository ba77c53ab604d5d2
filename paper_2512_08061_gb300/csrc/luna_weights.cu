// Attention weights of a block of query rows, for the conversion's stage 1
// (appendix: the feature-map parameters are trained so that the attention
// distribution induced by the kernel matches the one of the original softmax
// module; the loss is not fixed by the paper, so the library only produces
// the two distributions).
//
//   LUNA (Eq. kernel-attn read as a weighted average of the values):
//       a_ij = k(q_i, k_j) / (sum_j' k(q_i, k_j') + eps),  k(x, y) = phi(x)^T phi(y)
//   teacher: p_ij = exp(q_i . k_j / sqrt(d)) / sum_j' exp(q_i . k_j' / sqrt(d))
//
// over the valid keys (j <= i in the streaming form); masked keys, query rows
// at or past the valid length and rows whose guarded sum is exactly 0 get 0.
// One block owns 64 query rows of one head and sweeps every key in tiles of
// 64 rows (32 and 32 for short sequences); a thread owns the same 2 rows x 4
// columns of every tile.  Pass 1 writes the raw scores (the kernel values, or
// the scaled dot products) and accumulates each row's sum (LUNA, as a pair of
// floats) or its running maximum and rescaled exponential sum (teacher); pass 2
// rereads the thread's own entries, from L2, and normalises them.  A NaN score
// of the teacher makes the row's sum NaN and its scale 0, whichever tile holds
// it.  No scratch memory.  Measured at 48 heads of 512 x 512, d = D = 64: kernel
// weights 1567 -> 146 us, teacher 1198 -> 102 us against one score per thread
// from scalar shared loads.
#include <math.h>

#include "luna_prof.cuh"
#include "luna_tile.cuh"

namespace luna {
namespace {
using namespace simt;

// Tile of the kernel: W query rows per block and key rows per tile, RT rows x 4 columns per thread.  64 rows with two
// blocks per SM: one computes while the other loads and evaluates its key tile.  Sequences of at most kSmallN
// keys are one tile, whose time is the latency of its loads: 32-row tiles of one row per thread with four blocks
// per SM.  Tiles of 64 against 32 rows, us, kernel weights and teacher: 4096 heads of 32 keys 214 -> 129 and
// 122 -> 52, of 16 keys 200 -> 104 and 113 -> 34; 768 heads of 4 keys 48 -> 23 and 29 -> 11.
template <int W, int RT>
struct WTile {
    static constexpr int threads = W / RT * (W / 4);
    static constexpr int blocks = W == 64 ? 2 : 4;
};
constexpr int kSmallN = 32;

template <typename IO, int W, int RT>
__global__ void __launch_bounds__(WTile<W, RT>::threads, WTile<W, RT>::blocks)
    k_weights(AttnArgs a, int causal, int row0, int rows, int teacher, int64_t tstride, float *A) {
    constexpr int NC = W / 4;  // threads per row: columns f0 + NC m of every key tile
    extern __shared__ __align__(16) float smem[];
    Carve cv{smem};
    const TableLayout &lay = a.lay;
    const int D = a.D, d = a.d, n = a.n;
    SmemPhi s = {};
    if (!teacher) s = carve_phi_tile(cv, lay, 0);
    const Rows sX = take_rows(cv, W, d);                       // queries for phi, then keys
    const Rows sQ = take_rows(cv, W, teacher ? d : D);         // phi(q) (teacher: q)
    const Rows sP = teacher ? sX : take_rows(cv, W, D);        // phi(k) (teacher: k)
    if (!carve_fits(cv, smem)) return;
    const int bh = blockIdx.y;
    const int r_lo = blockIdx.x * W;                  // first output row of this block (relative to row0)
    const int nr = min(W, rows - r_lo);               // output rows of this block
    const int i_lo = row0 + r_lo;                      // its first query row
    const int len = head_length(a.lengths, bh / a.H, n);
    const int nq = max(0, min(nr, len - i_lo));        // of which valid query rows
    float *Ab = A + ((size_t)bh * rows + r_lo) * n;
    const IO *Qh = static_cast<const IO *>(a.Q) + (size_t)bh * n * d;
    const IO *Kh = static_cast<const IO *>(a.K) + (size_t)bh * n * d;
    // rows past the valid length: zeros
    for (size_t e = (size_t)nq * n + threadIdx.x; e < (size_t)nr * n; e += blockDim.x) Ab[e] = 0.0f;
    if (nq == 0) return;
    if (!teacher) load_phi_tile(s, lay, a.table + (size_t)(bh % a.H) * tstride);  // this head's table
    load_tile(teacher ? sQ : sX, Qh + (size_t)i_lo * d, nq, d, W);
    __syncthreads();
    if (!teacher) phi_rows(lay, s, sX, nq, W, sQ, nullptr, nullptr);
    const int r0 = RT * (threadIdx.x / NC), f0 = threadIdx.x % NC, K = ((teacher ? d : D) + 3) & ~3;
    const int jend = causal ? min(i_lo + nq, len) : len;  // keys the block needs
    int jmax[RT];                                         // keys each row sees
#pragma unroll
    for (int i = 0; i < RT; ++i) jmax[i] = r0 + i >= nq ? 0 : (causal ? min(i_lo + r0 + i + 1, len) : len);
    const float qscale = 1.0f / sqrtf((float)d);
    float sh[RT] = {}, sl[RT] = {};  // LUNA: row sums of the kernel values
    float mx[RT], es[RT] = {};       // teacher: maximum, exponential sum
#pragma unroll
    for (int i = 0; i < RT; ++i) mx[i] = -INFINITY;
    float *Ar = Ab + (size_t)r0 * n;
    for (int j0 = 0; j0 < n; j0 += W) {
        float h[RT][4] = {};
        if (j0 < jend) {
            __syncthreads();
            const int nk = min(min(W, n - j0), jend - j0);
            load_tile(sX, Kh + (size_t)j0 * d, nk, d, W);
            __syncthreads();
            if (!teacher) {
                phi_rows(lay, s, sX, nk, W, sP, nullptr, nullptr);
                __syncthreads();
            }
            const float *q = sQ[r0], *p = sP[f0];
            const int step = NC * sP.ld;
#pragma unroll 2
            for (int k = 0; k < (r0 < nq ? K : 0); k += 4) {
                float4 x[RT];
#pragma unroll
                for (int i = 0; i < RT; ++i) x[i] = ld4(q + i * sQ.ld + k);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float4 v = ld4(p + m * step + k);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                        for (int i = 0; i < RT; ++i) h[i][m] = fmaf(at(x[i], kk), at(v, kk), h[i][m]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            if (r0 + i >= nq) continue;
            float m2 = mx[i];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = j0 + f0 + NC * m;
                if (j >= jmax[i]) {
                    h[i][m] = 0.0f;
                } else if (teacher) {
                    h[i][m] *= qscale;
                    if (h[i][m] > m2) m2 = h[i][m];
                    if (h[i][m] != h[i][m]) es[i] = h[i][m];  // a NaN score: the row's sum is NaN from here on
                } else {
                    pair_mac_any(sh[i], sl[i], h[i][m], 1.0f);
                }
                if (j < n) Ar[(size_t)i * n + j] = h[i][m];
            }
            if (teacher && m2 > -INFINITY) {
                float e = es[i] * expf(mx[i] - m2);
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    if (j0 + f0 + NC * m < jmax[i]) e += expf(h[i][m] - m2);
                es[i] = e;
                mx[i] = m2;
            }
        }
    }
    // combine a row's threads (half a warp, or a quarter)
    float scale[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
#pragma unroll
        for (int o = NC / 2; o > 0; o >>= 1) {
            if (teacher) {
                const float m2 = __shfl_xor_sync(0xffffffffu, mx[i], o), e2 = __shfl_xor_sync(0xffffffffu, es[i], o);
                const float m = fmaxf(mx[i], m2);
                // (no maximum yet: both sums are 0, or NaN)
                es[i] = (m == -INFINITY) ? es[i] + e2 : es[i] * expf(mx[i] - m) + e2 * expf(m2 - m);
                mx[i] = m;
            } else {
                const float h2 = __shfl_xor_sync(0xffffffffu, sh[i], o), l2 = __shfl_xor_sync(0xffffffffu, sl[i], o);
                pair_add(sh[i], sl[i], h2, l2);
            }
        }
        if (teacher) {
            scale[i] = es[i] > 0.0f ? 1.0f / es[i] : 0.0f;
        } else {
            const double den = pair_double(sh[i], sl[i]) + (double)a.eps;
            scale[i] = den != 0.0 ? (float)(1.0 / den) : 0.0f;
        }
    }
    // pass 2: normalise this thread's own entries, written above
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        float *row = Ar + (size_t)i * n;
        for (int j = f0; j < jmax[i]; j += W) {  // four loads in flight
            float v[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) v[m] = j + NC * m < jmax[i] ? row[j + NC * m] : 0.0f;
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (j + NC * m < jmax[i]) row[j + NC * m] = teacher ? expf(v[m] - mx[i]) * scale[i] : v[m] * scale[i];
        }
    }
}

size_t smem_weights(const AttnArgs &a, int teacher, int W) {
    HostCarve cv;
    if (!teacher) carve_phi_tile_host(cv, a.lay, 0);
    take_rows_host(cv, W, a.d);
    take_rows_host(cv, W, teacher ? a.d : a.D);
    if (!teacher) take_rows_host(cv, W, a.D);
    return cv.bytes();
}

template <typename IO, int W, int RT>
cudaError_t weights_impl(const AttnArgs &a, int causal, int row0, int rows, int teacher, int64_t tstride, float *A,
                         cudaStream_t s) {
    const size_t sm = smem_weights(a, teacher, W);
    auto k = k_weights<IO, W, RT>;
    cudaError_t e = set_smem(k, sm);
    if (e != cudaSuccess) return e;
    const dim3 grid((rows + W - 1) / W, a.B * a.H);
    LUNA_LAUNCH("weights", k, grid, (WTile<W, RT>::threads), sm, s, a, causal, row0, rows, teacher, tstride, A);
    return cudaGetLastError();
}

template <typename IO>
cudaError_t weights_io(const AttnArgs &a, int causal, int row0, int rows, int teacher, int64_t tstride, float *A,
                       cudaStream_t s) {
    return a.n <= kSmallN ? weights_impl<IO, 32, 1>(a, causal, row0, rows, teacher, tstride, A, s)
                          : weights_impl<IO, 64, 2>(a, causal, row0, rows, teacher, tstride, A, s);
}

}  // namespace

size_t weights_max_smem(const AttnArgs &a) { return smem_weights(a, 0, 64); }

cudaError_t launch_weights(const AttnArgs &a, luna_dtype io, int causal, int row0, int rows, int teacher,
                           int64_t tstride, float *A, cudaStream_t s) {
    return io == LUNA_F32 ? weights_io<float>(a, causal, row0, rows, teacher, tstride, A, s)
                          : weights_io<__nv_bfloat16>(a, causal, row0, rows, teacher, tstride, A, s);
}

}  // namespace luna
