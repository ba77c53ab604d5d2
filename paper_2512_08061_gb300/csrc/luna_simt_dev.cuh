// Device helpers shared by the CUDA-core kernels (non-causal and causal).
#pragma once

#include "luna_simt.cuh"

namespace luna {
namespace simt {
namespace {  // internal linkage in every translation unit that includes this

constexpr int kThreads = 256;
constexpr int kPhiRows = 32;  // rows per tile of the variants' feature-map kernel

__host__ __device__ inline int r4(int x) { return (x + 3) & ~3; }

struct Carve {
    float *p;
    __device__ float *take(int n) {
        float *r = p;
        p += r4(n);
        return r;
    }
};

// True when the arrays carved so far fit in the block's dynamic shared memory (the host sizes the
// launch with a HostCarve of the same arrays; a kernel whose carve does not fit returns before it
// touches shared memory, so a mismatch shows as a wrong result, not as an out-of-bounds access).
__device__ __forceinline__ bool carve_fits(const Carve &cv, const float *base) {
    uint32_t dyn;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    return (size_t)(cv.p - base) * sizeof(float) <= (size_t)dyn;
}

struct HostCarve {
    int n = 0;
    void take(int k) { n += r4(k); }
    void at_least(int k) { n = n > k ? n : k; }
    size_t bytes() const { return (size_t)n * 4; }
};

// The feature map in shared memory: the sorted kinks T and the interval table AB (ReLU MLPs), or the
// MLP parameters themselves (another activation: direct evaluation); the projection; the variants'
// gate and coefficients with their per-row scratch.
struct SmemPhi {
    float *T, *AB, *W, *b;
    float *w1, *b1, *w2, *b2;  // channel MLPs (non-ReLU activation)
    float *We, *be, *coef;     // envelope gate, Bank+Coef coefficients
    float *E, *H, *dE;         // [cap][L], a row for each of the kernel's tile: e_l = h_l c_l, the gate h_l, dLoss/de_l
                               // (then the gate's pre-activation gradient)
};

// The (alpha, beta) table into shared memory at ab_stride(lay) words per interval.
__device__ void copy_ab(float *dst, const TableLayout &lay, const char *table) {
    const float *src = reinterpret_cast<const float *>(table + lay.off_AB);
    const int w = 2 * lay.L, st = ab_stride(lay);
    for (int e = threadIdx.x; e < lay.nint * w; e += blockDim.x) dst[(e / w) * st + e % w] = src[e];
}

// (alpha, beta) of channel l in the entry of one interval.
__device__ __forceinline__ float2 ab_pair(const float *entry, int l) { return reinterpret_cast<const float2 *>(entry)[l]; }

// The channel MLPs' hidden activation (luna_act) and its derivative da (ReLU'(0) = 0).
// GELU(a) = a Phi(a), Phi(a) = (1 + erf(a / sqrt 2)) / 2, GELU' = Phi(a) + a exp(-a^2 / 2) / sqrt(2 pi);
// SiLU(a) = a sigma(a), SiLU' = sigma (1 + a (1 - sigma)); tanh' = 1 - tanh^2.
__device__ __forceinline__ float act_eval(int act, float a, float &da) {
    switch (act) {
        case LUNA_ACT_GELU: {
            const float c = 0.5f * (1.0f + erff(a * 0.70710678118654752f));
            da = fmaf(a * 0.39894228040143268f, expf(-0.5f * a * a), c);
            return a * c;
        }
        case LUNA_ACT_SILU: {
            const float sg = 1.0f / (1.0f + expf(-a));
            da = sg * fmaf(a, 1.0f - sg, 1.0f);
            return a * sg;
        }
        case LUNA_ACT_TANH: {
            const float t = tanhf(a);
            da = fmaf(-t, t, 1.0f);
            return t;
        }
        default:
            da = a > 0.0f ? 1.0f : 0.0f;
            return fmaxf(a, 0.0f);
    }
}

// The 1/sqrt(M) of Eq. (phi-def-scalarenv), as the table folds it into alpha and beta.
__device__ __forceinline__ float phi_scale(const TableLayout &lay) { return 1.0f / sqrtf((float)lay.M); }

// Direct evaluation of channel l's MLP output y_l(u) = b2_l + sum_k w2_lk act(w1 u + b1) (before the outer
// ReLU and the scale); with dydu, also dy/du = sum_k w2_lk act'(w1 u + b1) w1.
__device__ __forceinline__ float channel_direct(const TableLayout &lay, const SmemPhi &s, int l, float u,
                                                float *dydu) {
    const int hid = lay.hid, base = lay.shared ? 0 : l * hid;
    const float *w2 = s.w2 + l * hid;
    float y = s.b2[l], t = 0.0f;
    for (int k = 0; k < hid; ++k) {
        float da;
        const float w1 = s.w1[base + k];
        const float av = act_eval(lay.act, fmaf(w1, u, s.b1[base + k]), da);
        y = fmaf(w2[k], av, y);
        t = fmaf(w2[k] * da, w1, t);
    }
    if (dydu) *dydu = t;
    return y;
}

// The ungated channel value phi0 = max(scale y_l(u), floor) of interval j (table) or by direct evaluation.
__device__ __forceinline__ float channel_value(const TableLayout &lay, const SmemPhi &s, float u, int j, int l,
                                               float fl) {
    if (lay.act) return fmaxf(phi_scale(lay) * channel_direct(lay, s, l, u, nullptr), fl);
    const float2 ab = ab_pair(s.AB + j * ab_stride(lay), l);
    return fmaxf(fmaf(ab.x, u, ab.y), fl);
}

// Per-row factors of the variants for rows [0, nr) of sX (row stride ldx): H = h_l(x) = sigmoid(We_l . x + be_l) (1 without the
// gate), E = h_l c_l (c_l = 1 without Bank+Coef).
__device__ void gate_rows(const TableLayout &lay, const SmemPhi &s, const float *sX, int ldx, int nr) {
    const int L = lay.L, d = lay.d;
    for (int e = threadIdx.x; e < nr * L; e += blockDim.x) {
        const int r = e / L, l = e - r * L;
        float h = 1.0f;
        if (lay.env) {
            float a = s.be[l];
            for (int c = 0; c < d; ++c) a = fmaf(s.We[l * d + c], sX[r * ldx + c], a);
            h = 1.0f / (1.0f + expf(-a));
        }
        s.H[e] = h;
        s.E[e] = lay.coef ? h * s.coef[l] : h;
    }
}

__device__ bool last_arrival(int *counter, int expected) {
    __shared__ int s_flag;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_flag = (atomicAdd(counter, 1) == expected - 1) ? 1 : 0;
    __syncthreads();
    if (s_flag) __threadfence();
    return s_flag != 0;
}

// out[e] = sum_p part[p][e] in order p = 0..nparts-1 (fp64, rounded once)
__device__ void ordered_sum(const float *part, int nparts, int count, float *out) {
    for (int e = threadIdx.x; e < count; e += blockDim.x) {
        double s = 0.0;
        for (int p0 = 0; p0 < nparts; p0 += 8) {  // eight loads in flight, added in order
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = (p0 + k < nparts) ? __ldcg(part + (size_t)(p0 + k) * count + e) : 0.0f;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (p0 + k < nparts) s += (double)v[k];
        }
        out[e] = (float)s;
    }
}

// Exclusive scan over partials in order: forward (out[p] = sum_{q<p} part[q],
// out[nparts] = total) or reverse (out[p] = sum_{q>p} part[q]); fp64 running sums, each output rounded once.
// Eight loads in flight: they cannot pass the stores by themselves.
__device__ void exclusive_scan(const float *part, int nparts, int count, float *out, bool reverse) {
    for (int e = threadIdx.x; e < count; e += blockDim.x) {
        double s = 0.0;
        for (int p0 = 0; p0 < nparts; p0 += 8) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int p = p0 + k;
                v[k] = p < nparts ? __ldcg(part + (size_t)(reverse ? nparts - 1 - p : p) * count + e) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int p = p0 + k;
                if (p < nparts) {
                    out[(size_t)(reverse ? nparts - 1 - p : p) * count + e] = (float)s;
                    s += (double)v[k];
                }
            }
        }
        if (!reverse) out[(size_t)nparts * count + e] = (float)s;
    }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}


}  // namespace
}  // namespace simt
}  // namespace luna
