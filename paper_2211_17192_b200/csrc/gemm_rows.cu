// Skinny weight-streaming GEMM on the FMA pipes: y[r] = x[r] . W^T for a few
// activation rows against an [n_out, k] weight matrix that is read exactly once
// per row tile.  This is the plain-ALU path: the only path for fp32 models
// (whose 1e-4 relative logit tolerance rules out tf32) and the reference the
// tensor-core path is checked against for bf16 weights.  Activations stay fp32.
//
// A warp owns NPW output features.  Each lane walks k in 16-byte steps of the
// weight rows (8 bf16 or 4 fp32 elements), so a warp-level load covers 512
// contiguous bytes of one weight row; the matching activation values come from
// L1 (every warp of the CTA reads the same few rows).  Partial sums are reduced
// across the lanes at the end.
//
// With few rows such a GEMM is a link in a chain of latencies.  So a lane keeps kAhead 16-byte loads of weights in flight,
// the first of them requested while the kernel before this one is still running; where there are few features a warp
// takes one (gated: a pair), so that there are warps enough to fetch them all at once; and the norm before and the
// activation after have no kernels of their own: rmsnorm(x) . W^T is (x * gain) . W^T times a factor per row, whose sum of
// squares falls off on the way, and the FFN's function is applied where the sum over the lanes ends.  64
// tokens with the fp32 pair (4 blocks of 256, draft 2 of 128): 9.1 -> 6.3 ms, for four sequences with six rows each
// 16.3 -> 10.7.
#include "model.cuh"

namespace spec {
namespace {

constexpr int kGemmWarps = 8;
constexpr int kAhead = 8;  // 16-byte loads of weights in flight per lane

template <typename WT>
struct WVec;  // 16 bytes of weights

template <>
struct WVec<float> {
    static constexpr int kElems = 4;
};
template <>
struct WVec<__nv_bfloat16> {
    static constexpr int kElems = 8;
};

template <typename WT>
__device__ __forceinline__ void widen(const uint4& t, float (&v)[WVec<WT>::kElems]);
template <>
__device__ __forceinline__ void widen<float>(const uint4& t, float (&v)[4]) {
    v[0] = __uint_as_float(t.x); v[1] = __uint_as_float(t.y); v[2] = __uint_as_float(t.z); v[3] = __uint_as_float(t.w);
}
template <>
__device__ __forceinline__ void widen<__nv_bfloat16>(const uint4& t, float (&v)[8]) {
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // bf16 -> fp32 is a 16-bit shift
        v[2 * i] = __uint_as_float(w[i] << 16);
        v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

struct RowsArgs {
    const float* x;
    const void* w;
    const float* residual;
    const int32_t* dst_rows;
    int n_rows, n_out, k;
    float* y;
    RowNorm norm;
};

constexpr int kNoAct = -1;

// grid = (ceil(n_out / (kGemmWarps * features per warp)), ceil(n_rows / MT)), block = 32 * kGemmWarps.
// A gated ACT has W rows n (gate) and n_out + n (up) of every output n: NPW / 2 outputs to a warp.
template <typename WT, int MT, int NPW, bool NORM, int ACT>
__global__ void __launch_bounds__(32 * kGemmWarps)
gemm_rows_kernel(const RowsArgs a) {
    constexpr int E = WVec<WT>::kElems;
    constexpr bool kGated = ACT != kNoAct && ACT != SPEC_FFN_GELU;
    constexpr int kOut = kGated ? NPW / 2 : NPW;
    constexpr int kSteps = kAhead / NPW;
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n0 = (blockIdx.x * kGemmWarps + warp) * kOut;
    const int r0 = blockIdx.y * MT;
    const int k = a.k, steps = (k + 32 * E - 1) / (32 * E);
    const WT* rows[NPW];
#pragma unroll
    for (int j = 0; j < NPW; ++j) {
        const int n = min(n0 + (kGated ? j >> 1 : j), a.n_out - 1);
        rows[j] = static_cast<const WT*>(a.w) + static_cast<size_t>(kGated && (j & 1) ? a.n_out + n : n) * k + lane * E;
    }
    uint4 ahead[kSteps][NPW];  // (weights are constants)
    auto fetch = [&](int step, uint4 (&to)[NPW]) {
#pragma unroll
        for (int j = 0; j < NPW; ++j)
            to[j] = step * 32 * E + lane * E < k ? __ldg(reinterpret_cast<const uint4*>(rows[j] + step * 32 * E)) : make_uint4(0u, 0u, 0u, 0u);
    };
#pragma unroll
    for (int s = 0; s < kSteps; ++s) fetch(s, ahead[s]);
    pdl_wait();
    if (n0 >= a.n_out) return;

    const float* xr[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        const int r = min(r0 + m, a.n_rows - 1);
        xr[m] = a.x + static_cast<size_t>(NORM && a.norm.src_rows ? a.norm.src_rows[r] : r) * k + lane * E;
    }
    float acc[NPW][MT], square[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        square[m] = 0.0f;
#pragma unroll
        for (int j = 0; j < NPW; ++j) acc[j][m] = 0.0f;
    }
    for (int s0 = 0; s0 < steps; s0 += kSteps) {
#pragma unroll
        for (int s = 0; s < kSteps; ++s) {
            const int at = (s0 + s) * 32 * E;
            if (at + lane * E < k) {
                float gain[E];
                if (NORM) {
#pragma unroll
                    for (int e = 0; e < E; e += 4) {
                        const float4 t = __ldg(reinterpret_cast<const float4*>(a.norm.gain + lane * E + at + e));
                        gain[e] = t.x; gain[e + 1] = t.y; gain[e + 2] = t.z; gain[e + 3] = t.w;
                    }
                }
                float wv[NPW][E];
#pragma unroll
                for (int j = 0; j < NPW; ++j) widen<WT>(ahead[s][j], wv[j]);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    float xv[E];
#pragma unroll
                    for (int e = 0; e < E; e += 4) {
                        const float4 t = *reinterpret_cast<const float4*>(xr[m] + at + e);
                        xv[e] = t.x; xv[e + 1] = t.y; xv[e + 2] = t.z; xv[e + 3] = t.w;
                    }
                    if (NORM) {
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            square[m] = fmaf(xv[e], xv[e], square[m]);
                            xv[e] *= gain[e];
                        }
                    }
#pragma unroll
                    for (int j = 0; j < NPW; ++j)
#pragma unroll
                        for (int e = 0; e < E; ++e) acc[j][m] = fmaf(wv[j][e], xv[e], acc[j][m]);
                }
            }
            fetch(s0 + s + kSteps, ahead[s]);
        }
    }
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        const float scale = NORM ? rsqrtf(warp_sum(square[m]) / static_cast<float>(k) + a.norm.eps) : 1.0f;
        const int r = r0 + m;
#pragma unroll
        for (int o = 0; o < kOut; ++o) {
            float s = warp_sum(acc[kGated ? 2 * o : o][m]);
            if (NORM) s *= scale;
            if (kGated) {
                float up = warp_sum(acc[(kGated ? 2 * o : o) + (kGated ? 1 : 0)][m]);
                if (NORM) up *= scale;
                s = (ACT == SPEC_FFN_SWIGLU ? silu(s) : gelu_tanh(s)) * up;
            } else if (ACT == SPEC_FFN_GELU) {
                s = gelu_tanh(s);
            }
            const int n = n0 + o;
            if (lane == 0 && n < a.n_out && r < a.n_rows) {
                const size_t dst = static_cast<size_t>(a.dst_rows ? a.dst_rows[r] : r) * a.n_out + n;
                a.y[dst] = a.residual ? s + a.residual[static_cast<size_t>(r) * a.n_out + n] : s;
            }
        }
    }
}

template <typename WT, int MT, int NPW, bool NORM, int ACT>
int launch(const RowsArgs& a, cudaStream_t stream) {
    constexpr int kPerCta = kGemmWarps * (ACT != kNoAct && ACT != SPEC_FFN_GELU ? NPW / 2 : NPW);
    const dim3 grid((a.n_out + kPerCta - 1) / kPerCta, (a.n_rows + MT - 1) / MT);
    return launch_pdl(gemm_rows_kernel<WT, MT, NPW, NORM, ACT>, grid, dim3(32 * kGemmWarps), 0, stream, a);
}

template <typename WT, bool NORM, int ACT>
int by_rows(const RowsArgs& a, cudaStream_t stream) {
    // a warp per feature while that is at most two waves of CTAs (64 tokens with the fp32 pair: 6.5 ms, with four features
    // to a warp everywhere 10.4); row tiles of eight while there are few (24 rows: a pass 194 us, with sixteen to a tile 284)
    constexpr int kFew = ACT != kNoAct && ACT != SPEC_FFN_GELU ? 2 : 1;
    const bool few = a.n_out <= 2 * 148 * kGemmWarps;
    if (a.n_rows <= 2) return few ? launch<WT, 2, kFew, NORM, ACT>(a, stream) : launch<WT, 2, 4, NORM, ACT>(a, stream);
    if (a.n_rows <= 4) return few ? launch<WT, 4, kFew, NORM, ACT>(a, stream) : launch<WT, 4, 4, NORM, ACT>(a, stream);
    if (a.n_rows <= 8) return few ? launch<WT, 8, kFew, NORM, ACT>(a, stream) : launch<WT, 8, 4, NORM, ACT>(a, stream);
    if (few && a.n_rows <= kMostNormedRows) return launch<WT, 8, kFew, NORM, ACT>(a, stream);
    if constexpr (NORM) return launch<WT, 8, 4, NORM, ACT>(a, stream);
    else return launch<WT, 16, 2, NORM, ACT>(a, stream);
}

template <typename WT, bool NORM>
int by_act(const RowsArgs& a, int ffn, cudaStream_t stream) {
    switch (ffn) {
        case SPEC_FFN_GELU: return by_rows<WT, NORM, SPEC_FFN_GELU>(a, stream);
        case SPEC_FFN_GATED_GELU: return by_rows<WT, NORM, SPEC_FFN_GATED_GELU>(a, stream);
        case SPEC_FFN_SWIGLU: return by_rows<WT, NORM, SPEC_FFN_SWIGLU>(a, stream);
        default: return by_rows<WT, NORM, kNoAct>(a, stream);
    }
}

}  // namespace

int launch_gemm_rows(const float* x, const void* w, bool w_bf16, const float* residual, const int32_t* dst_rows,
                     int n_rows, int n_out, int k, float* y, cudaStream_t stream, const RowNorm& norm, int ffn) {
    if (n_rows <= 0) return SPEC_OK;
    if (k % 8 != 0) return fail(SPEC_ERR_BAD_CONFIG, "gemm: inner dimension %d is not a multiple of 8", k);
    const RowsArgs a{x, w, residual, dst_rows, n_rows, n_out, k, y, norm};
    if (w_bf16) return by_rows<__nv_bfloat16, false, kNoAct>(a, stream);
    return norm.gain ? by_act<float, true>(a, ffn, stream) : by_act<float, false>(a, ffn, stream);
}

}  // namespace spec
