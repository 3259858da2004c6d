// The blocks of a tiny fp32 decoder (128 or 256 wide, heads of 64, an FFN of four widths) over a few rows as ONE thread-block
// cluster of sixteen CTAs.
//
// Such a pass is latency: a block of the 256-wide model holds 3 MB of weights, all of them in L2, and took six dependent kernels
// of 2 to 6 us each.  Sixteen SMs hold what they need of a whole block in shared memory (192 KB each), fetched by bulk copies
// a block ahead, and hand one another their results through distributed shared memory: every exchange is 16-byte stores that
// are counted in bytes on an mbarrier of the receiver (st.async), so nobody looks at a flag and nothing goes through L2.
// CTA c owns, of every block, a part of one head's rows of Wqkv (the CTAs of a head share its three times 64 rows), that
// many dimensions of the head's output, sixteenths of the rows of Wo and W_in and of W_out.  Five exchanges a block:
// q, k, v among the CTAs of a head; attention output, residual stream, FFN activations and residual stream again among all.  The
// products are fp32 multiply-adds, a lane's inputs in registers, a warp's features summed over its lanes; norms come as a
// factor per row on the sums.
//
// What is left is that chain: five trips between SMs and a dozen block barriers.  Two blocks of the draft (128 wide, one row)
// 29 -> 16 us, four of the target (256 wide, four rows) 84 -> 39; 64 tokens with the fp32 pair 5.93 -> 3.35 ms.
// More rows than kRows need more shared memory than there is (256 wide) or are better spread over the GPU: the chain of kernels
// takes them, as it takes contexts of more than kMaxKeys positions.
//
// Every wait is bounded.  One that runs out is recorded; the kernel goes on with whatever is there (the others count on it),
// further waits give up at once, nothing more is asked for, and at the end the copies and the announced exchanges that are still in
// flight are waited for, with a limit; what nobody announced any more has a grace time to arrive before the CTA leaves.
#include <cfloat>
#include <climits>
#include <vector>

#include "cluster_util.cuh"
#include "model.cuh"

namespace spec {
namespace {

constexpr int kCtas = 16;
constexpr int kWarps = 16;
constexpr int kThreads = 32 * kWarps;
constexpr int kDh = 64;
constexpr int kMaxKeys = 256;
constexpr uint32_t kSpin = 1u << 20;   // tries of a bounded wait: about a second
constexpr uint32_t kDrain = 1u << 14;  // and of the last ones of a pass that gave up
constexpr uint32_t kGraceNs = 20000;   // a store between two SMs takes about one microsecond

__device__ int g_cluster_error;  // a bounded wait expired

struct ClusterLayer {
    const float *ln1, *wqkv, *wo, *ln2, *w_in, *w_out;
};
constexpr int kMaxLayers = 16;
struct ClusterArgs {
    ClusterLayer layers[kMaxLayers];  // (as kernel parameters: a table in memory would be a trip to it at the start of every block)
    int n_layers, rows, batch, m_rows;
    const int32_t *token, *pos, *seq;
    const float *tok_emb, *pos_emb;
    int vocab, max_positions;
    float* kv;
    size_t layer_stride;
    const int32_t* page_table;
    int pages_per_seq, page_shift;
    float eps;
    float* h_out;
    uint32_t limit;  // of every wait, in tries
    int mute;        // spec_timeout_drill_pass: nothing is sent
};

// R: rows at most
template <int D, int R>
struct Shape {
    static constexpr int kHeads = D / kDh;
    static constexpr int kGroup = kCtas / kHeads;  // CTAs of a head
    static constexpr int kDv = kDh / kGroup;       // of its dimensions to each
    static constexpr int kO = D / kCtas;           // features of the residual stream to a CTA
    static constexpr int kF = 4 * D;
    static constexpr int kFc = kF / kCtas;
    static constexpr int kWq = 0, kWo = kWq + 3 * kDv * D, kWi = kWo + kO * D, kW2 = kWi + kFc * D;  // weights, in floats
    static constexpr int kH = kW2 + kO * kF;      // residual stream [R][D]
    static constexpr int kXq = kH + R * D;        // the head's q, k, v [R][192]
    static constexpr int kOut = kXq + R * 3 * kDh;  // attention output [R][D]
    static constexpr int kAct = kOut + R * D;     // FFN activations [R][kF]; at another time scores [R][kMaxKeys]
    static constexpr int kRed = kAct + R * kF;    // sums of the warps [16][R][kDv] or [4][R][kO], results to be sent [R][kFc]
    static constexpr int kRedFloats = kWarps * R * kDv > R * kFc ? kWarps * R * kDv : R * kFc;
    static constexpr int kMeta = kRed + kRedFloats;  // positions, sequences, cache rows [8 each]
    static constexpr int kBars = kMeta + 24;         // 8 barriers
    static constexpr int kBytes = (kBars + 2 * 8) * 4;
    static_assert(R <= 8 && R * kMaxKeys <= R * kF, "scores fit");
    static_assert(kBytes <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void expect_bytes(uint64_t* bar, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// The totals over the warp of V values (a power of two, at most 16): lane l returns that of value l / (32 / V).
template <int V>
__device__ __forceinline__ float sum_over_lanes(float (&v)[V], int lane) {
    int o = 16;
#pragma unroll
    for (int half = V / 2; half >= 1; half /= 2, o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(kFullMask, send, o);
        }
    }
    float s = v[0];
#pragma unroll
    for (; o >= 1; o /= 2) s += __shfl_xor_sync(kFullMask, s, o);
    return s;
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float c) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, c))));
}

template <int D, int R>
struct Worker {
    using S = Shape<D, R>;
    static constexpr int kV4 = D / 128;  // 16-byte groups of a row of D to a lane
    enum { kBarWq, kBarWo, kBarWi, kBarW2, kBarX, kBarO, kBarH, kBarA };
    const ClusterArgs& a;
    float* sm;
    uint64_t* bars;
    int tid, lane, warp, cta;
    uint32_t limit;  // of every wait; 1 after one ran out
    uint32_t turns;  // a bit per barrier: its parity
    // what divisions by runtime numbers give, once for the pass: warps per sequence, this warp's sequence and place in it; the
    // sequence of row `warp`; sequence and place in it of row tid / kDv
    int wps, b, wi, warp_seq, out_seq, out_row;

    __device__ __forceinline__ void arrived(int which) {
        if (!bar_wait(bars + which, (turns >> which) & 1, limit)) limit = 1;
        turns ^= 1u << which;
    }
    __device__ __forceinline__ void await_bytes(int which, int bytes) {
        if (tid == 0 && limit != 1) expect_bytes(bars + which, bytes);
    }
    // One thread, after a barrier that followed the last reads of what was there.
    __device__ __forceinline__ void fetch(int which, float* to, const float* from, int floats) {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(to)), "l"(from),
                     "r"(floats * 4), "r"(smem_u32(bars + which))
                     : "memory");
    }
    __device__ __forceinline__ void fetch_qkv(int layer) {
        const int head = cta / S::kGroup, j = cta % S::kGroup;
        const float* w = a.layers[layer].wqkv;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        expect_bytes(bars + kBarWq, 3 * S::kDv * D * 4);
        for (int part = 0; part < 3; ++part)
            fetch(kBarWq, sm + S::kWq + part * S::kDv * D, w + static_cast<size_t>((part * S::kHeads + head) * kDh + j * S::kDv) * D, S::kDv * D);
    }
    __device__ __forceinline__ void fetch_rest(int layer) {
        const ClusterLayer& l = a.layers[layer];
        const float *wo = l.wo, *wi = l.w_in, *w2 = l.w_out;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        expect_bytes(bars + kBarWo, S::kO * D * 4);
        fetch(kBarWo, sm + S::kWo, wo + static_cast<size_t>(cta) * S::kO * D, S::kO * D);
        expect_bytes(bars + kBarWi, S::kFc * D * 4);
        fetch(kBarWi, sm + S::kWi, wi + static_cast<size_t>(cta) * S::kFc * D, S::kFc * D);
        expect_bytes(bars + kBarW2, S::kO * S::kF * 4);
        fetch(kBarW2, sm + S::kW2, w2 + static_cast<size_t>(cta) * S::kO * S::kF, S::kO * S::kF);
    }
    // N features (rows of `stride` floats at w) against the rows at x (`ld` floats apart), D inputs: [feature][row], a lane's share.
    template <int N, int P>
    __device__ __forceinline__ void products(const float* w, int stride, const float4 (&x)[R][kV4], float (&out)[P]) {
#pragma unroll
        for (int i = 0; i < P; ++i) out[i] = 0.0f;
#pragma unroll
        for (int n = 0; n < N; ++n)
#pragma unroll
            for (int g = 0; g < kV4; ++g) {
                const float4 t = *reinterpret_cast<const float4*>(w + n * stride + 128 * g + 4 * lane);
#pragma unroll
                for (int r = 0; r < R; ++r) out[n * R + r] = dot4(t, x[r][g], out[n * R + r]);
            }
    }
    __device__ __forceinline__ void load_rows(float4 (&x)[R][kV4], const float* from, int ld) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int g = 0; g < kV4; ++g)
                x[r][g] = r < a.rows ? *reinterpret_cast<const float4*>(from + r * ld + 128 * g + 4 * lane) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // x = the residual stream times the gain; lane l returns the norm's factor of row l / (32 / R).
    __device__ __forceinline__ float normed(float4 (&x)[R][kV4], const float4 (&gain)[kV4]) {
        load_rows(x, sm + S::kH, D);
        float ss[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            ss[r] = 0.0f;
#pragma unroll
            for (int g = 0; g < kV4; ++g) {
                ss[r] = dot4(x[r][g], x[r][g], ss[r]);
                x[r][g] = make_float4(x[r][g].x * gain[g].x, x[r][g].y * gain[g].y, x[r][g].z * gain[g].z, x[r][g].w * gain[g].w);
            }
        }
        return rsqrtf(sum_over_lanes(ss, lane) / static_cast<float>(D) + a.eps);
    }
    __device__ __forceinline__ void send(const float* here, int which, int rank, const float4& v) {
        if (!a.mute) send4(here, bars + which, rank, v);
    }
    // [rows][WIDTH] results in kRed go to everyone, row r to to + r * LD; the whole CTA, between two barriers.
    template <int WIDTH, int LD>
    __device__ __forceinline__ void share(float* to, int which) {
        constexpr int kGroups = R * (WIDTH / 4);
#pragma unroll
        for (int i = tid; i < kGroups * kCtas; i += kThreads) {
            const int peer = i / kGroups, at = i % kGroups, r = at / (WIDTH / 4), f = at % (WIDTH / 4) * 4;
            if (r < a.rows) send(to + r * LD + f, which, peer, *reinterpret_cast<const float4*>(sm + S::kRed + r * WIDTH + f));
        }
    }
    __device__ __forceinline__ const int* row_pos() const { return reinterpret_cast<const int*>(sm + S::kMeta); }
    __device__ __forceinline__ const int* row_seq() const { return row_pos() + 8; }

    __device__ __forceinline__ void block(int layer) {
        const ClusterLayer& l = a.layers[layer];
        float4 gain1[kV4], gain2[kV4];
#pragma unroll
        for (int g = 0; g < kV4; ++g) {
            gain1[g] = __ldg(reinterpret_cast<const float4*>(l.ln1 + 128 * g + 4 * lane));
            gain2[g] = __ldg(reinterpret_cast<const float4*>(l.ln2 + 128 * g + 4 * lane));
        }
        const int head = cta / S::kGroup, j = cta % S::kGroup;
        float* red = sm + S::kRed;
        float* pool = a.kv + layer * a.layer_stride;
        // this warp's share of the keys: one sequence, every wps-th group of eight; the first are fetched ahead
        const bool live = b < a.batch;
        int cached = 0;
        const int32_t* pages = nullptr;
        if (live) {
            cached = min(max(row_pos()[b * a.m_rows], 0), kMaxKeys);
            pages = a.page_table + row_seq()[b * a.m_rows] * a.pages_per_seq;
        }
        const int total = live ? min(cached + a.m_rows, kMaxKeys) : 0;
        auto cache_row = [&](int key, int v) {
            const size_t page = pages[key >> a.page_shift];
            return pool + ((((page * 2 + v) * S::kHeads + head) << a.page_shift) + (key & ((1 << a.page_shift) - 1))) * kDh;
        };
        const int kk = lane >> 2, t = lane & 3;
        float4 k4[4];
        auto fetch_key = [&](int key) {
            if (key < cached) {
                const float* p = cache_row(key, 0);
#pragma unroll
                for (int i = 0; i < 4; ++i) k4[i] = __ldcg(reinterpret_cast<const float4*>(p + 16 * i + 4 * t));
            }
        };
        int key = 8 * wi + kk;
        fetch_key(key);

        // ---- q, k, v ----
        {
            constexpr int kN = 3 * S::kDv / kWarps + (3 * S::kDv % kWarps ? 1 : 0), kUsed = 3 * S::kDv / kN;
            constexpr int kP = kN * R <= 8 ? 8 : 16;
            static_assert(kN * kUsed == 3 * S::kDv && kN * R <= kP, "features over the warps");
            if (layer > 0) arrived(kBarH);
            arrived(kBarWq);
            float4 x[R][kV4];
            const float factor = normed(x, gain1);
            if (warp < kUsed) {
                float out[kP];
                products<kN>(sm + S::kWq + warp * kN * D, D, x, out);
                const float y = sum_over_lanes(out, lane);
                const int at = lane / (32 / kP), n = at / R, r = at % R;
                const float f = __shfl_sync(kFullMask, factor, r * (32 / R));
                if (lane % (32 / kP) == 0 && n < kN && r < a.rows) red[r * 3 * S::kDv + warp * kN + n] = y * f;
            }
        }
        await_bytes(kBarX, a.rows * 3 * kDh * 4);
        __syncthreads();
        if (tid == 0 && layer + 1 < a.n_layers && limit != 1) fetch_qkv(layer + 1);
        float* xq = sm + S::kXq;
        {
            constexpr int kGroups = 3 * S::kDv / 4;
#pragma unroll 1
            for (int i = tid; i < R * kGroups * S::kGroup; i += kThreads) {
                const int peer = i / (R * kGroups), at = i % (R * kGroups), r = at / kGroups, f = at % kGroups * 4;
                if (r >= a.rows) continue;
                const int part = f / S::kDv, dim = j * S::kDv + f % S::kDv;
                const float4 y = *reinterpret_cast<const float4*>(red + r * 3 * S::kDv + f);
                send(xq + r * 3 * kDh + part * kDh + dim, kBarX, head * S::kGroup + peer, y);
                const int p = row_pos()[r];
                if (peer == 0 && part > 0 && p >= 0) {
                    const size_t page = a.page_table[row_seq()[r] * a.pages_per_seq + (p >> a.page_shift)];
                    float* dst = pool + ((((page * 2 + part - 1) * S::kHeads + head) << a.page_shift) + (p & ((1 << a.page_shift) - 1))) * kDh + dim;
                    *reinterpret_cast<float4*>(dst) = y;
                }
            }
        }
        arrived(kBarX);
        // ---- attention: scores ----
        float* sc = sm + S::kAct;
#pragma unroll 1
        for (int first = 0; first < total; first += 8 * wps) {  // (the same for all lanes of a warp)
            key = first + 8 * wi + kk;
            if (first > 0) fetch_key(key);
            const int own = key - cached;
            if (own >= 0 && own < a.m_rows) {
                const float* p = xq + (b * a.m_rows + own) * 3 * kDh + kDh;
#pragma unroll
                for (int i = 0; i < 4; ++i) k4[i] = *reinterpret_cast<const float4*>(p + 16 * i + 4 * t);
            } else if (key >= total) {
#pragma unroll
                for (int i = 0; i < 4; ++i) k4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            // (an inactive row, at a position below 0, is nobody's key; what is not a row's key has a score of -inf, and a NaN is
            // a score like any other: it has to reach the logits, where it is reported)
            const int at = own < 0 ? key : own < a.m_rows ? row_pos()[b * a.m_rows + own] : -1;
#pragma unroll 1
            for (int i = 0; i < a.m_rows; ++i) {
                const int r = b * a.m_rows + i;
                float s = 0.0f;
#pragma unroll
                for (int g = 0; g < 4; ++g) s = dot4(k4[g], *reinterpret_cast<const float4*>(xq + r * 3 * kDh + 16 * g + 4 * t), s);
                s += __shfl_xor_sync(kFullMask, s, 1);
                s += __shfl_xor_sync(kFullMask, s, 2);
                if (t == 0 && key < total) sc[r * kMaxKeys + key] = at >= 0 && at <= row_pos()[r] ? s * 0.125f : -INFINITY;
            }
        }
        __syncthreads();
        if (warp < a.rows) {  // weights, a warp to a row
            const int n = min(min(max(row_pos()[warp_seq * a.m_rows], 0), kMaxKeys) + a.m_rows, kMaxKeys);
            float* p = sc + warp * kMaxKeys;
            float top = -FLT_MAX;
            for (int i = lane; i < n; i += 32) top = fmaxf(top, p[i]);
            top = warp_max(top);
            float sum = 0.0f;
            for (int i = lane; i < n; i += 32) {
                const float e = expf(p[i] - top);  // (top is finite where every score is -inf)
                p[i] = e;
                sum += e;
            }
            sum = warp_sum(sum);
            const float inv = sum == 0.0f ? 0.0f : 1.0f / sum;
            for (int i = lane; i < n; i += 32) p[i] *= inv;
        }
        __syncthreads();
        {  // this CTA's dimensions of the head's output: lanes are a dimension and one of kSubs keys
            constexpr int kSubs = 32 / S::kDv;
            const int dim = lane % S::kDv, sub = lane / S::kDv;
            float acc[R];
#pragma unroll
            for (int i = 0; i < R; ++i) acc[i] = 0.0f;
#pragma unroll 4
            for (int at = wi * kSubs + sub; at < total; at += wps * kSubs) {
                const int own = at - cached;
                const float v = own < 0 ? __ldcg(cache_row(at, 1) + j * S::kDv + dim)
                                        : xq[(b * a.m_rows + own) * 3 * kDh + 2 * kDh + j * S::kDv + dim];
                // (a row of the pass is nothing to those in front of it, not even 0 times its value, which may be no number)
                const int from = own < 0 ? INT_MIN : row_pos()[b * a.m_rows + own] < 0 ? INT_MAX : row_pos()[b * a.m_rows + own];
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (i < a.m_rows && row_pos()[b * a.m_rows + i] >= from)
                        acc[i] = fmaf(sc[(b * a.m_rows + i) * kMaxKeys + at], v, acc[i]);
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int o = S::kDv; o < 32; o *= 2) acc[i] += __shfl_xor_sync(kFullMask, acc[i], o);
            if (sub == 0)
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (i < a.m_rows) red[(warp * R + i) * S::kDv + dim] = acc[i];
        }
        await_bytes(kBarO, a.rows * D * 4);
        __syncthreads();
        if (tid < R * S::kDv) {  // (whole warps)
            const int r = tid / S::kDv, dim = tid % S::kDv;
            float o = 0.0f;
            if (r < a.rows) {
                const float* p = red + (out_seq * wps * R + out_row) * S::kDv + dim;
#pragma unroll 4
                for (int w = 0; w < wps; ++w) o += p[w * R * S::kDv];
            }
            spread(o, r, sm + S::kOut + r * D + head * kDh + j * S::kDv + (dim & ~3), kBarO);
        }
        // ---- output projection ----
        arrived(kBarO);
        arrived(kBarWo);
        float* stage = red;
        {
            float4 x[R][kV4];
            load_rows(x, sm + S::kOut, D);
            float y = 0.0f;
            if (warp < S::kO) {
                float out[R];
                products<1>(sm + S::kWo + warp * D, D, x, out);
                y = sum_over_lanes(out, lane);
            }
            __syncthreads();  // (the sums of the warps have been read)
            const int r = lane / (32 / R);
            if (warp < S::kO && lane % (32 / R) == 0 && r < a.rows) stage[r * S::kO + warp] = y + sm[S::kH + r * D + cta * S::kO + warp];
        }
        await_bytes(kBarH, a.rows * D * 4);
        __syncthreads();
        share<S::kO, D>(sm + S::kH + cta * S::kO, kBarH);
        arrived(kBarH);
        // ---- FFN ----
        arrived(kBarWi);
        {
            constexpr int kN = S::kFc / kWarps, kP = kN * R;
            static_assert(kP == 16, "features over the warps");
            float4 x[R][kV4];
            const float factor = normed(x, gain2);
            float out[kP];
            products<kN>(sm + S::kWi + warp * kN * D, D, x, out);
            const float y = sum_over_lanes(out, lane);
            const int at = lane / 2, n = at / R, r = at % R;
            const float f = __shfl_sync(kFullMask, factor, r * (32 / R));
            __syncthreads();  // (what was sent from here has been read)
            if (lane % 2 == 0 && r < a.rows) stage[r * S::kFc + warp * kN + n] = gelu_tanh(y * f);
        }
        await_bytes(kBarA, a.rows * S::kF * 4);
        __syncthreads();
        share<S::kFc, S::kF>(sm + S::kAct + cta * S::kFc, kBarA);
        arrived(kBarA);
        arrived(kBarW2);
        {  // a quarter of the inputs to a warp
            constexpr int kN = S::kO / 4, kP = kN * R;
            static_assert(kP == 16, "features over the warps");
            const int quarter = warp >> 2, n0 = (warp & 3) * kN;
            float4 x[R][kV4];
            load_rows(x, sm + S::kAct + quarter * D, S::kF);
            float out[kP];
            products<kN>(sm + S::kW2 + n0 * S::kF + quarter * D, S::kF, x, out);
            const float y = sum_over_lanes(out, lane);
            const int at = lane / 2, n = at / R, r = at % R;
            __syncthreads();  // (what was sent from here has been read)
            if (lane % 2 == 0) red[(quarter * R + r) * S::kO + n0 + n] = y;
        }
        const bool last = layer + 1 == a.n_layers;
        if (!last) await_bytes(kBarH, a.rows * D * 4);
        __syncthreads();
        if (tid == 0 && !last && limit != 1) fetch_rest(layer + 1);
        if (tid < R * S::kO) {  // (whole warps)
            const int r = tid / S::kO, f = tid % S::kO;
            float y = 0.0f;
            if (r < a.rows) {
                y = sm[S::kH + r * D + cta * S::kO + f];
#pragma unroll
                for (int q = 0; q < 4; ++q) y += red[(q * R + r) * S::kO + f];
                if (last) a.h_out[r * D + cta * S::kO + f] = y;
            }
            if (!last) spread(y, r, sm + S::kH + r * D + cta * S::kO + (f & ~3), kBarH);
        }
    }
    // Four lanes' values, 16 bytes of row r, to everyone: lane i of the four to peers 4 i .. 4 i + 3.
    __device__ __forceinline__ void spread(float v, int r, float* to, int which) {
        float4 q;
        q.x = __shfl_sync(kFullMask, v, lane & ~3);
        q.y = __shfl_sync(kFullMask, v, (lane & ~3) + 1);
        q.z = __shfl_sync(kFullMask, v, (lane & ~3) + 2);
        q.w = __shfl_sync(kFullMask, v, (lane & ~3) + 3);
        if (r < a.rows)
#pragma unroll
            for (int i = 0; i < 4; ++i) send(to, which, 4 * (lane & 3) + i, q);
    }
};

template <int D, int R>
__global__ void __launch_bounds__(kThreads, 1) cluster_pass_kernel(const __grid_constant__ ClusterArgs a) {
    extern __shared__ __align__(128) float sm[];
    using S = Shape<D, R>;
    using W = Worker<D, R>;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + S::kBars);
    const int tid = threadIdx.x;
    uint32_t cta;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(cta));
    if (tid == 0) {
        for (int i = 0; i < 8; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[i])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    W w{a, sm, bars, tid, tid & 31, tid >> 5, static_cast<int>(cta), a.limit, 0, kWarps / a.batch, 0, 0, 0, 0, 0};
    w.b = w.warp / w.wps;
    w.wi = w.warp % w.wps;
    w.warp_seq = w.warp / a.m_rows;
    w.out_seq = tid / S::kDv / a.m_rows;
    w.out_row = tid / S::kDv % a.m_rows;
    if (tid == 0) {  // (weights are constants)
        w.fetch_qkv(0);
        w.fetch_rest(0);
    }
    pdl_wait();
    pdl_trigger();
    for (int i = tid; i < a.rows * D / 4; i += kThreads) {
        const int r = 4 * i / D, e = 4 * i % D;
        const int tok = min(max(__ldcg(a.token + r), 0), a.vocab - 1), p = min(max(__ldcg(a.pos + r), 0), a.max_positions - 1);
        const float4 x = __ldg(reinterpret_cast<const float4*>(a.tok_emb + static_cast<size_t>(tok) * D + e));
        const float4 y = __ldg(reinterpret_cast<const float4*>(a.pos_emb + static_cast<size_t>(p) * D + e));
        *reinterpret_cast<float4*>(sm + S::kH + r * D + e) = make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w);
    }
    if (tid < a.rows) {
        int* meta = reinterpret_cast<int*>(sm + S::kMeta);
        meta[tid] = __ldcg(a.pos + tid);
        meta[8 + tid] = __ldcg(a.seq + tid);
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // (every peer's barriers are there)
    __syncthreads();
#pragma unroll 1
    for (int l = 0; l < a.n_layers; ++l) w.block(l);
    if (w.limit == 1) {
        atomicCAS(&g_cluster_error, 0, 1);
        if (tid == 0)  // what this thread asked for or announced: a barrier is past one of the two parities at any time
            for (int i = 0; i < 8; ++i) bar_wait(&bars[i], 0, kDrain), bar_wait(&bars[i], 1, kDrain);
    }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // nobody leaves while a peer may still write here
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // (a CTA whose waits have all been met has received everything; of the others some stores may be issued and not here yet)
    if (w.limit == 1) __nanosleep(kGraceNs);
}

using ClusterFn = void (*)(const ClusterArgs);
struct Variant {
    ClusterFn fn;
    int smem, rows;
};
Variant variant(int d) {
    return d == 256 ? Variant{cluster_pass_kernel<256, 4>, Shape<256, 4>::kBytes, 4} : Variant{cluster_pass_kernel<128, 8>, Shape<128, 8>::kBytes, 8};
}
cudaLaunchConfig_t launch_config(const Variant& v, cudaStream_t stream, cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCtas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = v.smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCtas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return cfg;
}

bool aligned(const void* p) { return p && (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

int cluster_pass_init(ClusterPass& s, const Model& m, int max_len) {
    s = ClusterPass{};
    const spec_model_cfg& c = m.cfg;
    if (m.bf16() || c.arch != SPEC_ARCH_GPT || c.ffn != SPEC_FFN_GELU || (c.d_model != 128 && c.d_model != 256) || c.d_head != kDh ||
        c.n_heads * kDh != c.d_model || c.n_kv_heads != c.n_heads || c.d_ff != 4 * c.d_model || m.kv_dtype != SPEC_DTYPE_FP32 ||
        c.n_layers > kMaxLayers || max_len > kMaxKeys || !aligned(m.tok_emb) || !aligned(m.pos_emb))
        return SPEC_OK;
    for (const spec_layer_weights& w : m.layers)
        for (const void* p : {static_cast<const void*>(w.ln1), w.wqkv, w.wo, static_cast<const void*>(w.ln2), w.w_in, w.w_out})
            if (!aligned(p)) return SPEC_OK;
    static std::atomic<unsigned long long> configured{0};
    static std::atomic<unsigned long long> fits[2];  // a bit per device: sixteen SMs side by side, with this much shared memory
    const int status = once_on_this_device(configured, []() -> int {
        for (int d = 128; d <= 256; d *= 2) {
            SPEC_CUDA_TRY(cudaFuncSetAttribute(variant(d).fn, cudaFuncAttributeMaxDynamicSharedMemorySize, variant(d).smem));
            SPEC_CUDA_TRY(cudaFuncSetAttribute(variant(d).fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            cudaLaunchAttribute attr[2];
            cudaLaunchConfig_t cfg = launch_config(variant(d), nullptr, attr);
            cfg.numAttrs = 1;
            int resident = 0, device = 0;
            if (cudaOccupancyMaxActiveClusters(&resident, variant(d).fn, &cfg) != cudaSuccess) cudaGetLastError();
            SPEC_CUDA_TRY(cudaGetDevice(&device));
            if (resident > 0 && device < 64) fits[d / 256].fetch_or(1ull << device);
        }
        return SPEC_OK;
    });
    if (status != SPEC_OK) return status;
    int device = 0;
    SPEC_CUDA_TRY(cudaGetDevice(&device));
    if (device >= 64 || !((fits[c.d_model / 256].load() >> device) & 1)) return SPEC_OK;
    s.rows = variant(c.d_model).rows;
    return SPEC_OK;
}

bool cluster_pass_serves(const ClusterPass& s, int batch, int m_rows) { return batch * m_rows <= s.rows; }

int launch_cluster_pass(const Model& m, const RowMeta& rows, const PassTables& t, int batch, int m_rows, float* h,
                        cudaStream_t stream, bool drill) {
    const spec_model_cfg& c = m.cfg;
    ClusterArgs a{};
    auto f = [](const void* p) { return static_cast<const float*>(p); };
    for (int l = 0; l < c.n_layers; ++l) {
        const spec_layer_weights& w = m.layers[l];
        a.layers[l] = ClusterLayer{w.ln1, f(w.wqkv), f(w.wo), w.ln2, f(w.w_in), f(w.w_out)};
    }
    a.n_layers = c.n_layers;
    a.rows = batch * m_rows;
    a.batch = batch;
    a.m_rows = m_rows;
    a.token = rows.token;
    a.pos = rows.pos;
    a.seq = rows.seq;
    a.tok_emb = static_cast<const float*>(m.tok_emb);
    a.pos_emb = static_cast<const float*>(m.pos_emb);
    a.vocab = c.vocab;
    a.max_positions = c.max_positions;
    a.kv = static_cast<float*>(m.kv);
    a.layer_stride = m.layer_stride / sizeof(float);
    a.page_table = t.page_table;
    a.pages_per_seq = t.pages_per_seq;
    while ((1 << a.page_shift) < t.page_size) ++a.page_shift;
    a.eps = c.rms_eps;
    a.h_out = h;
    a.limit = drill ? 64 : kSpin;
    a.mute = drill ? 1 : 0;
    const Variant v = variant(c.d_model);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = launch_config(v, stream, attr);
    SPEC_CUDA_TRY(cudaLaunchKernelEx(&cfg, v.fn, a));
    return SPEC_OK;
}

int* cluster_pass_error_word() { return symbol_address(g_cluster_error); }
int cluster_pass_take_error() {
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_cluster_error, sizeof(int)) != cudaSuccess) return -1;
    if (v) cudaMemcpyToSymbol(g_cluster_error, &zero, sizeof(int));
    return v;
}

}  // namespace spec
