// The blocks of a small decoder over a few rows as ONE kernel (bf16 models up to 768 wide with heads of 64: drafts,
// and targets of a hundred million parameters).
//
// Such a pass is latency: a block of the 160M shape streams 19 MB, three microseconds of HBM, through nine dependent
// kernels of three microseconds each.  Here the GPU is cut the way a tensor-parallel job cuts a model: 16 clusters of
// 8 CTAs, one per SM.  Cluster i < n_kv_heads owns KV head i - its rows of Wqkv, the attention of its queries, its
// columns of Wo - and every CTA owns some 16-column pieces of the FFN, the rows of W_in and the columns of W_out that
// belong to them.  Everything between two additions into the residual stream then stays inside a cluster, and the GPU
// meets twice per block (three times with cross-attention): CTA j of every cluster - the owner of feature slice j -
// publishes its partial sums of the branch as (value, epoch) pairs, CTA j of every other cluster polls the pairs
// themselves - no fence, no flag, one trip through L2 -, adds them up in a fixed order and hands the sum to its cluster
// through distributed shared memory (st.async, counted in bytes on an mbarrier of the receiver).
//
// The weights are packed once, per CTA, in the order in which the CTA uses them, as mma.sync m16n8k16 A fragments
// (16 features x 16 inputs, one 16-byte load per lane); bulk copies stream them through a ring of as many stages as the
// rows' buffers leave room for, refilled after every barrier that follows a read, which so runs ahead across every wait.
// The rows (at most 8) are the N side, as two bf16 terms.  With K cut over 16 warps the B fragments of a whole phase sit in
// registers.  The factor per row of the norms is applied to the projections' sums, not to their inputs: a projection
// starts when the residual stream is there.  The first keys of a warp load while the projection's sums are made.
//
// What is left is the length of the chain of such steps and instruction issue: in the CTAs that own a head a fifth to a
// quarter of a pass is waiting for another SM (8 to 10 % for other clusters, 12 to 15 within their own), 3 to 5 % for
// weights (clock() around the waits: 160M shape one row, 97M six rows, 6M one row).  The code runs once per block, straight through.  So every loop that is not a handful of instructions stays a loop, and what
// a division by a runtime number would give is prepared (written out, the waits alone made 90 KB of code, and the phases
// were two thirds slower).
//
// Every wait is bounded.  A wait that runs out is recorded and the kernel goes on with whatever is there (nobody leaves:
// the others count on it); further waits then give up at once, nothing more is asked for - a barrier whose bytes are still
// on their way must not be armed again -, and at the end the copies that are still in flight are waited for, with a limit.
//
// Measured, a whole pass with its head, chain of kernels against this: 160M shape, one row at context 1024 351 -> 199 us,
// four sequences at 777 397 -> 267, eight at 500 411 -> 340; 97M shape, six rows at 200 348 -> 245, eight sequences at 500
// 393 -> 324; 6M shape 56 -> 29; decoder of the small T5 shape, one row 257 -> 121, eight sequences 272 -> 193.  More rows
// would need a second column tile per fragment and twice the shared memory: the chain takes them.
#include <algorithm>
#include <cfloat>
#include <vector>

#include <cuda_fp16.h>

#include "cluster_util.cuh"
#include "model.cuh"

namespace spec {
namespace {

constexpr int kC = 8;             // CTAs per cluster
constexpr int kClusters = 16;     // at most: as many as are resident at once (15 on a B200 with one GPC short of 16 SMs)
constexpr int kWarps = 16;        // consumer warps
constexpr int kThreads = 32 * kWarps;
constexpr int kChunk = 8192;      // a fragment per warp; a ring stage is d / 256 of them: sixteen features over all inputs
constexpr int kMaxSmem = 227 * 1024;
constexpr int kRows = 8;
constexpr int kMaxD = 768;
constexpr int kMaxKi = kMaxD / 256;
constexpr int kDh = 64;
constexpr int kStateLen = 68;     // an attention state: max, sum, two of padding, 64 values
constexpr uint32_t kSpin = 1u << 20;  // tries of a bounded wait: about a second
constexpr uint32_t kDrain = 1u << 14;  // and of the last ones of a pass that gave up
constexpr float kLog2e = 1.4426950408889634f;

__device__ int g_small_error;  // first bounded wait that expired (0 = none)

struct SmallArgs {
    const uint8_t* stream;
    size_t cta_bytes, layer_stride, cross_stride;
    int n_layers, n_heads, n_kv_heads, units, gated, ffn, cross, clusters;
    int rows, batch, m_rows;
    const float* gains;  // [layers][3][d]: of attention, cross-attention, FFN
    const int32_t *token, *pos, *seq;
    const __nv_bfloat16 *tok_emb, *pos_emb;
    int vocab, max_positions;
    const float2* rope;
    __half *kv, *cross_kv;
    const int32_t *page_table, *src_page_table, *src_len;
    int pages_per_seq, src_pages_per_seq, page_size;
    const float* bias;
    int bias_span, bias_zero;
    float eps, inv_d;
    int per_group, per_rows, per_warp, warps_per_seq, page_shift;  // per_x: ceil(256 / x) of group, m_rows, warps_per_seq
    unsigned long long* exchanges;        // [4][16][8][d] pairs (value, epoch)
    unsigned* epoch;                      // exchanges of all passes so far
    float* last_part;                     // [clusters][rows][d]: the last FFN's partial sums
    float* h_out;
    uint32_t limit;                       // of every wait, in tries
    int mute;                             // spec_timeout_drill_pass: nothing is published
};

// ---- what a CTA streams, phase by phase (the packing kernel and the pass agree on it through these) ----
// tile lists: `qkv_tiles` 16-feature tiles of a head's projection, `wo` fragments, FFN units
__host__ __device__ inline int tiles_of(int n, int rank) { return n > rank ? (n - rank + kC - 1) / kC : 0; }  // tiles rank, rank + 8, ..
__host__ __device__ inline int qkv_tiles(int group) { return (group + 2) * 4; }
__host__ __device__ inline int units_of(int units, int cta, int ctas) {  // the last CTAs first: the ones without a head
    return units / ctas + (ctas - 1 - cta < units % ctas ? 1 : 0);
}
__host__ __device__ inline int unit_index(int cta, int i, int ctas) { return ctas - 1 - cta + i * ctas; }
__host__ __device__ inline int wo_stages(int group) { return (group + 1) / 2; }  // d / 128 * 4 group fragments, d / 16 to a stage

// KI = d / 256; R: rows at most.  What is left of the shared memory is the ring.
template <int KI, int R>
struct Smem {
    static constexpr int kD = 256 * KI;
    static constexpr int kRed = 0;  // cross-warp sums [4 tiles][16 warps][16][8] / attention states of the warps [16][8][68]
    static constexpr int kH = kRed + kWarps * 8 * kStateLen * 4;      // [2][R][d]
    // what the cluster's CTAs send: the rows' q, k, v [R][(group + 2) * 64] (group <= 4), the attention states
    // [8 ranks][8 queries][68]; over both, at another time, the FFN's partial sums [8 ranks][d / 8][R]
    static constexpr int kXq = kH + 2 * R * kD * 4;
    static constexpr int kState = kXq + R * 6 * kDh * 4;
    static constexpr int kFred = kXq;
    static constexpr int kAct = kState + kC * 8 * kStateLen * 4;      // act hi, lo [2 units][8][16]; attention output hi, lo [R][256]
    static constexpr int kGain = kAct + 2 * (R > 2 ? R : 2) * 256 * 2;  // [d]
    static constexpr int kSsq = kGain + kD * 4;                       // [8][16]
    static constexpr int kRope = kSsq + 16 * 8 * 4;                   // (cos, sin) [R][32]
    static constexpr int kMeta = kRope + R * 32 * 8;                  // positions, sequences, cache rows [8]; stages asked for
    static constexpr int kBars = kMeta + 28 * 4;                      // four for what the cluster sends, the ring's
    static constexpr int kStage = KI * kChunk;
    static constexpr int kRing = (kBars + (4 + 16) * 8 + 127) / 128 * 128;
    static constexpr int kFit = (kMaxSmem - kRing) / kStage;
    static constexpr int kStages = kFit < 16 ? kFit : 16;
    static constexpr int kTotal = kRing + kStages * kStage;
    static_assert(kD * R * 4 <= kAct - kXq, "the FFN's partial sums fit over q, k, v and the states");
    static_assert(kStages >= 4, "what a phase reads fits");
};

// A value and the exchange it belongs to in one 8-byte word.
__device__ __forceinline__ void publish(unsigned long long* at, float v, unsigned epoch) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(at), "l"((static_cast<unsigned long long>(epoch) << 32) | __float_as_uint(v)) : "memory");
}
// Two neighbouring words (each is whole, whichever of them is there first).
__device__ __forceinline__ ulonglong2 peek2(const unsigned long long* at) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(at) : "memory");
    return v;
}
__device__ __forceinline__ void sync_consumers() { __syncthreads(); }
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_half(float x, float y) {
    const __half2 h = __floats2half2_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void split_half(float x, float y, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(x, y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = pack_half(x - __low2float(h), y - __high2float(h));
}
__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float clamp_half(float x) { return __half2float(__float2half_rn(fminf(fmaxf(x, -65504.0f), 65504.0f))); }
// One CTA's view of the pass.  KI = d / 256: k-steps per warp.
template <int KI, int R>
struct Pass {
    using S = Smem<KI, R>;
    static constexpr int kBarH = 0, kBarQ = 1, kBarS = 2, kBarF = 3;  // residual stream; q, k, v; attention states; FFN sums
    static constexpr int kD = S::kD, kDs = kD / kC, kStages = S::kStages;
    const SmallArgs& a;
    uint8_t* sm;
    uint64_t *bars, *full;   // what the cluster sends (kBarH ..); ring stages
    int tid, lane, warp, rank, cluster;
    uint32_t limit;          // of every wait; 1 after one ran out
    int taken, ring;         // stages read; the next one to read, plus kStages in every second lap
    uint32_t turns;          // a bit per barrier of the cluster's: parity of its exchanges so far
    int cur;                 // which half of the residual stream is the present one
    unsigned epoch;          // the latest exchange of partial sums

    __device__ __forceinline__ void expect(bool ok) { limit = ok ? limit : 1; }  // (the waits that follow give up at once; nobody leaves)
    // Asks for as many stages as the ring has room for, a lane each.  Called where a barrier has just followed the last reads.
    __device__ __forceinline__ void refill() {
        if (warp == kWarps - 1 && !__any_sync(kFullMask, limit == 1)) {
            int* asked = reinterpret_cast<int*>(sm + S::kMeta) + 24;  // stages so far, and in all
            const int from = asked[0], n = min(taken + kStages, asked[1]) - from;
            __syncwarp();
            if (lane < n) {
                const int at = from + lane, s = at % kStages;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(S::kStage) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                 smem_u32(sm + S::kRing + s * S::kStage)),
                             "l"(a.stream + blockIdx.x * a.cta_bytes + static_cast<size_t>(at) * S::kStage), "r"(S::kStage), "r"(smem_u32(&full[s]))
                             : "memory");
            }
            if (lane == 0) asked[0] = from + max(n, 0);
            __syncwarp();
        }
    }
    // this warp's fragments of the next stage
    __device__ __forceinline__ void fragments(uint4 (&f)[KI]) {
        const bool lap = ring >= kStages;
        const int s = lap ? ring - kStages : ring;
        expect(bar_wait(&full[s], lap, limit));
        const uint8_t* p = sm + S::kRing + s * S::kStage + warp * 512 + lane * 16;
#pragma unroll
        for (int i = 0; i < KI; ++i) f[i] = *reinterpret_cast<const uint4*>(p + i * kChunk);
        ++taken;
        ring = ring + 1 == 2 * kStages ? 0 : ring + 1;
    }
    // `bytes` will be sent to this CTA on barrier `which`; one thread says so.
    __device__ __forceinline__ void await_bytes(int which, int bytes) {
        if (tid == 0 && limit != 1) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bars + which)), "r"(bytes) : "memory");
    }
    __device__ __forceinline__ void arrived(int which) {
        expect(bar_wait(bars + which, (turns >> which) & 1, limit));
        turns ^= 1u << which;
    }
    __device__ __forceinline__ float* red() const { return reinterpret_cast<float*>(sm + S::kRed); }
    __device__ __forceinline__ float* h(int half) const { return reinterpret_cast<float*>(sm + S::kH) + half * R * kD; }
    __device__ __forceinline__ const int* row_pos() const { return reinterpret_cast<const int*>(sm + S::kMeta); }
    __device__ __forceinline__ const int* row_seq() const { return row_pos() + 8; }
    __device__ __forceinline__ const int* row_at() const { return row_pos() + 16; }  // where a row goes in the cache
    __device__ __forceinline__ int by_group(int q) const { return q * a.per_group >> 8; }  // q / group, q < 8

    // v += the `count` published values of two neighbouring elements, in cluster order.
    __device__ __forceinline__ void gather(const unsigned long long* at, int count, unsigned when, float2& v) {
        constexpr int kStride = kRows * kD;  // (known here: the addresses take no registers)
        const unsigned long long nobody = static_cast<unsigned long long>(when) << 32;  // 0.0f
        ulonglong2 w[kClusters];
#pragma unroll 1
        for (uint32_t spin = 0;; ++spin) {
            bool all = true;
#pragma unroll
            for (int c = 0; c < kClusters; ++c) w[c] = c < count ? peek2(at + c * kStride) : make_ulonglong2(nobody, nobody);
#pragma unroll
            for (int c = 0; c < kClusters; ++c) all &= static_cast<unsigned>(w[c].x >> 32) == when && static_cast<unsigned>(w[c].y >> 32) == when;
            if (all) break;
            if (spin >= limit) {
                limit = 1;
                break;
            }
        }
#pragma unroll
        for (int c = 0; c < kClusters; ++c) {
            v.x += __uint_as_float(static_cast<unsigned>(w[c].x));
            v.y += __uint_as_float(static_cast<unsigned>(w[c].y));
        }
    }
    // The exchange buffer of an epoch.  Four take turns: whoever publishes an exchange has, since the one four before it,
    // waited for an FFN's sums of every cluster, and they have read what came before.
    __device__ __forceinline__ unsigned long long* exchange(unsigned when) const {
        return a.exchanges + (when & 3) * static_cast<size_t>(kClusters * kRows * kD);
    }
    // Adds the latest `n` exchanges, of which the first is an FFN's where `ffn_first`, to this CTA's slice of the residual
    // stream and spreads it over the cluster.
    // The gain of the norm that follows comes with it.
    __device__ __forceinline__ void collect(int n, bool ffn_first, const float* gain) {
        await_bytes(kBarH, ((n ? a.rows : 0) + 1) * kD * 4);
        if (tid == 0 && limit != 1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(sm + S::kGain)),
                         "l"(gain), "r"(kD * 4), "r"(smem_u32(bars + kBarH))
                         : "memory");
        }
        if (n) {
            // (two features to a thread, so that eight rows of 768 are one trip, not two: 128 tokens of the 97M shape at six rows a pass,
            // with what else takes pairs below, 33.9 -> 32.1 ms)
            const int items = a.rows * (kDs / 2);
#pragma unroll 1
            for (int i = tid; (i & ~31) < items; i += kThreads) {  // (whole warps)
                const bool on = i < items;
                const int at = on ? i : 0, r = at / (kDs / 2), f = rank * kDs + at % (kDs / 2) * 2;
                float2 v = *reinterpret_cast<const float2*>(h(cur) + r * kD + f);
                if (on) {
#pragma unroll 1
                    for (int k = 0; k < n; ++k) {
                        const unsigned when = epoch - (n - 1 - k);
                        gather(exchange(when) + r * kD + f, ffn_first && k == 0 ? a.clusters : a.n_kv_heads, when, v);
                    }
                }
                __syncwarp();
                // two lanes' values: the even one sends them to peers 0 .. 3, the odd one to 4 .. 7
                const float ox = __shfl_xor_sync(kFullMask, v.x, 1), oy = __shfl_xor_sync(kFullMask, v.y, 1);
                const float4 q = lane & 1 ? make_float4(ox, oy, v.x, v.y) : make_float4(v.x, v.y, ox, oy);
                const float* to = h(cur ^ 1) + r * kD + (f & ~3);
                if (on)
#pragma unroll
                    for (int p = 0; p < 4; ++p) send4(to, bars + kBarH, 4 * (lane & 1) + p, q);
            }
            cur ^= 1;
        }
        arrived(kBarH);
    }
    // The residual stream times the norm's gain as this warp's B fragments (k-steps warp, warp + 16, ..), two bf16 terms,
    // and its share of the rows' sums of squares: the rest of the norm, a factor per row, waits until the sums over the
    // warps (row_scale).
    __device__ __forceinline__ void weighted(uint32_t (&bh)[KI][2], uint32_t (&bl)[KI][2]) {
        const int n = lane >> 2, t = lane & 3;
        float ss = 0.0f;
#pragma unroll
        for (int i = 0; i < KI; ++i) {
            const int e = (warp + 16 * i) * 16 + 2 * t;
            const float *p = h(cur) + n * kD + e, *w = reinterpret_cast<const float*>(sm + S::kGain) + e;
            const float2 w0 = *reinterpret_cast<const float2*>(w), w1 = *reinterpret_cast<const float2*>(w + 8);
            float2 x0 = make_float2(0.f, 0.f), x1 = x0;
            if (n < a.rows) {
                x0 = *reinterpret_cast<const float2*>(p);
                x1 = *reinterpret_cast<const float2*>(p + 8);
            }
            ss += (x0.x * x0.x + x0.y * x0.y) + (x1.x * x1.x + x1.y * x1.y);
            split2(x0.x * w0.x, x0.y * w0.y, bh[i][0], bl[i][0]);
            split2(x1.x * w1.x, x1.y * w1.y, bh[i][1], bl[i][1]);
        }
        ss += __shfl_xor_sync(kFullMask, ss, 1);
        ss += __shfl_xor_sync(kFullMask, ss, 2);
        if (t == 0) reinterpret_cast<float*>(sm + S::kSsq)[n * 16 + warp] = ss;
    }
    __device__ __forceinline__ float row_scale(int row) const {
        const float4* p = reinterpret_cast<const float4*>(sm + S::kSsq) + row * 4;
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = p[i];
            s += (v.x + v.y) + (v.z + v.w);
        }
        return rsqrtf(s * a.inv_d + a.eps);
    }
    // `tiles` 16-feature tiles against the weighted rows; every warp leaves its share in
    // red()[slot0 + tile][warp][feature * 8 + row].
    __device__ __forceinline__ void project(int slot0, int tiles, const uint32_t (&bh)[KI][2], const uint32_t (&bl)[KI][2]) {
        const int g = lane >> 2, t = lane & 3;
#pragma unroll 1
        for (int tile = 0; tile < tiles; ++tile) {
            float c[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};
            uint4 f[KI];
            fragments(f);
#pragma unroll
            for (int i = 0; i < KI; ++i) {
                mma_bf16(c, f[i], bh[i][0], bh[i][1]);
                mma_bf16(e, f[i], bl[i][0], bl[i][1]);
            }
            float* to = red() + ((slot0 + tile) * kWarps + warp) * 128;
            *reinterpret_cast<float2*>(to + g * 8 + 2 * t) = make_float2(c[0] + e[0], c[1] + e[1]);
            *reinterpret_cast<float2*>(to + (g + 8) * 8 + 2 * t) = make_float2(c[2] + e[2], c[3] + e[3]);
        }
    }
    // sums over lanes 4 i .. 4 i + 3
    __device__ __forceinline__ static void sum_four(float& s, float4& o) {
#pragma unroll
        for (int i = 1; i <= 2; i *= 2) {
            s += __shfl_xor_sync(kFullMask, s, i);
            o.x += __shfl_xor_sync(kFullMask, o.x, i);
            o.y += __shfl_xor_sync(kFullMask, o.y, i);
            o.z += __shfl_xor_sync(kFullMask, o.z, i);
            o.w += __shfl_xor_sync(kFullMask, o.w, i);
        }
    }
    __device__ __forceinline__ float summed(int tile, int v) const {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += red()[(tile * kWarps + w) * 128 + v];
        return s;
    }

    // The K,V rows of sixteen keys as B fragments of the two contractions.  Lane (g, t) holds, for the scores, dims
    // 8 t .. and 32 + 8 t .. of keys g and 8 + g; for the sum over the keys, dims 8 g .. of keys 2 t, 2 t + 1, and
    // those two + 8: the order of the contraction's index is free, so every load is 16 bytes of one row.
    struct Keys {
        uint4 k[4], v[4];
    };
    // Sixteen keys from a multiple of sixteen on share a page; keys beyond the last repeat it.
    struct KeyRows {
        const __half* at;  // the first key's K row; V rows are `to_v` further
        int last;          // of the sixteen
    };
    __device__ __forceinline__ KeyRows key_rows(const __half* pool, int page, int n_keys, int first) const {
        const uint32_t row = (static_cast<uint32_t>(page) * 2 * a.n_kv_heads + cluster) * a.page_size + (first & (a.page_size - 1));
        return KeyRows{pool + static_cast<size_t>(row) * kDh, n_keys - 1 - first};
    }
    __device__ __forceinline__ void load_k(uint4 (&k)[4], const KeyRows& r) const {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const __half* p = r.at + min(8 * i + (lane >> 2), r.last) * kDh + 8 * (lane & 3);
            k[2 * i] = __ldcg(reinterpret_cast<const uint4*>(p));
            k[2 * i + 1] = __ldcg(reinterpret_cast<const uint4*>(p + 32));
        }
    }
    __device__ __forceinline__ void load_v(uint4 (&v)[4], const KeyRows& r) const {
        const __half* p = r.at + a.n_kv_heads * a.page_size * kDh + 8 * (lane >> 2);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __ldcg(reinterpret_cast<const uint4*>(p + min(2 * (lane & 3) + (i & 1) + 8 * (i >> 1), r.last) * kDh));
    }

    // The rows' own keys, all as the first eight of sixteen.
    __device__ __forceinline__ void own_keys(Keys& x, int (&kp)[4], const float* own, int width, int first_row) const {
        const int g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int at = 2 * t + (i & 1);
            const bool have = i < 2 && at < a.m_rows;
            kp[i] = have ? row_pos()[first_row + at] : -1;
            x.k[i] = x.v[i] = make_uint4(0u, 0u, 0u, 0u);
            if (have) {
                const float4 lo = *reinterpret_cast<const float4*>(own + at * width + kDh + 8 * g);
                const float4 hi = *reinterpret_cast<const float4*>(own + at * width + kDh + 8 * g + 4);
                x.v[i] = make_uint4(pack_half(lo.x, lo.y), pack_half(lo.z, lo.w), pack_half(hi.x, hi.y), pack_half(hi.z, hi.w));
            }
        }
        if (g < a.m_rows) {
            float4 w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const float4*>(own + g * width + 16 * t + 4 * i);
            x.k[0] = make_uint4(pack_half(w[0].x, w[0].z), pack_half(w[1].x, w[1].z), pack_half(w[2].x, w[2].z), pack_half(w[3].x, w[3].z));
            x.k[1] = make_uint4(pack_half(w[0].y, w[0].w), pack_half(w[1].y, w[1].w), pack_half(w[2].y, w[2].w), pack_half(w[3].y, w[3].w));
        }
    }

    // One attention branch: projection of the normed rows, attention of this cluster's head, its share of the output
    // projection, published as the next exchange.  Self-attention appends the rows' K,V to the cache.  Scores and the sums over the
    // keys are mma.sync m16n8k16 in fp16, the type of the cache: the eight queries (q scaled by a power of two, and the
    // weights times 2^10, so that the small ones keep their bits) are two fp16 terms each, which are rows g and g + 8 of
    // the A operand.
    __device__ __forceinline__ void attention(bool cross, const float* gain, __half* pool, bool first_block) {
        const int group = a.n_heads / a.n_kv_heads;
        const int g = lane >> 2, t = lane & 3;
        // this warp's share of the keys: one sequence, every (8 wps)-th group of sixteen
        const int wps = a.warps_per_seq, b = warp * a.per_warp >> 8, wi = warp - b * wps;
        const bool live = b < a.batch;
        const int step = 16 * kC * wps;
        int key = 16 * (rank + kC * wi);
        int n_keys = 0;
        const int32_t* pages = nullptr;
        KeyRows kr{};
        int page = 0;
        Keys x;
        if (live) {
            const int s = row_seq()[b * a.m_rows];
            n_keys = cross ? a.src_len[s] : max(row_pos()[b * a.m_rows], 0);
            pages = cross ? a.src_page_table + s * a.src_pages_per_seq : a.page_table + s * a.pages_per_seq;
            if (key < n_keys) page = pages[key >> a.page_shift];
            // on their way to L2 while the residual stream is awaited: a row of 128 bytes to a lane
#pragma unroll 1
            for (int at = key, p = page; at < n_keys; at += step, p = at < n_keys ? pages[at >> a.page_shift] : 0) {
                const KeyRows r = key_rows(pool, p, n_keys, at);
                const __half* row = r.at + min(lane & 15, r.last) * kDh + (lane < 16 ? 0 : a.n_kv_heads * a.page_size * kDh);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(row));
            }
        }
        collect(first_block ? 0 : 1, !cross, gain);
        ++epoch;
        uint32_t bh[KI][2], bl[KI][2];
        weighted(bh, bl);
        const int n_tiles = cross ? group * 4 : qkv_tiles(group);
        const int tiles = tiles_of(n_tiles, rank);
        const int width = (group + 2) * kDh;
        await_bytes(kBarQ, a.rows * n_tiles * 16 * 4);
        project(0, tiles, bh, bl);
        if (key < n_keys) {  // (back by the time that the scores need them; asked for earlier they only cost registers)
            kr = key_rows(pool, page, n_keys, key);
            load_k(x.k, kr);
            load_v(x.v, kr);
        }
        sync_consumers();
        refill();
        // Rotary positions, the scale of the scores (in base-2 units), the rounding of cached rows, and off to the cluster.
        // Features 2 k and 2 k + 1 of a q or k tile are dims k and 32 + k of its eight (pack_small_kernel).
        float* xq = reinterpret_cast<float*>(sm + S::kXq);
#pragma unroll 1
        for (int i = tid; i < tiles * 128; i += kThreads) {
            const int v = i & 127, row = v & 7, f = v >> 3, n = rank + kC * (i >> 7), part = n >> 2;
            float y = summed(i >> 7, v) * row_scale(row);
            const float other = __shfl_xor_sync(kFullMask, y, 8);
            const int dim = part == group + 1 ? 16 * (n & 3) + f : 8 * (n & 3) + (f >> 1) + 32 * (f & 1);
            const int p = row < a.rows ? row_pos()[row] : -1;
            if (a.rope && !cross && p >= 0 && part <= group) {
                const float2 w = reinterpret_cast<const float2*>(sm + S::kRope)[row * 32 + (dim & 31)];
                y = (f & 1) ? y * w.x + other * w.y : y * w.x - other * w.y;
            }
            if (part < group) {
                y *= 0.125f * kLog2e;
            } else {
                y = clamp_half(y);
                if (p >= 0) {
                    pool[static_cast<size_t>(static_cast<uint32_t>(row_at()[row]) + ((part - group) * a.n_kv_heads + cluster) * a.page_size) * kDh + dim] =
                        __float2half_rn(y);
                }
            }
            float4 q;  // four features of a row: lanes row, 8 + row, ..; the j-th sends them to peers j and j + 4
            q.x = __shfl_sync(kFullMask, y, lane & 7);
            q.y = __shfl_sync(kFullMask, y, (lane & 7) + 8);
            q.z = __shfl_sync(kFullMask, y, (lane & 7) + 16);
            q.w = __shfl_sync(kFullMask, y, (lane & 7) + 24);
            if (row < a.rows) {
                const float* to = xq + row * width + n * 16 + (f & ~3);
                send4(to, bars + kBarQ, lane >> 3, q);
                send4(to, bars + kBarQ, (lane >> 3) + 4, q);
            }
        }
        arrived(kBarQ);
        // ---- attention: states per warp, then per CTA, then the cluster's ----
        const int nq = a.m_rows * group;  // queries of a sequence on this head: query q is row q / group
        const bool query = live && g < nq;
        const int q_row = query ? b * a.m_rows + by_group(g) : 0, q_head = query ? g - by_group(g) * group : 0;
        const int q_pos = query ? row_pos()[q_row] : -1;
        const bool own_rows = !cross && rank == kC - 1 && wi == wps - 1;
        float mx = -FLT_MAX, l = 0.0f, acc[8][4];
        uint32_t qa[4][4];
        float unscale;
        float* st = red();  // states [warp][query]
        auto queries = [&]() {
            float v[16];
            float top = 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w = query ? *reinterpret_cast<const float4*>(xq + q_row * width + q_head * kDh + 16 * t + 4 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * i] = w.x;
                v[4 * i + 1] = w.y;
                v[4 * i + 2] = w.z;
                v[4 * i + 3] = w.w;
                top = fmaxf(fmaxf(fmaxf(top, fabsf(w.x)), fabsf(w.y)), fmaxf(fabsf(w.z), fabsf(w.w)));
            }
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 1));
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 2));
            const uint32_t e = max(__float_as_uint(top) >> 23, 14u);  // the largest becomes 2^13 ..
            const float scale = __uint_as_float((267u - e) << 23);
            unscale = __uint_as_float((e - 13u) << 23);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                split_half(v[4 * i] * scale, v[4 * i + 2] * scale, qa[i][0], qa[i][1]);
                split_half(v[4 * i + 1] * scale, v[4 * i + 3] * scale, qa[i][2], qa[i][3]);
            }
        };
        // sixteen keys; kp: positions of keys 2 t, 2 t + 1 and those two + 8 (< 0: none)
        auto scores = [&](float (&sc)[4], const int (&kp)[4]) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < 4; ++k) mma_f16(c, qa[k], word(x.k[2 * i], k), word(x.k[2 * i + 1], k));
                sc[2 * i] = (c[0] + c[2]) * unscale;
                sc[2 * i + 1] = (c[1] + c[3]) * unscale;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool sees = kp[i] >= 0 && q_pos >= 0 && (cross || kp[i] <= q_pos);
                if (sees && a.bias && !cross)
                    sc[i] += kLog2e * a.bias[static_cast<size_t>(cluster * group + q_head) * a.bias_span + kp[i] - q_pos + a.bias_zero];
                if (!sees) sc[i] = -FLT_MAX;
            }
        };
        auto values = [&](const float (&sc)[4], int first) {
            float top = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 1));
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 2));
            const float now = fmaxf(mx, top), keep = exp2_fast(mx - now);
            mx = now;
            float p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = sc[i] != -FLT_MAX ? exp2_fast(sc[i] - now) * 1024.0f : 0.0f;
            l = l * keep + ((p[0] + p[1]) + (p[2] + p[3]));
            uint32_t pa[4];
            split_half(p[0], p[1], pa[0], pa[1]);
            split_half(p[2], p[3], pa[2], pa[3]);
            if (first) {
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[j][i] *= keep;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t sel = (j & 1) ? 0x7632 : 0x5410;
                mma_f16(acc[j], pa, __byte_perm(word(x.v[0], j >> 1), word(x.v[1], j >> 1), sel),
                        __byte_perm(word(x.v[2], j >> 1), word(x.v[3], j >> 1), sel));
            }
        };
        if (live && (key < n_keys || own_rows)) {
            queries();
#pragma unroll 1
            for (int first = 1, again = 1; again; first = 0) {
                int kp[4];
                if (key < n_keys) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int at = key + 2 * t + (i & 1) + 8 * (i >> 1);
                        kp[i] = at < n_keys ? at : -1;
                    }
                } else {
                    own_keys(x, kp, xq + b * a.m_rows * width + group * kDh, width, b * a.m_rows);
                }
                float sc[4];
                scores(sc, kp);
                again = key < n_keys && (own_rows || key + step < n_keys);
                key += step;
                const bool more = key < n_keys;
                asm volatile("" : "+r"(first), "+r"(again));  // (hidden from the compiler, which would write the loop out for each case)
                if (more) {
                    kr = key_rows(pool, pages[key >> a.page_shift], n_keys, key);
                    load_k(x.k, kr);
                }
                values(sc, first);
                if (more) load_v(x.v, kr);
            }
            l += __shfl_xor_sync(kFullMask, l, 1);
            l += __shfl_xor_sync(kFullMask, l, 2);
            if (query) {  // (column n of tile j is dim 8 n + j)
                float* to = st + (warp * 8 + g) * kStateLen;
                if (t == 0) *reinterpret_cast<float2*>(to) = make_float2(mx, l);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 8; j += 4)
                        *reinterpret_cast<float4*>(to + 4 + 16 * t + 8 * i + j) =
                            make_float4(acc[j][i] + acc[j][2 + i], acc[j + 1][i] + acc[j + 1][2 + i], acc[j + 2][i] + acc[j + 2][2 + i],
                                        acc[j + 3][i] + acc[j + 3][2 + i]);
            }
        } else if (query && t == 0) {
            st[(warp * 8 + g) * kStateLen] = -FLT_MAX;  // no keys here
        }
        sync_consumers();
        // Four lanes per query and four dims: each takes four of the warps, then two of the peers.
        float* state = reinterpret_cast<float*>(sm + S::kState);
        const int all_q = a.rows * group;
        await_bytes(kBarS, kC * all_q * (kDh + 2) * 4);
        const int part = tid & 3, dim = ((tid >> 2) & 15) * 4, mq = tid >> 6;
        if (mq < all_q) {
            const int sb = by_group(mq) * a.per_rows >> 8, sq = mq - sb * nq;
            float m[4], top = -FLT_MAX;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int w = part + 4 * i;
                m[i] = w / wps == sb ? st[(w * 8 + sq) * kStateLen] : -FLT_MAX;
                top = fmaxf(top, m[i]);
            }
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 1));
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 2));
            float s = 0.0f;
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (m[i] > -FLT_MAX) {
                    const float* p = st + ((part + 4 * i) * 8 + sq) * kStateLen;
                    const float e = exp2_fast(m[i] - top);
                    const float4 v = *reinterpret_cast<const float4*>(p + 4 + dim);
                    s += p[1] * e;
                    o.x += v.x * e;
                    o.y += v.y * e;
                    o.z += v.z * e;
                    o.w += v.w * e;
                }
            }
            sum_four(s, o);
            const float* dest = state + (rank * 8 + mq) * kStateLen;
#pragma unroll
            for (int i = 0; i < kC; i += 4) {
                send4(dest + 4 + dim, bars + kBarS, part + i, o);
                if (dim == 0) send2(dest, bars + kBarS, part + i, top, s);
            }
        }
        arrived(kBarS);
        __nv_bfloat16* oh = reinterpret_cast<__nv_bfloat16*>(sm + S::kAct);
        __nv_bfloat16* ol = oh + R * 256;
        const int kw = group * kDh;  // width of the head's output
        if (mq < all_q) {  // and two of the cluster's states each
            const float *p0 = state + (part * 8 + mq) * kStateLen, *p1 = p0 + 4 * 8 * kStateLen;
            const float2 s0 = *reinterpret_cast<const float2*>(p0), s1 = *reinterpret_cast<const float2*>(p1);
            const float4 v0 = *reinterpret_cast<const float4*>(p0 + 4 + dim), v1 = *reinterpret_cast<const float4*>(p1 + 4 + dim);
            float top = fmaxf(s0.x, s1.x);
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 1));
            top = fmaxf(top, __shfl_xor_sync(kFullMask, top, 2));
            const float e0 = exp2_fast(s0.x - top), e1 = exp2_fast(s1.x - top);
            float s = s0.y * e0 + s1.y * e1;
            float4 o = make_float4(v0.x * e0 + v1.x * e1, v0.y * e0 + v1.y * e1, v0.z * e0 + v1.z * e1, v0.w * e0 + v1.w * e1);
            sum_four(s, o);
            const float mine = part == 0 ? o.x : part == 1 ? o.y : part == 2 ? o.z : o.w;
            const float y = s > 0.0f ? mine / s : 0.0f;  // an inactive row has no keys
            const __nv_bfloat16 hi = __float2bfloat16_rn(y);
            const int at = by_group(mq) * 256 + (mq - by_group(mq) * group) * kDh + dim + part;
            oh[at] = hi;
            ol[at] = __float2bfloat16_rn(y - __bfloat162float(hi));
        }
        sync_consumers();
        // ---- output projection: the CTA's d / 8 features over the head's inputs ----
        // (fragment fi of the list: k-step fi / kWo, sixteen features fi % kWo)
        constexpr int kWo = kDs / 16;
        const int ks = kw / 16, frags = kWo * ks;
#pragma unroll 1
        for (int f0 = 0; f0 < frags; f0 += KI * kWarps) {
            uint4 f[KI];
            fragments(f);
#pragma unroll
            for (int i = 0; i < KI; ++i) {
                const int fi = f0 + i * kWarps + warp, k = fi / kWo;
                if (fi < frags) {
                    uint32_t b0 = 0, b1 = 0, e0 = 0, e1 = 0;
                    if (g < a.rows) {
                        const int at = g * 256 + k * 16 + 2 * t;
                        b0 = *reinterpret_cast<const uint32_t*>(oh + at);
                        b1 = *reinterpret_cast<const uint32_t*>(oh + at + 8);
                        e0 = *reinterpret_cast<const uint32_t*>(ol + at);
                        e1 = *reinterpret_cast<const uint32_t*>(ol + at + 8);
                    }
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_bf16(c, f[i], b0, b1);
                    mma_bf16(c, f[i], e0, e1);
                    float* to = red() + fi * 128;
                    *reinterpret_cast<float2*>(to + g * 8 + 2 * t) = make_float2(c[0], c[1]);
                    *reinterpret_cast<float2*>(to + (g + 8) * 8 + 2 * t) = make_float2(c[2], c[3]);
                }
            }
        }
        sync_consumers();
        refill();
#pragma unroll 1
        for (int i = tid; i < kDs * ((a.rows + 1) / 2); i += kThreads) {  // (two rows to a thread)
            const int f = i % kDs, row = i / kDs * 2;
            float2 s = make_float2(0.0f, 0.0f);
            const float* p = red() + (f >> 4) * 128 + (f & 15) * 8 + row;
#pragma unroll 1
            for (int k = 0; k < ks; k += 4, p += 4 * kWo * 128) {
                float2 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const float2*>(p + j * kWo * 128);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    s.x += v[j].x;
                    s.y += v[j].y;
                }
            }
            publish_rows(row, rank * kDs + f, s);
        }
    }
    // The sums of rows `row` and `row` + 1 (if there is one) of a feature.
    __device__ __forceinline__ void publish_rows(int row, int feature, const float2& v) {
        if (a.mute) return;
        unsigned long long* at = exchange(epoch) + (cluster * kRows + row) * kD + feature;
        publish(at, v.x, epoch);
        if (row + 1 < a.rows) publish(at + kD, v.y, epoch);
    }

    // The FFN of the rows: the cluster's share of W_out act(W_in x), published, or as plain sums after the last block.
    __device__ __forceinline__ void ffn(int units, float* plain) {
        const int g = lane >> 2, t = lane & 3;
        uint32_t bh[KI][2], bl[KI][2];
        weighted(bh, bl);
        float out[KI][4];
#pragma unroll
        for (int i = 0; i < KI; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) out[i][j] = 0.0f;
        await_bytes(kBarF, kD * (R > 2 ? (a.rows + 3) / 4 * 4 : 2) * 4);
        const int per = a.gated ? 2 : 1;
        __nv_bfloat16* ah = reinterpret_cast<__nv_bfloat16*>(sm + S::kAct);
        __nv_bfloat16* al = ah + 2 * kRows * 16;
#pragma unroll 1
        for (int u0 = 0; u0 < units; u0 += 2) {
            const int nu = min(2, units - u0);
            project(0, per, bh, bl);
            if (nu == 2) {
                if (kStages < 6) {  // (else both units' chunks fit)
                    sync_consumers();
                    refill();
                }
                project(per, per, bh, bl);
            }
            sync_consumers();
            refill();
            if (tid < nu * 128) {
                const int u = tid >> 7, v = tid & 127, row = v & 7, f = v >> 3;
                const float scale = row_scale(row);
                float y = summed(u * per, v) * scale;
                if (a.gated) {
                    const float up = summed(u * per + 1, v) * scale;
                    y = (a.ffn == SPEC_FFN_SWIGLU ? silu(y) : gelu_tanh(y)) * up;
                } else {
                    y = gelu_tanh(y);
                }
                const __nv_bfloat16 hi = __float2bfloat16_rn(y);
                ah[(u * kRows + row) * 16 + f] = hi;
                al[(u * kRows + row) * 16 + f] = __float2bfloat16_rn(y - __bfloat162float(hi));
            }
            sync_consumers();
#pragma unroll 1
            for (int u = 0; u < nu; ++u) {
                const int at = (u * kRows + g) * 16 + 2 * t;
                const uint32_t b0 = *reinterpret_cast<const uint32_t*>(ah + at), b1 = *reinterpret_cast<const uint32_t*>(ah + at + 8);
                const uint32_t e0 = *reinterpret_cast<const uint32_t*>(al + at), e1 = *reinterpret_cast<const uint32_t*>(al + at + 8);
                uint4 f[KI];
                fragments(f);
#pragma unroll
                for (int i = 0; i < KI; ++i) {
                    mma_bf16(out[i], f[i], b0, b1);
                    mma_bf16(out[i], f[i], e0, e1);
                }
            }
        }
        // to the owners of the feature slices: [rank][feature][8 rows]
        float* fred = reinterpret_cast<float*>(sm + S::kFred);
        if constexpr (R > 2) {
            // lanes t and t ^ 1 hold two rows each of features g and g + 8: the even one takes the four of g, the odd one of g + 8
            const int odd = t & 1, quad = t >> 1 << 2;
#pragma unroll
            for (int i = 0; i < KI; ++i) {
                const float x = __shfl_xor_sync(kFullMask, odd ? out[i][0] : out[i][2], 1), y = __shfl_xor_sync(kFullMask, odd ? out[i][1] : out[i][3], 1);
                const float4 q = odd ? make_float4(x, y, out[i][2], out[i][3]) : make_float4(out[i][0], out[i][1], x, y);
                const int f = (i * kWarps + warp) * 16 + g + 8 * odd;
                if (quad < a.rows) send4(fred + (rank * kDs + f % kDs) * R + quad, bars + kBarF, f / kDs, q);
            }
        } else if (t == 0) {
#pragma unroll
            for (int i = 0; i < KI; ++i)
#pragma unroll
                for (int up = 0; up < 2; ++up) {
                    const int f = (i * kWarps + warp) * 16 + g + 8 * up;
                    send2(fred + (rank * kDs + f % kDs) * R, bars + kBarF, f / kDs, out[i][2 * up], out[i][2 * up + 1]);
                }
        }
        sync_consumers();  // (every warp has read its fragments)
        refill();
        arrived(kBarF);
#pragma unroll 1
        for (int i = tid; i < kDs * ((a.rows + 1) / 2); i += kThreads) {
            const int row = i / kDs * 2, f = i % kDs;
            float2 v[kC];
#pragma unroll
            for (int c = 0; c < kC; ++c) v[c] = *reinterpret_cast<const float2*>(fred + (c * kDs + f) * R + row);
            float2 s = v[0];
#pragma unroll
            for (int c = 1; c < kC; ++c) {
                s.x += v[c].x;
                s.y += v[c].y;
            }
            if (plain) {
                float* at = plain + (cluster * a.rows + row) * kD + rank * kDs + f;
                at[0] = s.x;
                if (row + 1 < a.rows) at[kD] = s.y;
            } else {
                publish_rows(row, rank * kDs + f, s);
            }
        }
    }
};

template <int KI, int R>
__global__ void __cluster_dims__(kC, 1, 1) __launch_bounds__(kThreads, 1)
small_pass_kernel(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(1024) uint8_t sm[];
    using P = Pass<KI, R>;
    using S = typename P::S;
    constexpr int kD = P::kD;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + S::kBars);  // residual stream, q k v, states, FFN sums
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = blockIdx.x, rank = cta % kC, cluster = cta / kC;
    if (tid == 0) {
        for (int s = 0; s < S::kStages + 4; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[s])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const int group = a.n_heads / a.n_kv_heads;
    const bool head = cluster < a.n_kv_heads;
    const int units = units_of(a.units, cta, a.clusters * kC);
    if (tid == 0) {
        int stages = units * (a.gated ? 3 : 2);
        if (head) {
            stages += tiles_of(qkv_tiles(group), rank) + wo_stages(group);
            if (a.cross) stages += tiles_of(group * 4, rank) + wo_stages(group);
        }
        int* asked = reinterpret_cast<int*>(sm + S::kMeta) + 24;
        asked[0] = 0;
        asked[1] = stages * a.n_layers;
    }
    __syncthreads();
    P p{a, sm, bars, bars + 4, tid, lane, warp, rank, cluster, a.limit, 0, 0, 0, 0, *a.epoch};
    p.refill();
    // the embedding, every CTA for itself; the rows' positions, sequences and rotations
#pragma unroll 1
    for (int i = tid; i < a.rows * kD / 2; i += kThreads) {
        const int r = 2 * i / kD, e = 2 * i % kD;
        const int tok = min(max(a.token[r], 0), a.vocab - 1);
        float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(a.tok_emb + static_cast<size_t>(tok) * kD + e));
        if (a.pos_emb) {
            const int pos = min(max(a.pos[r], 0), a.max_positions - 1);
            const float2 w = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(a.pos_emb + static_cast<size_t>(pos) * kD + e));
            v.x += w.x;
            v.y += w.y;
        }
        *reinterpret_cast<float2*>(p.h(0) + r * kD + e) = v;
    }
    if (tid < a.rows) {
        int* meta = reinterpret_cast<int*>(sm + S::kMeta);
        const int pos = a.pos[tid], seq = a.seq[tid];
        meta[tid] = pos;
        meta[8 + tid] = seq;
        if (pos >= 0) meta[16 + tid] = a.page_table[seq * a.pages_per_seq + pos / a.page_size] * 2 * a.n_kv_heads * a.page_size + pos % a.page_size;
    }
    if (a.rope)
#pragma unroll 1
        for (int i = tid; i < a.rows * 32; i += kThreads)
            reinterpret_cast<float2*>(sm + S::kRope)[i] = a.rope[static_cast<size_t>(max(a.pos[i >> 5], 0)) * 32 + (i & 31)];
    // (CTA 0 advances the epoch at its end.  By then every CTA has read it: from two blocks on, CTA 0 has gathered an FFN's sums
    // of its peer in every cluster, each of which needed something of every CTA of that cluster.  shape_fits has the rest)
    sync_consumers();
#pragma unroll 1
    for (int l = 0; l < a.n_layers; ++l) {
        const float* gain = a.gains + static_cast<size_t>(l) * 3 * kD;
        if (head) {
#pragma unroll 1
            for (int x = 0; x <= a.cross; ++x) {  // self-attention, cross-attention
                asm volatile("" : "+r"(x));       // (hidden from the compiler, which would write both out)
                p.attention(x != 0, gain + x * kD, x ? a.cross_kv + l * a.cross_stride : a.kv + l * a.layer_stride, l + x == 0);
            }
        } else {
            p.epoch += 1 + a.cross;
        }
        // (a cluster without a head has the whole block before it to catch up with)
        const int pending = head ? 1 : 1 + a.cross + (l > 0 ? 1 : 0);
        p.collect(pending, pending == 2 + a.cross, gain + 2 * kD);
        ++p.epoch;
        p.ffn(units, l + 1 == a.n_layers ? a.last_part : nullptr);
    }
    // the residual stream without the last branch, whose partial sums the kernel that follows adds
    if (cta == 0) {
#pragma unroll 1
        for (int i = tid; i < a.rows * kD; i += kThreads) a.h_out[i] = p.h(p.cur)[i];
        if (tid == 0) *a.epoch = p.epoch;
    }
    if (p.limit == 1) {
        atomicCAS(&g_small_error, 0, 1);
        // the copies that this thread or warp asked for: a barrier is past one of the two parities at any time
        if (tid == 0) bar_wait(bars + P::kBarH, 0, kDrain), bar_wait(bars + P::kBarH, 1, kDrain);
        if (warp == kWarps - 1 && lane < S::kStages) bar_wait(&p.full[lane], 0, kDrain), bar_wait(&p.full[lane], 1, kDrain);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // nobody leaves while a peer may still write here
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---- packing ------------------------------------------------------------------------
struct PackLayer {
    const __nv_bfloat16 *wqkv, *wo, *w_in, *w_out, *wq_x, *wo_x;
    const float *ln1, *lnx, *ln2;
};

// rows `row` and `row + below` are the lane's
__device__ __forceinline__ void pack_fragment(const __nv_bfloat16* w, int ld, int row, int below, int col, int lane, uint8_t* to) {
    const __nv_bfloat16* p = w + static_cast<size_t>(row) * ld + col + 2 * (lane & 3);
    uint4 f;
    f.x = *reinterpret_cast<const uint32_t*>(p);
    f.y = *reinterpret_cast<const uint32_t*>(p + static_cast<size_t>(below) * ld);
    f.z = *reinterpret_cast<const uint32_t*>(p + 8);
    f.w = *reinterpret_cast<const uint32_t*>(p + static_cast<size_t>(below) * ld + 8);
    *reinterpret_cast<uint4*>(to + lane * 16) = f;
}

// grid = (CTAs of the pass, layers), block = 512: writes the stream of one CTA and layer in the order of Pass's reads.
__global__ void pack_small_kernel(const PackLayer* layers, int d, int n_heads, int n_kv_heads, int d_ff, int units, int gated, int cross,
                                  size_t cta_bytes, uint8_t* stream, float* gains) {
    const int cta = blockIdx.x, rank = cta % kC, cluster = cta / kC, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = n_heads / n_kv_heads, ki = d / 256;
    const PackLayer& w = layers[blockIdx.y];
    if (cta == 0)
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            float* to = gains + static_cast<size_t>(blockIdx.y) * 3 * d + i;
            to[0] = w.ln1[i];
            if (cross) to[d] = w.lnx[i];
            to[2 * d] = w.ln2[i];
        }
    const bool head = cluster < n_kv_heads;
    const int ctas = gridDim.x, my_units = units_of(units, cta, ctas);
    int per_layer = my_units * (gated ? 3 : 2);
    if (head) {
        per_layer += tiles_of(qkv_tiles(group), rank) + wo_stages(group);
        if (cross) per_layer += tiles_of(group * 4, rank) + wo_stages(group);
    }
    uint8_t* out = stream + static_cast<size_t>(cta) * cta_bytes + static_cast<size_t>(blockIdx.y) * per_layer * ki * kChunk + warp * 512;
    const int g = lane >> 2;
    auto tile = [&](const __nv_bfloat16* m, int row) {
        for (int i = 0; i < ki; ++i, out += kChunk) pack_fragment(m, d, row + g, 8, (warp + 16 * i) * 16, lane, out);
    };
    auto paired = [&](const __nv_bfloat16* m, int row, int quarter) {  // features 2 k, 2 k + 1: dims k, 32 + k of the quarter's eight
        for (int i = 0; i < ki; ++i, out += kChunk)
            pack_fragment(m, d, row + 8 * quarter + (g >> 1) + 32 * (g & 1), 4, (warp + 16 * i) * 16, lane, out);
    };
    auto out_projection = [&](const __nv_bfloat16* m) {
        const int tiles = d / (16 * kC), frags = tiles * 4 * group;
        for (int f0 = 0; f0 < wo_stages(group) * ki * kWarps; f0 += kWarps, out += kChunk) {
            const int f = f0 + warp;
            if (f < frags) pack_fragment(m, n_heads * kDh, rank * (d / kC) + (f % tiles) * 16 + g, 8, cluster * group * kDh + (f / tiles) * 16, lane, out);
            else *reinterpret_cast<uint4*>(out + lane * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
    };
    if (head) {
        for (int i = rank; i < qkv_tiles(group); i += kC) {
            const int part = i / 4;  // 64 rows each: the query heads, K, V
            const int row = part < group ? (cluster * group + part) * kDh : (n_heads + (part - group) * n_kv_heads + cluster) * kDh;
            if (part <= group) paired(w.wqkv, row, i % 4);
            else tile(w.wqkv, row + i % 4 * 16);
        }
        out_projection(w.wo);
        if (cross) {
            for (int i = rank; i < group * 4; i += kC) paired(w.wq_x, (cluster * group + i / 4) * kDh, i % 4);
            out_projection(w.wo_x);
        }
    }
    for (int u0 = 0; u0 < my_units; u0 += 2) {
        const int nu = min(2, my_units - u0);
        for (int u = 0; u < nu; ++u) {
            const int f = unit_index(cta, u0 + u, ctas) * 16;
            tile(w.w_in, f);
            if (gated) tile(w.w_in, d_ff + f);
        }
        for (int u = 0; u < nu; ++u) {
            const int f = unit_index(cta, u0 + u, ctas) * 16;
            for (int i = 0; i < ki; ++i, out += kChunk) pack_fragment(w.w_out, d_ff, (i * kWarps + warp) * 16 + g, 8, f, lane, out);
        }
    }
}

using SmallFn = void (*)(const SmallArgs);
struct Variant {
    SmallFn fn;
    int smem;
};
template <int KI>
Variant pick(int rows) {
    return rows <= 2   ? Variant{small_pass_kernel<KI, 2>, Smem<KI, 2>::kTotal}
           : rows <= 4 ? Variant{small_pass_kernel<KI, 4>, Smem<KI, 4>::kTotal}
                       : Variant{small_pass_kernel<KI, 8>, Smem<KI, 8>::kTotal};
}
// fewer rows leave room for a longer ring
Variant pick(int ki, int rows) { return ki == 1 ? pick<1>(rows) : ki == 2 ? pick<2>(rows) : pick<3>(rows); }

bool shape_fits(const Model& m) {
    const spec_model_cfg& c = m.cfg;
    // In a model of one block nothing makes CTA 0 wait for the clusters without a head: one that starts late would read the
    // epoch of the next pass and poll for exchanges that never come.
    if (c.n_layers < 2) return false;
    if (!m.bf16() || (c.arch != SPEC_ARCH_GPT && c.arch != SPEC_ARCH_LLAMA && c.arch != SPEC_ARCH_T5)) return false;
    const int group = c.n_heads / c.n_kv_heads;
    return c.d_head == kDh && c.d_model % 256 == 0 && c.d_model <= kMaxD && c.n_kv_heads <= kClusters && group <= 4 && c.d_ff % 16 == 0 &&
           m.kv_dtype == SPEC_DTYPE_FP16 && (c.d_model / (16 * kC)) * 4 * group <= 64;
}

}  // namespace

int small_pass_init(SmallPass& s, const Model& m, std::vector<void*>& allocations, size_t& spare, cudaStream_t stream) {
    s = SmallPass{};
    if (!shape_fits(m)) return SPEC_OK;
    const spec_model_cfg& c = m.cfg;
    const int ki = c.d_model / 256, group = c.n_heads / c.n_kv_heads, units = c.d_ff / 16, gated = c.ffn != SPEC_FFN_GELU ? 1 : 0;
    static std::atomic<unsigned long long> configured{0};
    const int status = once_on_this_device(configured, []() -> int {
        for (int k = 1; k <= kMaxKi; ++k)
            for (int rows = 2; rows <= 8; rows *= 2)
                SPEC_CUDA_TRY(cudaFuncSetAttribute(pick(k, rows).fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
        return SPEC_OK;
    });
    if (status != SPEC_OK) return status;
    // all clusters have to be resident at once
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kC * kClusters);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kMaxSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kC;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int resident = 0;
    if (cudaOccupancyMaxActiveClusters(&resident, pick(ki, kRows).fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return SPEC_OK;
    }
    s.clusters = std::min(resident, kClusters);
    if (s.clusters < c.n_kv_heads) return SPEC_OK;
    const int ctas = s.clusters * kC;
    size_t most = 0;
    for (int cta = 0; cta < ctas; ++cta) {
        size_t n = static_cast<size_t>(units_of(units, cta, ctas)) * (gated ? 3 : 2);
        if (cta / kC < c.n_kv_heads) {
            n += tiles_of(qkv_tiles(group), cta % kC) + wo_stages(group);
            if (m.t5()) n += tiles_of(group * 4, cta % kC) + wo_stages(group);
        }
        most = std::max(most, n);
    }
    s.cta_bytes = most * c.n_layers * ki * kChunk;
    // one allocation: gains, the epoch, exchange buffers, the last partial sums, the stream
    const size_t gain_bytes = static_cast<size_t>(c.n_layers) * 3 * c.d_model * sizeof(float), epoch_bytes = 256;
    const size_t ll_bytes = static_cast<size_t>(4) * kClusters * kRows * c.d_model * sizeof(unsigned long long);
    const size_t part_bytes = static_cast<size_t>(kClusters) * kRows * c.d_model * sizeof(float);
    // (the packing kernel's pointers pass through the partial sums' memory, which nothing uses yet; 1820 blocks of the narrowest
    // model fit)
    std::vector<PackLayer> pack(c.n_layers);
    if (pack.size() * sizeof(PackLayer) > part_bytes) return SPEC_OK;
    char* base = nullptr;
    const size_t bytes = gain_bytes + epoch_bytes + ll_bytes + part_bytes + s.cta_bytes * ctas;
    // a third copy of the weights, for speed alone: without room for it the chain of kernels serves the model
    if (bytes > spare || cudaMalloc(reinterpret_cast<void**>(&base), bytes) != cudaSuccess) {
        cudaGetLastError();
        return SPEC_OK;
    }
    allocations.push_back(base);
    spare -= bytes;
    s.gains = reinterpret_cast<float*>(base);
    s.epoch = reinterpret_cast<unsigned*>(base + gain_bytes);
    s.exchanges = reinterpret_cast<unsigned long long*>(base + gain_bytes + epoch_bytes);
    s.last_part = reinterpret_cast<float*>(base + gain_bytes + epoch_bytes + ll_bytes);
    s.stream = base + gain_bytes + epoch_bytes + ll_bytes + part_bytes;
    auto b = [](const void* p) { return static_cast<const __nv_bfloat16*>(p); };
    for (int l = 0; l < c.n_layers; ++l) {
        const spec_layer_weights& w = m.layers[l];
        pack[l] = PackLayer{b(w.wqkv), b(w.wo), b(w.w_in), b(w.w_out), b(w.wq_x), b(w.wo_x), w.ln1, w.lnx, w.ln2};
    }
    SPEC_CUDA_TRY(cudaMemcpyAsync(s.last_part, pack.data(), pack.size() * sizeof(PackLayer), cudaMemcpyHostToDevice, stream));
    // (no epoch is 0: the pairs start as nobody's)
    SPEC_CUDA_TRY(cudaMemsetAsync(s.epoch, 0, epoch_bytes + ll_bytes, stream));
    pack_small_kernel<<<dim3(ctas, c.n_layers), kThreads, 0, stream>>>(reinterpret_cast<const PackLayer*>(s.last_part), c.d_model,
                                                                               c.n_heads, c.n_kv_heads, c.d_ff, units, gated, m.t5() ? 1 : 0,
                                                                               s.cta_bytes, reinterpret_cast<uint8_t*>(s.stream), s.gains);
    SPEC_CUDA_TRY(cudaGetLastError());
    SPEC_CUDA_TRY(cudaStreamSynchronize(stream));
    return SPEC_OK;
}

bool small_pass_serves(const SmallPass& s, const Model& m, int batch, int m_rows) {
    return s.stream && batch * m_rows <= kRows && batch * m_rows * (m.cfg.n_heads / m.cfg.n_kv_heads) <= 8;
}

int launch_small_pass(const SmallPass& s, const Model& m, const RowMeta& rows, const PassTables& t, int batch, int m_rows, float* h,
                      cudaStream_t stream, bool drill) {
    const spec_model_cfg& c = m.cfg;
    const int group = c.n_heads / c.n_kv_heads;
    SmallArgs a{};
    a.stream = static_cast<const uint8_t*>(s.stream);
    a.cta_bytes = s.cta_bytes;
    a.layer_stride = m.layer_stride / sizeof(__half);
    a.cross_stride = m.cross_stride / sizeof(__half);
    a.n_layers = c.n_layers;
    a.n_heads = c.n_heads;
    a.n_kv_heads = c.n_kv_heads;
    a.units = c.d_ff / 16;
    a.gated = c.ffn != SPEC_FFN_GELU ? 1 : 0;
    a.ffn = c.ffn;
    a.cross = m.t5() ? 1 : 0;
    a.clusters = s.clusters;
    a.rows = batch * m_rows;
    a.batch = batch;
    a.m_rows = m_rows;
    a.gains = s.gains;
    a.warps_per_seq = kWarps / batch;
    auto inverse = [](int n) { return (256 + n - 1) / n; };  // x * inverse(n) >> 8 == x / n for x < 16 and n <= 16
    a.per_group = inverse(group);
    a.per_rows = inverse(m_rows);
    a.per_warp = inverse(a.warps_per_seq);
    a.inv_d = 1.0f / static_cast<float>(c.d_model);
    a.token = rows.token;
    a.pos = rows.pos;
    a.seq = rows.seq;
    a.tok_emb = static_cast<const __nv_bfloat16*>(m.tok_emb);
    a.pos_emb = c.arch == SPEC_ARCH_GPT ? static_cast<const __nv_bfloat16*>(m.pos_emb) : nullptr;
    a.vocab = c.vocab;
    a.max_positions = c.max_positions;
    a.rope = c.arch == SPEC_ARCH_LLAMA ? m.rope_table : nullptr;
    a.kv = static_cast<__half*>(m.kv);
    a.cross_kv = static_cast<__half*>(m.cross_kv);
    a.page_table = t.page_table;
    a.pages_per_seq = t.pages_per_seq;
    a.page_size = t.page_size;
    while ((1 << a.page_shift) < t.page_size) ++a.page_shift;
    a.src_page_table = t.src_page_table;
    a.src_pages_per_seq = t.src_pages_per_seq;
    a.src_len = t.src_len;
    a.bias = m.t5() ? m.dec_bias : nullptr;
    a.bias_span = t.bias_span;
    a.bias_zero = t.bias_zero;
    a.eps = c.rms_eps;
    a.exchanges = s.exchanges;
    a.epoch = s.epoch;
    a.last_part = s.last_part;
    a.h_out = h;
    a.limit = drill ? 64 : kSpin;
    a.mute = drill ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kC * s.clusters);
    cfg.blockDim = dim3(kThreads);
    const Variant v = pick(c.d_model / 256, a.rows);
    cfg.dynamicSmemBytes = v.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;  // every CTA resident at once: they wait for one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SPEC_CUDA_TRY(cudaLaunchKernelEx(&cfg, v.fn, a));
    return SPEC_OK;
}

PartialPlan small_pass_plan(const SmallPass& s) {
    PartialPlan p{};
    p.slots = s.clusters;
    return p;
}

int* small_pass_error_word() { return symbol_address(g_small_error); }
int small_pass_take_error() {
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_small_error, sizeof(int)) != cudaSuccess) return -1;
    if (v) cudaMemcpyToSymbol(g_small_error, &zero, sizeof(int));
    return v;
}

}  // namespace spec
