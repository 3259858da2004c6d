// Speculative sampling (Section 2.3 / Algorithm 1, accept-adjust-draw part),
// plain standardised sampling (Section 2.2) and the method's uniforms.
//
// spec_verify_sample is two kernels on one stream (few logits: one; with a cut: another first one; see below):
//   1. verify_stats_kernel streams every logit of p_1..p_{gamma+1} and
//      q_1..q_gamma exactly once from HBM.  A CTA reduces one chunk of one row
//      to (max, sum exp) with an online rescale, and also picks up the row's
//      logit at the drafted token.  No CTA talks to another: the kernel is a
//      pure map-reduce and runs at streaming bandwidth.
//   2. verify_finish_kernel, one cluster of CTAs per sequence, merges the chunk
//      statistics, runs the gamma accept tests, and re-reads only row n+1 of p
//      and q (still in L2) to normalise the residual max(0, p - q) and draw from
//      it by inverse CDF: every warp keeps the weights of its segment in
//      registers, the segment totals are scanned once across the cluster, and
//      the warp whose segment holds the target walks it without another trip to
//      memory.  It is chained with programmatic dependent launch, so its launch
//      latency and prologue overlap the tail of the first kernel.
// With few logits, where launches are what a call costs, one kernel does both (one_kernel); with a cut the selection kernel
// leaves the statistics (cut_floor_kernel).
#include <algorithm>
#include <cfloat>
#include <cstddef>
#include <mutex>

#include <cooperative_groups.h>

#include "model.cuh"

namespace cg = cooperative_groups;

namespace spec {
namespace {

constexpr int kStatThreads = 256;
constexpr int kStatWarps = kStatThreads / 32;
constexpr int kUnroll = 4;              // 128-bit loads in flight per thread while streaming
constexpr int kMinChunkGroups = 1000;   // a CTA streams at least 4000 logits (unless the row is shorter)
constexpr int kTargetCtas = 148 * 48;   // about six waves of resident CTAs (eight of 256 threads per SM), so that the last wave
                                        // costs little; smaller CTAs stagger their reduce-and-restart pauses (512 threads: +0.8 us)
constexpr int kFinishThreads = 512;
constexpr int kCdfBatch = 8;            // groups fetched per thread before any is consumed (inverse CDF, one CTA)
constexpr int kClusterCdfBatch = 4;     // the same when a cluster shares the row
constexpr int kWalkBatch = 4;           // 128-element steps fetched at once by the final walk
constexpr int kMaxCluster = 4;          // CTAs per sequence in the finishing kernel
constexpr int kMostParts = 128;         // warps that share an inverse CDF: eight CTAs of 16
constexpr int kSampleThreads = 512;
constexpr int kMaxGamma = 64;
constexpr int kMaxRows = 2 * kMaxGamma + 1;
constexpr float kLog2e = 1.4426950408889634f;

// 2^x with one MUFU instruction (2 ulp; results below 2^-126 flush to zero,
// which is far below anything a sum over the vocabulary can see).
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A row of fp32 logits addressed in groups of four elements.  VEC: the vocabulary
// is a multiple of four and every row starts on a 16-byte boundary, so a group
// is one unconditional 128-bit load.  Logits below `floor` read
// as -inf: that is top-k standardisation (Section 2.2) with `floor` the row's
// k-th largest logit, and no change with floor = -inf.
//
// Without VEC a row may begin anywhere (a vocabulary that is not a multiple of four): `shift`, 0 to 3, is how many
// elements before the row its first group starts, group g holds elements 4g - shift .., and elements outside the row
// read as `pad`.  With the shift of its own address a row is read in 128-bit loads; of two rows that are paired element
// by element the second takes the first one's shift, and is read in 32-bit loads unless it happens to be its own
// (30 x 11 rows of 50003, statistics and draw: 27.4 us with guarded loads of both rows, 26.6 so).
__host__ __device__ __forceinline__ int row_shift(const float* row) { return static_cast<int>((reinterpret_cast<uintptr_t>(row) >> 2) & 3u); }

template <bool VEC, bool CUT = false>
struct Row {
    const float* base;
    int vocab;
    float floor;  // used only with CUT, so that the usual path pays nothing for it
    int shift;
    bool own;  // shift is that of the row's own address

    __device__ __forceinline__ int groups() const { return (vocab + shift + 3) >> 2; }
    __device__ __forceinline__ float kept(float v) const { return (!CUT || v >= floor) ? v : -INFINITY; }
    __device__ __forceinline__ float4 raw(int g, float pad) const {
        if (VEC) return __ldg(reinterpret_cast<const float4*>(base) + g);
        const int j = 4 * g - shift;
        if (j >= 0 && j + 4 <= vocab) {
            if (own) return __ldg(reinterpret_cast<const float4*>(base + j));
            return make_float4(__ldg(base + j), __ldg(base + j + 1), __ldg(base + j + 2), __ldg(base + j + 3));
        }
        float4 v;
        v.x = j + 0 >= 0 && j + 0 < vocab ? __ldg(base + j + 0) : pad;
        v.y = j + 1 >= 0 && j + 1 < vocab ? __ldg(base + j + 1) : pad;
        v.z = j + 2 >= 0 && j + 2 < vocab ? __ldg(base + j + 2) : pad;
        v.w = j + 3 >= 0 && j + 3 < vocab ? __ldg(base + j + 3) : pad;
        return v;
    }
    __device__ __forceinline__ float4 load(int g, float pad) const {
        const float4 v = raw(g, pad);
        if (!CUT) return v;
        return make_float4(kept(v.x), kept(v.y), kept(v.z), kept(v.w));
    }
};

template <bool VEC, bool CUT = false>
__device__ __forceinline__ Row<VEC, CUT> make_row(const float* base, int vocab, float floor = -INFINITY, int shift = -1) {
    Row<VEC, CUT> r;
    const int own = VEC ? 0 : row_shift(base);
    r.shift = VEC ? 0 : shift < 0 ? own : shift;
    r.own = r.shift == own;
    r.base = base;
    r.vocab = vocab;
    r.floor = floor;
    return r;
}

// Weight functors for the inverse-CDF draw.  fetch() only loads, weigh() only
// computes, so that a caller can put several fetches in flight before it
// consumes any of them.

// Unnormalised softmax weights exp((l - max) / T) of one row; c2 = log2(e) / T.
template <bool VEC, bool CUT = false>
struct PlainWeights {
    struct Raw { float4 a; };
    Row<VEC, CUT> p;
    float max_p, c2;
    __device__ __forceinline__ Raw fetch(int g) const { return Raw{p.load(g, -INFINITY)}; }
    __device__ __forceinline__ Raw nothing() const {
        return Raw{make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY)};
    }
    __device__ __forceinline__ int groups() const { return p.groups(); }
    __device__ __forceinline__ int shift() const { return p.shift; }
    __device__ __forceinline__ float one(float lp) const { return fast_exp2((lp - max_p) * c2); }
    __device__ __forceinline__ float4 weigh(const Raw& r) const {
        return make_float4(one(r.a.x), one(r.a.y), one(r.a.z), one(r.a.w));
    }
    __device__ __forceinline__ float4 operator()(int g) const { return weigh(fetch(g)); }
};

// max(0, p - q) with p, q the normalised softmaxes of two rows (Algorithm 1's
// adjusted distribution before normalisation).
template <bool VEC, bool CUT = false>
struct ResidualWeights {
    struct Raw { float4 a, b; };
    Row<VEC, CUT> p, q;
    float max_p, max_q, inv_sum_p, inv_sum_q, c2;
    __device__ __forceinline__ Raw fetch(int g) const { return Raw{p.load(g, -INFINITY), q.load(g, -INFINITY)}; }
    __device__ __forceinline__ Raw nothing() const {
        const float4 z = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        return Raw{z, z};
    }
    __device__ __forceinline__ int groups() const { return p.groups(); }
    __device__ __forceinline__ int shift() const { return p.shift; }
    __device__ __forceinline__ float one(float lp, float lq) const {
        // (both products are rounded before the subtraction: contracted into a multiply-add, one of them would not
        // be, and p = q would leave rounding residue instead of the exact zero that the fallback to p tests for)
        const float pv = __fmul_rn(fast_exp2((lp - max_p) * c2), inv_sum_p);
        const float qv = __fmul_rn(fast_exp2((lq - max_q) * c2), inv_sum_q);
        return fmaxf(0.0f, pv - qv);
    }
    __device__ __forceinline__ float4 weigh(const Raw& r) const {
        return make_float4(one(r.a.x, r.b.x), one(r.a.y, r.b.y), one(r.a.z, r.b.z), one(r.a.w, r.b.w));
    }
    __device__ __forceinline__ float4 operator()(int g) const { return weigh(fetch(g)); }
};

template <int WARPS>
struct CdfScratch {
    float part[WARPS];              // per-warp totals of the level being scanned
    float all[kMostParts];          // the same for every CTA of a cluster
    float pick_before, pick_total;   // outcome of the cluster-wide scan
    int pick_part_index, pick_hit;
    int result;
    int last_positive;
};

// Sum of the weights of groups [g0, g1) by one warp, lane-strided so that every
// load instruction covers 512 contiguous bytes; BATCH fetches are in flight
// per lane before any is consumed.
template <int BATCH, class Weights>
__device__ __forceinline__ float warp_range_sum(const Weights& w, int g0, int g1, int lane) {
    float acc = 0.0f;
    for (int base = g0 + lane; base < g1; base += 32 * BATCH) {
        typename Weights::Raw raw[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const int g = base + 32 * i;
            raw[i] = g < g1 ? w.fetch(g) : w.nothing();
        }
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const float4 v = w.weigh(raw[i]);
            acc += (v.x + v.y) + (v.z + v.w);
        }
    }
    return warp_sum(acc);
}

// Which of `count` consecutive parts holds `target`: the first part whose
// running sum exceeds it (the same arithmetic in every thread, so every thread
// agrees).  Returns -1 if none does; *before gets the running sum in front of
// the chosen part; *fallback is the last part with positive weight (0 if none),
// for the case where rounding leaves no part above the target.
template <class PartAt>
__device__ __forceinline__ int pick_part(PartAt part_at, int count, float target, float* before, int* fallback) {
    float run = 0.0f;
    int hit = -1, last = 0;
    for (int i = 0; i < count; ++i) {
        const float v = part_at(i);
        const float next = run + v;
        if (hit < 0 && next > target) {
            hit = i;
            *before = run;
        }
        if (v > 0.0f) last = i;
        run = next;
    }
    *fallback = last;
    return hit;
}

// One step of the walk: the 128 elements of groups gs .. gs + 31 (lane l holds the four weights of group
// gs + l), in index order after the weight `run` already passed.  Sets `found` to the first index whose running
// sum exceeds `rem` (if want_hit), keeps `last_pos` = the last index with positive weight so far.
__device__ __forceinline__ void walk_step(const float4& v, int gs, int lane, bool want_hit, float rem, float& run, int& found,
                                          int& last_pos) {
    const float mine = (v.x + v.y) + (v.z + v.w);
    const float incl = warp_inclusive_scan(mine, lane);
    const unsigned over = want_hit ? __ballot_sync(kFullMask, run + incl > rem) : 0u;
    const unsigned pos = __ballot_sync(kFullMask, mine > 0.0f);
    if (pos) {
        const int pl = 31 - __clz(pos);  // last lane with positive weight in this step
        const float py = __shfl_sync(kFullMask, v.y, pl), pz = __shfl_sync(kFullMask, v.z, pl),
                    pw = __shfl_sync(kFullMask, v.w, pl);
        const int pg = 4 * (gs + pl);
        last_pos = pw > 0.f ? pg + 3 : pz > 0.f ? pg + 2 : py > 0.f ? pg + 1 : pg;
    }
    if (over) {
        const int hl = __ffs(over) - 1;
        const float excl = __shfl_sync(kFullMask, incl - mine, hl) + run;
        const float hx = __shfl_sync(kFullMask, v.x, hl), hy = __shfl_sync(kFullMask, v.y, hl),
                    hz = __shfl_sync(kFullMask, v.z, hl);
        const int hg = 4 * (gs + hl);
        float c = excl + hx;
        if (c > rem) found = hg;
        else if ((c += hy) > rem) found = hg + 1;
        else if ((c += hz) > rem) found = hg + 2;
        else found = hg + 3;
    }
    run += __shfl_sync(kFullMask, incl, 31);
}

// The draw inside one contiguous range of groups [r0, r1) by a whole CTA: `rem`
// is the target minus the weight in front of the range.  Long ranges are first
// cut into one sub-range per warp; warp 0 then walks the chosen (sub-)range 128
// elements at a time with a warp scan.  With want_hit false the answer is the
// last index of the range with positive weight.  Returns the index (or -1) to
// all threads.
template <int WARPS, class Weights>
__device__ int locate_in_range(const Weights& w, int r0, int r1, float rem, bool want_hit, CdfScratch<WARPS>& s) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s.result = -1;
        s.last_positive = -1;
    }
    if (r1 - r0 > 4 * 32) {  // uniform across the CTA
        const int sub = (r1 - r0 + WARPS - 1) / WARPS;
        const int g0 = min(r1, r0 + warp * sub), g1 = min(r1, g0 + sub);
        const float acc = warp_range_sum<2>(w, g0, g1, lane);
        __syncthreads();  // previous users of s.part are done
        if (lane == 0) s.part[warp] = acc;
        __syncthreads();
        float before = 0.0f;
        int fallback = 0;
        int hit = pick_part([&](int i) { return s.part[i]; }, WARPS, rem, &before, &fallback);
        if (!want_hit || hit < 0) {
            want_hit = false;
            hit = fallback;
        }
        rem -= before;
        r0 = min(r1, r0 + hit * sub);
        r1 = min(r1, r0 + sub);
    }
    __syncthreads();
    if (warp == 0) {
        float run = 0.0f;
        int found = -1, last_pos = -1;
        for (int gb = r0; gb < r1 && found < 0; gb += 32 * kWalkBatch) {
            typename Weights::Raw raw[kWalkBatch];  // the whole batch is fetched before the serial scan
#pragma unroll
            for (int i = 0; i < kWalkBatch; ++i) {
                const int g = gb + 32 * i + lane;
                raw[i] = g < r1 ? w.fetch(g) : w.nothing();
            }
#pragma unroll
            for (int i = 0; i < kWalkBatch; ++i) {
                const int gs = gb + 32 * i;
                if (gs >= r1 || found >= 0) break;
                walk_step(w.weigh(raw[i]), gs, lane, want_hit, rem, run, found, last_pos);
            }
        }
        if (lane == 0) {
            s.result = found;
            s.last_positive = last_pos;
        }
    }
    __syncthreads();
    const int k = s.result >= 0 ? s.result : s.last_positive;
    __syncthreads();  // scratch may be reused by the caller
    return k;
}

// Inverse-CDF draw by one CTA of 32 * WARPS threads: the smallest index k whose
// running weight sum exceeds u * (sum of all weights); the last index with
// positive weight if rounding leaves none.  The vocabulary is cut into WARPS
// contiguous segments (one per warp); the segment holding the target is then
// resolved by locate_in_range.  Returns the index to all threads, the total
// through *total_out.  `mine`: the sum over this warp's segment, where it is known already.
template <int WARPS, class Weights>
__device__ int block_inverse_cdf(const Weights& w, int vocab, float u, CdfScratch<WARPS>& s, float* total_out, const float* mine = nullptr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int groups = w.groups();
    const int seg = (groups + WARPS - 1) / WARPS;
    const int g0 = min(groups, warp * seg), g1 = min(groups, g0 + seg);
    const float acc = mine ? *mine : warp_range_sum<kCdfBatch>(w, g0, g1, lane);
    if (lane == 0) s.part[warp] = acc;
    __syncthreads();
    float total = 0.0f;
#pragma unroll
    for (int i = 0; i < WARPS; ++i) total += s.part[i];
    const float target = u * total;
    float before = 0.0f;
    int fallback = 0;
    int hit = pick_part([&](int i) { return s.part[i]; }, WARPS, target, &before, &fallback);
    const bool want_hit = hit >= 0;
    if (!want_hit) hit = fallback;
    const int r0 = min(groups, hit * seg), r1 = min(groups, r0 + seg);
    const int k = locate_in_range<WARPS>(w, r0, r1, target - before, want_hit, s);
    *total_out = total;
    return max(0, min(k - w.shift(), vocab - 1));
}

// The same draw by a thread-block cluster: CTA `rank` of `nctas` owns a
// contiguous slice of the vocabulary, the per-warp totals of all CTAs are read
// through distributed shared memory, and only the CTA whose slice holds the
// target goes on to resolve it.  Returns the index in that CTA and -1 in the
// others; the total is returned to all.
template <int WARPS, class Weights>
__device__ int cluster_inverse_cdf(const Weights& w, int vocab, float u, CdfScratch<WARPS>& s, float* total_out, const float* own = nullptr) {
    cg::cluster_group cluster = cg::this_cluster();
    const int nctas = static_cast<int>(cluster.num_blocks());
    const int rank = static_cast<int>(cluster.block_rank());
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int groups = w.groups();
    const int slice = (groups + nctas - 1) / nctas;
    const int seg = (slice + WARPS - 1) / WARPS;
    auto seg_begin = [&](int part) {  // part = cta * WARPS + warp
        const int c0 = min(groups, (part / WARPS) * slice), c1 = min(groups, c0 + slice);
        return min(c1, c0 + (part % WARPS) * seg);
    };
    auto seg_end = [&](int part) {
        const int c0 = min(groups, (part / WARPS) * slice), c1 = min(groups, c0 + slice);
        return min(c1, seg_begin(part) + seg);
    };
    const int mine = rank * WARPS + warp;
    const int b0 = seg_begin(mine), b1 = seg_end(mine);
    // When a warp's segment fits one batch of fetches, the weights stay in registers: the warp whose segment
    // holds the target then walks it without going back to memory.
    const bool keep = !own && seg <= 32 * kClusterCdfBatch;  // (uniform across the cluster)
    float4 kept[kClusterCdfBatch];
    float acc;
    if (keep) {
        typename Weights::Raw raw[kClusterCdfBatch];
#pragma unroll
        for (int i = 0; i < kClusterCdfBatch; ++i) {
            const int g = b0 + lane + 32 * i;
            raw[i] = g < b1 ? w.fetch(g) : w.nothing();
        }
        acc = 0.0f;
#pragma unroll
        for (int i = 0; i < kClusterCdfBatch; ++i) {
            kept[i] = w.weigh(raw[i]);
            acc += (kept[i].x + kept[i].y) + (kept[i].z + kept[i].w);
        }
        acc = warp_sum(acc);
    } else {
        acc = own ? *own : warp_range_sum<kClusterCdfBatch>(w, b0, b1, lane);
    }
    if (lane == 0) s.part[warp] = acc;
    cluster.sync();
    // warp 0 copies every CTA's totals into this CTA's shared memory ...
    const int parts = nctas * WARPS;
    if (warp == 0)
        for (int i = lane; i < parts; i += 32) s.all[i] = cluster.map_shared_rank(s.part, i / WARPS)[i % WARPS];
    __syncthreads();
    // (this CTA has read its peers' totals: it arrives at the cluster barrier now and waits for the others only
    // when it is about to leave, so the CTA that resolves the draw does not stand still meanwhile)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    // ... and scans them: lane l takes the consecutive parts [l*per, (l+1)*per)
    if (warp == 0) {
        const int per = (parts + 31) / 32;
        float mine_sum = 0.0f;
        for (int i = lane * per; i < min(parts, (lane + 1) * per); ++i) mine_sum += s.all[i];
        const float incl = warp_inclusive_scan(mine_sum, lane);
        const float tot = __shfl_sync(kFullMask, incl, 31);
        const float tgt = u * tot;
        const unsigned over = __ballot_sync(kFullMask, incl > tgt);
        const unsigned pos = __ballot_sync(kFullMask, mine_sum > 0.0f);
        const int hl = over ? __ffs(over) - 1 : (pos ? 31 - __clz(pos) : 0);
        if (lane == hl) {
            float run = incl - mine_sum;
            int hit = -1, last = lane * per;
            for (int i = lane * per; i < min(parts, (lane + 1) * per); ++i) {
                if (s.all[i] > 0.0f) last = i;
                if (over && hit < 0 && run + s.all[i] > tgt) { hit = i; break; }
                run += s.all[i];
            }
            if (hit < 0) { hit = last; s.pick_hit = 0; run = 0.0f; } else { s.pick_hit = 1; }
            s.pick_part_index = hit;
            s.pick_before = run;
            s.pick_total = tot;
        }
    }
    __syncthreads();
    const float total = s.pick_total;
    const float target = u * total;
    const float before = s.pick_before;
    const int hit = s.pick_part_index;
    const bool want_hit = s.pick_hit != 0;
    *total_out = total;
    int k = -1;
    if (hit / WARPS == rank) {  // (uniform across the CTA)
        if (keep) {
            if (warp == hit % WARPS) {
                float run = 0.0f;
                int found = -1, last_pos = -1;
#pragma unroll
                for (int i = 0; i < kClusterCdfBatch; ++i) {
                    const int gs = b0 + 32 * i;
                    if (gs >= b1 || found >= 0) break;
                    walk_step(kept[i], gs, lane, want_hit, target - before, run, found, last_pos);
                }
                if (lane == 0) {
                    s.result = found;
                    s.last_positive = last_pos;
                }
            }
            __syncthreads();
            k = s.result >= 0 ? s.result : s.last_positive;
        } else {
            k = locate_in_range<WARPS>(w, seg_begin(hit), seg_end(hit), target - before, want_hit, s);
        }
        k = max(0, min(k - w.shift(), vocab - 1));
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // nobody reads this CTA's totals any more
    return k;
}

// (max, lowest index attaining it) across a CTA of 32 * WARPS threads; the
// result is valid in thread 0.
template <int WARPS>
__device__ __forceinline__ void block_argmax(float& m, int& arg, float* red, int* red_i) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float om = __shfl_xor_sync(kFullMask, m, o);
        const int oa = __shfl_xor_sync(kFullMask, arg, o);
        if (om > m || (om == m && oa < arg)) { m = om; arg = oa; }
    }
    if (lane == 0) { red[warp] = m; red_i[warp] = arg; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < WARPS; ++i)
            if (red[i] > m || (red[i] == m && red_i[i] < arg)) { m = red[i]; arg = red_i[i]; }
    }
}

// One chunk of one row, as written by verify_stats_kernel.
struct __align__(16) ChunkStat {
    float max;     // chunk maximum
    float aux;     // T > 0: sum exp((l - max) / T) over the chunk; T = 0: argmax index as int bits
    float xlogit;  // the row's logit at the drafted token, if that token falls in this chunk
    float bad;     // T = 0: non-zero if the chunk holds a NaN or +inf logit (T > 0: the sums show it)
};

template <int W>
struct StatShared {
    float max[W], sum[W];
    int index[W];
};

// The statistics of groups [g0, g1) of a row by a CTA of T threads; valid in thread 0, the logit at the drafted token left out.
template <int T, bool GREEDY, bool VEC>
__device__ __forceinline__ float4 chunk_statistics(const Row<VEC>& r, int g0, int g1, float c2, StatShared<T / 32>& sh) {
    constexpr int W = T / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Every thread streams groups g0+tid, g0+tid+T, ... with kUnroll 128-bit
    // loads in flight and keeps a running (max, sum exp) pair that is rescaled
    // when the maximum moves; one block-wide merge at the end.
    constexpr float kPad = -INFINITY;
    float m = -FLT_MAX;  // finite, so that (m - new_max) never becomes inf - inf
    float s = 0.0f;
    int arg = 0x7fffffff;
    bool bad = false;  // T = 0 only: a NaN or +inf logit (the comparisons below would pass over a NaN in silence)
    for (int base = g0 + tid; base < g1; base += kUnroll * T) {
        float4 v[kUnroll];
#pragma unroll
        for (int i = 0; i < kUnroll; ++i) {
            const int g = base + i * T;
            v[i] = g < g1 ? r.load(g, kPad) : make_float4(kPad, kPad, kPad, kPad);
        }
        if (GREEDY) {
#pragma unroll
            for (int i = 0; i < kUnroll; ++i) {
                const int j = 4 * (base + i * T) - r.shift;  // indices grow with i: '>' keeps the lowest on ties
                if (v[i].x > m) { m = v[i].x; arg = j; }
                if (v[i].y > m) { m = v[i].y; arg = j + 1; }
                if (v[i].z > m) { m = v[i].z; arg = j + 2; }
                if (v[i].w > m) { m = v[i].w; arg = j + 3; }
                bad |= !(v[i].x < INFINITY) | !(v[i].y < INFINITY) | !(v[i].z < INFINITY) | !(v[i].w < INFINITY);
            }
        } else {
            float bm = m;
#pragma unroll
            for (int i = 0; i < kUnroll; ++i)
                bm = fmaxf(bm, fmaxf(fmaxf(v[i].x, v[i].y), fmaxf(v[i].z, v[i].w)));
            s *= fast_exp2((m - bm) * c2);
            m = bm;
            // exp2(v * c2 - m * c2): one multiply-add per logit (the kernel is close to issue-bound).  A thread that has
            // seen only padding keeps m = -FLT_MAX: the product is clamped so that -inf * c2 + it stays -inf.
            const float mc = fminf(-m * c2, FLT_MAX);
#pragma unroll
            for (int i = 0; i < kUnroll; ++i)
                s += (fast_exp2(fmaf(v[i].x, c2, mc)) + fast_exp2(fmaf(v[i].y, c2, mc))) +
                     (fast_exp2(fmaf(v[i].z, c2, mc)) + fast_exp2(fmaf(v[i].w, c2, mc)));
        }
    }
    if (GREEDY) {
        const int any_bad = __syncthreads_or(bad ? 1 : 0);
        block_argmax<W>(m, arg, sh.max, sh.index);
        return make_float4(m, __int_as_float(arg), 0.0f, any_bad ? 1.0f : 0.0f);
    } else {
        const float wm = warp_max(m);
        s = warp_sum(s * fast_exp2((m - wm) * c2));
        if (lane == 0) { sh.max[warp] = wm; sh.sum[warp] = s; }
        __syncthreads();
        float bm = sh.max[0], t = 0.0f;
        if (tid == 0) {
#pragma unroll
            for (int i = 1; i < W; ++i) bm = fmaxf(bm, sh.max[i]);
#pragma unroll
            for (int i = 0; i < W; ++i) t += sh.sum[i] * fast_exp2((sh.max[i] - bm) * c2);
        }
        return make_float4(bm, t, 0.0f, 0.0f);
    }
}

// The logits of row `row` of a sequence: p_1..p_{gamma+1}, q_1..q_gamma.
__device__ __forceinline__ const float* verify_row(const float* target_logits, const float* draft_logits, int b, int row, int gamma, int vocab) {
    return row <= gamma ? target_logits + (static_cast<size_t>(b) * (gamma + 1) + row) * vocab
                        : draft_logits + (static_cast<size_t>(b) * gamma + (row - gamma - 1)) * vocab;
}
// Its logit at the drafted token (none for p_{gamma+1}) if that lies in groups [g0, g1): the accept test then needs no further
// trip to memory.
template <bool VEC>
__device__ __forceinline__ float verify_logit(const Row<VEC>& r, const int32_t* draft_tokens, int b, int row, int gamma, int g0, int g1) {
    if (row == gamma) return 0.0f;
    const int x = draft_tokens[static_cast<size_t>(b) * gamma + (row < gamma ? row : row - gamma - 1)];
    return x >= 0 && x < r.vocab && x + r.shift >= 4 * g0 && x + r.shift < 4 * g1 ? __ldg(r.base + x) : 0.0f;
}

// grid = (chunks, rows, batch); rows = 2*gamma+1 (T > 0: p_1..p_{gamma+1}, q_1..q_gamma)
// or gamma+1 (T = 0: only p is read).
template <bool GREEDY, bool VEC>
__global__ void __launch_bounds__(kStatThreads)
verify_stats_kernel(const float* target_logits, const float* draft_logits, const int32_t* draft_tokens, int gamma, int vocab,
                    float c2, ChunkStat* stats) {
    __shared__ StatShared<kStatWarps> sh;
    pdl_wait();
    pdl_trigger();  // after the wait: the finishing kernel, which may take its places as this grid drains, fetches inputs at once
    target_logits = after_wait(target_logits);
    draft_logits = after_wait(draft_logits);
    draft_tokens = after_wait(draft_tokens);
    const int chunk = blockIdx.x, chunks = gridDim.x, row = blockIdx.y, rows = gridDim.y, b = blockIdx.z;
    const Row<VEC> r = make_row<VEC>(verify_row(target_logits, draft_logits, b, row, gamma, vocab), vocab);
    const int groups = r.groups();
    const int per_chunk = (groups + chunks - 1) / chunks;
    const int g0 = chunk * per_chunk, g1 = min(groups, g0 + per_chunk);
    float xlogit = 0.0f;
    if (threadIdx.x == 0 && !GREEDY) xlogit = verify_logit(r, draft_tokens, b, row, gamma, g0, g1);
    float4 found = chunk_statistics<kStatThreads, GREEDY, VEC>(r, g0, g1, c2, sh);
    if (threadIdx.x == 0) {
        if (!GREEDY) found.z = xlogit;
        *reinterpret_cast<float4*>(stats + (static_cast<size_t>(b) * rows + row) * chunks + chunk) = found;
    }
}

struct FinishShared {
    float row_max[kMaxRows];
    float row_aux[kMaxRows];
    float row_x[kMaxRows];
    CdfScratch<kFinishThreads / 32> cdf;
    float u_cand[kMaxGamma + 1];
    float u_final;
    int n;
};

// grid = batch * cluster size, one thread-block cluster per sequence.  Everything
// after the statistics: merge, accept tests, adjusted distribution, draw.  The
// cheap decision part is repeated in every CTA of the cluster; the pass over
// row n+1 is split between them.
// ALONE: the statistics too, a row at a time to each CTA (one_kernel).
template <bool GREEDY, bool VEC, bool CUT, bool ALONE>
__global__ void __launch_bounds__(kFinishThreads, 2)
verify_finish_kernel(const float* __restrict__ target_logits, const float* __restrict__ draft_logits,
                     const int32_t* __restrict__ draft_tokens, const float* __restrict__ uniforms, int gamma,
                     int vocab, float inv_t, int chunks, int cluster_size, ChunkStat* stats,
                     const float* __restrict__ final_uniforms, float lenience, const float* floors,
                     int32_t* __restrict__ n_accepted, int32_t* __restrict__ next_token, int* __restrict__ nonfinite) {
    __shared__ FinishShared sh;
    if (ALONE) {  // (all of its inputs may come from the kernel in front)
        pdl_wait();
        pdl_trigger();
        target_logits = after_wait(target_logits);
        draft_logits = after_wait(draft_logits);
        draft_tokens = after_wait(draft_tokens);
        uniforms = after_wait(uniforms);
    }
    const int tid = threadIdx.x;
    const int b = blockIdx.x / cluster_size;
    const int rank = blockIdx.x % cluster_size;
    const int rows = GREEDY ? gamma + 1 : 2 * gamma + 1;
    const float c2 = inv_t * kLog2e;
    const float* tl = target_logits + static_cast<size_t>(b) * (gamma + 1) * vocab;
    const float* ql = GREEDY ? nullptr : draft_logits + static_cast<size_t>(b) * gamma * vocab;

    // Inputs that the kernel before does not produce can be fetched before waiting for it: it lets this one start when its
    // own wait is over, and so what came before it is complete.
    if (ALONE) {
        __shared__ StatShared<kFinishThreads / 32> stat;
        for (int row = rank; row < rows; row += cluster_size) {
            const Row<VEC> r = make_row<VEC>(verify_row(target_logits, draft_logits, b, row, gamma, vocab), vocab);
            float4 found = chunk_statistics<kFinishThreads, GREEDY, VEC>(r, 0, r.groups(), c2, stat);
            if (tid == 0) {
                if (!GREEDY) found.z = verify_logit(r, draft_tokens, b, row, gamma, 0, r.groups());
                *reinterpret_cast<float4*>(stats + static_cast<size_t>(b) * rows + row) = found;
            }
            __syncthreads();  // (`stat` is used again)
        }
    }
    float my_uniform = 0.5f;
    if (!GREEDY && tid <= gamma) my_uniform = __ldg(uniforms + static_cast<size_t>(b) * (gamma + 1) + tid);
    int my_x = -1;
    if (tid < rows && tid != gamma)
        my_x = draft_tokens[static_cast<size_t>(b) * gamma + (tid < gamma ? tid : tid - gamma - 1)];
    // lenient argmax decoding compares the target's logit at the drafted token with the row maximum
    float my_xlogit = 0.0f;
    if (GREEDY && lenience < 1.0f && tid < gamma && my_x >= 0 && my_x < vocab) my_xlogit = __ldg(tl + static_cast<size_t>(tid) * vocab + my_x);
    // The generation loop keys the final draw by the position it decides, which depends on n: it passes one
    // candidate uniform per possible n; all of them are fetched now.
    if (!GREEDY && final_uniforms && tid <= gamma) sh.u_cand[tid] = __ldg(final_uniforms + static_cast<size_t>(b) * (gamma + 1) + tid);
    if (ALONE) {
        cg::this_cluster().sync();  // (every CTA sees the others' statistics)
    } else {
        pdl_trigger();
        pdl_wait();
        floors = after_wait(floors);
    }

    // merge the chunk statistics of row `tid` (eight loads in flight at a time)
    if (tid < rows) {
        const ChunkStat* st_r = stats + (static_cast<size_t>(b) * rows + tid) * chunks;
        float M = -FLT_MAX, A = 0.0f, X = 0.0f;
        int best = 0x7fffffff;
        bool bad = false;
        // (the chunks of this row, as the statistics kernel cut it)
        const int shift = VEC || GREEDY ? 0 : row_shift(tid <= gamma ? tl + static_cast<size_t>(tid) * vocab : ql + static_cast<size_t>(tid - gamma - 1) * vocab);
        const int per_chunk = (((vocab + shift + 3) >> 2) + chunks - 1) / chunks;
        const int xchunk = (my_x >= 0 && my_x < vocab) ? ((my_x + shift) >> 2) / per_chunk : -1;
        constexpr int kMergeBatch = 8;  // chunk statistics fetched together
        for (int c0 = 0; c0 < chunks; c0 += kMergeBatch) {
            float4 st[kMergeBatch];
#pragma unroll
            for (int i = 0; i < kMergeBatch; ++i)
                st[i] = c0 + i < chunks ? __ldcg(reinterpret_cast<const float4*>(st_r + c0 + i))
                                        : make_float4(-FLT_MAX, __int_as_float(0x7fffffff), 0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < kMergeBatch; ++i) {
                if (c0 + i >= chunks) break;
                if (GREEDY) {
                    const int ci = __float_as_int(st[i].y);
                    if (st[i].x > M || (st[i].x == M && ci < best)) { M = st[i].x; best = ci; }
                    bad |= st[i].w != 0.0f;
                } else {
                    const float nm = fmaxf(M, st[i].x);
                    A = A * fast_exp2((M - nm) * c2) + st[i].y * fast_exp2((st[i].x - nm) * c2);
                    M = nm;
                    if (c0 + i == xchunk) X = st[i].z;
                }
            }
        }
        // a NaN or +inf logit (or a row without a finite logit) leaves a sum that is not a positive number
        if (!GREEDY) bad = !(A > 0.0f) || !isfinite(A) || !isfinite(M);
        if (bad && nonfinite && rank == 0) atomicExch(nonfinite, 1);
        sh.row_max[tid] = M;
        sh.row_aux[tid] = GREEDY ? __int_as_float(best) : A;
        sh.row_x[tid] = X;
    }
    if (tid == 0) sh.n = gamma;
    __syncthreads();

    // the gamma accept tests (Algorithm 1: n = index of the first rejection)
    if (tid < gamma) {
        bool reject = true;
        if (my_x >= 0 && my_x < vocab) {
            if (GREEDY) {
                // strict: x must be the lowest-index maximum; lenient (Appendix A.5 at T = 0):
                // p(x) >= l max p before standardising, i.e. logit(x) >= max logit + ln l
                reject = lenience < 1.0f ? !(my_xlogit - sh.row_max[tid] - logf(lenience) >= 0.0f)
                                         : my_x != __float_as_int(sh.row_aux[tid]);
            } else {
                const float ep = expf((sh.row_x[tid] - sh.row_max[tid]) * inv_t);
                const float eq = expf((sh.row_x[gamma + 1 + tid] - sh.row_max[gamma + 1 + tid]) * inv_t);
                // r * l * q(x) > p(x) with p = ep / Sp, q = eq / Sq, cross-multiplied (l = 1: Algorithm 1)
                reject = my_uniform * lenience * eq * sh.row_aux[tid] > ep * sh.row_aux[gamma + 1 + tid];
            }
        }
        if (reject) atomicMin(&sh.n, tid);
    }
    if (tid == gamma) sh.u_final = my_uniform;
    __syncthreads();
    const int n = sh.n;

    int token = -1;
    if (GREEDY) {
        if (rank == 0) token = __float_as_int(sh.row_aux[n]);
    } else {
        constexpr int W = kFinishThreads / 32;
        const float u = final_uniforms ? sh.u_cand[n] : sh.u_final;
        PlainWeights<VEC, CUT> pw;
        const float* fl = CUT ? floors + static_cast<size_t>(b) * rows : nullptr;
        pw.p = make_row<VEC, CUT>(tl + static_cast<size_t>(n) * vocab, vocab, CUT ? __ldcg(fl + n) : -INFINITY);
        pw.max_p = sh.row_max[n];
        pw.c2 = c2;
        float total = 0.0f;
        bool plain = n == gamma;
        if (!plain) {
            ResidualWeights<VEC, CUT> rw;
            rw.p = pw.p;
            rw.q = make_row<VEC, CUT>(ql + static_cast<size_t>(n) * vocab, vocab, CUT ? __ldcg(fl + gamma + 1 + n) : -INFINITY, pw.p.shift);
            rw.max_p = sh.row_max[n];
            rw.max_q = sh.row_max[gamma + 1 + n];
            rw.inv_sum_p = 1.0f / sh.row_aux[n];
            rw.inv_sum_q = 1.0f / sh.row_aux[gamma + 1 + n];
            rw.c2 = c2;
            token = cluster_inverse_cdf<W>(rw, vocab, u, sh.cdf, &total);
            plain = !(total > 0.0f) || !isfinite(total);  // vanished residual: draw from p_{n+1}
        }
        if (plain) token = cluster_inverse_cdf<W>(pw, vocab, u, sh.cdf, &total);
    }
    if (tid == 0) {
        if (rank == 0) n_accepted[b] = n;
        if (token >= 0) next_token[b] = token;  // exactly one CTA of the cluster holds the draw
    }
}

// One CTA per row: tokens[r] ~ softmax(logits[r] / T), or argmax at T = 0.
template <bool VEC>
__global__ void __launch_bounds__(kSampleThreads)
sample_kernel(const float* logits, size_t logit_stride, const float* uniforms, int uniform_stride, int vocab, float inv_t, bool greedy,
              int32_t* tokens, int token_stride, int* nonfinite) {
    constexpr int W = kSampleThreads / 32;
    __shared__ float red[W];
    __shared__ int red_i[W];
    __shared__ CdfScratch<W> cdf;
    __shared__ float s_max;
    __shared__ int s_arg;
    pdl_trigger();
    pdl_wait();
    logits = after_wait(logits);
    uniforms = after_wait(uniforms);
    const int tid = threadIdx.x;
    const Row<VEC> r = make_row<VEC>(logits + static_cast<size_t>(blockIdx.x) * logit_stride, vocab);
    const int groups = r.groups();
    float m = -FLT_MAX;
    int arg = 0x7fffffff;
    bool bad = false;  // a NaN or +inf logit
#pragma unroll 4
    for (int g = tid; g < groups; g += kSampleThreads) {
        const float4 v = r.load(g, -INFINITY);
        const int j = 4 * g - r.shift;
        if (v.x > m) { m = v.x; arg = j; }
        if (v.y > m) { m = v.y; arg = j + 1; }
        if (v.z > m) { m = v.z; arg = j + 2; }
        if (v.w > m) { m = v.w; arg = j + 3; }
        bad |= !(v.x < INFINITY) | !(v.y < INFINITY) | !(v.z < INFINITY) | !(v.w < INFINITY);
    }
    if (nonfinite && bad) atomicExch(nonfinite, 1);
    block_argmax<W>(m, arg, red, red_i);
    if (tid == 0) { s_max = m; s_arg = arg; }
    __syncthreads();
    int token = s_arg;
    if (!greedy) {
        PlainWeights<VEC> pw;
        pw.p = r;
        pw.max_p = s_max;
        pw.c2 = inv_t * kLog2e;
        float total;
        token = block_inverse_cdf<W>(pw, vocab, uniforms[blockIdx.x * uniform_stride], cdf, &total);
    }
    if (tid == 0) tokens[blockIdx.x * token_stride] = max(0, min(token, vocab - 1));
}

// ---- top-k and nucleus: the lowest logit that each row keeps ---------------------
// One CTA per row, several CTAs per SM, or, where that would leave SMs idle or unevenly loaded, a cluster of up to four
// (cut_shape).  Both cuts are a selection: the largest
// value t such that the logits at or above t number at least k (top-k), or carry
// at least top_p of the mass (nucleus).  The row is never sorted or held:
//   1. one pass finds the range [lo, hi] of the logits still in play;
//   2. one pass drops them into kSelBins equal-width bins counted from the top
//      (a count per bin, for the nucleus also the mass), a scan finds the bin in
//      which the target is crossed;
//   3. if that bin holds few logits they are copied out and ranked against each
//      other exactly; otherwise the bin's own range becomes [lo, hi] and step 2
//      repeats (heavy ties end when lo == hi).
// The bin of a logit is a monotone function of it, so the bins partition the row
// by value and the result is exact (comparisons of the logits themselves decide;
// -inf, +inf and NaN logits are never in play).  Mass is summed in fixed point
// (units of 2^-32 of the largest weight) with integer atomics, so every order of
// summation gives the same totals: a row always gives the same floor, however the
// threads interleave, however many CTAs share it and whether it was listed (below).  The kernel is bound by instruction issue, not by memory
// (the passes after the first hit L2), so the per-logit work is kept short: no
// float-to-int conversion for the bin, one 32-bit atomic plus a rare carry for
// the mass (a 64-bit shared-memory atomic cost 48 us of 180 on 960 rows of 32000),
// a two-instruction test before a logit is asked whether it is in the chosen bin.
//
// The CTAs of a cluster take a slice of the row each, and what they find goes through distributed shared memory: the range
// and the warps' maxima to all of them; of the bins the sums of 32 at a time, then only the 32 where the target is
// crossed (with all bins read by everyone a cluster of four cost 40 us more on 200 rows of 100000); the lists, made
// locally, to the CTA of rank 0, which ranks them.
constexpr int kSelMostWarps = 16;  // of a CTA: T / 32, T = 256 or 512 threads
constexpr int kSelBins = 2048;
constexpr int kSelSegments = kSelBins / 32;
constexpr int kSelCap = 1024;   // logits ranked against each other at the end
constexpr int kSelLevels = 40;  // every level shrinks the range; fp32 allows far fewer than this
constexpr int kMostCtas = 4;    // per row
static_assert(kSelSegments == 64, "two segments to a lane");

struct SelShared {
    unsigned mass_lo[kSelBins], mass_hi[kSelBins];  // a bin's mass, low and high word (apart: the low words then spread over all banks)
    float cand[kSelCap];
    unsigned long long cand_mass[kSelCap];
    unsigned long long segment[kSelSegments];       // counts or masses of 32 bins
    unsigned long long warp_mass[kSelMostWarps];
    unsigned warp_cnt[kSelMostWarps];
    float warp_lo[kSelMostWarps], warp_hi[kSelMostWarps], warp_top[kSelMostWarps];
    unsigned long long below[kSelMostWarps];        // mass that is not listed, of what the warps went over
    int found[kSelMostWarps];                       // candidates of the warps
    float kept[kSelMostWarps];                      // of what the warps have listed, the weights that the cut leaves
    float cta_max[kMostCtas], cta_sum[kMostCtas];  // (in the CTA of rank 0)
    unsigned n_cand, n_hit, n_list;  // listed here; threads that reach the pivot; listed in all CTAs (in rank 0's)
    float floor;    // what rank 0 found
    float row_top;  // the largest logit, +inf included
    // where the scan found the target crossed
    int bin;
    unsigned in_bin;
    unsigned long long before, target;
    unsigned cnt[kSelBins];  // (last: a nucleus from its candidates has no use for it)
};

// The CTAs that share a row.
template <bool SOLO>
struct Team {
    int rank, size;
    __device__ __forceinline__ Team() {
        rank = SOLO ? 0 : static_cast<int>(cg::this_cluster().block_rank());
        size = SOLO ? 1 : static_cast<int>(cg::this_cluster().num_blocks());
    }
    __device__ __forceinline__ void sync() const {
        if (SOLO) __syncthreads();
        else cg::this_cluster().sync();
    }
    __device__ __forceinline__ SelShared& of(SelShared& sh, int r) const { return SOLO ? sh : *cg::this_cluster().map_shared_rank(&sh, r); }
};

// A CTA's slice of a row; LOADS 128-bit loads are in flight per thread when it is gone over.
template <bool VEC, int LOADS>
struct Slice {
    static constexpr bool kList = false;
    Row<VEC> row;
    int g0, g1;
};

// Logits that can be kept, if they are few: values in sh.cand, their places in list_index.
__device__ __forceinline__ unsigned* list_index(SelShared& sh) { return sh.cnt + kSelBins / 2; }

__device__ __forceinline__ void list_group(const float4& v, int j, float at_least, SelShared& sh) {
    if (!(fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)) >= at_least)) return;
    const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (e[i] >= at_least) {
            const unsigned at = atomicAdd(&sh.n_cand, 1u);
            if (at < kSelCap) {
                sh.cand[at] = e[i];
                list_index(sh)[at] = static_cast<unsigned>(j + i);
            }
        }
    }
}

// Brings the CTAs' lists together in the first one's, with their masses or their places.  Returns how many there are, to all;
// -1, and nothing is brought together, if that is more than kSelCap.
template <int T, bool SOLO>
__device__ int gather_list(const Team<SOLO>& team, bool masses, SelShared& sh) {
    team.sync();
    unsigned total = 0;
    for (int r = 0; r < team.size; ++r) total += team.of(sh, r).n_cand;
    if (total > kSelCap) return -1;
    if (team.rank == 0) {
        if (!SOLO) {
            unsigned at = sh.n_cand;
            for (int r = 1; r < team.size; ++r) {
                SelShared& from = team.of(sh, r);
                const unsigned n = from.n_cand;
                for (unsigned i = threadIdx.x; i < n; i += T) {
                    sh.cand[at + i] = from.cand[i];
                    if (masses) sh.cand_mass[at + i] = from.cand_mass[i];
                    else list_index(sh)[at + i] = list_index(from)[i];
                }
                at += n;
            }
        }
        if (threadIdx.x == 0) sh.n_list = total;
        __syncthreads();
    }
    return static_cast<int>(total);
}

// f(LOADS times four logits, the first ones' group) over the slice; the others are T groups apart.
template <int T, bool VEC, int LOADS, class F>
__device__ __forceinline__ void for_each_batch(const Slice<VEC, LOADS>& s, F f) {
    for (int base = s.g0 + threadIdx.x; base < s.g1; base += LOADS * T) {
        float4 v[LOADS];
#pragma unroll
        for (int i = 0; i < LOADS; ++i) {
            const int g = base + i * T;
            v[i] = g < s.g1 ? s.row.raw(g, -INFINITY) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
        f(v, base);
    }
}
// f(four logits, their group) over the slice.
template <int T, bool VEC, int LOADS, class F>
__device__ __forceinline__ void for_each_group(const Slice<VEC, LOADS>& s, F f) {
    for_each_batch<T>(s, [&](const float4 (&v)[LOADS], int base) {
#pragma unroll
        for (int i = 0; i < LOADS; ++i) f(v[i], base + i * T);
    });
}
template <int T, bool VEC, int LOADS, class F>
__device__ __forceinline__ void for_each_logit(const Slice<VEC, LOADS>& s, F f) {
    for_each_group<T>(s, [&](const float4& v, int) {
        f(v.x);
        f(v.y);
        f(v.z);
        f(v.w);
    });
}

// What a warp has listed of its row: at[0] .. at[n - 1].
template <bool VEC, int LOADS>
struct Listed {
    static constexpr bool kList = true;
    static constexpr int kLoads = LOADS;
    const Slice<VEC, LOADS>& slice;
    const float* at;
    int n, first, step;
    float from, most;  // what is listed reaches `from`; the thread's largest logit (+inf for a NaN)
    bool all;          // the warp's candidates all found a place
};
template <int T, bool VEC, int LOADS, class F>
__device__ __forceinline__ void for_each_logit(const Listed<VEC, LOADS>& s, F f) {
    for (int i = s.first; i < s.n; i += s.step) f(s.at[i]);
}

// NaN if either is.
__device__ __forceinline__ float max_or_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The floor among the finite logits >= kf: MASS = false, the k-th largest of
// them; MASS = true, the nucleus of mass top_p with weights exp2((l - max) * c2).
// Every thread of the team returns the same value; -inf means "keep everything".
// Of a Source that is not the row but its listed candidates: the nucleus of the row, NaN where the list does not decide it.
template <int T, bool MASS, bool SOLO, class Source>
__device__ float select_floor(Source& s, const Team<SOLO>& team, float kf, unsigned k, float top_p, float c2, SelShared& sh) {
    constexpr bool LIST = Source::kList;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // 1. range and number of the logits in play
    float lo = INFINITY, hi = -INFINITY, all = -INFINITY;
    unsigned n = 0;
    if constexpr (LIST) {
        lo = s.from;
        hi = all = s.most;
        n = s.all ? 0 : 1;
    } else {
        for_each_logit<T>(s, [&](float v) {
            all = fmaxf(all, v);
            const bool in_play = fabsf(v) < INFINITY && v >= kf;
            const float u = in_play ? v : __int_as_float(0x7fc00000);  // (fminf and fmaxf pass over a NaN operand)
            lo = fminf(lo, u);
            hi = fmaxf(hi, u);
            n += in_play;
        });
    }
    // what the warps of the whole team found
    auto of_all = [&](float& least, float& most, float& top, unsigned& count) {
        least = warp_min(least);
        most = warp_max(most);
        top = warp_max(top);
        count = __reduce_add_sync(0xffffffffu, count);
        if (lane == 0) { sh.warp_lo[warp] = least; sh.warp_hi[warp] = most; sh.warp_top[warp] = top; sh.warp_cnt[warp] = count; }
        team.sync();
        least = INFINITY; most = top = -INFINITY; count = 0;
        for (int i = lane; i < team.size * (T / 32); i += 32) {
            const SelShared& from = team.of(sh, i / (T / 32));
            const int w = i % (T / 32);
            least = fminf(least, from.warp_lo[w]);
            most = fmaxf(most, from.warp_hi[w]);
            top = fmaxf(top, from.warp_top[w]);
            count += from.warp_cnt[w];
        }
        least = warp_min(least);
        most = warp_max(most);
        top = warp_max(top);
        count = __reduce_add_sync(0xffffffffu, count);
    };
    if (!LIST) team.sync();  // (the shared arrays may still be read by a previous call)
    of_all(lo, hi, all, n);
    if (tid == 0) sh.row_top = all;
    if constexpr (LIST) {
        s.all = n == 0;
        if (n > 0 || !(hi < INFINITY && hi >= lo)) return NAN;
    } else {
        if (n == 0 || (!MASS && k > n)) return kf;  // nothing to cut
    }
    // weight exp2((l - max) * c2) of a logit in units of 2^-32 (the largest float below 2^32, so that the row's
    // maximum still fits 32 bits): a bin's mass is then one 32-bit shared-memory atomic and, rarely, a carry
    const float mc = fminf(-hi * c2, FLT_MAX);
    auto units = [&](float v) { return fast_exp2(fmaf(v, c2, mc)) * 4294967040.0f; };
    auto fixed_mass = [&](float v) { return __float2uint_rz(units(v)); };
    if constexpr (LIST) {
        // what is not listed, in the same units: the total below is then the one that bins of the whole row come to, to the last
        // bit.  As a rule all of it is far below the maximum, where adding 2^23 with rounding toward zero is the conversion.
        unsigned long long below = 0;
        auto rest = [&](float v) { return v < s.from ? units(v) : 0.0f; };
        if (units(s.from) < 4194304.0f) {
            auto whole = [&](float v) { return __float_as_uint(__fadd_rz(rest(v), 8388608.0f)) - 0x4b000000u; };
            for_each_batch<T>(s.slice, [&](const float4 (&v)[Source::kLoads], int) {
                unsigned part = 0;  // (each below 2^23, four to a load)
#pragma unroll
                for (int i = 0; i < Source::kLoads; ++i) part += (whole(v[i].x) + whole(v[i].y)) + (whole(v[i].z) + whole(v[i].w));
                below += part;
            });
        } else {
            for_each_logit<T>(s.slice, [&](float v) { below += __float2uint_rz(rest(v)); });
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
        if (lane == 0) sh.below[warp] = below;
    }

    unsigned long long before = 0, target = k;  // counts, or masses
    for (int level = 0; level < kSelLevels; ++level) {
        if (lo == hi && !(LIST && level == 0)) return hi;  // everything left is one value: it stays whole
        const float top = hi, bottom = lo;
        // (top - v) * scale stays below kSelBins for every v >= bottom: the quarter bin absorbs the roundings
        const float scale = fminf((static_cast<float>(kSelBins) - 0.25f) / (top - bottom), FLT_MAX);
        // bin of a logit in [bottom, top], counted from the top; anything else gets no bin.  The floor is taken by
        // adding 2^23 with rounding toward zero (the sum's last bit is then worth one) instead of a conversion.
        auto bin_of = [&](float v) {
            const int b = __float_as_int(__fmaf_rz(top - v, scale, 8388608.0f)) & 0x7fffff;
            return (v >= bottom && v <= top) ? b : -1;
        };
        // 2. counts (and masses) per bin
        for (int i = tid; i < kSelBins; i += T) {
            if (MASS) { sh.mass_lo[i] = 0; sh.mass_hi[i] = 0; } else { sh.cnt[i] = 0; }
        }
        if (tid == 0) { sh.n_cand = sh.in_bin = 0; sh.bin = kSelBins - 1; sh.before = before; }
        __syncthreads();
        for_each_logit<T>(s, [&](float v) {
            const int b = bin_of(v);
            if (b >= 0) {
                if (MASS) {
                    const unsigned m = fixed_mass(v);
                    const unsigned was = atomicAdd(&sh.mass_lo[b], m);
                    if (was + m < was) atomicAdd(&sh.mass_hi[b], 1u);
                } else {
                    atomicAdd(&sh.cnt[b], 1u);
                }
            }
        });
        __syncthreads();
        {
            unsigned long long sum = 0;
#pragma unroll
            for (int i = 0; i < (kSelBins / T); ++i) {
                const int b = tid * (kSelBins / T) + i;
                sum += MASS ? (static_cast<unsigned long long>(sh.mass_hi[b]) << 32) | sh.mass_lo[b] : sh.cnt[b];
            }
            constexpr int kThreads = 32 * T / kSelBins;  // to a segment
#pragma unroll
            for (int d = 1; d < kThreads; d *= 2) sum += __shfl_xor_sync(0xffffffffu, sum, d);
            if (lane % kThreads == 0) sh.segment[tid / kThreads] = sum;
        }
        team.sync();
        if (warp == 0) {  // scan from the top: over the segments of all CTAs, then over the bins of one of them
            auto scan = [&](unsigned long long v) {
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned long long o = __shfl_up_sync(0xffffffffu, v, d);
                    if (lane >= d) v += o;
                }
                return v;
            };
            unsigned long long a = 0, b = 0;
            for (int r = 0; r < team.size; ++r) {
                const unsigned long long* from = team.of(sh, r).segment + 2 * lane;
                a += from[0];
                b += from[1];
            }
            const unsigned long long upto = scan(a + b), all_of_it = __shfl_sync(0xffffffffu, upto, 31);
            if (MASS && level == 0) {  // the first level sees every logit in play: top_p of their mass is the target
                unsigned long long mass = all_of_it;
                if constexpr (LIST) {  // .. and what is not listed
                    unsigned long long below = 0;
                    for (int i = lane; i < team.size * (T / 32); i += 32) below += team.of(sh, i / (T / 32)).below[i % (T / 32)];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
                    mass += below;
                }
                target = static_cast<unsigned long long>(ceil(static_cast<double>(top_p) * static_cast<double>(mass)));
                if (LIST && target > all_of_it) target = 0;  // (not decided)
            }
            const unsigned long long above = before + upto - (a + b);
            const unsigned who = __ballot_sync(0xffffffffu, above < target && above + a + b >= target);
            if (who) {
                const int at = __ffs(who) - 1;
                const bool second = __shfl_sync(0xffffffffu, above + a < target ? 1 : 0, at) != 0;
                const unsigned long long over = __shfl_sync(0xffffffffu, second ? above + a : above, at);
                const int bin = 32 * (2 * at + (second ? 1 : 0)) + lane;
                unsigned long long mine = 0;
                for (int r = 0; r < team.size; ++r) {
                    const SelShared& from = team.of(sh, r);
                    mine += MASS ? (static_cast<unsigned long long>(from.mass_hi[bin]) << 32) | from.mass_lo[bin] : from.cnt[bin];
                }
                const unsigned long long ex = over + scan(mine) - mine;
                if (ex < target && ex + mine >= target) {
                    sh.bin = bin;
                    sh.before = ex;
                    sh.in_bin = static_cast<unsigned>(mine);
                }
            }
            if (lane == 0) sh.target = target;
        }
        __syncthreads();
        const int bin = sh.bin;
        before = sh.before;
        target = sh.target;
        if (LIST && target == 0) return NAN;
        // top-k knows how many logits the bin holds; the nucleus keeps no counts and finds out by copying them
        const bool few = MASS || sh.in_bin <= kSelCap;
        // a cheap test that no logit of the bin fails (its centre, half its width and the roundings of bin_of, with
        // room to spare); the few that pass are then asked for their bin
        const float centre = top - (static_cast<float>(bin) + 0.5f) / scale;
        const float reach = 0.51f / scale + 2e-6f * fmaxf(fabsf(top), fabsf(bottom));
        auto in_the_bin = [&](float v) { return fabsf(v - centre) <= reach && bin_of(v) == bin; };
        if (few) {
            // 3. copy the bin's logits out and rank them against each other
            for_each_logit<T>(s, [&](float v) {
                if (in_the_bin(v)) {
                    const unsigned at = atomicAdd(&sh.n_cand, 1u);
                    if (at < kSelCap) { sh.cand[at] = v; if (MASS) sh.cand_mass[at] = fixed_mass(v); }
                }
            });
            const int count = gather_list<T>(team, MASS, sh);
            if (count >= 0) {  // (always so for top-k)
                if (team.rank == 0) {
                    float best = -INFINITY;
                    for (int i = tid; i < count; i += T) {
                        const float mine = sh.cand[i];
                        unsigned long long m = before;
#pragma unroll 8
                        for (int j = 0; j < count; ++j) {
                            const unsigned long long w = MASS ? sh.cand_mass[j] : 1ull;
                            m += sh.cand[j] >= mine ? w : 0ull;
                        }
                        if (m >= target) best = fmaxf(best, mine);
                    }
                    best = warp_max(best);
                    if (lane == 0) sh.warp_hi[warp] = best;
                    __syncthreads();
                    best = -INFINITY;
#pragma unroll
                    for (int w = 0; w < (T / 32); ++w) best = fmaxf(best, sh.warp_hi[w]);
                    best = best > -INFINITY ? best : bottom;
                    if (SOLO) return best;
                    if (tid < team.size) team.of(sh, tid).floor = best;
                }
                team.sync();
                return sh.floor;
            }
        }
        // the bin is crowded: its own range is searched next
        float new_lo = INFINITY, new_hi = -INFINITY, unused = -INFINITY;
        unsigned none = 0;
        for_each_logit<T>(s, [&](float v) {
            const bool here = in_the_bin(v);
            new_lo = fminf(new_lo, here ? v : INFINITY);
            new_hi = fmaxf(new_hi, here ? v : -INFINITY);
        });
        team.sync();  // (everyone has read the others' counts and bins)
        of_all(new_lo, new_hi, unused, none);
        lo = new_lo;
        hi = new_hi;
    }
    return lo;
}

template <int T>
__device__ __forceinline__ float block_max(float v, float* per_warp) {
    v = warp_max(v);
    if ((threadIdx.x & 31) == 0) per_warp[threadIdx.x >> 5] = v;
    __syncthreads();
    v = per_warp[0];
#pragma unroll
    for (int w = 1; w < (T / 32); ++w) v = fmaxf(v, per_warp[w]);
    return v;
}
// ---- the nucleus from a list of candidates ----
// A nucleus is a few per cent of a row as a rule, so the row is read once: a sample of it, four groups at a time and spread over
// the row, says above which logit its mass lies with room to spare; the pass lists what reaches that, every warp for
// itself.  A second pass, over what L2 holds by then, adds up the mass of the rest, now that the row's maximum is known.  The selection,
// the statistics and the draw's sums then go over the list, in shared memory.  A list that overflows or carries less than top_p of the
// mass decides nothing: the row is then binned as it lies.
// Masses are in the units of the bins, integers, so a row has one floor, from a list and from bins, to the last bit.  (Added up in fp32
// while the row was listed, against the sample's maximum, the mass of the rest moved one floor in several hundred at T = 1, and one in 80 of rows
// around 100 at T = 0.05.  The second pass costs
// nothing where L2 holds the rows already, 200 x 100000 46.3 -> 45.1 us, with other rows at every call 46.4 -> 50.2, cold 53 -> 61.)
// A warp lists its own part of the row, and large logits may all lie in one part (ids in order of frequency, say): a row of
// which a warp finds more than its share is listed once more, as one list.  Binned, listed where they lie by chance, and sorted, us
// call after call, rows N(0, 3^2), p = 0.9, with the draw: 200 x 100000 68, 46, 64; 64 x 100000 33, 28, 38; 1 x 50000 23, 18,
// 22; 200 x 32000 25, 22, 28; 960 x 32000 82, 58, 78; 24 x 9 rows of 50003, verified, 61, 42, 53.
// A flat row (N(0, 1), or p = 0.99) is no row for a list, which the sample sees; it costs that row the sample, and its bins the
// threads that the list's memory and registers keep off the SM: 64 x 100000 36 us binned, 37 so; 200 x 100000 72, 72; 600 x 20000
// 39, 48; 256 x 128000, which a pair of CTAs shares for the list's sake, 94, 120.
// What bounded the bins was an atomic per logit and three passes over the row behind the one that read it; now it is issue of
// the passes (a dozen instructions per logit in the first) and the barriers of the selection.  (Bins for the sampled range alone, no
// list: one pass over the row fewer than bins, but its atomics, in a few lanes of every warp, cost as much as in all of them:
// 200 x 100000, cold, 72 against 57.  One list for all warps from the start, filled in runs that the warps ask for: 60 for 46.)
constexpr int kSampleBins = 256;
constexpr float kSampleRange = 24.0f;  // of the bins, in powers of two below the largest
// Of the sampled logits as many are listed as carry all but half of (1 - top_p) of their mass, but a tenth at least: a sample of
// logits N(0, 3^2) holds few of those that carry the mass, and with a sixty-fourth as the least one row in 20 was listed too short.
// Where the most that can be listed carries less than all but 0.7 of (1 - top_p), nothing is (at 0.9 one row in six N(0, 3^2) at
// p = 0.98 was listed in vain).
constexpr float kListLeast = 0.10f, kListShare = 0.15f;
// Slots per warp: kListShare of its logits, 5 standard deviations (two CTAs with 100000 logits each then share an SM).  A CTA of several
// has room for the whole row's candidates where two of them still fit an SM, for they need not be spread evenly.
constexpr size_t kTwoListsBytes = 80 * 1024;  // of each of two CTAs on an SM
inline int list_slots(int vocab, int ctas, int threads) {
    auto of = [&](int warps) {
        const float most = kListShare * (static_cast<float>(vocab) / warps + 256.0f);
        return static_cast<int>(most + 5.0f * sqrtf(most)) + 1;
    };
    const int warps = threads / 32;
    return std::max(of(ctas * warps), std::min(of(warps), static_cast<int>(kTwoListsBytes / sizeof(float)) / warps));
}

// The logit from which on candidates are listed; +inf where the sample says that a list would not do.  *ref: the sample's
// largest.  The same in all CTAs of a row.
template <int T, bool VEC, int LOADS>
__device__ float candidate_floor(const Slice<VEC, LOADS>& s, float top_p, float c2, SelShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, groups = s.row.groups();
    const int g = groups > T ? static_cast<int>(static_cast<long long>(groups - 4) * (tid / 4) / (T / 4 - 1)) + tid % 4 : tid;
    const float4 v = g < groups ? s.row.raw(g, -INFINITY) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    for (int i = tid; i < kSampleBins; i += T) sh.mass_lo[i] = 0;
    const float most = block_max<T>(fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)), sh.warp_hi);  // (the bins are clear)
    if (!(fabsf(most) < INFINITY)) return INFINITY;  // (uniform)
    const float scale = c2 * (kSampleBins / kSampleRange);
    auto count = [&](float x) {
        const float b = (most - x) * scale;
        if (b < static_cast<float>(kSampleBins)) atomicAdd(&sh.mass_lo[max(static_cast<int>(b), 0)], 1u);  // (not for a NaN)
    };
    count(v.x);
    count(v.y);
    count(v.z);
    count(v.w);
    __syncthreads();
    if (warp == 0) {
        constexpr int kEach = kSampleBins / 32;
        float n[kEach], m[kEach], all_n = 0.0f, all_m = 0.0f;
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const int bin = lane * kEach + i;
            n[i] = static_cast<float>(sh.mass_lo[bin]);
            m[i] = n[i] * fast_exp2((static_cast<float>(bin) + 0.5f) * (-kSampleRange / kSampleBins));
            all_n += n[i];
            all_m += m[i];
        }
        float upto_n = warp_inclusive_scan(all_n, lane), upto_m = warp_inclusive_scan(all_m, lane);
        const float total = __shfl_sync(kFullMask, upto_m, 31);
        const float enough = (1.0f - 0.5f * (1.0f - top_p)) * total, least = (1.0f - 0.7f * (1.0f - top_p)) * total;
        upto_n -= all_n;
        upto_m -= all_m;
        int bin = -1;
        bool good = false;
#pragma unroll
        for (int i = 0; i < kEach; ++i) {  // the first bin down to which there is mass enough, or as many logits as can be listed
            upto_n += n[i];
            upto_m += m[i];
            if (bin < 0 && ((upto_m >= enough && upto_n >= kListLeast * 4 * T) || upto_n > kListShare * 4 * T)) {
                bin = lane * kEach + i;
                good = upto_m >= least && upto_n <= 1.2f * kListShare * 4 * T;
            }
        }
        const unsigned who = __ballot_sync(kFullMask, bin >= 0);
        if (who == 0) {  // fewer logits within the bins than are listed at least
            if (lane == 0) sh.floor = most - kSampleRange / c2;
        } else if (lane == __ffs(who) - 1) {
            sh.floor = good ? most - static_cast<float>(bin + 1) / scale : INFINITY;
        }
    }
    __syncthreads();
    return sh.floor;
}

// Lists the candidates of this warp's part of the slice, as the inverse CDF cuts it, two steps of two loads ahead (200 x 100000:
// 47 us a call; one step of four at a time 50, of eight 53; four ahead of four 51, and eight ahead of eight spill: 70; all with the
// mass of the rest in the same pass).
constexpr int kListLoads = 2;
template <int T, bool VEC, int LOADS>
__device__ Listed<VEC, LOADS> list_candidates(const Slice<VEC, LOADS>& s, int each, float from, int slots, float* lists) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned before_me = (1u << lane) - 1;
    const int seg = (each + T / 32 - 1) / (T / 32);
    const int b0 = min(s.g1, s.g0 + warp * seg), b1 = min(s.g1, b0 + seg);
    float* list = lists + warp * slots;
    float most = -INFINITY;
    int n = 0;
    const int last = slots - 1;  // (what does not fit goes to the last slot)
    float4 v[kListLoads];
    auto fetch = [&](int base) {
#pragma unroll
        for (int i = 0; i < kListLoads; ++i) {
            const int g = base + 32 * i + lane;
            v[i] = g < b1 ? s.row.raw(g, -INFINITY) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
    };
    if (b0 < b1) fetch(b0);
    for (int base = b0; base < b1; base += 32 * kListLoads) {
        float4 now[kListLoads];
#pragma unroll
        for (int i = 0; i < kListLoads; ++i) now[i] = v[i];
        if (base + 32 * kListLoads < b1) fetch(base + 32 * kListLoads);  // (on its way while these are looked at)
#pragma unroll
        for (int i = 0; i < kListLoads; ++i) {
            const float x[4] = {now[i].x, now[i].y, now[i].z, now[i].w};
            int at = 0, own = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                at += __popc(__ballot_sync(kFullMask, x[j] >= from) & before_me);
                most = max_or_nan(most, x[j]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool in = x[j] >= from;
                if (in) list[min(n + at + own, last)] = x[j];
                own += in ? 1 : 0;
            }
            n += __shfl_sync(kFullMask, at + own, 31);
        }
    }
    __syncwarp();
    return Listed<VEC, LOADS>{s, list, n, lane, 32, from, most == most ? most : INFINITY, n <= slots};
}

// Top-k for k up to 128, without bins: every warp gives its largest lane maxima, 3 k of them in all; the k-th largest of
// these is a value that at least k logits reach, so the k-th largest logit of the row is among those that reach it - a
// few more than k as a rule.  One pass for the maxima; only the threads whose maximum reaches the pivot have such
// logits, and what they read is read again, by all warps, and listed.
// Returns how many are listed, or -1, having decided nothing, when fewer than k lanes hold a finite logit, when there is a
// +inf, or when more than kSelCap logits reach the pivot (heavy ties): the binned selection then does the row.
constexpr int kMostTops = 512;

// One CTA to a row: a list has few passes, which a cluster does not pay for (cut_shape).
template <int T, bool VEC, int LOADS>
__device__ int top_k_list(const Slice<VEC, LOADS>& s, unsigned k, SelShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // (measured on 960 rows of 32000: k = 40 66 us per call against 82 binned, k = 128 71, k = 200 92: the pivot sinks
    // with k and lets ever more logits through)
    if (k > 128) return -1;
    float* tops = reinterpret_cast<float*>(sh.cand_mass);
    constexpr int kWarps = T / 32;
    const int per_warp = min(min(32, kMostTops / kWarps), (3 * static_cast<int>(k) + kWarps - 1) / kWarps);
    const int n_tops = per_warp * kWarps;
    float mine = -INFINITY;
    for_each_logit<T>(s, [&](float v) { mine = fmaxf(mine, v); });
    {
        // (keys: the floats' order as unsigned integers, for the warp-wide integer maximum; 0 marks a lane that is out)
        const unsigned u = __float_as_uint(mine);
        unsigned key = u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u), top = 0;
        float given = -INFINITY;
        for (int i = 0; i < per_warp; ++i) {
            top = __reduce_max_sync(0xffffffffu, key);
            const unsigned who = __ballot_sync(0xffffffffu, key == top);
            if (lane == __ffs(who) - 1) key = 0;
            if (lane == i && top != 0) given = __uint_as_float(top ^ ((top >> 31) ? 0x80000000u : 0xffffffffu));
        }
        if (lane < per_warp) tops[warp * per_warp + lane] = given;
    }
    if (tid == 0) { sh.n_cand = 0; sh.n_hit = 0; }
    __syncthreads();
    // the k-th largest of the maxima: the largest one that at least k of them reach; `per` threads count for each
    int per = 1;
    while (per * 2 * n_tops <= T && per < 32) per *= 2;
    float pivot = -INFINITY, most = -INFINITY;
    for (int base = 0; base < n_tops; base += T / per) {
        const int i = base + tid / per;
        const float top = i < n_tops ? tops[i] : INFINITY;
        unsigned reach = 0;
#pragma unroll 8
        for (int j = tid % per; j < n_tops; j += per) reach += tops[j] >= top;
        for (int o = per / 2; o > 0; o >>= 1) reach += __shfl_xor_sync(0xffffffffu, reach, o);
        if (i < n_tops) {
            most = fmaxf(most, top);
            if (reach >= k) pivot = fmaxf(pivot, top);
        }
    }
    pivot = warp_max(pivot);
    most = warp_max(most);
    if (lane == 0) { sh.warp_hi[warp] = pivot; sh.warp_top[warp] = most; }
    __syncthreads();
    pivot = most = -INFINITY;
#pragma unroll
    for (int w = 0; w < (T / 32); ++w) {
        pivot = fmaxf(pivot, sh.warp_hi[w]);
        most = fmaxf(most, sh.warp_top[w]);
    }
    if (!(pivot > -INFINITY) || most == INFINITY) return -1;
    if (mine >= pivot) sh.cnt[atomicAdd(&sh.n_hit, 1u)] = tid;
    __syncthreads();
    const int hits = static_cast<int>(sh.n_hit);
    for (int h = warp; h < hits; h += (T / 32))  // a warp goes over what one of those threads has read
        for (int g = s.g0 + sh.cnt[h] + lane * T; g < s.g1; g += 32 * T)
            list_group(s.row.raw(g, -INFINITY), 4 * g - s.row.shift, pivot, sh);
    return gather_list<T>(Team<true>(), false, sh);
}

// The k-th largest of the listed logits.  In the first CTA.
template <int T>
__device__ float top_k_of_list(unsigned k, SelShared& sh) {
    const int tid = threadIdx.x, count = static_cast<int>(sh.n_list);
    float best = -INFINITY;
    for (int i = tid; i < count; i += T) {
        const float c = sh.cand[i];
        unsigned at_least = 0;
#pragma unroll 8
        for (int j = 0; j < count; ++j) at_least += sh.cand[j] >= c;
        if (at_least >= k) best = fmaxf(best, c);
    }
    best = warp_max(best);
    if ((tid & 31) == 0) sh.warp_lo[tid >> 5] = best;
    __syncthreads();
    best = -INFINITY;
#pragma unroll
    for (int w = 0; w < (T / 32); ++w) best = fmaxf(best, sh.warp_lo[w]);
    return best;
}

// Lists the logits that reach kf > -inf, after a top-k that found it by bins.  Returns how many, or -1 if they are more than
// kSelCap (a large tie at kf) or one of them is +inf.
template <int T, bool VEC, int LOADS, bool SOLO>
__device__ int list_row(const Slice<VEC, LOADS>& s, const Team<SOLO>& team, float kf, SelShared& sh) {
    team.sync();  // (the shared arrays may still be read by a previous call)
    if (sh.row_top == INFINITY) return -1;
    if (threadIdx.x == 0) sh.n_cand = 0;
    __syncthreads();
    for_each_group<T>(s, [&](const float4& v, int g) { list_group(v, 4 * g - s.row.shift, kf, sh); });
    return gather_list<T>(team, false, sh);
}

template <int T>
__device__ __forceinline__ unsigned long long block_sum(unsigned long long v, unsigned long long* per_warp) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) per_warp[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0;
#pragma unroll
    for (int w = 0; w < (T / 32); ++w) v += per_warp[w];
    return v;
}

// What is left of a listed row: the nucleus of the logits that reach *floor (if `nucleus`, which raises *floor), ranked
// against each other, the largest logit and the sum of the kept weights.  Weights are summed in units of 2^-40 of the
// largest, so that the order in which the list was made does not matter.  In the first CTA.
template <int T>
__device__ void finish_list(bool nucleus, float top_p, float c2, SelShared& sh, float* floor, float* row_max, float* sum) {
    const int tid = threadIdx.x, count = static_cast<int>(sh.n_list);
    const float kf = *floor;
    float m = -INFINITY;
    for (int i = tid; i < count; i += T) m = fmaxf(m, sh.cand[i]);
    m = block_max<T>(m, sh.warp_hi);
    unsigned long long mine_sum = 0;
    for (int i = tid; i < count; i += T) {
        const unsigned long long w = sh.cand[i] >= kf ? __float2ull_rz(fast_exp2((sh.cand[i] - m) * c2) * 1099511627776.0f) : 0ull;  // 2^40
        sh.cand_mass[i] = w;
        mine_sum += w;
    }
    unsigned long long kept = block_sum<T>(mine_sum, sh.warp_mass);  // (and cand_mass is complete)
    if (nucleus) {
        const unsigned long long goal = static_cast<unsigned long long>(ceil(static_cast<double>(top_p) * static_cast<double>(kept)));
        float best = -INFINITY;
        for (int i = tid; i < count; i += T) {
            const float mine = sh.cand[i];
            if (!(mine >= kf)) continue;
            unsigned long long above = 0;
#pragma unroll 8
            for (int j = 0; j < count; ++j) above += sh.cand[j] >= mine ? sh.cand_mass[j] : 0ull;
            if (above >= goal) best = fmaxf(best, mine);
        }
        best = block_max<T>(best, sh.warp_lo);
        *floor = best > -INFINITY ? best : kf;
        mine_sum = 0;
        for (int i = tid; i < count; i += T)
            if (sh.cand[i] >= *floor) mine_sum += sh.cand_mass[i];
        kept = block_sum<T>(mine_sum, sh.warp_mass);  // (everyone has read the first sums: a barrier ago)
    }
    *row_max = m;
    *sum = static_cast<float>(static_cast<double>(kept) * (1.0 / 1099511627776.0));
}

// The draw from a listed row: the kept logits in the order of their places, walked by one warp.  In the first CTA.
template <int T>
__device__ int draw_from_list(float floor, float row_max, float c2, float u, SelShared& sh) {
    const int tid = threadIdx.x, count = static_cast<int>(sh.n_list);
    unsigned* index = list_index(sh);
    float* weight = reinterpret_cast<float*>(sh.cand_mass);  // in order
    unsigned* place = sh.mass_lo;
    __syncthreads();  // (cand_mass has been read by everyone)
    if (tid == 0) sh.n_hit = 0;
    for (int i = tid; i < count; i += T)
        if (!(sh.cand[i] >= floor)) index[i] = 0xffffffffu;  // (behind every place of the row)
    __syncthreads();
    for (int i = tid; i < count; i += T) {
        if (!(sh.cand[i] >= floor)) continue;
        unsigned rank = 0;
#pragma unroll 8
        for (int j = 0; j < count; ++j) rank += index[j] < index[i];
        weight[rank] = fast_exp2((sh.cand[i] - row_max) * c2);
        place[rank] = index[i];
        atomicMax(&sh.n_hit, rank + 1);
    }
    __syncthreads();
    int token = 0;
    if (tid < 32) {
        const int kept = static_cast<int>(sh.n_hit);
        float total = 0.0f;
        for (int base = 0; base < kept; base += 32) total += warp_sum(base + tid < kept ? weight[base + tid] : 0.0f);
        const float target = u * total;
        float run = 0.0f;
        int found = -1, last = 0;
        for (int base = 0; base < kept && found < 0; base += 32) {
            const float w = base + tid < kept ? weight[base + tid] : 0.0f;
            const float incl = warp_inclusive_scan(w, tid);
            const unsigned over = __ballot_sync(kFullMask, base + tid < kept && run + incl > target), some = __ballot_sync(kFullMask, w > 0.0f);
            if (some) last = base + 31 - __clz(some);
            if (over) found = base + __ffs(over) - 1;
            run += __shfl_sync(kFullMask, incl, 31);
        }
        token = static_cast<int>(place[found >= 0 ? found : last]);
    }
    return token;  // (valid in the first warp)
}

// (max, sum of exp2((l - max) * c2)) of the kept logits, online, in a fixed order.  Valid in thread 0 of the first CTA.
template <int T, bool VEC, int LOADS, bool SOLO>
__device__ void row_statistics(const Slice<VEC, LOADS>& s, const Team<SOLO>& team, float floor, float c2, SelShared& sh, float* row_max, float* sum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    Row<VEC, true> r;
    r.base = s.row.base;
    r.vocab = s.row.vocab;
    r.floor = floor;
    r.shift = s.row.shift;
    r.own = s.row.own;
    float m = -FLT_MAX, t = 0.0f;  // (finite, so that m - new maximum never becomes inf - inf)
    for (int base = s.g0 + tid; base < s.g1; base += LOADS * T) {
        float4 v[LOADS];
        float bm = m;
#pragma unroll
        for (int i = 0; i < LOADS; ++i) {
            const int g = base + i * T;
            v[i] = g < s.g1 ? r.load(g, -INFINITY) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
#pragma unroll
        for (int i = 0; i < LOADS; ++i) bm = fmaxf(bm, fmaxf(fmaxf(v[i].x, v[i].y), fmaxf(v[i].z, v[i].w)));
        t *= fast_exp2((m - bm) * c2);
        m = bm;
        const float mc = fminf(-m * c2, FLT_MAX);  // (-inf * c2 + it stays -inf)
#pragma unroll
        for (int i = 0; i < LOADS; ++i)
            t += (fast_exp2(fmaf(v[i].x, c2, mc)) + fast_exp2(fmaf(v[i].y, c2, mc))) +
                 (fast_exp2(fmaf(v[i].z, c2, mc)) + fast_exp2(fmaf(v[i].w, c2, mc)));
    }
    const float wm = warp_max(m);
    t = warp_sum(t * fast_exp2((m - wm) * c2));
    team.sync();  // (the shared arrays may still be read)
    if (lane == 0) { sh.warp_hi[warp] = wm; sh.warp_lo[warp] = t; }
    __syncthreads();
    auto merge = [&](const float* max, const float* part, int count) {
        float bm = max[0], all = 0.0f;
        for (int w = 1; w < count; ++w) bm = fmaxf(bm, max[w]);
        for (int w = 0; w < count; ++w) all += part[w] * fast_exp2((max[w] - bm) * c2);
        *row_max = bm;
        *sum = all;
    };
    if (tid == 0) {
        merge(sh.warp_hi, sh.warp_lo, (T / 32));
        SelShared& first = team.of(sh, 0);
        first.cta_max[team.rank] = *row_max;
        first.cta_sum[team.rank] = *sum;
    }
    if (!SOLO) {
        team.sync();
        if (tid == 0 && team.rank == 0) merge(sh.cta_max, sh.cta_sum, team.size);
    }
}

// What else to find out about a row while it is at hand.
struct CutWork {
    // verification: its statistics, at the drafted token too
    const int32_t* draft_tokens;
    ChunkStat* stats;
    // sampling: a token
    const float* uniforms;
    int uniform_stride;
    int32_t* tokens;
    int token_stride;
    int* nonfinite;
};
// (ordering a list by place takes a comparison per pair; beyond this it is cheaper to go over the row, as without a list:
// one row of 32000, k = 400, p = 0.95 39 us with the list, 48 without)
constexpr int kDrawList = 512;
constexpr int kFloorsOnly = 0, kWithStats = 1, kWithDraw = 2;

// floors[s * (a_rows + b_rows) + r] for sequence s's a_rows rows of `a`, then its
// b_rows rows of `b`: top-k first (0 < top_k < vocab), then the nucleus (0 < top_p < 1)
// of what top-k left.  The statistics of the verification and the draw of the sampling follow in the same CTAs: after a
// top-k they cost nothing, the list is there (24 x 9 rows of 50003, k = 40, p = 0.9: 66 us with kernels of their own, 40 so
// with 1024 threads to a row, 32 with 512; 200 rows of 100000, k = 40, with the draw: 73, 28 and 22; one of 32000: 16, 9 and
// 8), and after a nucleus one pass less and no second kernel (200 rows of 100000: 99, 91 and 70).
// LIST: the nucleus alone, from a list of `slots` candidates per warp.
template <int T, int LOADS, bool VEC, bool SOLO, int WORK, bool LIST>
__global__ void __launch_bounds__(T, LIST ? 1024 / T : T == 256 ? 5 : LOADS == 8 ? 2 : 3)
cut_floor_kernel(const float* a, size_t a_stride, int a_rows, const float* b, size_t b_stride, int b_rows, int vocab, int top_k,
                 float top_p, float c2, float* floors, CutWork work, int slots) {
    extern __shared__ float lists[];
    __shared__ __align__(16) unsigned char shared[LIST ? offsetof(SelShared, cnt) : sizeof(SelShared)];
    SelShared& sh = *reinterpret_cast<SelShared*>(shared);
    pdl_wait();
    pdl_trigger();  // after the wait: the finishing kernel fetches inputs at once
    a = after_wait(a);
    b = after_wait(b);
    const Team<SOLO> team;
    const int at = blockIdx.x / team.size;
    const int per_seq = a_rows + b_rows;
    const int seq = at / per_seq, row = at % per_seq;
    const float* src = row < a_rows ? a + (static_cast<size_t>(seq) * a_rows + row) * a_stride
                                    : b + (static_cast<size_t>(seq) * b_rows + (row - a_rows)) * b_stride;
    Slice<VEC, LOADS> s;
    s.row = make_row<VEC>(src, vocab);
    const int groups = s.row.groups(), each = (groups + team.size - 1) / team.size;
    s.g0 = min(groups, team.rank * each);
    s.g1 = min(groups, s.g0 + each);
    const bool first = team.rank == 0;
    float floor = -INFINITY, row_max = 0.0f, sum = 0.0f;
    int listed = -1;  // logits listed (the same in all CTAs; floor, row_max and sum of a listed row are the first one's)
    const bool nucleus = top_p > 0.0f && top_p < 1.0f;
    Listed<VEC, LOADS> found{s};
    found.first = threadIdx.x % 32;
    found.step = 32;
    bool candidates = false;  // the nucleus came from them
    if constexpr (LIST) {
        const float from = candidate_floor<T>(s, top_p, c2, sh);
        if (from < INFINITY) {
            Listed<VEC, LOADS> listed = list_candidates<T>(s, each, from, slots, lists);
            found.at = listed.at;
            found.n = listed.n;
            if (threadIdx.x % 32 == 0) sh.found[threadIdx.x / 32] = listed.n;
            // A warp has more than its share of slots: listed once more, one warp's candidates behind another's, if the CTA has room for
            // all of them, and the selection shares them out evenly.  (A loop, so that the selection is there once: with a second
            // copy of it for this case 200 x 100000 were 52 us, as a function of its own 58, and 46 so.)
            float f;
#pragma unroll 1
            for (bool again = false;; again = true) {
                f = select_floor<T, true>(listed, team, -INFINITY, 0u, top_p, c2, sh);
                if (again || listed.all) break;  // (the same for the team)
                team.sync();  // (what the warps found has been read)
                int total = 0, before = 0;
#pragma unroll
                for (int w = 0; w < T / 32; ++w) {
                    if (w == static_cast<int>(threadIdx.x / 32)) before = total;
                    total += sh.found[w];
                }
                const bool room = total <= slots * (T / 32);
                if (room) list_candidates<T>(s, each, from, found.n, lists + before - static_cast<int>(threadIdx.x / 32) * found.n);
                found.at = lists + before;
                listed.all = room;
                listed.at = lists;
                listed.first = threadIdx.x;
                listed.step = T;
                listed.n = total;
            }
            candidates = f == f;
            if (candidates) floor = f;
        }
    } else if (top_k > 0 && top_k < vocab) {
        if constexpr (SOLO) listed = top_k_list<T>(s, static_cast<unsigned>(top_k), sh);
        if (listed >= 0) {
            if (first) floor = top_k_of_list<T>(static_cast<unsigned>(top_k), sh);
        } else {
            floor = select_floor<T, false>(s, team, -INFINITY, static_cast<unsigned>(top_k), 0.0f, 0.0f, sh);
            if (nucleus && floor > -INFINITY && top_k <= kSelCap) listed = list_row<T>(s, team, floor, sh);
        }
    }
    if (listed >= 0) {
        if (first) finish_list<T>(nucleus, top_p, c2, sh, &floor, &row_max, &sum);
    } else if (nucleus && !candidates) {
        floor = select_floor<T, true>(s, team, floor, 0u, top_p, c2, sh);
    }
    if (threadIdx.x == 0 && first && floors) floors[at] = floor;
    float kept = 0.0f;  // the candidates that are kept, of this warp
    if (LIST && WORK != kFloorsOnly && candidates) {
        row_max = sh.row_top;
        for_each_logit<T>(found, [&](float v) { kept += v >= floor ? fast_exp2((v - row_max) * c2) : 0.0f; });
        kept = warp_sum(kept);
    }
    if (WORK == kWithStats) {
        if (LIST && candidates) {
            if (threadIdx.x % 32 == 0) sh.kept[threadIdx.x / 32] = kept;
            team.sync();
            if (threadIdx.x == 0 && first)
                for (int i = 0; i < team.size * (T / 32); ++i) sum += team.of(sh, i / (T / 32)).kept[i % (T / 32)];
        } else if (listed < 0) {
            row_statistics<T>(s, team, floor, c2, sh, &row_max, &sum);
        }
        if (threadIdx.x == 0 && first) {
            float at_x = 0.0f;  // (none for p_{gamma+1})
            if (row != a_rows - 1) {
                const int x = work.draft_tokens[static_cast<size_t>(seq) * b_rows + (row < a_rows ? row : row - a_rows)];
                if (x >= 0 && x < vocab) at_x = __ldg(src + x) >= floor ? __ldg(src + x) : -INFINITY;
            }
            *reinterpret_cast<float4*>(work.stats + at) = make_float4(row_max, sum, at_x, 0.0f);
        }
    }
    if (WORK == kWithDraw) {
        __shared__ CdfScratch<T / 32> cdf;
        const float u = work.uniforms[static_cast<size_t>(at) * work.uniform_stride];
        int token = -1;
        if (listed >= 0 && listed <= kDrawList) {
            if (first) token = draw_from_list<T>(floor, row_max, c2, u, sh);
        } else {
            if (listed >= 0) {  // the others need what the first one found
                if (first && threadIdx.x < team.size) {
                    team.of(sh, threadIdx.x).floor = floor;
                    team.of(sh, threadIdx.x).row_top = row_max;
                }
                team.sync();
                floor = sh.floor;
            }
            __syncthreads();
            if (threadIdx.x == 0 && first && work.nonfinite && sh.row_top == INFINITY) atomicExch(work.nonfinite, 1);
            PlainWeights<VEC, true> pw;
            pw.p = make_row<VEC, true>(src, vocab, floor);
            pw.max_p = fmaxf(sh.row_top, -FLT_MAX);
            pw.c2 = c2;
            float total;
            const float* mine = LIST && candidates ? &kept : nullptr;
            token = SOLO ? block_inverse_cdf<T / 32>(pw, vocab, u, cdf, &total, mine) : cluster_inverse_cdf<T / 32>(pw, vocab, u, cdf, &total, mine);
        }
        // (of a cluster one CTA has drawn, and the others have -1)
        if (threadIdx.x == 0 && (SOLO || token >= 0)) work.tokens[static_cast<size_t>(at) * work.token_stride] = max(0, min(token, vocab - 1));
    }
    if (!SOLO) team.sync();  // nobody leaves while another may still look here
}

__global__ void uniforms_kernel(uint64_t seed, const int32_t* __restrict__ positions,
                                const int32_t* __restrict__ sequences, uint32_t purpose, int count,
                                float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count)
        out[i] = method_uniform(seed, static_cast<uint32_t>(positions[i]), static_cast<uint32_t>(sequences[i]), purpose);
}

// Chunks per row: one unless the batch is too small to fill the GPU with
// whole-row CTAs; never more than the workspace was sized for.
int max_chunks(int vocab) {
    const int groups = (vocab + 3) / 4;
    return std::max(1, groups / kMinChunkGroups);
}

// CTAs per cluster in the finishing kernel: each CTA should still have a few
// thousand elements of row n+1 to sum.
int finish_cluster_size(int vocab) {
    int c = 1;
    while (c < kMaxCluster && vocab / (2 * c) >= 2048) c *= 2;
    return c;
}

// One kernel for statistics and decision, where a call is bound by its launches and not by the GPU: a lone decision of
// 4 x 8192 logits takes the host one launch less, 1.8 us, at 7.9 us of the GPU instead of 6.5 (a cluster of eight SMs reads all
// rows); call after call 7.7 us, with the checks in Python and without programmatic launch 10.5.  The line is where the GPU's time meets the host's: 7 rows of 32000
// 9.6, 11 rows of 32000 11.7, 17 of 32000 13.7, 7 of 50003 11.9 (two kernels: 12.3 of the host); at T = 0, 4 x 128000
// 8.7, 9 x 128000 14.1.  The generation loop replays a graph, to which only the GPU's time matters: never there.
constexpr int kMostAlone = 8;  // CTAs to a sequence
bool one_kernel(int batch, int rows, int vocab, bool greedy) {
    return batch <= 8 && static_cast<long long>((rows + kMostAlone - 1) / kMostAlone) * vocab <= (greedy ? 128 * 1024 : 32 * 1024);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int chunks_for(int vocab, int rows_total) {
    const int want = (kTargetCtas + rows_total - 1) / std::max(1, rows_total);
    const int most = std::max(1, std::min(want, max_chunks(vocab)));
    // the fewest chunks of as many steps of the streaming loop: with 12 of 1042 groups each, a row of 50003 took a second
    // step for 18 groups, with 7 that step is nearly full (30 x 11 such rows, with the draw 26.6 ->
    // 23.4 us; rows of 100000 40.0 -> 33.3, of 128000 43.8 -> 38.5)
    const int groups = (vocab + 3) / 4, step = kUnroll * kStatThreads;
    const int steps = ((groups + most - 1) / most + step - 1) / step;
    return (groups + steps * step - 1) / (steps * step);
}

size_t stats_bytes(int batch, int gamma, int vocab) {
    const size_t rows = 2 * static_cast<size_t>(gamma) + 1;
    return (static_cast<size_t>(batch) * rows * max_chunks(vocab) * sizeof(ChunkStat) + 255) & ~static_cast<size_t>(255);
}

}  // namespace

// Shared with the generation loop: same launches, no argument checks.
// Layout: chunk statistics, then one top-k floor per row.
size_t verify_sample_workspace_bytes(int batch, int gamma, int vocab) {
    const size_t rows = 2 * static_cast<size_t>(gamma) + 1;
    return stats_bytes(batch, gamma, vocab) + static_cast<size_t>(batch) * rows * sizeof(float) + 256;
}

constexpr size_t kMostListBytes = 160 * 1024;  // of candidates; a longer row is binned as it lies
size_t list_bytes(int vocab, int ctas, int threads) { return static_cast<size_t>(list_slots(vocab, ctas, threads)) * (threads / 32) * sizeof(float); }

// How the rows of a cut are shared out.
struct CutShape {
    int threads, loads, ctas;  // of a CTA; in flight per thread; CTAs per row
};
// Both ways measured (us per call, with what follows the cut):
// - 512 threads with eight loads each, two rows to an SM, while that is one wave (200 x 100000, p = 0.9: 70, with 1024 threads
//   90, with 256 103; 216 x 32000: 31, with four loads and three rows to an SM 37); with more rows four loads (330 x
//   50003: 98, 74), and with many short ones 256 threads (960 x 32000 88, 512 threads 98; 960 x 8192 32, 50; but 960 x
//   50003 157, 223).  A short row that is binned is all barriers: 256 threads (64 x 8192: 10, 12; 64 x 16000: 15, 14).
// - a cluster pays where few rows are long and binned (4 x 512 threads against 512: 16 x 50003 26, 37; 16 x 128000 29, 53;
//   64 x 100000 32, 50; 2 x 512: 128 x 100000 51, 66), not on more rows (200 x 100000 with two: 87, 70), shorter ones (16 x
//   32000: 19, 18) or a list, whose passes are few (16 x 100000, k = 50: 13, 13).
// - of the nucleus from lists, 200 x 100000 are one row to a CTA and two CTAs to an SM, with four loads (eight were 64 us to 57
//   when loads were not yet requested two steps ahead); with lists so long that one CTA fills the SM, a pair (256 x 128000: 82, 512
//   threads alone 90, likewise).
CutShape cut_shape(int rows, int vocab, int top_k) {
    const bool listed = top_k <= 0 || top_k >= vocab;
    const bool binned = top_k <= 0 || top_k > 128 || top_k >= vocab, long_row = vocab >= 48 * 1024;
    if (rows > 4 * 148 && !long_row) return CutShape{256, 4, 1};
    if (binned && vocab < 12 * 1024) return CutShape{256, 4, 1};
    if (rows > 2 * 148) return CutShape{512, 4, 1};
    if (listed && long_row && rows > 148)
        return list_bytes(vocab, 1, 512) <= kTwoListsBytes ? CutShape{512, 4, 1} : CutShape{512, 8, 2};
    return CutShape{512, 8, binned && long_row ? (rows <= 74 ? 4 : rows <= 148 ? 2 : 1) : 1};
}

bool cut_is_on(int vocab, float temperature, int top_k, float top_p) {
    return temperature > 0.0f && ((top_k > 0 && top_k < vocab) || (top_p > 0.0f && top_p < 1.0f));
}

// Top-k, then the nucleus of what is left (Section 2.2): one floor per row, one kernel.
// floors[s * (a_rows + b_rows) + r] belongs to sequence s's row r (its a_rows rows of `a`,
// then its b_rows rows of `b`).
template <int WORK>
int launch_cut(const float* a, size_t a_stride, int a_rows, const float* b, size_t b_stride, int b_rows, int seqs, int vocab,
               int top_k, float top_p, float inv_t, float* floors, const CutWork& work, cudaStream_t stream) {
    const int total = seqs * (a_rows + b_rows);
    if (total == 0) return SPEC_OK;
    const bool vec = vocab % 4 == 0 && a_stride % 4 == 0 && aligned16(a) && (b_rows == 0 || (b_stride % 4 == 0 && aligned16(b)));
    const float c2 = inv_t * kLog2e;
    const CutShape shape = cut_shape(total, vocab, top_k);
    const int ctas = shape.ctas;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(total * ctas);
    cfg.blockDim = dim3(shape.threads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (pdl_enabled()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (ctas > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = ctas;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    // (short rows are all barriers, of which the list has more, unless they are many: binned and listed, 16 x 8192 11 us, 11;
    // 600 x 4099 18, 20; 600 x 8192 19, 20; 1600 x 8192 40, 37; 96 x 17 x 8192, verified, 50, 45)
    const bool listed = !(top_k > 0 && top_k < vocab) && (vocab >= 12 * 1024 || (vocab >= 6 * 1024 && total > 1024)) &&
                        list_bytes(vocab, ctas, shape.threads) <= kMostListBytes;
    int slots = 0;
    if (listed) {
        slots = list_slots(vocab, ctas, shape.threads);
        cfg.dynamicSmemBytes = list_bytes(vocab, ctas, shape.threads);
    }
    auto launch = [&](auto kernel) -> int {
        SPEC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, a, a_stride, a_rows, b, b_stride, b_rows, vocab, top_k, top_p, c2, floors, work, slots));
        return SPEC_OK;
    };
    auto launch_listed = [&](std::atomic<unsigned long long>& done, auto kernel) -> int {
        const int status = allow_shared_memory(done, kernel, static_cast<int>(kMostListBytes));
        return status != SPEC_OK ? status : launch(kernel);
    };
#define SPEC_LAUNCH_CUT(T, L, S)                                                                                                   \
    do {                                                                                                                           \
        static std::atomic<unsigned long long> done[2];                                                                            \
        if (listed)                                                                                                                \
            return vec ? launch_listed(done[0], cut_floor_kernel<T, L, true, S, WORK, true>)                                       \
                       : launch_listed(done[1], cut_floor_kernel<T, L, false, S, WORK, true>);                                     \
        return vec ? launch(cut_floor_kernel<T, L, true, S, WORK, false>) : launch(cut_floor_kernel<T, L, false, S, WORK, false>); \
    } while (0)
    if (ctas > 1) SPEC_LAUNCH_CUT(512, 8, false);
    if (shape.threads == 256) SPEC_LAUNCH_CUT(256, 4, true);
    if (shape.loads == 4) SPEC_LAUNCH_CUT(512, 4, true);
    SPEC_LAUNCH_CUT(512, 8, true);
#undef SPEC_LAUNCH_CUT
}

int launch_verify_sample(const float* target_logits, const float* draft_logits, const int32_t* draft_tokens,
                         const float* uniforms, const float* final_uniforms, int batch, int gamma, int vocab,
                         float temperature, float lenience, int top_k, float top_p, int32_t* n_accepted,
                         int32_t* next_token, void* workspace, cudaStream_t stream, int* nonfinite) {
    const bool greedy = temperature == 0.0f;
    const int rows = greedy ? gamma + 1 : 2 * gamma + 1;
    const float inv_t = greedy ? 0.0f : 1.0f / temperature;
    ChunkStat* stats = static_cast<ChunkStat*>(workspace);
    const bool cut = cut_is_on(vocab, temperature, top_k, top_p);  // never with greedy
    const bool alone = !cut && !final_uniforms && one_kernel(batch, rows, vocab, greedy);
    const int chunks = cut || alone ? 1 : chunks_for(vocab, rows * batch);
    const dim3 grid(chunks, rows, batch);
    const bool vec = vocab % 4 == 0 && aligned16(target_logits) && (greedy || gamma == 0 || aligned16(draft_logits));
    const float c2 = inv_t * kLog2e;
    const float* floors = nullptr;
    int status = SPEC_OK;
#define SPEC_LAUNCH_STATS(G, V)                                                                                  \
    status = launch_pdl(verify_stats_kernel<G, V>, grid, dim3(kStatThreads), 0, stream, target_logits, draft_logits, \
                        draft_tokens, gamma, vocab, c2, stats)
    if (cut) {
        // top-k and nucleus (Section 2.2): both models' rows are cut at their own floors
        float* f = reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + stats_bytes(batch, gamma, vocab));
        CutWork work{};
        work.draft_tokens = draft_tokens;
        work.stats = stats;
        status = launch_cut<kWithStats>(target_logits, static_cast<size_t>(vocab), gamma + 1, draft_logits, static_cast<size_t>(vocab),
                                        gamma, batch, vocab, top_k, top_p, inv_t, f, work, stream);
        floors = f;
    } else if (alone) {
    } else if (greedy && vec) SPEC_LAUNCH_STATS(true, true);
    else if (greedy) SPEC_LAUNCH_STATS(true, false);
    else if (vec) SPEC_LAUNCH_STATS(false, true);
    else SPEC_LAUNCH_STATS(false, false);
#undef SPEC_LAUNCH_STATS
    if (status != SPEC_OK) return status;

    // One cluster per sequence; more CTAs per cluster for longer rows.
    const int cluster_size = alone ? std::min(kMostAlone, rows) : greedy ? 1 : finish_cluster_size(vocab);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(batch * cluster_size);
    cfg.blockDim = dim3(kFinishThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster_size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
#define SPEC_LAUNCH_FINISH(G, V, C, A)                                                                                  \
    SPEC_CUDA_TRY(cudaLaunchKernelEx(&cfg, verify_finish_kernel<G, V, C, A>, target_logits, draft_logits, draft_tokens, \
                                     uniforms, gamma, vocab, inv_t, chunks, cluster_size, stats, final_uniforms,       \
                                     lenience, floors, n_accepted, next_token, nonfinite))
    if (alone && greedy && vec) SPEC_LAUNCH_FINISH(true, true, false, true);
    else if (alone && greedy) SPEC_LAUNCH_FINISH(true, false, false, true);
    else if (alone && vec) SPEC_LAUNCH_FINISH(false, true, false, true);
    else if (alone) SPEC_LAUNCH_FINISH(false, false, false, true);
    else if (greedy && vec) SPEC_LAUNCH_FINISH(true, true, false, false);
    else if (greedy) SPEC_LAUNCH_FINISH(true, false, false, false);
    else if (vec && cut) SPEC_LAUNCH_FINISH(false, true, true, false);
    else if (vec) SPEC_LAUNCH_FINISH(false, true, false, false);
    else if (cut) SPEC_LAUNCH_FINISH(false, false, true, false);
    else SPEC_LAUNCH_FINISH(false, false, false, false);
#undef SPEC_LAUNCH_FINISH
    return SPEC_OK;
}

// Row r reads logits + r * logit_stride and uniforms[r * uniform_stride] and
// writes tokens[r * token_stride].
// With a cut (0 < top_k < vocab or 0 < top_p < 1, and T > 0) `floor_scratch` must hold `rows` floats.
int launch_sample_strided(const float* logits, size_t logit_stride, const float* uniforms, int uniform_stride,
                          int rows, int vocab, float temperature, int top_k, float top_p, float* floor_scratch,
                          int32_t* tokens, int token_stride, cudaStream_t stream, int* nonfinite) {
    const bool greedy = temperature == 0.0f;
    const float inv_t = greedy ? 0.0f : 1.0f / temperature;
    if (cut_is_on(vocab, temperature, top_k, top_p)) {
        CutWork work{};
        work.uniforms = uniforms;
        work.uniform_stride = uniform_stride;
        work.tokens = tokens;
        work.token_stride = token_stride;
        work.nonfinite = nonfinite;
        return launch_cut<kWithDraw>(logits, logit_stride, 1, nullptr, 0, 0, rows, vocab, top_k, top_p, inv_t, floor_scratch, work, stream);
    }
    const bool vec = vocab % 4 == 0 && logit_stride % 4 == 0 && aligned16(logits);
#define SPEC_LAUNCH_SAMPLE(V)                                                                                      \
    return launch_pdl(sample_kernel<V>, dim3(rows), dim3(kSampleThreads), 0, stream, logits, logit_stride, uniforms,     \
                      uniform_stride, vocab, inv_t, greedy, tokens, token_stride, nonfinite)
    if (vec) SPEC_LAUNCH_SAMPLE(true);
    SPEC_LAUNCH_SAMPLE(false);
#undef SPEC_LAUNCH_SAMPLE
}

int launch_sample(const float* logits, const float* uniforms, int rows, int vocab, float temperature, int top_k,
                  float top_p, float* floor_scratch, int32_t* tokens, cudaStream_t stream) {
    return launch_sample_strided(logits, static_cast<size_t>(vocab), uniforms, 1, rows, vocab, temperature, top_k, top_p,
                                 floor_scratch, tokens, 1, stream, nullptr);
}

}  // namespace spec

extern "C" size_t spec_verify_sample_workspace_bytes(int batch, int gamma, int vocab) {
    if (batch < 0 || gamma < 0 || vocab < 1) return 0;
    return spec::verify_sample_workspace_bytes(batch, gamma, vocab);
}

extern "C" int spec_verify_sample_truncated(const float* target_logits, const float* draft_logits,
                                            const int32_t* draft_tokens, const float* uniforms, int batch, int gamma,
                                            int vocab, float temperature, float lenience, int top_k, float top_p,
                                            int32_t* n_accepted, int32_t* next_token, void* workspace,
                                            size_t workspace_bytes, void* stream) {
    using namespace spec;
    if (top_k < 0 || !(top_p == top_p)) return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: top_k must be >= 0 and top_p a number");
    if (!(lenience > 0.0f) || !(lenience <= 1.0f)) return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: lenience must be in (0, 1]");
    if (batch < 0 || gamma < 0 || gamma > kMaxGamma || vocab < 1)
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: batch=%d gamma=%d (max %d) vocab=%d", batch, gamma, kMaxGamma, vocab);
    if (!(temperature >= 0.0f) || !isfinite(temperature))
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: temperature must be finite and >= 0");
    if (batch == 0) return SPEC_OK;
    if (batch > 65535) return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: batch %d exceeds 65535", batch);
    const bool greedy = temperature == 0.0f;
    if (!target_logits || !n_accepted || !next_token || !workspace || (gamma > 0 && !draft_tokens) ||
        (!greedy && (!uniforms || (gamma > 0 && !draft_logits))))
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: null pointer");
    if (workspace_bytes < spec_verify_sample_workspace_bytes(batch, gamma, vocab) ||
        (reinterpret_cast<uintptr_t>(workspace) & 255u))
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample: workspace too small (%zu bytes) or not 256-byte aligned", workspace_bytes);
    return launch_verify_sample(target_logits, draft_logits, draft_tokens, uniforms, nullptr, batch, gamma, vocab,
                                temperature, lenience, top_k, top_p, n_accepted, next_token, workspace,
                                static_cast<cudaStream_t>(stream));
}

extern "C" int spec_verify_sample_lenient(const float* target_logits, const float* draft_logits,
                                          const int32_t* draft_tokens, const float* uniforms, int batch, int gamma,
                                          int vocab, float temperature, float lenience, int32_t* n_accepted,
                                          int32_t* next_token, void* workspace, size_t workspace_bytes, void* stream) {
    return spec_verify_sample_truncated(target_logits, draft_logits, draft_tokens, uniforms, batch, gamma, vocab,
                                        temperature, lenience, 0, 1.0f, n_accepted, next_token, workspace,
                                        workspace_bytes, stream);
}

extern "C" int spec_verify_sample(const float* target_logits, const float* draft_logits, const int32_t* draft_tokens,
                                  const float* uniforms, int batch, int gamma, int vocab, float temperature,
                                  int32_t* n_accepted, int32_t* next_token, void* workspace, size_t workspace_bytes,
                                  void* stream) {
    return spec_verify_sample_lenient(target_logits, draft_logits, draft_tokens, uniforms, batch, gamma, vocab, temperature,
                                      1.0f, n_accepted, next_token, workspace, workspace_bytes, stream);
}

// ---- spec_verify_sample without any allocation ---------------------------------
// The chunk statistics that the two kernels hand to each other normally live in a
// caller-provided workspace.  This variant keeps them in a fixed array inside the
// library image instead, so the call needs no device memory beyond its inputs and
// outputs.  Every GPU that loads the library holds the array until the process
// exits.
namespace {

constexpr size_t kStaticStatsBytes = 1u << 20;  // 65536 chunk statistics
static __device__ __align__(256) unsigned char g_static_stats[kStaticStatsBytes];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};  // device address of g_static_stats, per device

// The array's name is only a host-side handle; kernels need its device address,
// which differs per device and is looked up once per device.
int static_stats_address(void** out) {
    int device = -1;
    SPEC_CUDA_TRY(cudaGetDevice(&device));
    if (device < 0 || device >= kMaxDevices) return spec::fail(SPEC_ERR_BAD_CONFIG, "device ordinal %d not supported", device);
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[device]) {
        void* p = nullptr;
        SPEC_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_stats));
        g_static_ptr[device] = p;
    }
    *out = g_static_ptr[device];
    return SPEC_OK;
}

}  // namespace

extern "C" size_t spec_verify_sample_static_capacity(void) { return kStaticStatsBytes; }

extern "C" int spec_verify_sample_static(const float* target_logits, const float* draft_logits,
                                         const int32_t* draft_tokens, const float* uniforms, int batch, int gamma,
                                         int vocab, float temperature, int32_t* n_accepted, int32_t* next_token,
                                         void* stream) {
    using namespace spec;
    if (batch < 0 || gamma < 0 || gamma > kMaxGamma || vocab < 1)
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample_static: batch=%d gamma=%d (max %d) vocab=%d", batch, gamma, kMaxGamma, vocab);
    if (!(temperature >= 0.0f) || !isfinite(temperature))
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample_static: temperature must be finite and >= 0");
    if (batch == 0) return SPEC_OK;
    if (batch > 65535) return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample_static: batch %d exceeds 65535", batch);
    const bool greedy = temperature == 0.0f;
    if (!target_logits || !n_accepted || !next_token || (gamma > 0 && !draft_tokens) ||
        (!greedy && (!uniforms || (gamma > 0 && !draft_logits))))
        return fail(SPEC_ERR_BAD_ARG, "spec_verify_sample_static: null pointer");
    const size_t need = verify_sample_workspace_bytes(batch, gamma, vocab);
    if (need > kStaticStatsBytes)
        return fail(SPEC_ERR_CAPACITY,
                    "spec_verify_sample_static: batch %d x gamma %d x vocab %d needs %zu bytes of statistics, the built-in "
                    "array holds %zu; use spec_verify_sample with a workspace", batch, gamma, vocab, need, kStaticStatsBytes);
    void* scratch = nullptr;
    const int status = static_stats_address(&scratch);
    if (status != SPEC_OK) return status;
    return launch_verify_sample(target_logits, draft_logits, draft_tokens, uniforms, nullptr, batch, gamma, vocab,
                                temperature, 1.0f, 0, 1.0f, n_accepted, next_token, scratch, static_cast<cudaStream_t>(stream));
}

extern "C" int spec_sample(const float* logits, const float* uniforms, int rows, int vocab, float temperature,
                           int32_t* tokens, void* stream) {
    using namespace spec;
    if (rows < 0 || vocab < 1) return fail(SPEC_ERR_BAD_ARG, "spec_sample: rows=%d vocab=%d", rows, vocab);
    if (!(temperature >= 0.0f) || !isfinite(temperature))
        return fail(SPEC_ERR_BAD_ARG, "spec_sample: temperature must be finite and >= 0");
    if (rows == 0) return SPEC_OK;
    if (!logits || !tokens || (temperature > 0.0f && !uniforms)) return fail(SPEC_ERR_BAD_ARG, "spec_sample: null pointer");
    return launch_sample(logits, uniforms, rows, vocab, temperature, 0, 1.0f, nullptr, tokens, static_cast<cudaStream_t>(stream));
}

extern "C" int spec_sample_truncated(const float* logits, const float* uniforms, int rows, int vocab, float temperature,
                                     int top_k, float top_p, int32_t* tokens, float* floors, void* stream) {
    using namespace spec;
    if (rows < 0 || vocab < 1 || top_k < 0 || !(top_p == top_p))
        return fail(SPEC_ERR_BAD_ARG, "spec_sample_truncated: rows=%d vocab=%d top_k=%d top_p=%g", rows, vocab, top_k, top_p);
    if (!(temperature >= 0.0f) || !isfinite(temperature))
        return fail(SPEC_ERR_BAD_ARG, "spec_sample_truncated: temperature must be finite and >= 0");
    if (rows == 0) return SPEC_OK;
    if (!logits || !tokens || (temperature > 0.0f && !uniforms) || (cut_is_on(vocab, temperature, top_k, top_p) && !floors))
        return fail(SPEC_ERR_BAD_ARG, "spec_sample_truncated: null pointer");
    return launch_sample(logits, uniforms, rows, vocab, temperature, top_k, top_p, floors, tokens,
                         static_cast<cudaStream_t>(stream));
}

extern "C" int spec_truncation_floors(const float* logits, int rows, int vocab, float temperature, int top_k, float top_p,
                                      float* floors, void* stream) {
    using namespace spec;
    if (rows < 0 || vocab < 1 || top_k < 0 || !(top_p == top_p))
        return fail(SPEC_ERR_BAD_ARG, "spec_truncation_floors: rows=%d vocab=%d top_k=%d top_p=%g", rows, vocab, top_k, top_p);
    if (!(temperature > 0.0f) || !isfinite(temperature))
        return fail(SPEC_ERR_BAD_ARG, "spec_truncation_floors: temperature must be finite and > 0");
    if (!cut_is_on(vocab, temperature, top_k, top_p))
        return fail(SPEC_ERR_BAD_ARG, "spec_truncation_floors: neither 0 < top_k < vocab nor 0 < top_p < 1");
    if (rows == 0) return SPEC_OK;
    if (!logits || !floors) return fail(SPEC_ERR_BAD_ARG, "spec_truncation_floors: null pointer");
    return launch_cut<kFloorsOnly>(logits, static_cast<size_t>(vocab), 1, nullptr, 0, 0, rows, vocab, top_k, top_p,
                                   1.0f / temperature, floors, CutWork{}, static_cast<cudaStream_t>(stream));
}

extern "C" int spec_uniforms(uint64_t seed, const int32_t* positions, const int32_t* sequences, int purpose, int count,
                             float* out, void* stream) {
    using namespace spec;
    if (count < 0 || purpose < 0 || purpose > 2) return fail(SPEC_ERR_BAD_ARG, "spec_uniforms: count=%d purpose=%d", count, purpose);
    if (count == 0) return SPEC_OK;
    if (!positions || !sequences || !out) return fail(SPEC_ERR_BAD_ARG, "spec_uniforms: null pointer");
    uniforms_kernel<<<(count + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(
        seed, positions, sequences, static_cast<uint32_t>(purpose), count, out);
    SPEC_CUDA_TRY(cudaGetLastError());
    return SPEC_OK;
}
