// The weight-streaming GEMM for passes of many rows (prompt chunks, batched verification):
//   partial[slot][r][n] = sum over a range of k of x[r][k] * W[n][k],  x = hi + lo in bf16, W bf16.
//
// A pair of CTAs on neighbouring SMs (tcgen05 cta_group::2) owns 256 output features by up to 256 rows.  Each CTA
// holds the weights of its own 128 features and half of the activation tile: the even CTA the hi terms of the rows,
// the odd CTA their lo terms.  To the MMA the two halves are one operand of N = 2 x rows columns, so a k-step is
// one instruction (M = 256, N up to 256) whose accumulator holds W.hi and W.lo side by side; the epilogue adds
// them.  Against one CTA issuing W.hi and W.lo by itself, the weight operand is read from shared memory once
// instead of twice and a CTA fetches half the activation bytes.  More than 128 rows are two such accumulators fed
// by the same weight tile.
//
// The kernel is persistent, one CTA per SM: a warp feeds a ring of stages by TMA, a warp of the even CTA issues the
// MMAs, eight warps drain the accumulators (up to 128 rows there are two in tensor memory: the next tile is multiplied
// while the last one is written).  Work is a list of (256-feature, row) tiles.  The first `dp_tiles` are dealt out
// whole; the k-blocks of the rest are dealt out in equal contiguous runs (stream-K), so that every pair multiplies
// the same amount whatever the shape; a tile that several pairs share has a partial sum per pair, in slots 0, 1, .. in
// k order, which the consumer adds up in that order (no atomics: the same bits every time).
//
// Every wait is bounded; on expiry the kernel records an error code and unwinds (tensor memory is freed on every
// path, and a CTA waits, with a limit, for the copies it has asked for).
#include <algorithm>

#include "model.cuh"
#include "tc_util.cuh"

namespace spec {
namespace {

using namespace tc;

constexpr int kEpilogueWarps = 8;
constexpr int kWideThreads = 32 * (2 + kEpilogueWarps);  // producer warp, MMA warp, epilogue warps
constexpr int kMaxSub = 128;       // rows per accumulator: 2 x 128 columns
constexpr int kWeightBytes = kTileM * kTileK * 2;
constexpr int kMaxStages = 12;
constexpr int kSmemBudget = 227 * 1024 - 1024 /* alignment */ - 512 /* barriers */;
constexpr int kDrainLimit = 1 << 14;

__device__ int g_wide_error;  // first device-side time-out (0 = none)

struct WideArgs {
    PartialPlan plan;
    int n_out, n_rows, stages, packed, fill, stream_once;
    int subs, sub_rows;  // a tile's rows are `subs` accumulators of sub_rows rows each
    uint32_t limit;      // of every wait
    int drill;           // spec_timeout_drill: the producers ask for nothing and arm no barrier
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t in_cta(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void pair_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A box into this CTA's shared memory, its bytes counted on `bar` (an address in either CTA of the pair).
__device__ __forceinline__ void tma_load_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t"
        "}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// One arrival on the barrier at this offset in both CTAs once every MMA issued so far has finished.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(smem_u32(bar)), "h"(static_cast<uint16_t>(3))
        : "memory");
}
__device__ __forceinline__ void arrive_at(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// The segments of one CTA pair, in order: whole tiles first, then its run of the shared ones.
struct WideWork {
    int tile_dp, u, u1;
    __device__ __forceinline__ WideWork(const WideArgs& a, int pair) : tile_dp(pair) {
        const PartialPlan& p = a.plan;
        u = static_cast<int>(static_cast<long long>(pair) * p.units / p.pairs);
        u1 = static_cast<int>(static_cast<long long>(pair + 1) * p.units / p.pairs);
    }
    __device__ __forceinline__ bool next(const PartialPlan& p, int& tile, int& k0, int& k1) {
        if (tile_dp < p.dp_tiles) {
            tile = tile_dp;
            k0 = 0;
            k1 = p.kb;
            tile_dp += p.pairs;
            return true;
        }
        if (u >= u1) return false;
        tile = u / p.kb;
        k0 = u - tile * p.kb;
        k1 = min(p.kb, k0 + (u1 - u));
        tile += p.dp_tiles;
        u += k1 - k0;
        return true;
    }
};

// grid = 2 * pairs, clusters of 2, block = kWideThreads.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kWideThreads, 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_hi,
                 const __grid_constant__ CUtensorMap map_lo, float* __restrict__ partial, const __grid_constant__ WideArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const PartialPlan& p = a.plan;
    const int stages = a.stages;
    const int sub_bytes = a.sub_rows * kTileK * 2;
    const int stage_bytes = kWeightBytes + a.subs * sub_bytes;
    const int n_buf = 3 - a.subs;  // accumulator buffers: two of one accumulator or one of two
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + stages * stage_bytes);  // (the even CTA's count both CTAs' bytes)
    uint64_t* empty_bar = full_bar + kMaxStages;
    uint64_t* acc_full = empty_bar + kMaxStages;   // [2]
    uint64_t* acc_empty = acc_full + 2;            // [2], the even CTA's count both CTAs' epilogue warps
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);

    const int warp = __shfl_sync(kFullMask, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // (uniform for the compiler)
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], 2 * kEpilogueWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    pair_sync();  // both CTAs' barriers exist
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    bool ok = true;

    if (warp == 0) {
        // ---- producer: this CTA's weight tile and its half (hi or lo) of the activation tile per stage ----
        const bool leader = elect_one() && !a.drill;
        uint64_t policy_w, policy_x;
        if (a.stream_once) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy_w));
        else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy_w));
        asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy_x));
        const CUtensorMap* map_x = rank == 0 ? &map_hi : &map_lo;
        const uint32_t full0 = in_cta(smem_u32(full_bar), 0);
        auto load_w = [&](int s, int tile, int kb) {
            const int f = (tile / p.token_tiles) * 2 + static_cast<int>(rank);  // 128-feature tile
            if (!leader) return;
            if (rank == 0) mbar_expect_tx(&full_bar[s], 2 * stage_bytes);
            if (a.packed) tma_load_pair(smem + s * stage_bytes, &map_w, 0, (f * p.kb + kb) * kTileM, full0 + 8 * s, policy_w);
            else tma_load_pair(smem + s * stage_bytes, &map_w, kb * kTileK, f * kTileM, full0 + 8 * s, policy_w);
        };
        auto load_x = [&](int s, int tile, int kb) {
            if (!leader) return;
            for (int sub = 0; sub < a.subs; ++sub)
                tma_load_pair(smem + s * stage_bytes + kWeightBytes + sub * sub_bytes, map_x, kb * kTileK,
                              (tile % p.token_tiles) * p.tok_tile + sub * a.sub_rows, full0 + 8 * s, policy_x);
        };
        int tile, k0, k1;
        // the first ring of weights does not depend on the kernel before this one
        int ahead = 0;
        for (WideWork w(a, pair); ahead < stages && w.next(p, tile, k0, k1);)
            for (int kb = k0; kb < k1 && ahead < stages; ++kb) load_w(ahead++, tile, kb);
        pdl_wait();
        int it = 0;
        int s = 0, use = 0;  // stage of block `it` and how often the ring has gone round
        for (WideWork w(a, pair); ok && w.next(p, tile, k0, k1);)
            for (int kb = k0; kb < k1; ++kb) {
                if (it >= ahead) {
                    if (!mbar_wait_warp(&empty_bar[s], (use - 1) & 1, a.limit)) { ok = false; break; }
                    load_w(s, tile, kb);
                }
                load_x(s, tile, kb);
                ++it;
                if (++s == stages) { s = 0; ++use; }
            }
        pdl_trigger();  // (after the wait: kernels behind this one count on what lies in front of it, common.cuh)
        if (!ok && rank == 0)  // nothing may still be on its way when the CTAs leave
            for (int i = 0; i < stages; ++i) {
                mbar_wait(&full_bar[i], 0, kDrainLimit);
                mbar_wait(&full_bar[i], 1, kDrainLimit);
            }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---- MMA issuer (for both CTAs) ----
            const bool leader = elect_one();
            const uint32_t idesc = instr_desc(2 * kTileM, 2 * a.sub_rows);
            const uint32_t base = smem_u32(smem);
            int s = 0, use = 0;     // stage, and how often the ring has gone round
            int buf = 0, turn = 0;  // accumulator buffer, and how often the buffers have gone round
            int tile, k0, k1;
            for (WideWork w(a, pair); ok && w.next(p, tile, k0, k1);) {
                if (turn > 0 && !mbar_wait_warp(&acc_empty[buf], (turn - 1) & 1, a.limit)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem + buf * 256;
                for (int kb = k0; kb < k1; ++kb) {
                    if (!mbar_wait_warp(&full_bar[s], use & 1, a.limit)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t a_desc = smem_desc_sw128(base + s * stage_bytes);
                    const uint64_t b_desc = smem_desc_sw128(base + s * stage_bytes + kWeightBytes);
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < kTileK / kMmaK; ++k) {
                            const uint64_t step = static_cast<uint64_t>((k * kMmaK * 2) >> 4);
                            mma_pair(acc, a_desc + step, b_desc + step, idesc, (kb > k0 || k > 0) ? 1u : 0u);
                            if (a.subs == 2)
                                mma_pair(acc + 256, a_desc + step, b_desc + (sub_bytes >> 4) + step, idesc, (kb > k0 || k > 0) ? 1u : 0u);
                        }
                        commit_pair(&empty_bar[s]);
                    }
                    __syncwarp();
                    if (++s == stages) { s = 0; ++use; }
                }
                if (ok && leader) commit_pair(&acc_full[buf]);
                __syncwarp();
                if (++buf == n_buf) { buf = 0; ++turn; }
            }
        }
    } else {
        // ---- epilogue: warp w reads accumulator lanes 32 (w % 4) .. + 31 ----
        pdl_wait();  // (the partial sums of the GEMM before may still be read by the kernel before this one)
        const int quarter = warp & 3, first_col = ((warp - 2) >> 2) * 16;
        const size_t slot_stride = static_cast<size_t>(a.n_rows) * a.n_out;
        int buf = 0, turn = 0;
        int tile, k0, k1;
        for (WideWork w(a, pair); w.next(p, tile, k0, k1);) {
            if (!mbar_wait_warp(&acc_full[buf], turn & 1, a.limit)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int feature = ((tile / p.token_tiles) * 2 + static_cast<int>(rank)) * kTileM + quarter * 32 + lane;
            const int slot = partial_slot(p, tile, k0);
            for (int sub = 0; sub < a.subs; ++sub) {
                const int row0 = (tile % p.token_tiles) * p.tok_tile + sub * a.sub_rows;
                const uint32_t acc = tmem + (buf + sub) * 256 + (static_cast<uint32_t>(quarter * 32) << 16);
                for (int c0 = first_col; c0 < a.sub_rows && row0 + c0 < a.n_rows; c0 += 32) {
                    uint32_t vh[16], vl[16];
                    tmem_ld16(acc + c0, vh);
                    tmem_ld16(acc + a.sub_rows + c0, vl);
                    tmem_ld_wait();
                    if (feature >= a.n_out) continue;
                    float* out = partial + slot * slot_stride + static_cast<size_t>(row0 + c0) * a.n_out + feature;
                    if (row0 + c0 + 16 <= a.n_rows) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) out[static_cast<uint32_t>(i * a.n_out)] = __uint_as_float(vh[i]) + __uint_as_float(vl[i]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (row0 + c0 + i < a.n_rows) out[static_cast<uint32_t>(i * a.n_out)] = __uint_as_float(vh[i]) + __uint_as_float(vl[i]);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive_at(in_cta(smem_u32(&acc_empty[buf]), 0));
            if (a.fill && k1 == p.kb && feature < a.n_out) {  // zeros where a caller wants the same number of sums everywhere
                const int row0 = (tile % p.token_tiles) * p.tok_tile;
                for (int f = slot + 1; f < p.slots; ++f)
                    for (int r = row0 + (warp - 2) / 4; r < min(a.n_rows, row0 + p.tok_tile); r += 2)
                        partial[f * slot_stride + static_cast<size_t>(r) * a.n_out + feature] = 0.0f;
            }
            if (++buf == n_buf) { buf = 0; ++turn; }
        }
    }
    if (!ok) atomicCAS(&g_wide_error, 0, 16 + warp);
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    pair_sync();  // nobody leaves while its peer may still signal or read its shared memory
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

int wide_subs(int n_rows) { return n_rows <= kMaxSub ? 1 : 2; }

}  // namespace

PartialPlan gemm_wide_plan(int n_out, int k, int n_rows) {
    PartialPlan p{};
    const int features = (n_out + 2 * kTileM - 1) / (2 * kTileM);
    const int subs = wide_subs(n_rows);
    p.token_tiles = (n_rows + kMaxSub * subs - 1) / (kMaxSub * subs);
    const int unit = 16 * subs;
    p.tok_tile = ((n_rows + p.token_tiles - 1) / p.token_tiles + unit - 1) / unit * unit;
    p.kb = (k + kTileK - 1) / kTileK;
    const int tiles = features * p.token_tiles;
    constexpr int kPairs = 74;  // one CTA per SM
    p.pairs = std::max(1, static_cast<int>(std::min<long long>(kPairs, static_cast<long long>(tiles) * p.kb / 4)));
    // Whole tiles only from 16 rounds on (the last round then costs little), one to two rounds' worth of tiles shared
    // below that, everything shared when there are fewer tiles than pairs.
    if (tiles >= 16 * p.pairs) p.dp_tiles = tiles;
    else p.dp_tiles = std::max(0, tiles / p.pairs - 1) * p.pairs;
    p.units = (tiles - p.dp_tiles) * p.kb;
    p.slots = 1;
    for (int t = p.dp_tiles; t < tiles; ++t) p.slots = std::max(p.slots, partial_slots_of_tile(p, t));
    return p;
}

int launch_gemm_wide(const __nv_bfloat16* hi, const __nv_bfloat16* lo, int hi_rows, const void* w, bool packed, int n_rows,
                     int n_out, int k, float* partial, bool fill, cudaStream_t stream) {
    WideArgs a{};
    a.plan = gemm_wide_plan(n_out, k, n_rows);
    a.n_out = n_out;
    a.n_rows = n_rows;
    a.packed = packed ? 1 : 0;
    a.fill = fill ? 1 : 0;
    a.stream_once = a.plan.token_tiles == 1 ? 1 : 0;
    a.subs = wide_subs(n_rows);
    a.sub_rows = a.plan.tok_tile / a.subs;
    a.limit = kSpinLimit;
    const int stage_bytes = kWeightBytes + a.plan.tok_tile * kTileK * 2;
    a.stages = std::min(kMaxStages, kSmemBudget / stage_bytes);
    const int smem = a.stages * stage_bytes + 1024 + 512;
    const int tiles = (n_out + kTileM - 1) / kTileM;
    CUtensorMap mw, mhi, mlo;
    int status = packed ? cached_bf16_map(w, tiles * a.plan.kb * kTileM, kTileK, kTileM, false, &mw)
                        : cached_bf16_map(w, n_out, k, kTileM, true, &mw);
    if (status == SPEC_OK) status = cached_bf16_map(hi, hi_rows, k, a.sub_rows, true, &mhi);
    if (status == SPEC_OK) status = cached_bf16_map(lo, hi_rows, k, a.sub_rows, true, &mlo);
    if (status != SPEC_OK) return status;
    static std::atomic<unsigned long long> configured{0};
    status = allow_shared_memory(configured, gemm_wide_kernel, 227 * 1024);
    if (status != SPEC_OK) return status;
    return launch_pdl(gemm_wide_kernel, dim3(2 * a.plan.pairs), dim3(kWideThreads), smem, stream, mw, mhi, mlo, partial, a);
}

// One pair of CTAs, one tile of one k-block, nothing requested, waits of `limit` polls; `base`: 16 KB that are never read.
int launch_gemm_wide_drill(void* base, uint32_t limit, cudaStream_t stream) {
    WideArgs a{};
    a.plan = gemm_wide_plan(kTileM, kTileK, 16);
    a.n_out = kTileM;
    a.n_rows = a.sub_rows = 16;
    a.subs = 1;
    a.stages = 2;
    a.limit = limit;
    a.drill = 1;
    CUtensorMap mw, mx;
    int status = cached_bf16_map(base, kTileM, kTileK, kTileM, true, &mw);
    if (status == SPEC_OK) status = cached_bf16_map(base, 16, kTileK, 16, true, &mx);
    if (status != SPEC_OK) return status;
    const int smem = a.stages * (kWeightBytes + a.sub_rows * kTileK * 2) + 1024 + 512;
    return launch_pdl(gemm_wide_kernel, dim3(2 * a.plan.pairs), dim3(kWideThreads), smem, stream, mw, mx, mx, static_cast<float*>(base), a);
}

int* gemm_wide_error_word() { return symbol_address(g_wide_error); }

int gemm_wide_take_error() {
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_wide_error, sizeof(int)) != cudaSuccess) return -1;
    if (v) cudaMemcpyToSymbol(g_wide_error, &zero, sizeof(int));
    return v;
}

}  // namespace spec
