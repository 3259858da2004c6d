// The small kernels between the weight-streaming GEMMs of a decoder block.
// Each one also finishes the GEMM before it (adds up the split-K partial sums
// in a fixed order, adds the residual) and prepares the input of the GEMM after
// it (fp32, and/or split into two bf16 terms for the tensor-core path), so that
// a block is nine launches: norm, qkv GEMM, rope + KV append, attention,
// out-projection GEMM, norm, FFN-in GEMM, activation, FFN-out GEMM; ten where
// attention's key slices are merged by a kernel of their own (long contexts).
// fp32 models have the norms and the activation inside their GEMMs
// (gemm_rows.cu), few rows of a small bf16 model all of it in one kernel
// (small_pass.cu).
#include <cmath>

#include "attn_unit.cuh"

namespace spec {
namespace {

// No pointer here is __restrict__: a load through a const __restrict__ pointer may be moved in front of pdl_wait(), where
// what the kernel before writes is not there yet.

__device__ __forceinline__ float load_elem(const void* base, size_t i, bool bf16) {
    return bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(base)[i]) : static_cast<const float*>(base)[i];
}

__device__ __forceinline__ float4 add4(const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// Sums of the split-K partial results of the N groups of four elements that start at i[0], .., i[N-1], in split order;
// BATCH splits' loads of every group are in flight at a time.
template <int N, int BATCH>
__device__ __forceinline__ void sum_partials(const float* partial, int splits, size_t stride, const size_t (&i)[N],
                                             float4 (&out)[N]) {
    for (int s0 = 0; s0 < splits; s0 += BATCH) {
        float4 p[BATCH][N];
#pragma unroll
        for (int k = 0; k < BATCH; ++k)
#pragma unroll
            for (int n = 0; n < N; ++n)
                p[k][n] = s0 + k < splits ? *reinterpret_cast<const float4*>(partial + static_cast<size_t>(s0 + k) * stride + i[n])
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < BATCH; ++k)
            if (s0 + k < splits) {
#pragma unroll
                for (int n = 0; n < N; ++n) out[n] = (s0 + k == 0) ? p[k][n] : add4(out[n], p[k][n]);
            }
    }
}

// x = hi + lo with hi = bf16(x), lo = bf16(x - hi): 16 mantissa bits survive.  Four elements at once.
__device__ __forceinline__ void store_split4(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t i, const float4& x) {
    const float v[4] = {x.x, x.y, x.z, x.w};
    __align__(8) __nv_bfloat16 h[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        h[e] = __float2bfloat16_rn(v[e]);
        l[e] = __float2bfloat16_rn(v[e] - __bfloat162float(h[e]));
    }
    *reinterpret_cast<uint2*>(hi + i) = *reinterpret_cast<const uint2*>(h);
    *reinterpret_cast<uint2*>(lo + i) = *reinterpret_cast<const uint2*>(l);
}

// four consecutive elements (i a multiple of four) of an fp32 or bf16 array
__device__ __forceinline__ float4 load_elem4(const void* base, size_t i, bool bf16) {
    if (!bf16) return *reinterpret_cast<const float4*>(static_cast<const float*>(base) + i);
    const uint2 t = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(base) + i);
    return make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u), __uint_as_float(t.y << 16),
                       __uint_as_float(t.y & 0xffff0000u));
}

// grid = (ceil(d / 512), rows), block = 128: four elements per thread.
__global__ void embed_kernel(const void* tok_emb, const void* pos_emb, bool bf16,
                             bool add_pos, const int32_t* token, const int32_t* pos, int d,
                             int vocab, int max_positions, float* h) {
    pdl_trigger();
    pdl_wait();
    const int r = blockIdx.y;
    const int t = min(max(token[r], 0), vocab - 1);
    const int p = min(max(pos[r], 0), max_positions - 1);
    const int i = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= d) return;
    float4 v = load_elem4(tok_emb, static_cast<size_t>(t) * d + i, bf16);
    if (add_pos) v = add4(v, load_elem4(pos_emb, static_cast<size_t>(p) * d + i, bf16));
    *reinterpret_cast<float4*>(h + static_cast<size_t>(r) * d + i) = v;
}

// grid = rows, block = THREADS; d is a multiple of 4, at most 4 * THREADS * PER.  Row r of the output is
// RMSNorm(h[src(r)]) * gain.  If `partial` is given, h[r] += sum of the partial
// results first (the residual add of the GEMM that produced them) and the new h
// is stored.  A thread holds up to PER float4 of the row in registers.
// With CTAS > 1 a cluster of that many CTAs shares a row (d at most 4 * THREADS * CTAS, PER = 1, grid = rows * CTAS): a
// row of 4096 with its eight partial sums is 147 KB, a microsecond of what one SM takes in, and nothing else runs
// meanwhile.  The CTAs give one another their warps' sums of squares through distributed shared memory.
// DEFER: they do not.  W . (rmsnorm(h) gain) is W . (h gain) times a factor per row, so the terms are of h * gain, the warps' sums of
// squares go to `squares`, [row][32], and the kernel that adds up the GEMM's partial sums forms the factor (DeferredRow).  The
// norm is a stop between two weight streams of which only the first 24 MB of the second is on its way meanwhile, and the
// exchange between the CTAs was a fifth of it (7B shape, three rows: 7.0 -> 5.5 us behind the GEMM).  The terms have the same 16 bits
// either way: logits of nine shapes of pass are off 64 bits by 6.87e-4 (mean; 6.88e-4 with the factor applied here).
constexpr int kNormMaxWidth = 4 * 1024 * 4;
constexpr int kNormCtas = 8;  // of a cluster that shares a row
// The activation kernel gives a thread several rows where one each is more threads than the GPU holds at once: below that the
// rows of a thread only lengthen it (96 rows of the 160M shape: a pass 625 us with a row each, 699 with four).
constexpr long long kResidentThreads = 148 * 2048;
constexpr int kNormFourRows = 296;  // at most for a cluster of four: eight CTAs of 256 threads to an SM
constexpr int kNormClusterRows = kDeferredRows;  // at most (launch_norm has both sides)

template <int THREADS, int PER, int CTAS = 1, bool DEFER = false>
__global__ void __launch_bounds__(THREADS)
norm_kernel(float* h, const float* partial, const PartialPlan plan, int n_rows, const float* gain,
            const int32_t* src_rows, int d, float eps, float* out,
            __nv_bfloat16* out_hi, __nv_bfloat16* out_lo, float* squares) {
    static_assert(CTAS == 1 || (PER == 1 && CTAS * THREADS / 32 == 32), "a lane per warp of the cluster");
    __shared__ float red[CTAS * THREADS / 32];
    const int r = blockIdx.x / CTAS;
    const int groups = d / 4;
    const int first = CTAS > 1 ? blockIdx.x % CTAS * THREADS + threadIdx.x : threadIdx.x;
    if constexpr (CTAS > 1 && !DEFER) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // (its peers are there)
    // the gains are constants: fetched while the kernel before this one is still finishing
    float4 gg[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int g = first + j * THREADS;
        gg[j] = g < groups ? *reinterpret_cast<const float4*>(gain + 4 * g) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    pdl_wait();
    // The GEMM that follows is released only now, when the GEMM before this kernel is complete: released earlier, its CTAs
    // take the places of that GEMM's leaving CTAs and their first weight tiles compete with the tail of its stream
    // (measured per 7B block: 94.5 -> 93.1 us; releasing at the end of this kernel instead: 95.1).
    pdl_trigger();
    const int src_row = src_rows ? src_rows[r] : r;
    const size_t src = static_cast<size_t>(src_row) * d;
    const size_t stride = static_cast<size_t>(n_rows) * d;
    float4 v[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int g = first + j * THREADS;
        v[j] = g < groups ? *reinterpret_cast<const float4*>(h + src + 4 * g) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (partial) {
        constexpr int kBatch = PER == 1 ? 8 : 2;  // splits in flight at a time, added in split order
        int splits[PER], most = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int g = first + j * THREADS;
            splits[j] = g < groups ? partial_count(plan, src_row, 4 * g) : 0;
            most = max(most, splits[j]);
        }
        for (int s0 = 0; s0 < most; s0 += kBatch) {
            float4 p[kBatch][PER];
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
#pragma unroll
                for (int j = 0; j < PER; ++j)
                    p[k][j] = s0 + k < splits[j] ? *reinterpret_cast<const float4*>(partial + static_cast<size_t>(s0 + k) * stride + src +
                                                                                    4 * (first + j * THREADS))
                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
#pragma unroll
                for (int j = 0; j < PER; ++j)
                    if (s0 + k < splits[j]) v[j] = add4(v[j], p[k][j]);
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int g = first + j * THREADS;
            if (g < groups) *reinterpret_cast<float4*>(h + src + 4 * g) = v[j];
        }
    }
    float ss = 0.0f;
#pragma unroll
    for (int j = 0; j < PER; ++j) ss += (v[j].x * v[j].x + v[j].y * v[j].y) + (v[j].z * v[j].z + v[j].w * v[j].w);
    ss = warp_sum(ss);
    float total = 0.0f;
    if constexpr (DEFER) {
        if ((threadIdx.x & 31) == 0) squares[32 * r + (first >> 5)] = ss;
    } else if constexpr (CTAS > 1) {
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        const int lane = threadIdx.x & 31;
        if (lane < CTAS) {
            const uint32_t here = static_cast<uint32_t>(__cvta_generic_to_shared(&red[first >> 5]));
            asm volatile("{\n\t.reg .b32 there;\n\tmapa.shared::cluster.u32 there, %0, %1;\n\tst.shared::cluster.f32 [there], %2;\n\t}"
                         ::"r"(here), "r"(lane), "f"(ss)
                         : "memory");
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        total = warp_sum(red[lane]);
    } else {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < THREADS / 32; ++i) total += red[i];
    }
    const float scale = DEFER ? 1.0f : rsqrtf(total / static_cast<float>(d) + eps);
    const size_t dst = static_cast<size_t>(r) * d;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int g = first + j * THREADS;
        if (g < groups) {
            const float4 y = DEFER ? make_float4(v[j].x * gg[j].x, v[j].y * gg[j].y, v[j].z * gg[j].z, v[j].w * gg[j].w)
                                   : make_float4(v[j].x * scale * gg[j].x, v[j].y * scale * gg[j].y, v[j].z * scale * gg[j].z,
                                         v[j].w * scale * gg[j].w);
            if (out) *reinterpret_cast<float4*>(out + dst + 4 * g) = y;
            if (out_hi) store_split4(out_hi, out_lo, dst + 4 * g, y);
        }
    }
}

// The factor of a deferred norm in row r (1 without one): what the norm kernel would have multiplied the row with.  All lanes.
struct DeferredRow {
    float square = 0.0f;  // this lane's, on its way while other loads are
    __device__ __forceinline__ void fetch(const RowFactor& f, int r) {
        if (f.squares) square = f.squares[32 * r + (threadIdx.x & 31)];
    }
    __device__ __forceinline__ float factor(const RowFactor& f) const { return f.squares ? rsqrtf(warp_sum(square) / f.width + f.eps) : 1.0f; }
};

template <typename KV>
__device__ __forceinline__ void store_cached4(KV* dst, const float (&v)[4]) {
    __align__(16) KV t[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] = to_cached<KV>(v[e]);
    if (sizeof(KV) == 4) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(t);
    else *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(t);
}

// grid = (ceil(heads * d_head / 8 / block), rows), heads = n_heads + 2 n_kv_heads.  qkv row layout:
// [q heads | k heads | v heads], d_head each.  A thread finishes elements j .. j+3 and
// j + d_head/2 .. of one head of one row of the qkv GEMM (optional partial sums), applies
// rotary positions (q and k heads; they pair j with j + d_head/2), leaves q in `qkv` for the
// attention kernel, and appends K or V to the paged cache.  A row to a thread at any number of rows: four, as in ffn_act_kernel, changed
// nothing (a block of the 7B shape, us: 448 rows 372 with four, 370; 1024 rows 782, 783; 16 prompts of 500 to 1000 tokens with their
// answers 1.5 % longer with four in one run, 0.8 % shorter in another).
template <typename KV>
__global__ void qkv_kernel(float* qkv, const float* partial, const PartialPlan plan, int n_rows,
                           const int32_t* pos, const int32_t* seq, int n_heads,
                           int n_kv_heads, int d_head, const float2* rope_table,
                           KV* kv_layer, const int32_t* page_table, int pages_per_seq,
                           int page_shift, const RowFactor norm) {
    pdl_trigger();
    // (with partial sums the kernel in front is a tensor-core GEMM, which releases this one only after its own wait: the rows'
    // positions, rotations and pages are older than that, and are fetched ahead of this kernel's)
    if (!partial) pdl_wait();
    const int half = d_head / 2, per_head = half / 4;
    const int task = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
    const int head = task / per_head, j = 4 * (task % per_head);
    if (blockIdx.x * blockDim.x + (threadIdx.x & ~31) >= (n_heads + 2 * n_kv_heads) * per_head) return;  // (whole warps)
    const bool out = head >= n_heads + 2 * n_kv_heads;
    const bool is_q = head < n_heads, is_k = !is_q && head < n_heads + n_kv_heads;
    const int width = (n_heads + 2 * n_kv_heads) * d_head;
    const int p = pos[r];
    const bool rotate = rope_table && p >= 0 && (is_q || is_k);
    float4 t0, t1;  // (cos, sin) of position p for the four pairs
    if (rotate) {
        const float4* at = reinterpret_cast<const float4*>(rope_table + static_cast<size_t>(p) * half + j);
        t0 = at[0];
        t1 = at[1];
    }
    size_t cached = 0;  // where K or V goes
    if (p >= 0 && !is_q && !out) {
        const int kv_head = is_k ? head - n_heads : head - n_heads - n_kv_heads;
        const int page = page_table[seq[r] * pages_per_seq + (p >> page_shift)];
        const size_t block = (static_cast<size_t>(page) * 2 + (is_k ? 0 : 1)) * n_kv_heads + kv_head;
        cached = ((block << page_shift) + (p & ((1 << page_shift) - 1))) * d_head + j;
    }
    if (partial) pdl_wait();
    DeferredRow deferred;
    deferred.fetch(norm, r);
    const size_t at = static_cast<size_t>(r) * width + (out ? 0 : head * d_head + j);
    const size_t where[2] = {at, at + half};
    float4 x[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    if (partial) {
        // (a head of 64 or 128 columns lies inside one 256-column tile)
        sum_partials<2, 4>(partial, partial_count(plan, r, out ? 0 : head * d_head), static_cast<size_t>(n_rows) * width, where, x);
    } else {
        x[0] = *reinterpret_cast<const float4*>(qkv + where[0]);
        x[1] = *reinterpret_cast<const float4*>(qkv + where[1]);
    }
    const float factor = deferred.factor(norm);
    if (out) return;
    float a[4] = {x[0].x, x[0].y, x[0].z, x[0].w}, b[4] = {x[1].x, x[1].y, x[1].z, x[1].w};
    if (norm.squares) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            a[e] *= factor;
            b[e] *= factor;
        }
    }
    if (rotate) {
        const float c[4] = {t0.x, t0.z, t1.x, t1.z}, s[4] = {t0.y, t0.w, t1.y, t1.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float y1 = a[e] * c[e] - b[e] * s[e], y2 = b[e] * c[e] + a[e] * s[e];
            a[e] = y1;
            b[e] = y2;
        }
    }
    if (is_q) {
        *reinterpret_cast<float4*>(qkv + where[0]) = make_float4(a[0], a[1], a[2], a[3]);
        *reinterpret_cast<float4*>(qkv + where[1]) = make_float4(b[0], b[1], b[2], b[3]);
        return;
    }
    if (p < 0) return;  // inactive row: nothing is cached
    KV* dst = kv_layer + cached;
    store_cached4<KV>(dst, a);
    store_cached4<KV>(dst + half, b);
}

// logits[dst(i)] = table[token[src(i)]] for a table model: grid = (chunks, rows), block = 256.
__global__ void table_logits_kernel(const void* table, bool bf16, int vocab, const int32_t* token,
                                    const int32_t* src_rows, const int32_t* dst_rows,
                                    float* logits) {
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.y;
    const int t = min(max(token[src_rows ? src_rows[i] : i], 0), vocab - 1);
    float* out = logits + static_cast<size_t>(dst_rows ? dst_rows[i] : i) * vocab;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < vocab; v += gridDim.x * blockDim.x)
        out[v] = load_elem(table, static_cast<size_t>(t) * vocab + v, bf16);
}

// Copy-from-context draft: logits row i is one-hot (0 at the guess, -inf elsewhere), the
// guess being what followed the most recent earlier occurrence of the last `ngram`
// tokens of the sequence up to the row's position, or the last token again if there is
// none.  Positions below length[seq] read the committed tokens, later ones this
// iteration's guesses.  grid = (chunks, rows): every CTA repeats the search (a few
// thousand token compares) and writes its share of the row.  An inactive row (position < 0) has no
// last token; its guess, which nobody looks at, is token 0.
__global__ void copy_logits_kernel(const int32_t* tokens, int max_len, const int32_t* length,
                                   const int32_t* draft_tokens, int gamma, const int32_t* row_pos,
                                   const int32_t* row_seq, const int32_t* src_rows,
                                   const int32_t* dst_rows, int ngram, int vocab, float* logits) {
    __shared__ int best[32];
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.y;
    const int r = src_rows ? src_rows[i] : i;
    const int b = row_seq[r], last = row_pos[r];
    const int committed = length[b];
    const int32_t* seq = tokens + static_cast<size_t>(b) * max_len;
    const int32_t* guesses = draft_tokens + static_cast<size_t>(b) * gamma;
    auto at = [&](int p) { return p < committed ? seq[p] : guesses[min(p - committed, gamma - 1)]; };
    // j = end of an earlier occurrence of the suffix: ngram-1 <= j <= last-1
    int found = -1;
    for (int j = last - 1 - static_cast<int>(threadIdx.x); j >= ngram - 1; j -= blockDim.x) {
        bool same = true;
        for (int k = 0; k < ngram && same; ++k) same = at(j - k) == at(last - k);
        if (same) { found = j; break; }  // this thread's later candidates are all older
    }
    found = __reduce_max_sync(0xffffffffu, found);
    if ((threadIdx.x & 31) == 0) best[threadIdx.x >> 5] = found;
    __syncthreads();
    for (int w = 0; w < static_cast<int>(blockDim.x) / 32; ++w) found = max(found, best[w]);
    const int guess = last < 0 ? 0 : min(max(at(found >= 0 ? found + 1 : last), 0), vocab - 1);
    float* out = logits + static_cast<size_t>(dst_rows ? dst_rows[i] : i) * vocab;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < vocab; v += gridDim.x * blockDim.x)
        out[v] = v == guess ? 0.0f : -INFINITY;
}

// f = gelu(u)  |  gelu(gate) * up  |  silu(gate) * up, with u the partial sums of the FFN-in GEMM, as two bf16 terms.
// grid = (ceil(d_ff / 4 / block), ceil(rows / ROWS)): four columns of ROWS rows per thread.  Of few rows each is a thread's own
// (the kernel is then one trip to memory); of many ROWS share what is not arithmetic - how many partial sums there are takes
// four integer divisions - and their loads are in flight together.  One row to a thread was bound by issue (940 instructions
// a warp, 12.5 us behind the GEMM for 224 rows of the 7B shape, 9.8 with four).
constexpr int kActRows = 4;  // (a tile's rows are a multiple of 16: these share their partial sums' number)
template <int FFN, int ROWS>
__global__ void ffn_act_kernel(const float* partial, const PartialPlan plan, int n_rows, int d_ff, __nv_bfloat16* f_hi,
                               __nv_bfloat16* f_lo, const RowFactor norm) {
    pdl_trigger();
    pdl_wait();
    const int mine = 4 * (blockIdx.x * blockDim.x + threadIdx.x), r0 = ROWS * blockIdx.y;
    if (mine - 4 * static_cast<int>(threadIdx.x & 31) >= d_ff) return;  // (whole warps)
    const bool beyond = mine >= d_ff;
    const int c = beyond ? 0 : mine;
    DeferredRow deferred[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) deferred[i].fetch(norm, min(r0 + i, n_rows - 1));
    constexpr bool kGated = FFN != SPEC_FFN_GELU;
    const int width = kGated ? 2 * d_ff : d_ff;
    const size_t stride = static_cast<size_t>(n_rows) * width;
    const int n_gate = partial_count(plan, r0, c), n_up = kGated ? partial_count(plan, r0, c + d_ff) : 0;
    float4 g[ROWS], up[ROWS];
    if constexpr (ROWS == 1) {
        const size_t at = static_cast<size_t>(r0) * width + c;
        g[0] = up[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kGated && n_gate == n_up) {
            const size_t where[2] = {at, at + d_ff};
            float4 both[2] = {g[0], g[0]};
            sum_partials<2, 4>(partial, n_gate, stride, where, both);
            g[0] = both[0];
            up[0] = both[1];
        } else {
            const size_t where[1] = {at};
            sum_partials<1, 8>(partial, n_gate, stride, where, g);
            if (kGated) {
                const size_t where_up[1] = {at + d_ff};
                sum_partials<1, 8>(partial, n_up, stride, where_up, up);
            }
        }
    } else {
        const float* at[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            at[i] = partial + static_cast<size_t>(min(r0 + i, n_rows - 1)) * width + c;
            g[i] = up[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int k = 0; k < max(n_gate, n_up); ++k) {
            float4 p[ROWS], q[ROWS];
#pragma unroll
            for (int i = 0; i < ROWS; ++i) {
                p[i] = k < n_gate ? *reinterpret_cast<const float4*>(at[i]) : make_float4(0.f, 0.f, 0.f, 0.f);
                if (kGated) q[i] = k < n_up ? *reinterpret_cast<const float4*>(at[i] + d_ff) : make_float4(0.f, 0.f, 0.f, 0.f);
                at[i] += stride;
            }
#pragma unroll
            for (int i = 0; i < ROWS; ++i) {
                g[i] = add4(g[i], p[i]);
                if (kGated) up[i] = add4(up[i], q[i]);
            }
        }
    }
    if (norm.squares) {
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const float f = deferred[i].factor(norm);
            g[i] = make_float4(g[i].x * f, g[i].y * f, g[i].z * f, g[i].w * f);
            up[i] = make_float4(up[i].x * f, up[i].y * f, up[i].z * f, up[i].w * f);
        }
    }
    if (beyond) return;
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        if (ROWS > 1 && r0 + i >= n_rows) break;
        const float4 x = g[i], u = up[i];
        float4 y;
        if (FFN == SPEC_FFN_GELU) y = make_float4(gelu_tanh(x.x), gelu_tanh(x.y), gelu_tanh(x.z), gelu_tanh(x.w));
        else if (FFN == SPEC_FFN_SWIGLU) y = make_float4(silu(x.x) * u.x, silu(x.y) * u.y, silu(x.z) * u.z, silu(x.w) * u.w);
        else y = make_float4(gelu_tanh(x.x) * u.x, gelu_tanh(x.y) * u.y, gelu_tanh(x.z) * u.z, gelu_tanh(x.w) * u.w);
        store_split4(f_hi, f_lo, static_cast<size_t>(r0 + i) * d_ff + c, y);
    }
}

}  // namespace

int launch_embed(const Model& m, const RowMeta& rows, int n_rows, float* h, cudaStream_t stream) {
    return launch_pdl(embed_kernel, dim3((m.cfg.d_model / 4 + 127) / 128, n_rows), dim3(128), 0, stream, m.tok_emb, m.pos_emb, m.bf16(),
                      m.cfg.arch == SPEC_ARCH_GPT, rows.token, rows.pos, m.cfg.d_model, m.cfg.vocab,
                      m.cfg.max_positions, h);
}

int launch_table_logits(const void* table, bool bf16, int vocab, const int32_t* token, const int32_t* src_rows,
                        const int32_t* dst_rows, int n_rows, float* logits, cudaStream_t stream) {
    const int chunks = std::max(1, std::min((vocab + 255) / 256, 32));
    return launch_pdl(table_logits_kernel, dim3(chunks, n_rows), dim3(256), 0, stream, table, bf16, vocab, token, src_rows,
                      dst_rows, logits);
}

int launch_copy_logits(const int32_t* tokens, int max_len, const int32_t* length, const int32_t* draft_tokens, int gamma,
                       const RowMeta& rows, const int32_t* src_rows, const int32_t* dst_rows, int n_rows, int ngram,
                       int vocab, float* logits, cudaStream_t stream) {
    const int chunks = std::max(1, std::min((vocab + 255) / 256, 16));
    return launch_pdl(copy_logits_kernel, dim3(chunks, n_rows), dim3(256), 0, stream, tokens, max_len, length, draft_tokens,
                      gamma, rows.pos, rows.seq, src_rows, dst_rows, ngram, vocab, logits);
}

bool norm_defers(int d, int n_rows) { return d % 4 == 0 && d > 2048 && d <= 512 * kNormCtas && n_rows <= kNormClusterRows; }

int launch_norm(float* h, const float* partial, const PartialPlan& plan, int rows_total, const float* gain, const int32_t* src_rows,
                int n_rows, int d, float eps, float* out, __nv_bfloat16* out_hi, __nv_bfloat16* out_lo,
                cudaStream_t stream, float* squares) {
    if (d % 4 || d > kNormMaxWidth)
        return fail(SPEC_ERR_BAD_CONFIG, "norm: width %d is not a multiple of 4 or exceeds %d", d, kNormMaxWidth);
#define SPEC_LAUNCH_NORM(T, P)                                                                                              \
    return launch_pdl(norm_kernel<T, P>, dim3(n_rows), dim3(T), 0, stream, h, partial, plan, rows_total, gain, src_rows, d, \
                      eps, out, out_hi, out_lo, static_cast<float*>(nullptr))
    if (squares && !norm_defers(d, n_rows)) return fail(SPEC_ERR_BAD_CONFIG, "norm: %d rows of %d are not deferred", n_rows, d);
    // a thread per 128-bit group of the row (fewer warps to reduce over where the row is narrow); with more rows than
    // SMs, small CTAs with several groups per thread, so that the CTAs of an SM wait for memory side by side.
    // Wide rows that leave SMs idle go to a cluster each.  Whole pass of the 7B shape at 500 cached tokens, a CTA of 1024
    // threads per row against a cluster, ms: 1 row 2.779 / 2.761, 3 rows 2.865 / 2.839, 7 rows 2.937 / 2.915, 16 rows
    // 3.111 / 3.123 (the runs of one side differ by as much), 32 rows 3.196 / 3.152, 64 rows 3.748 / 3.734, 126 rows
    // 5.232 / 5.216; beyond, four larger CTAs (eight partial sums in flight, not two: 224 rows 11.0 -> 9.8 us behind the GEMM), and
    // where those no longer fit side by side a CTA per row (us a block, a CTA per row against four: 160 rows 177 / 173, 224 rows
    // 212 / 211, 259 rows 292 / 292, 296 rows 296 / 297).
    const int groups = d / 4;
    if (squares)
        return launch_cluster(norm_kernel<128, 1, kNormCtas, true>, 0, dim3(n_rows * kNormCtas), dim3(128), 0, stream, h, partial,
                              plan, rows_total, gain, src_rows, d, eps, out, out_hi, out_lo, squares);
    if (groups > 512 && groups <= 128 * kNormCtas && n_rows <= kNormClusterRows)
        return launch_cluster(norm_kernel<128, 1, kNormCtas>, kNormCtas, dim3(n_rows * kNormCtas), dim3(128), 0, stream, h, partial,
                              plan, rows_total, gain, src_rows, d, eps, out, out_hi, out_lo, static_cast<float*>(nullptr));
    if (groups > 512 && groups <= 1024 && n_rows <= kNormFourRows)
        return launch_cluster(norm_kernel<256, 1, 4>, 4, dim3(n_rows * 4), dim3(256), 0, stream, h, partial, plan, rows_total, gain,
                              src_rows, d, eps, out, out_hi, out_lo, static_cast<float*>(nullptr));
    if (groups <= 128) SPEC_LAUNCH_NORM(128, 1);
    if (groups <= 256) SPEC_LAUNCH_NORM(256, 1);
    if (groups <= 1024 && n_rows > 148) SPEC_LAUNCH_NORM(256, 4);
    if (groups <= 1024) SPEC_LAUNCH_NORM(1024, 1);
    SPEC_LAUNCH_NORM(1024, 4);
#undef SPEC_LAUNCH_NORM
}

int launch_qkv(int n_heads, int n_kv_heads, int d_head, const float2* rope, const KvPool& pool, const RowMeta& rows,
               int n_rows, float* qkv, const float* partial, const PartialPlan& plan, cudaStream_t stream, const RowFactor& norm) {
    const int tasks = (n_heads + 2 * n_kv_heads) * (d_head / 8);
    const int threads = n_rows <= 16 ? 64 : 256;
    const dim3 grid((tasks + threads - 1) / threads, n_rows);
    int page_shift = 0;  // (pages are a power of two)
    while ((1 << page_shift) < pool.page_size) ++page_shift;
#define SPEC_LAUNCH_QKV(KV)                                                                                                      \
    return launch_pdl(qkv_kernel<KV>, grid, dim3(threads), 0, stream, qkv, partial, plan, n_rows, rows.pos, rows.seq, n_heads,   \
                      n_kv_heads, d_head, rope, static_cast<KV*>(pool.kv), pool.page_table, pool.pages_per_seq, page_shift, norm)
    if (pool.dtype == SPEC_DTYPE_FP16) SPEC_LAUNCH_QKV(__half);
    if (pool.dtype == SPEC_DTYPE_BF16) SPEC_LAUNCH_QKV(__nv_bfloat16);
    SPEC_LAUNCH_QKV(float);
#undef SPEC_LAUNCH_QKV
}

int launch_ffn_act(const float* partial, const PartialPlan& plan, int n_rows, int d_ff, int ffn, __nv_bfloat16* f_hi,
                   __nv_bfloat16* f_lo, cudaStream_t stream, const RowFactor& norm) {
    const bool many = static_cast<long long>(n_rows) * (d_ff / 4) > kResidentThreads;
    const int threads = n_rows <= 16 ? 64 : 256;
    const dim3 grid((d_ff / 4 + threads - 1) / threads, many ? (n_rows + kActRows - 1) / kActRows : n_rows);
#define SPEC_LAUNCH_ACT(F)                                                                                                     \
    return many ? launch_pdl(ffn_act_kernel<F, kActRows>, grid, dim3(threads), 0, stream, partial, plan, n_rows, d_ff, f_hi, f_lo, norm) \
                : launch_pdl(ffn_act_kernel<F, 1>, grid, dim3(threads), 0, stream, partial, plan, n_rows, d_ff, f_hi, f_lo, norm)
    if (ffn == SPEC_FFN_GELU) SPEC_LAUNCH_ACT(SPEC_FFN_GELU);
    if (ffn == SPEC_FFN_SWIGLU) SPEC_LAUNCH_ACT(SPEC_FFN_SWIGLU);
    SPEC_LAUNCH_ACT(SPEC_FFN_GATED_GELU);
#undef SPEC_LAUNCH_ACT
}

// (cos, sin) of position * base^(-2j / d_head), evaluated in double precision on
// the host and rounded once to fp32: [positions][d_head / 2].
void fill_rope_table(std::vector<float2>& table, int positions, int d_head, double base) {
    const int half = d_head / 2;
    table.resize(static_cast<size_t>(positions) * half);
    for (int j = 0; j < half; ++j) {
        const double inv_freq = std::pow(base, -2.0 * j / static_cast<double>(d_head));
        for (int p = 0; p < positions; ++p) {
            const double a = static_cast<double>(p) * inv_freq;
            table[static_cast<size_t>(p) * half + j] = make_float2(static_cast<float>(std::cos(a)), static_cast<float>(std::sin(a)));
        }
    }
}

}  // namespace spec
