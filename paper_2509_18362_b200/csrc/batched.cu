// Batched draft path (Sec. 2.1 recursion, Sec. 2.2 Eq. 3 compressed head) for groups of up to 64
// sequences: per step, six weight-streaming tcgen05 GEMMs (skinny_gemm.cuh) and the small
// row-wise kernels between them (norms, rotary embedding + cache append, attention, residuals).
// All kernels of a call are enqueued on the caller's stream; none waits on another CTA.
#include "batched.cuh"
#include "skinny_gemm.cuh"

namespace fmtp {

namespace {

constexpr uint32_t kDevBadToken = 0x1u, kDevBadPage = 0x2u, kDevBadPos = 0x4u, kDevAllNan = 0x10u;
constexpr int kRowThreads = 512;

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

__device__ __forceinline__ float block_sum(float v, float *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < nw; ++w) t += red[w];     // same order on every thread
    return t;
}

__device__ __forceinline__ void store_hilo(bf16_t *xop, int ld, int r, int j, float v) {
    uint16_t hi, lo;
    split_bf16(v, hi, lo);
    xop[(size_t)(2 * r) * ld + j] = hi;
    xop[(size_t)(2 * r + 1) * ld + j] = lo;
}

// ---- rows of a launch. Row r belongs to sequence r / M. In a target step the M rows of a sequence sit at
// positions L .. L+M-1. In draft step 0 they are the sequence's extend rows (Sec. 2.3 "Drafting phase":
// the pairs of target hidden state and next token committed since the last call), n = n_ext[seq] of them
// at positions L .. L+n-1, the last one being draft step 1; rows beyond n are padding (computed, never
// stored or published). A later draft step has one row per sequence at position L + n - 1 + step.
struct RowGeo {
    int M;                   // rows per sequence in this launch
    int M0;                  // rows per sequence of draft step 0 (the bound of n_ext); target step: M
    int step;                // draft step (0 in a target step)
    const int32_t *n_ext;    // [sequences] or NULL (= M0 for every sequence)
};
constexpr int kMaxLen = 1 << 30;      // a longer committed length is the caller's error: flagged like any position without a slot
__device__ __forceinline__ int geo_len(const KvPtrs &kv, int seq) { return min(max(kv.seq_lens[seq], 0), kMaxLen); }
__device__ __forceinline__ int geo_next(const RowGeo &g, int seq) { return g.n_ext ? min(max(g.n_ext[seq], 1), g.M0) : g.M0; }
// Position of row r (before clamping to the cache's capacity); *valid = false for a padding row.
__device__ __forceinline__ int geo_pos(const RowGeo &g, const KvPtrs &kv, int r, bool *valid) {
    const int seq = r / g.M, m = r - seq * g.M;
    const int L = geo_len(kv, seq);
    if (g.step > 0) { *valid = true; return L + geo_next(g, seq) - 1 + g.step; }
    const int n = geo_next(g, seq);
    *valid = m < n;
    return L + min(m, n - 1);
}
// Extend step of a draft: only the last extend row of a sequence publishes its result (hidden state, head
// operand), under the sequence's index; -1 for every other row.
__device__ __forceinline__ int geo_out_seq(const RowGeo &g, int r) {
    const int seq = r / g.M, m = r - seq * g.M;
    return m == geo_next(g, seq) - 1 ? seq : -1;
}

// ---- step input: [rms(h; g_h) ; rms(Emb(tok); g_e)] as the projection's operand; also turns the
// previous step's argmax key into its draft token. One block per sequence.
struct PrologueArgs {
    int step, K, d, V, ld, only_tokens;
    RowGeo geo;                  // step 0 of a draft with extend rows: which rows are padding
    float eps;
    const bf16_t *h_last;
    const int32_t *tok_last;
    const float *hout;
    const unsigned long long *keys_prev;
    int32_t *out_drafts;
    const bf16_t *embed, *g_h, *g_e;
    bf16_t *xop;
    uint32_t *status, *user_status;
};

// eight consecutive values -> hi/lo bf16, one 16-byte store each
__device__ __forceinline__ void store_hilo8(bf16_t *xop, int ld, int r, int j, const float (&v)[8]) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint16_t h0, l0, h1, l1;
        split_bf16(v[2 * i], h0, l0);
        split_bf16(v[2 * i + 1], h1, l1);
        hi[i] = (uint32_t)h0 | ((uint32_t)h1 << 16);
        lo[i] = (uint32_t)l0 | ((uint32_t)l1 << 16);
    }
    *reinterpret_cast<uint4 *>(xop + (size_t)(2 * r) * ld + j) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4 *>(xop + (size_t)(2 * r + 1) * ld + j) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}
__device__ __forceinline__ void unpack_bf16x8(const uint4 &u, float (&v)[8]) {
    v[0] = bf16lo_f32(u.x); v[1] = bf16hi_f32(u.x); v[2] = bf16lo_f32(u.y); v[3] = bf16hi_f32(u.y);
    v[4] = bf16lo_f32(u.z); v[5] = bf16hi_f32(u.z); v[6] = bf16lo_f32(u.w); v[7] = bf16hi_f32(u.w);
}
__device__ __forceinline__ void load_f32x8(const float *p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// Each thread owns U groups of eight consecutive columns (d % 64 == 0), kept in registers: every load and store is 16 bytes,
// all loads are issued before the first use and made once (re-reading the row and fetching the gains after the
// reduction were two more round trips to L2: draft calls 611 -> 603 us at 16 sequences, 765 -> 756 at 4).
template <int U>
__global__ void __launch_bounds__(kRowThreads) prologue_kernel(const PrologueArgs a) {
    chain_release();
    __shared__ float red[32];
    __shared__ int s_tok;
    const int r = blockIdx.x, tid = threadIdx.x;
    uint4 gh[U], ge[U];                          // weights, and in step 0 the caller's hidden state: nothing to wait for
    float h[U][8];
    if (!a.only_tokens) {
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int j = (tid + q * kRowThreads) * 8;
            if (j < a.d) {
                gh[q] = *reinterpret_cast<const uint4 *>(a.g_h + j);
                ge[q] = *reinterpret_cast<const uint4 *>(a.g_e + j);
                if (a.step == 0) unpack_bf16x8(*reinterpret_cast<const uint4 *>(a.h_last + (size_t)r * a.d + j), h[q]);
            }
        }
    }
    chain_wait();
    if (tid == 0) {
        int tok;
        if (a.step == 0) {
            const int seq = r / a.geo.M;                   // a padding row's token is never looked at
            tok = (r - seq * a.geo.M < geo_next(a.geo, seq)) ? a.tok_last[r] : 0;
        } else {
            tok = 0;
            if (a.out_drafts) {
                const unsigned long long key = a.keys_prev[r];
                if ((key >> 32) == 0ull) atomicOr(a.status, kDevAllNan);
                tok = (int)argmax_key_id(key);
                a.out_drafts[(size_t)r * a.K + (a.step - 1)] = tok;
            }
        }
        if ((unsigned)tok >= (unsigned)a.V) { atomicOr(a.status, kDevBadToken); tok = 0; }
        s_tok = tok;
    }
    __syncthreads();
    if (a.only_tokens) {
        // last kernel of the call: hand the status word (earlier kernels' flags and this block's) to the caller
        if (tid == 0 && a.user_status) {
            __threadfence();
            const uint32_t st = *reinterpret_cast<volatile uint32_t *>(a.status);
            if (st) atomicOr(a.user_status, st);
        }
        return;
    }
    const bf16_t *erow = a.embed + (size_t)s_tok * a.d;
    float e[U][8], sh = 0.f, se = 0.f;
#pragma unroll
    for (int q = 0; q < U; ++q) {
        const int j = (tid + q * kRowThreads) * 8;
        if (j < a.d) {
            if (a.step > 0) load_f32x8(a.hout + (size_t)r * a.d + j, h[q]);
            unpack_bf16x8(*reinterpret_cast<const uint4 *>(erow + j), e[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < U; ++q)
        if ((tid + q * kRowThreads) * 8 < a.d) {
#pragma unroll
            for (int i = 0; i < 8; ++i) { sh += h[q][i] * h[q][i]; se += e[q][i] * e[q][i]; }
        }
    sh = block_sum(sh, red);
    se = block_sum(se, red);
    const float rh = 1.0f / sqrtf(sh / (float)a.d + a.eps), re = 1.0f / sqrtf(se / (float)a.d + a.eps);
#pragma unroll
    for (int q = 0; q < U; ++q) {
        const int j = (tid + q * kRowThreads) * 8;
        if (j < a.d) {
            float g[8];
            unpack_bf16x8(gh[q], g);
#pragma unroll
            for (int i = 0; i < 8; ++i) h[q][i] = h[q][i] * rh * g[i];
            unpack_bf16x8(ge[q], g);
#pragma unroll
            for (int i = 0; i < 8; ++i) e[q][i] = e[q][i] * re * g[i];
            store_hilo8(a.xop, a.ld, r, j, h[q]);
            store_hilo8(a.xop, a.ld, r, a.d + j, e[q]);
        }
    }
}

// ---- after a split-K GEMM: x = (residual ? x : 0) + sum of the partials; operand of the next
// GEMM = rms(x; gain) as hi/lo. With `final`: the normed vector is the step's output hidden state.
struct PostArgs {
    int d, splits, rows, ldp, ld, residual, final, K, step;
    int map_out, seq0;           // final norm of a draft's extend step: row r publishes as sequence seq0 + geo_out_seq(r)
    RowGeo geo;
    float eps;
    const float *partial;
    float *x, *hout;
    bf16_t *out_h;
    const bf16_t *gain;
    bf16_t *xop;
};

template <int U>
__global__ void __launch_bounds__(kRowThreads) post_kernel(const PostArgs a) {
    chain_release();
    __shared__ float red[32];
    const int r = blockIdx.x, tid = threadIdx.x;
    float v[U][8], ss = 0.f;
    uint4 gn[U];                                 // (weights: nothing to wait for)
#pragma unroll
    for (int q = 0; q < U; ++q)
        if ((tid + q * kRowThreads) * 8 < a.d) gn[q] = *reinterpret_cast<const uint4 *>(a.gain + (tid + q * kRowThreads) * 8);
    chain_wait();
#pragma unroll
    for (int q = 0; q < U; ++q) {
        const int j = (tid + q * kRowThreads) * 8;
        if (j < a.d) {
            float part[kBatchMaxSplits][8];
            // every load of a group is issued before the first use
#pragma unroll
            for (int s = 0; s < kBatchMaxSplits; ++s)
                if (s < a.splits) load_f32x8(a.partial + ((size_t)s * a.rows + r) * a.ldp + j, part[s]);
            if (a.residual) load_f32x8(a.x + (size_t)r * a.d + j, v[q]);
            else {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[q][i] = 0.f;
            }
#pragma unroll
            for (int s = 0; s < kBatchMaxSplits; ++s)
                if (s < a.splits) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[q][i] += part[s][i];
                }
            *reinterpret_cast<float4 *>(a.x + (size_t)r * a.d + j) = make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
            *reinterpret_cast<float4 *>(a.x + (size_t)r * a.d + j + 4) = make_float4(v[q][4], v[q][5], v[q][6], v[q][7]);
#pragma unroll
            for (int i = 0; i < 8; ++i) ss += v[q][i] * v[q][i];
        }
    }
    ss = block_sum(ss, red);
    const float rs = 1.0f / sqrtf(ss / (float)a.d + a.eps);
    int dst = r;
    if (a.map_out) {
        const int o = geo_out_seq(a.geo, r);
        if (o < 0) return;                       // an extend row that is not its sequence's last: nothing to publish
        dst = a.seq0 + o;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
        const int j = (tid + q * kRowThreads) * 8;
        if (j < a.d) {
            float g[8];
            unpack_bf16x8(gn[q], g);
#pragma unroll
            for (int i = 0; i < 8; ++i) v[q][i] = v[q][i] * rs * g[i];
            store_hilo8(a.xop, a.ld, dst, j, v[q]);
            if (a.final) {
                *reinterpret_cast<float4 *>(a.hout + (size_t)dst * a.d + j) = make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
                *reinterpret_cast<float4 *>(a.hout + (size_t)dst * a.d + j + 4) = make_float4(v[q][4], v[q][5], v[q][6], v[q][7]);
                if (a.out_h) {
                    uint32_t o[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) o[i] = (uint32_t)f32_bf16bits(v[q][2 * i]) | ((uint32_t)f32_bf16bits(v[q][2 * i + 1]) << 16);
                    *reinterpret_cast<uint4 *>(a.out_h + ((size_t)dst * a.K + a.step) * a.d + j) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
        }
    }
}

// ---- after the QKV GEMM: sum the partials, rotate q and k at the row's position, keep q as bf16 pairs,
// append k and v (rounded to bf16) to the paged cache. Block = (head, sequence), dh/2 threads.
struct QkvArgs {
    int qdim, kvdim, dh, Hq, Hkv, splits, rows, ldp, page, max_ctx;
    RowGeo geo;                  // which sequence and position a row has
    const float *partial;
    bf16_t *q;                   // layout: AttnArgs::q
    KvPtrs kv;
    const float *rope_cos, *rope_sin;
    uint32_t *status;
};

// Positions, rotary factors and the block table are inputs of the call: they are read before the wait for the predecessor.
__global__ void qkv_finish_kernel(const QkvArgs a) {
    chain_release();
    const int head = blockIdx.x, r = blockIdx.y, e = threadIdx.x, half = a.dh >> 1;
    const int max_tokens = min(a.kv.max_pages * a.page, a.max_ctx);
    const int seq = r / a.geo.M;
    bool valid;
    const int pos_true = geo_pos(a.geo, a.kv, r, &valid);
    const int pos = min(pos_true, max_tokens - 1);
    const int col = head * a.dh;              // q heads, then k heads, then v heads: the GEMM's row order
    const bool rotate = head < a.Hq + a.Hkv;
    const float cs = rotate ? a.rope_cos[(size_t)pos * half + e] : 1.f, sn = rotate ? a.rope_sin[(size_t)pos * half + e] : 0.f;
    int page = head >= a.Hq ? a.kv.block_table[(size_t)seq * a.kv.max_pages + pos / a.page] : 0;
    chain_wait();
    float lo = 0.f, hi = 0.f;
    {
        float x[kBatchMaxSplits], y[kBatchMaxSplits];
#pragma unroll
        for (int s = 0; s < kBatchMaxSplits; ++s)
            if (s < a.splits) {
                const float *pp = a.partial + ((size_t)s * a.rows + r) * a.ldp + col;
                x[s] = pp[e];
                y[s] = pp[e + half];
            }
#pragma unroll
        for (int s = 0; s < kBatchMaxSplits; ++s)
            if (s < a.splits) { lo += x[s]; hi += y[s]; }
    }
    if (rotate) {
        const float x = lo, y = hi;
        lo = x * cs - y * sn;
        hi = y * cs + x * sn;
    }
    if (head < a.Hq) {
        // stored ready for the attention MMA (see AttnArgs::q): scaled by log2(e) / sqrt(dh), split into two bf16 parts
        const float sc = (1.0f / sqrtf((float)a.dh)) * 1.4426950408889634f;
        const int gq = a.Hq / a.Hkv, kvh = head / gq, h = head - kvh * gq;
        bf16_t *qh = a.q + (((size_t)r * a.Hkv + kvh) * 2 * gq + h) * a.dh, *ql = qh + (size_t)gq * a.dh;
        auto at = [&](int i) -> int { return (((i >> 3) ^ (h & 7)) << 3) | (i & 7); };
        split_bf16(lo * sc, qh[at(e)], ql[at(e)]);
        split_bf16(hi * sc, qh[at(e + half)], ql[at(e + half)]);
        return;
    }
    if (!valid) return;                       // padding row: nothing to store
    if (pos_true >= max_tokens) {             // no slot for this position: flagged, nothing written
        if (head == a.Hq && e == 0) atomicOr(a.status, kDevBadPos);
        return;
    }
    const bool is_k = rotate;
    const int kvh = is_k ? head - a.Hq : head - a.Hq - a.Hkv;
    if ((unsigned)page >= (unsigned)a.kv.num_pages) { atomicOr(a.status, kDevBadPage); page = 0; }
    bf16_t *dst = (is_k ? a.kv.k_pages : a.kv.v_pages) + (((size_t)page * a.Hkv + kvh) * a.page + (pos % a.page)) * a.dh;
    dst[e] = f32_bf16bits(lo);
    dst[e + half] = f32_bf16bits(hi);
}

// ---- attention. A work item is one 256-token chunk of one (sequence, KV head) for up to ROWS rows of the sequence: the
// M rows of a target step or of a draft's extend step share the K/V stream (ROWS = 4), later draft steps have one row
// (ROWS = 1). The Hq/Hkv query heads of the group share it as well. One persistent CTA per SM; its eight compute warps
// form two groups, each with a ring of its own, fed by its own copy warp, and each walking its own items, so one
// group's serial work (softmax, barriers, the partial's write) hides behind the other's and behind both streams.
//
// Scores and the weighted sum run on mma.sync.m16n8k16 with the query heads (and the probabilities) as the A operand,
// rows 0-7 the high bf16 parts of the heads and rows 8-15 the low parts, so both products carry fp32-accurate inputs.
// One row: within a group warp w computes the scores of tokens 16w .. 16w+15 of a 64-token block; the warps exchange the
// block maximum and the probabilities through shared memory, then warp w adds up its quarter of the head dimension over all
// 64 tokens. Several rows: one warp per row, all 64 tokens and the whole head dimension, its probabilities never leave
// its registers. A row goes through the same operations, in the same order, either way and whatever rows share its item.
//
// The K/V pool is a stack of page x head-dim tiles: one TMA copy brings 16 tokens of K or V (4 KB at head dim 128) in the
// 128-byte-swizzled layout ldmatrix reads without bank conflicts. The copies used to be 16-byte cp.async from 128 threads
// that also read the block table: those reads queued behind the copies, and a block could not be requested before the
// read of its table entries came back (1.2 us per 32 KB block). Now a warp holds the table entries of a whole item in
// registers, one item ahead.
// Bound: the K/V stream for one row; the tensor-core issue, shared-memory reads and the softmax for four. Measured at the
// 7B shape, before -> now: 64 rows with contexts in [512, 8192] (618 MB) 154 -> 95 us (6.5 TB/s); 16 sequences x 4 rows at
// 2048 (67 MB) 82 -> 24 us (28 with four rows split over the warps like one: two barriers per block, and the queries
// re-read from shared memory for every block).
//
// Committed K/V (positions below seq_lens) is immutable during a call, so the first ring stages are requested before the
// wait for the predecessor kernel; blocks with positions this call writes, and the queries, come after it.
// Output per item and row: unnormalised o, running max m (log2 units) and sum l per head.
struct AttnArgs {
    int Hq, Hkv, dh, page, max_ctx, max_chunks, B;    // B: sequences
    int tma;                     // pages are whole 16-token tiles: TMA copies (else 16-byte copies, any page size)
    int extra_arrivals;          // self-test only: arrivals a ring stage expects beyond the copies that are made
    RowGeo geo;                  // which positions a sequence's rows have
    unsigned long long wait_limit_ns;   // a ring wait gives up after this long
    const bf16_t *q;             // [rows][Hkv][2][Hq/Hkv][dh]: scaled queries, high parts then low parts, 16-byte pieces of head
                                 // h (of its group) stored at piece ^ (h & 7)
    KvPtrs kv;
    float *att_part;             // [rows][Hq][max_chunks][dh+2]
    uint32_t *status;
};

constexpr int kAttnBlk = 64;                 // tokens per ring stage
constexpr int kAttnBox = 16;                 // tokens per TMA copy, and per warp in the score product
constexpr int kAttnCompute = 256;            // compute threads (warps 0-7); warps 8-11: two copy warps per group
constexpr int kAttnThreads = kAttnCompute + 128;
constexpr int kAttnRows = 4;                 // rows of an item in calls with several rows per sequence

struct AttnItem {                            // one (sequence, KV head, chunk, row set), group-uniform
    int seq, kvh, chunk, set, t0, n_ctx, n_blk;
};

template <int DH, int ROWS>
struct AttnSmem {
    static constexpr int BOX = kAttnBox * DH * 2;                // bytes of one copy: [DH / 64][16 tokens][128 bytes]
    static constexpr int VOFF = 4 * BOX;                         // a stage: four K boxes, four V boxes
    static constexpr int STAGE = 8 * BOX;
    static constexpr int SG = 3;                                 // stages per group
    static constexpr int NQ = ROWS == 1 ? 2 : 1;                 // items per group whose queries are held (they go to registers at once)
    static constexpr int QROW = 16 * DH * 2;                     // room for a row's queries (8 heads, two parts)
    static constexpr int PROW = ROWS == 1 ? 16 * 128 : 0;        // a row's probabilities: 16 operand rows x 64 tokens
    static constexpr int O_Q = 2 * SG * STAGE;
    static constexpr int O_P = O_Q + 2 * NQ * ROWS * QROW;
    static constexpr int O_RED = O_P + 2 * PROW;                 // per group, one row: [4 warps][8 heads] maxima, then sums
    static constexpr int O_BAR = O_RED + (ROWS == 1 ? 2 * 2 * 32 * 4 : 0);
    static constexpr int O_TAB = O_BAR + (2 * (2 * SG + NQ) + 1) * 8;
    static constexpr int BYTES = O_TAB + (4 * kBatchRows + 1) * 4;
    static constexpr int TOTAL = BYTES + 1024;                   // the ring starts on a 1024-byte boundary
};

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
// Two values as two packed bf16 pairs: their high parts and what is left of them (two conversions for the four).
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
    const float ra = a - bf16lo_f32(hi), rb = b - bf16hi_f32(hi);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(rb), "f"(ra));
}
// 2^x for x <= 0 (results below the normal range are zero, as is 2^-inf).
__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int DH, int ROWS>
__global__ void __launch_bounds__(kAttnThreads, 1) attn_kernel(const __grid_constant__ AttnArgs a, const __grid_constant__ CUtensorMap kmap,
                                                               const __grid_constant__ CUtensorMap vmap) {
    chain_release();
    using L = AttnSmem<DH, ROWS>;
    constexpr int SG = L::SG, NQ = L::NQ;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::O_BAR);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(bars + 2 * (2 * SG + NQ));
    int *prefix = reinterpret_cast<int *>(smem + L::O_TAB);                // [B + 1] items before a sequence
    int *tpos = prefix + kBatchRows + 1;                                   // position of a sequence's row 0
    int *tval = tpos + kBatchRows;                                         // its rows that count
    int *tlen = tval + kBatchRows;                                         // its committed positions
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp < 8 ? warp >> 2 : (warp - 8) >> 1;                // copy warps 8, 9 serve group 0; 10, 11 group 1
    uint64_t *full = bars + grp * (2 * SG + NQ), *empty = full + SG, *qempty = empty + SG;
    unsigned char *ring = smem + (size_t)grp * SG * L::STAGE;
    const int max_tokens = min(a.kv.max_pages * a.page, a.max_ctx);
    const int gq = a.Hq / a.Hkv;
    if (threadIdx.x == 0) {
        for (int g = 0; g < 2; ++g) {
            uint64_t *b = bars + g * (2 * SG + NQ);
            for (int s = 0; s < SG; ++s) { mbar_init(&b[s], (a.tma ? 1 : 65) + a.extra_arrivals); mbar_init(&b[SG + s], 4); }
            for (int s = 0; s < NQ; ++s) mbar_init(&b[2 * SG + s], 4);
        }
        *abort_flag = 0;
        mbar_fence_init();
    }
    // visible positions 0 .. n-1 of row m of a sequence
    auto row_ctx = [&](int pos0, int m) -> int { return min(pos0 + m, max_tokens - 1) + 1; };
    if (warp == 0) {             // two sequences per lane; seq_lens and n_ext are inputs of the call: nothing to wait for
        int cnt[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int s = 2 * lane + u;
            cnt[u] = 0;
            if (s < a.B) {
                const int len = geo_len(a.kv, s), nx = geo_next(a.geo, s);
                const int pos0 = a.geo.step > 0 ? len + nx - 1 + a.geo.step : len;
                const int nv = a.geo.step > 0 ? 1 : nx;
                tpos[s] = pos0; tval[s] = nv; tlen[s] = len;
                cnt[u] = (row_ctx(pos0, nv - 1) + kBatchAttnChunk - 1) / kBatchAttnChunk * a.Hkv * ((nv + ROWS - 1) / ROWS);
            }
        }
        int incl = cnt[0] + cnt[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (2 * lane <= a.B) prefix[2 * lane] = incl - cnt[0] - cnt[1];
        if (2 * lane + 1 <= a.B) prefix[2 * lane + 1] = incl - cnt[1];
        if (lane == 31 && a.B == 2 * 32) prefix[a.B] = incl;
    }
    __syncthreads();
    const int n_items = prefix[a.B], worker = grp * (int)gridDim.x + (int)blockIdx.x, stride = 2 * (int)gridDim.x;

    // a wait that gives up after two seconds (or when another thread has), so a logic error cannot hang the device;
    // after that no wait blocks any more and every role runs to its end
    auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        const unsigned long long t_begin = global_timer_ns();
        uint32_t polls = 0;
        while (!mbar_try_wait(bar, parity)) {
            if ((++polls & 63u) == 0) {
                if (*abort_flag) return false;
                if (global_timer_ns() - t_begin > a.wait_limit_ns) { *abort_flag = 1u; return false; }
            }
        }
        return true;
    };
    auto load_item = [&](AttnItem &it, int item) {
        int s = it.seq;                      // a worker's items come in ascending order: search on from the last one
        while (prefix[s + 1] <= item) ++s;
        it.seq = s;
        int rem = item - prefix[s];
        it.kvh = rem % a.Hkv;
        rem /= a.Hkv;
        const int nv = tval[s], sets = (nv + ROWS - 1) / ROWS;
        it.chunk = rem / sets;
        it.set = rem - it.chunk * sets;
        it.t0 = it.chunk * kBatchAttnChunk;
        it.n_ctx = row_ctx(tpos[s], min(nv, (it.set + 1) * ROWS) - 1);             // of the set's last row
        it.n_blk = max(0, (min(kBatchAttnChunk, it.n_ctx - it.t0) + kAttnBlk - 1) / kAttnBlk);   // 0: no row of the set sees the chunk
    };
    const uint32_t qbytes = (uint32_t)(2 * gq * DH * 2);
    auto copy_queries = [&](const AttnItem &it, int slot, int stage, int i) {      // thread i copies the queries of the set's row i
        if (i < min(ROWS, tval[it.seq] - it.set * ROWS)) {
            const size_t r = (size_t)it.seq * a.geo.M + it.set * ROWS + i;
            bulk_load(smem_u32(smem + L::O_Q + ((size_t)(grp * NQ + slot) * ROWS + i) * L::QROW),
                      a.q + (r * a.Hkv + it.kvh) * 2 * gq * DH, qbytes, &full[stage]);
        }
    };
    auto query_bytes = [&](const AttnItem &it) -> uint32_t { return qbytes * (uint32_t)min(ROWS, tval[it.seq] - it.set * ROWS); };

    if (warp >= 8) {
    const int ct = threadIdx.x - kAttnCompute - grp * 64;                 // thread among the group's 64 copy threads
    const uint64_t policy = l2_evict_first();
    AttnItem it, nx;
    it.seq = 0;
    int stage = 0, li = 0;
    uint32_t phase = 0;
    bool ok = true;
    if (a.tma) {
        if (ct < 32) {
            // ---- lane i holds where 16-token tile i of the item's chunk is: its row in the pool seen as [.., dh]
            auto tile_row = [&](const AttnItem &i_) -> int {
                const int pos = min(i_.t0 + (lane & 15) * kAttnBox, i_.n_ctx - 1) & ~(kAttnBox - 1), pgi = pos / a.page;
                int page = a.kv.block_table[(size_t)i_.seq * a.kv.max_pages + pgi];
                if ((unsigned)page >= (unsigned)a.kv.num_pages) { atomicOr(a.status, kDevBadPage); page = 0; }
                return (page * a.Hkv + i_.kvh) * a.page + (pos - pgi * a.page);
            };
            // lanes 0-3 copy the K tiles of a block, lanes 4-7 its V tiles
            auto copy_block = [&](const AttnItem &i_, int blk, int rows) {
                const int n = min(4, (i_.n_ctx - i_.t0 - blk * kAttnBlk + kAttnBox - 1) / kAttnBox);
                const int y = __shfl_sync(0xffffffffu, rows, blk * 4 + (lane & 3));
                if (lane == 0) mbar_arrive_expect_tx(&full[stage], (uint32_t)(2 * n * L::BOX) + (blk == 0 ? query_bytes(i_) : 0u));
                __syncwarp();
                if (lane < 8 && (lane & 3) < n)
                    tma_load_3d_hint(smem_u32(ring + (size_t)stage * L::STAGE + (lane >> 2) * L::VOFF + (lane & 3) * L::BOX),
                                     lane < 4 ? &kmap : &vmap, 0, y, 0, &full[stage], policy);
            };
            int item = worker, pre = 0, rows = 0, nrows = 0;
            // the first item with work
            for (; item < n_items; item += stride) { load_item(it, item); if (it.n_blk > 0) break; }
            if (item < n_items) {
                rows = tile_row(it);
                for (; pre < SG && pre < it.n_blk && it.t0 + (pre + 1) * kAttnBlk <= tlen[it.seq]; ++pre) { stage = pre; copy_block(it, pre, rows); }
            }
            chain_wait();
            stage = 0;
            while (item < n_items && ok) {
                // the next item with work, and its tiles
                int nitem = item + stride;
                nx = it;
                for (; nitem < n_items; nitem += stride) { load_item(nx, nitem); if (nx.n_blk > 0) break; }
                if (nitem < n_items) nrows = tile_row(nx);
                for (int blk = 0; blk < it.n_blk; ++blk) {
                    if (lane == 0) ok = wait(&empty[stage], phase ^ 1u) && (blk > 0 || wait(&qempty[li % NQ], ((li / NQ) & 1) ^ 1));
                    ok = __shfl_sync(0xffffffffu, ok, 0);
                    if (!ok) break;
                    if (pre > 0) --pre;                 // this block's K/V is already on its way
                    else copy_block(it, blk, rows);
                    if (blk == 0) copy_queries(it, li % NQ, stage, lane);
                    if (++stage == SG) { stage = 0; phase ^= 1u; }
                }
                ++li;
                it = nx; item = nitem; rows = nrows;
            }
        }
    } else {
        // ---- any page size: 16-byte copies into the same layout, zeros beyond the visible positions
        constexpr int PIECES = DH / 8;
        chain_wait();
        for (int item = worker; item < n_items && ok; item += stride) {
            load_item(it, item);
            if (it.n_blk == 0) continue;
            for (int blk = 0; blk < it.n_blk; ++blk) {
                if (!wait(&empty[stage], phase ^ 1u) || (blk == 0 && !wait(&qempty[li % NQ], ((li / NQ) & 1) ^ 1))) { ok = false; break; }
                const uint32_t sb = smem_u32(ring + (size_t)stage * L::STAGE);
                for (int i = ct; i < kAttnBlk * PIECES; i += 64) {
                    const int t = i / PIECES, c = i - t * PIECES;
                    const int pos = it.t0 + blk * kAttnBlk + t, pc = min(pos, it.n_ctx - 1), pgi = pc / a.page;
                    int page = a.kv.block_table[(size_t)it.seq * a.kv.max_pages + pgi];
                    if ((unsigned)page >= (unsigned)a.kv.num_pages) { atomicOr(a.status, kDevBadPage); page = 0; }
                    const size_t off = (((size_t)page * a.Hkv + it.kvh) * a.page + (pc - pgi * a.page)) * DH + c * 8;
                    const uint32_t d = sb + (uint32_t)((t >> 4) * L::BOX + (c >> 3) * 2048 + (t & 15) * 128 + (((c & 7) ^ (t & 7)) << 4));
                    const uint32_t n = pos < it.n_ctx ? 16u : 0u;
                    cp_async16_off_hint<0>(d, a.kv.k_pages + off, n, policy);
                    cp_async16_off_hint<0>(d + L::VOFF, a.kv.v_pages + off, n, policy);
                }
                if (ct == 0) mbar_arrive_expect_tx(&full[stage], blk == 0 ? query_bytes(it) : 0u);
                if (blk == 0) copy_queries(it, li % NQ, stage, ct);
                cp_async_arrive(&full[stage]);
                if (++stage == SG) { stage = 0; phase ^= 1u; }
            }
            ++li;
        }
        cp_async_wait_all();
    }
    // The copies of the last stages (K/V tiles, queries) land before the CTA exits, also after a timeout, when nobody else
    // waits for them any more: 1 ms at most
    if (ct == 0) {
        const unsigned long long t_begin = global_timer_ns();
        for (int s = 0; s < SG; ++s) {
            stage = stage == 0 ? SG - 1 : stage - 1;
            if (stage == SG - 1) phase ^= 1u;
            while (!mbar_try_wait(&full[stage], phase) && global_timer_ns() - t_begin < 1000000ull) { }
        }
    }
    } else {

    // ---- compute side
    const int wi = warp & 3, hrow = lane >> 2, kq = (lane & 3) * 2;
    constexpr int KS = DH / 16;                              // 16-wide slices of the head dimension
    // ldmatrix row addresses. K: tokens as the operand's n; V (transposed): tokens as its k
    const int ktok = (lane & 7) + ((lane >> 4) << 3), vtok = (lane & 7) + (((lane >> 3) & 1) << 3);
    const uint32_t kbase = (uint32_t)(ktok * 128), ksw = (uint32_t)(ktok & 7), kpc = (uint32_t)((lane >> 3) & 1);
    const uint32_t vbase = (uint32_t)(L::VOFF + vtok * 128), vsw = (uint32_t)(vtok & 7);
    // queries: operand rows 0-7 = high parts, 8-15 = low parts (a head that does not exist repeats the last one: not used)
    const int qh = min(lane & 7, gq - 1);
    const uint32_t qlane = (uint32_t)((((lane >> 3) & 1) * gq + qh) * DH * 2), qsw = (uint32_t)(qh & 7), qpc = (uint32_t)(lane >> 4);
    AttnItem it;
    it.seq = 0;
    int stage = 0, li = 0;
    uint32_t phase = 0;
    auto load_q = [&](int row, int slot, uint32_t (&q)[KS][4]) {
        const uint32_t b = smem_u32(smem + L::O_Q + ((size_t)(grp * NQ + slot) * ROWS + row) * L::QROW) + qlane;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) ldsm4(b + ((((uint32_t)(2 * ks) + qpc) ^ qsw) << 4), q[ks]);
    };
    auto load_k = [&](uint32_t sb, int tile, int ks, uint32_t (&k)[4]) {
        ldsm4(sb + kbase + (uint32_t)(tile * L::BOX + (ks >> 2) * 2048) + ((((uint32_t)(2 * (ks & 3)) + kpc) ^ ksw) << 4), k);
    };
    auto load_v = [&](uint32_t sb, int tile, uint32_t half, uint32_t piece, uint32_t (&v)[4]) {    // 16 head dims from 64 half + 8 piece on
        ldsm4_trans(sb + vbase + (uint32_t)(tile * L::BOX) + half * 2048u + (((piece + (uint32_t)(lane >> 4)) ^ vsw) << 4), v);
    };
    // scores of a tile's 16 tokens: thread: head hrow, tokens nt*8 + kq + {0,1} of the tile
    auto scores = [&](const uint32_t (&q)[KS][4], const uint32_t (&kf)[KS][4], float (&sc)[4]) {
        float s[2][2][4];                                    // [n-tile of 8 tokens][even / odd slices]: four independent chains
#pragma unroll
        for (int i = 0; i < 4; ++i) s[0][0][i] = s[0][1][i] = s[1][0][i] = s[1][1][i] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            mma_bf16_pure(s[0][ks & 1], q[ks][0], q[ks][1], q[ks][2], q[ks][3], kf[ks][0], kf[ks][1]);
            mma_bf16_pure(s[1][ks & 1], q[ks][0], q[ks][1], q[ks][2], q[ks][3], kf[ks][2], kf[ks][3]);
        }
        // hi-part product in [0],[1], lo-part in [2],[3]
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int j = 0; j < 2; ++j) sc[nt * 2 + j] = (s[nt][0][j] + s[nt][1][j]) + (s[nt][0][j + 2] + s[nt][1][j + 2]);
    };
    if constexpr (ROWS == 1) {
    constexpr int NT = DH / 32;                              // 8-wide tiles of this warp's quarter of the head dimension
    float *mx_s = reinterpret_cast<float *>(smem + L::O_RED) + grp * 64, *l_s = mx_s + 32;
    const uint32_t vhalf = (uint32_t)(wi * NT / 8), vpiece = (uint32_t)((wi * NT) & 7);
    // probabilities: [16 operand rows][64 tokens], pieces of 8 tokens swizzled by the row
    const uint32_t pbase = smem_u32(smem + L::O_P) + (uint32_t)(grp * L::PROW);
    const uint32_t plane = (uint32_t)(((lane & 7) + ((lane >> 3) & 1) * 8) * 128), psw = (uint32_t)(lane & 7), ppc = (uint32_t)(lane >> 4);
    const uint32_t pst = pbase + (uint32_t)(hrow * 128 + kq * 2);
    // value rows nothing has written may hold anything: zeros, so that a probability of 0 meets a finite number
    auto clear_values = [&](int tile, int tokens) {
        for (int i = lane; i < (kAttnBox - tokens) * (DH / 8); i += 32) {
            const int tok = tokens + i / (DH / 8), c = i % (DH / 8);
            *reinterpret_cast<uint4 *>(ring + (size_t)stage * L::STAGE + L::VOFF + tile * L::BOX + (c >> 3) * 2048 + tok * 128 + (c & 7) * 16) =
                make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async();                                 // before a later TMA copy overwrites them
    };
    for (int item = worker; item < n_items; item += stride) {
        load_item(it, item);
        if (it.n_blk == 0) continue;
        const int slot = li % NQ;
        ++li;
        uint32_t qa[KS][4];
        float m_run = -INFINITY, l_run = 0.f, o[NT][4];      // o: [0],[1] the hi-part products, [2],[3] the lo-part ones
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
        for (int blk = 0; blk < it.n_blk; ++blk) {
            wait(&full[stage], phase);
            const uint32_t sb = smem_u32(ring + (size_t)stage * L::STAGE);
            const int tb = it.t0 + blk * kAttnBlk, tw = tb + wi * kAttnBox;
            if (blk == 0) load_q(0, slot, qa);
            uint32_t kf[KS][4];
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) load_k(sb, wi, ks, kf[ks]);
            const int over = it.n_ctx - tw;                  // of this warp's 16 tokens, those that exist
            if (over > 0 && over < kAttnBox) clear_values(wi, over);
            float sc[4], mx = -INFINITY;
            scores(qa, kf, sc);
            const bool edge = over < kAttnBox;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (edge && (i >> 1) * 8 + kq + (i & 1) >= over) sc[i] = -INFINITY;
                mx = fmaxf(mx, sc[i]);
            }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            if ((lane & 3) == 0) mx_s[wi * 8 + hrow] = mx;
            if (blk == 0) {                                  // the queries are in registers
                __syncwarp();
                if (lane == 0) mbar_arrive(&qempty[slot]);
            }
            bar_sync(1 + grp, 128);
            const float *mk = mx_s + hrow;
            const float m_new = fmaxf(m_run, fmaxf(fmaxf(mk[0], mk[8]), fmaxf(mk[16], mk[24])));
            const float corr = exp2_fast(m_run - m_new);     // 0 on the item's first block (m_run = -inf)
            float p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = exp2_fast(sc[i] - m_new);
            // each thread keeps its own tokens' share of the sum; the shares are added at the end of the item
            l_run = l_run * corr + ((p[0] + p[1]) + (p[2] + p[3]));
            m_run = m_new;
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                uint32_t hi, lo;
                split2(p[2 * nt], p[2 * nt + 1], hi, lo);
                const uint32_t d = pst + (((uint32_t)(wi * 2 + nt) ^ (uint32_t)hrow) << 4);
                sts32(d, hi);
                sts32(d + 1024, lo);
            }
            if (__any_sync(0xffffffffu, corr != 1.0f)) {
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) { o[nt][0] *= corr; o[nt][1] *= corr; o[nt][2] *= corr; o[nt][3] *= corr; }
            }
            uint32_t vf[4][NT / 2][4];                       // all value fragments are requested before the barrier
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (tb + s * kAttnBox < it.n_ctx) {
#pragma unroll
                    for (int j = 0; j < NT / 2; ++j) load_v(sb, s, vhalf, vpiece + (uint32_t)(2 * j), vf[s][j]);
                }
            bar_sync(1 + grp, 128);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (tb + s * kAttnBox >= it.n_ctx) continue;
                uint32_t pf[4];
                ldsm4(pbase + plane + ((((uint32_t)(2 * s) + ppc) ^ psw) << 4), pf);
#pragma unroll
                for (int j = 0; j < NT / 2; ++j) {
                    mma_bf16_pure(o[2 * j], pf[0], pf[1], pf[2], pf[3], vf[s][j][0], vf[s][j][1]);
                    mma_bf16_pure(o[2 * j + 1], pf[0], pf[1], pf[2], pf[3], vf[s][j][2], vf[s][j][3]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[stage]);        // this warp has read all it needs from the stage
            if (++stage == SG) { stage = 0; phase ^= 1u; }
        }
        // ---- the chunk's partial
        l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
        l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
        if ((lane & 3) == 0) l_s[wi * 8 + hrow] = l_run;
        bar_sync(1 + grp, 128);
        if (hrow < gq) {
            const size_t r = (size_t)it.seq * a.geo.M + it.set;
            float *out = a.att_part + ((r * a.Hq + (size_t)it.kvh * gq + hrow) * a.max_chunks + it.chunk) * (DH + 2);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
                *reinterpret_cast<float2 *>(out + wi * (DH / 4) + nt * 8 + kq) = make_float2(o[nt][0] + o[nt][2], o[nt][1] + o[nt][3]);
            if (wi == 0 && (lane & 3) == 0) {
                const float *lk = l_s + hrow;
                *reinterpret_cast<float2 *>(out + DH) = make_float2(m_run, ((lk[0] + lk[8]) + lk[16]) + lk[24]);
            }
        }
    }
    } else {
    // One warp per row: its scores are its own probabilities' operand (an accumulator's lanes are an A operand's), so nothing
    // is exchanged and the group's warps meet nowhere but at the ring. The other group starts with another warp's
    // scheduler, so that two rows use all four.
    static_assert(ROWS == 4, "one row per warp");
    constexpr int ND = DH / 16;
    const int row = (wi + 2 * grp) & 3;
    for (int item = worker; item < n_items; item += stride) {
        load_item(it, item);
        if (it.n_blk == 0) continue;
        const int slot = li % NQ;
        ++li;
        const int m = it.set * ROWS + row;
        const int n = m < tval[it.seq] ? row_ctx(tpos[it.seq], m) : 0;             // visible positions, 0 for a row that does not exist
        const bool active = n > it.t0;
        uint32_t qa[KS][4];
        float m_run = -INFINITY, l_run[4], o[2 * ND][4];     // l_run: by tile of a block
#pragma unroll
        for (int s = 0; s < 4; ++s) l_run[s] = 0.f;
#pragma unroll
        for (int nt = 0; nt < 2 * ND; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
        for (int blk = 0; blk < it.n_blk; ++blk) {
            wait(&full[stage], phase);
            if (blk == 0) {
                if (active) load_q(row, slot, qa);
                __syncwarp();
                if (lane == 0) mbar_arrive(&qempty[slot]);
            }
            const uint32_t sb = smem_u32(ring + (size_t)stage * L::STAGE);
            const int left = n - (it.t0 + blk * kAttnBlk);   // positions of the block that the row sees
            if (active && left > 0) {
                float sc[4][4], mx = -INFINITY;
#pragma unroll
                for (int s = 0; s < 4; ++s) {                // a tile that was not copied is whatever is there: masked
                    uint32_t kf[KS][4];
#pragma unroll
                    for (int ks = 0; ks < KS; ++ks) load_k(sb, s, ks, kf[ks]);
                    scores(qa, kf, sc[s]);
                }
                if (left < kAttnBlk) {
#pragma unroll
                    for (int s = 0; s < 4; ++s)
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (s * kAttnBox + (i >> 1) * 8 + kq + (i & 1) >= left) sc[s][i] = -INFINITY;
                }
#pragma unroll
                for (int s = 0; s < 4; ++s) mx = fmaxf(mx, fmaxf(fmaxf(sc[s][0], sc[s][1]), fmaxf(sc[s][2], sc[s][3])));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float m_new = fmaxf(m_run, mx);
                const float corr = exp2_fast(m_run - m_new);
                m_run = m_new;
                if (__any_sync(0xffffffffu, corr != 1.0f)) {
#pragma unroll
                    for (int nt = 0; nt < 2 * ND; ++nt) { o[nt][0] *= corr; o[nt][1] *= corr; o[nt][2] *= corr; o[nt][3] *= corr; }
                }
                uint32_t pf[4][4];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    float p[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) p[i] = exp2_fast(sc[s][i] - m_new);
                    l_run[s] = l_run[s] * corr + ((p[0] + p[1]) + (p[2] + p[3]));
                    split2(p[0], p[1], pf[s][0], pf[s][1]);
                    split2(p[2], p[3], pf[s][2], pf[s][3]);
                }
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    if ((s + 1) * kAttnBox > left) break;
#pragma unroll
                    for (int j = 0; j < ND; ++j) {
                        uint32_t v[4];
                        load_v(sb, s, (uint32_t)(j >> 2), (uint32_t)(2 * (j & 3)), v);
                        mma_bf16_pure(o[2 * j], pf[s][0], pf[s][1], pf[s][2], pf[s][3], v[0], v[1]);
                        mma_bf16_pure(o[2 * j + 1], pf[s][0], pf[s][1], pf[s][2], pf[s][3], v[2], v[3]);
                    }
                }
                if (left < kAttnBlk && (left & (kAttnBox - 1))) {
                    // the tile in which the row's context ends: what lies beyond is another row's value, or what an unwritten
                    // slot holds, and need not be finite. A probability of 0 meets a 0 there
                    const int s = left / kAttnBox, seen = left & (kAttnBox - 1);
                    const uint32_t keep0 = (kq < seen ? 0xffffu : 0u) | (kq + 1 < seen ? 0xffff0000u : 0u);
                    const uint32_t keep1 = (kq + 8 < seen ? 0xffffu : 0u) | (kq + 9 < seen ? 0xffff0000u : 0u);
                    uint32_t pe[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) pe[i] = s == 0 ? pf[0][i] : s == 1 ? pf[1][i] : s == 2 ? pf[2][i] : pf[3][i];
#pragma unroll
                    for (int j = 0; j < ND; ++j) {
                        uint32_t v[4];
                        load_v(sb, s, (uint32_t)(j >> 2), (uint32_t)(2 * (j & 3)), v);
                        mma_bf16_pure(o[2 * j], pe[0], pe[1], pe[2], pe[3], v[0] & keep0, v[1] & keep1);
                        mma_bf16_pure(o[2 * j + 1], pe[0], pe[1], pe[2], pe[3], v[2] & keep0, v[3] & keep1);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[stage]);        // this warp has read all it needs from the stage
            if (++stage == SG) { stage = 0; phase ^= 1u; }
        }
        if (!active) continue;
        // ---- the chunk's partial of the row
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            l_run[s] += __shfl_xor_sync(0xffffffffu, l_run[s], 1);
            l_run[s] += __shfl_xor_sync(0xffffffffu, l_run[s], 2);
        }
        if (hrow < gq) {
            const size_t r = (size_t)it.seq * a.geo.M + m;
            float *out = a.att_part + ((r * a.Hq + (size_t)it.kvh * gq + hrow) * a.max_chunks + it.chunk) * (DH + 2);
#pragma unroll
            for (int nt = 0; nt < 2 * ND; ++nt)
                *reinterpret_cast<float2 *>(out + nt * 8 + kq) = make_float2(o[nt][0] + o[nt][2], o[nt][1] + o[nt][3]);
            if ((lane & 3) == 0) *reinterpret_cast<float2 *>(out + DH) = make_float2(m_run, ((l_run[0] + l_run[1]) + l_run[2]) + l_run[3]);
        }
    }
    }
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicOr(a.status, 0x8u);
}

// ---- combine a head's chunk partials in ascending order; write the O-projection's operand.
struct MergeArgs {
    int Hq, dh, page, max_ctx, max_chunks, ld;
    RowGeo geo;
    KvPtrs kv;
    const float *att_part;
    bf16_t *xop;
};

// A warp's lanes hold the chunks' maxima and sums, 32 chunks at a time, and
// the chunks' values are requested before the maxima are known, so a row of up to 8192 positions is one round trip to L2
// (eight chunks at a time behind a block-wide maximum took 12.5 us at 64 rows with contexts in [512, 8192] and 8.2 us at
// four rows of 500 to 3000; draft call of five steps at the latter 781 -> 770 us). G: chunks whose values are in flight.
template <int G>
__device__ __forceinline__ float merge_chunks(const float *base, int n_chunks, int stride, int dh, int j) {
    const int lane = threadIdx.x & 31;
    float v[G];
    auto load_values = [&](int c0) {
#pragma unroll
        for (int u = 0; u < G; ++u) v[u] = c0 + u < n_chunks ? base[(size_t)(c0 + u) * stride + j] : 0.f;
    };
    load_values(0);
    float m = -INFINITY;
    for (int c = lane; c < n_chunks; c += 32) m = fmaxf(m, base[(size_t)c * stride + dh]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    // weighted sums in ascending chunk order; the denominator adds each group of 32 by a fixed tree
    float acc = 0.f, l = 0.f;
    for (int c0 = 0; c0 < n_chunks; c0 += 32) {
        const int c = c0 + lane;
        const float w = c < n_chunks ? exp2f(base[(size_t)c * stride + dh] - m) : 0.f;
        float lw = c < n_chunks ? base[(size_t)c * stride + dh + 1] * w : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o);
        l += lw;
        if (c0 > 0) load_values(c0);
#pragma unroll
        for (int u = 0; u < G; ++u) acc += v[u] * __shfl_sync(0xffffffffu, w, u);
    }
    return acc / l;
}

// Block = (head, row), a thread per output element.
__global__ void attn_merge_kernel(const MergeArgs a) {
    chain_release();
    const int head = blockIdx.x, r = blockIdx.y, j = threadIdx.x;
    const int max_tokens = min(a.kv.max_pages * a.page, a.max_ctx);
    bool valid;
    const int n_ctx = min(geo_pos(a.geo, a.kv, r, &valid), max_tokens - 1) + 1;
    chain_wait();
    if (!valid) {                // padding row: attention skipped it
        store_hilo(a.xop, a.ld, r, head * a.dh + j, 0.f);
        return;
    }
    const int n_chunks = (n_ctx + kBatchAttnChunk - 1) / kBatchAttnChunk;
    const int stride = a.dh + 2;
    const float *base = a.att_part + ((size_t)r * a.Hq + head) * a.max_chunks * stride;
    const float o = n_chunks <= 8 ? merge_chunks<8>(base, n_chunks, stride, a.dh, j) : merge_chunks<32>(base, n_chunks, stride, a.dh, j);
    store_hilo(a.xop, a.ld, r, head * a.dh + j, o);
}

// ---- target step input: x = Emb(token) per row (fp32 residual stream). One block per row.
__global__ void __launch_bounds__(kRowThreads) embed_kernel(const int32_t *tokens, const bf16_t *embed, int d, int V, float *x,
                                                            uint32_t *status) {
    chain_release();
    chain_wait();
    const int r = blockIdx.x;
    int tok = tokens[r];
    if ((unsigned)tok >= (unsigned)V) { if (threadIdx.x == 0) atomicOr(status, kDevBadToken); tok = 0; }
    const bf16_t *erow = embed + (size_t)tok * d;
    for (int j = threadIdx.x * 8; j < d; j += kRowThreads * 8) {
        float e[8];
        unpack_bf16x8(*reinterpret_cast<const uint4 *>(erow + j), e);
        *reinterpret_cast<float4 *>(x + (size_t)r * d + j) = make_float4(e[0], e[1], e[2], e[3]);
        *reinterpret_cast<float4 *>(x + (size_t)r * d + j + 4) = make_float4(e[4], e[5], e[6], e[7]);
    }
}

// ---- the subset in ascending id order. The argmax over the subset does not depend on the order of
// its rows, and gathering head rows in address order keeps the 128 rows of a GEMM tile within a few
// memory pages (an unsorted subset spreads them over the whole matrix and the address translation
// misses cost ~25 % of the head's stream rate). Membership bitmap, then a one-block compaction.
// (The two kernels stand before step 0: its first kernel waits for them as for any predecessor, and only its launch and the first
// weight copies of the projection overlap them. The head GEMM, the only reader of the sorted ids, waits for the whole
// chain before it looks at them.)
__global__ void ids_mark_kernel(const int32_t *ids, int N, int V, uint32_t *bitmap, uint32_t *status) {
    chain_release();
    chain_wait();
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
        int id = ids[j];
        if ((unsigned)id >= (unsigned)V) { atomicOr(status, kDevBadToken); id = 0; }
        atomicOr(&bitmap[id >> 5], 1u << (id & 31));
    }
}

// Compaction of the membership bitmap into ascending ids. Block b owns a contiguous range of bitmap words; the
// number of ids before its range is the population count of all earlier words, which every block sums for itself
// (the whole bitmap is 19 KB at V = 152064), so no block waits for another. Duplicates in the caller's array leave
// fewer distinct ids than N: the tail repeats `fill` (a member of the subset; a repeated row cannot change an argmax).
constexpr int kCompactThreads = 256;
__global__ void __launch_bounds__(kCompactThreads) ids_compact_kernel(const uint32_t *bitmap, int n_words, int32_t *sorted, int N,
                                                                      const int32_t *ids, int V) {
    chain_release();
    chain_wait();
    __shared__ int wsum[kCompactThreads / 32];
    __shared__ int s_base, s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w0 = (int)(((long long)blockIdx.x * n_words) / gridDim.x), w1 = (int)(((long long)(blockIdx.x + 1) * n_words) / gridDim.x);
    // ids before this block's words, and in the whole bitmap
    int before = 0, all = 0;
    for (int w = tid; w < n_words; w += kCompactThreads) {
        const int c = __popc(bitmap[w]);
        all += c;
        if (w < w0) before += c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { before += __shfl_xor_sync(0xffffffffu, before, o); all += __shfl_xor_sync(0xffffffffu, all, o); }
    if (lane == 0) wsum[warp] = before;
    __syncthreads();
    if (tid == 0) { int t = 0; for (int w = 0; w < kCompactThreads / 32; ++w) t += wsum[w]; s_base = t; }
    __syncthreads();
    if (lane == 0) wsum[warp] = all;
    __syncthreads();
    if (tid == 0) { int t = 0; for (int w = 0; w < kCompactThreads / 32; ++w) t += wsum[w]; s_total = t; }
    __syncthreads();
    // this block's words: one word per thread and round, exclusive scan of the counts within the block
    int run = s_base;
    for (int r0 = w0; r0 < w1; r0 += kCompactThreads) {
        const int w = r0 + tid;
        uint32_t bits = w < w1 ? bitmap[w] : 0u;
        const int cnt = __popc(bits);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        __syncthreads();
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int base = run;
        for (int q = 0; q < warp; ++q) base += wsum[q];
        int pos = base + incl - cnt;
        while (bits) {
            const int b = __ffs(bits) - 1;
            bits &= bits - 1;
            if (pos < N) sorted[pos] = w * 32 + b;
            ++pos;
        }
        for (int q = 0; q < kCompactThreads / 32; ++q) run += wsum[q];
    }
    if (blockIdx.x == 0) {
        int fill = ids[0];
        if ((unsigned)fill >= (unsigned)V) fill = 0;
        for (int j = min(s_total, N) + tid; j < N; j += kCompactThreads) sorted[j] = fill;
    }
}

// Tensor map of a paged K or V pool seen as rows of head_dim values: a copy brings 16 rows as [dh / 64][16][64], each
// 128-byte row swizzled. Encoded per call (a host computation): the pool is the caller's.
int attn_encode_map(CUtensorMap *map, const bf16_t *pool, const BatchedShape &sh, int num_pages) {
    TmapEncodeFn encode;
    if (int rc = tmap_encoder(&encode)) return rc;
    const cuuint64_t dims[3] = {64, (cuuint64_t)num_pages * sh.Hkv * sh.page, (cuuint64_t)(sh.dh / 64)};
    const cuuint64_t strides[2] = {(cuuint64_t)sh.dh * 2, 128};
    const cuuint32_t box[3] = {64, kAttnBox, (cuuint32_t)(sh.dh / 64)};
    const cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16_t *>(pool), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : (int)cudaErrorInvalidValue;
}

template <int DH, int ROWS>
int attn_launch(const AttnArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int n_sm, TmapCache *cache, cudaStream_t st) {
    bool &raised = cache->attn_raised[ROWS > 1];
    if (!raised) {                                // once per context (every context of this kernel sets the same limit)
        cudaError_t e = cudaFuncSetAttribute(attn_kernel<DH, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<DH, ROWS>::TOTAL);
        if (e != cudaSuccess) return (int)e;
        raised = true;
    }
    return (int)launch_chained(attn_kernel<DH, ROWS>, dim3(n_sm), dim3(kAttnThreads), (size_t)AttnSmem<DH, ROWS>::TOTAL, st, a, kmap, vmap);
}

// Attention and chunk merge of a pass over `rows` rows (geo.M per sequence).
int attention(const BatchedShape &sh, const BatchedWs &ws, const KvPtrs &kv, const RowGeo &geo, int rows, int n_sm,
              unsigned long long wait_limit_ns, int extra_arrivals, TmapCache *cache, cudaStream_t st, long long *launches) {
    AttnArgs a{};
    a.extra_arrivals = extra_arrivals;
    a.Hq = sh.Hq; a.Hkv = sh.Hkv; a.dh = sh.dh; a.page = sh.page; a.max_ctx = sh.max_ctx; a.geo = geo;
    a.max_chunks = ws.max_chunks; a.q = ws.q; a.kv = kv; a.att_part = ws.att_part; a.status = ws.status;
    a.B = rows / geo.M; a.wait_limit_ns = wait_limit_ns;
    a.tma = sh.page % kAttnBox == 0 && (long long)kv.num_pages * sh.Hkv * sh.page < (1ll << 31);
    CUtensorMap kmap{}, vmap{};
    int rc = 0;
    if (a.tma) {
        if ((rc = attn_encode_map(&kmap, kv.k_pages, sh, kv.num_pages))) return rc;
        if ((rc = attn_encode_map(&vmap, kv.v_pages, sh, kv.num_pages))) return rc;
    }
    if (geo.M > 1) rc = sh.dh == 128 ? attn_launch<128, kAttnRows>(a, kmap, vmap, n_sm, cache, st) : attn_launch<64, kAttnRows>(a, kmap, vmap, n_sm, cache, st);
    else rc = sh.dh == 128 ? attn_launch<128, 1>(a, kmap, vmap, n_sm, cache, st) : attn_launch<64, 1>(a, kmap, vmap, n_sm, cache, st);
    if (rc) return rc;
    MergeArgs m{};
    m.Hq = sh.Hq; m.dh = sh.dh; m.page = sh.page; m.max_ctx = sh.max_ctx; m.geo = geo; m.max_chunks = ws.max_chunks;
    m.ld = ws.ld0; m.kv = kv; m.att_part = ws.att_part; m.xop = ws.xop0;
    *launches += 2;
    return (int)launch_chained(attn_merge_kernel, dim3(sh.Hq, rows), dim3(sh.dh), 0, st, m);
}

// The row-wise kernels by how many groups of eight columns a thread owns (d <= 4096 / 8192 / 24576).
int launch_prologue(const PrologueArgs &a, int rows, cudaStream_t st) {
    auto kern = a.d <= kRowThreads * 8 ? prologue_kernel<1> : a.d <= kRowThreads * 16 ? prologue_kernel<2> : prologue_kernel<6>;
    return a.d <= kRowThreads * 48 ? (int)launch_chained(kern, dim3(rows), dim3(kRowThreads), 0, st, a) : (int)cudaErrorInvalidConfiguration;
}
int launch_post(const PostArgs &a, int rows, cudaStream_t st) {
    auto kern = a.d <= kRowThreads * 8 ? post_kernel<1> : a.d <= kRowThreads * 16 ? post_kernel<2> : post_kernel<6>;
    return a.d <= kRowThreads * 48 ? (int)launch_chained(kern, dim3(rows), dim3(kRowThreads), 0, st, a) : (int)cudaErrorInvalidConfiguration;
}

int pick_splits(int n_tiles, int n_kb, int n_sm) {
    int best = 1;
    double best_eff = 0.0;
    for (int s = 1; s <= kBatchMaxSplits; ++s) {
        if (s > 1 && n_kb / s < 8) break;
        const int items = n_tiles * s;
        const int waves = (items + n_sm - 1) / n_sm;
        const double eff = (double)items / ((double)waves * n_sm);
        if (eff > best_eff + 0.02) { best_eff = eff; best = s; }
    }
    return best;
}

// Rows and K ranges of a GEMM's work items; a function of the matrix and the SM count only, never of the batch.
void pick_items(GemmArgs &g, int n_sm) {
    const int n_kb = (g.K + kGemmBK - 1) / kGemmBK;
    g.splits = 1;
    g.item_rows = kGemmTileM;
    g.n_ranges = 0;
    if (g.epi == EPI_ARGMAX) {
        // equal shares of the rows in the fewest rounds over the SMs
        const int most = 2 * kGemmTileM, rounds = (g.n_rows + most * n_sm - 1) / (most * n_sm);
        g.item_rows = ((g.n_rows + rounds * n_sm - 1) / (rounds * n_sm) + 7) / 8 * 8;
        g.n_ranges = (g.n_rows + g.item_rows - 1) / g.item_rows;
    } else {
        for (int s = 0; s < g.n_seg; ++s) g.n_ranges += (g.a_rows[s] + g.item_rows - 1) / g.item_rows;
        if (g.epi == EPI_PARTIAL) g.splits = pick_splits(g.n_ranges, n_kb, n_sm);
    }
    g.kb_per_split = (n_kb + g.splits - 1) / g.splits;
    g.splits = (n_kb + g.kb_per_split - 1) / g.kb_per_split;      // no empty range
}

}  // namespace

size_t batched_layout(BatchedWs &ws, unsigned char *base, const BatchedShape &sh) {
    const int rows = sh.max_rows < kBatchRows ? sh.max_rows : kBatchRows;
    const int qdim = sh.Hq * sh.dh, kvdim = sh.Hkv * sh.dh;
    const int widest_in = 2 * sh.d > qdim ? 2 * sh.d : qdim;
    const int widest_out = sh.d > qdim + 2 * kvdim ? sh.d : qdim + 2 * kvdim;
    ws.rows = rows;
    ws.ld0 = (int)align_up((size_t)widest_in, 64);
    ws.ldF = (int)align_up((size_t)sh.F, 64);
    ws.ldp = (int)align_up((size_t)widest_out, 128);
    ws.max_chunks = (sh.max_ctx + kBatchAttnChunk - 1) / kBatchAttnChunk;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = align_up(off, 256);
        unsigned char *p = base ? base + off : nullptr;
        off += bytes;
        return p;
    };
    ws.xop0 = reinterpret_cast<bf16_t *>(take((size_t)128 * ws.ld0 * 2));
    ws.xopF = reinterpret_cast<bf16_t *>(take((size_t)128 * ws.ldF * 2));
    ws.xopH = reinterpret_cast<bf16_t *>(take((size_t)128 * ws.ld0 * 2));
    ws.partial = reinterpret_cast<float *>(take((size_t)kBatchMaxSplits * rows * ws.ldp * 4));
    ws.x = reinterpret_cast<float *>(take((size_t)rows * sh.d * 4));
    ws.hout = reinterpret_cast<float *>(take((size_t)rows * sh.d * 4));
    ws.q = reinterpret_cast<bf16_t *>(take((size_t)rows * 2 * qdim * 2));
    ws.att_part = reinterpret_cast<float *>(take((size_t)rows * sh.Hq * ws.max_chunks * (sh.dh + 2) * 4));
    ws.keys_bytes = (size_t)(sh.max_K > 1 ? sh.max_K : 1) * kBatchRows * 8 + 256;
    ws.keys = reinterpret_cast<unsigned long long *>(take(ws.keys_bytes));
    ws.id_bitmap = reinterpret_cast<uint32_t *>(take((size_t)((sh.V + 31) / 32) * 4));
    ws.sorted_ids = reinterpret_cast<int32_t *>(take((size_t)sh.V * 4));
    ws.status = reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned char *>(ws.keys) + ws.keys_bytes - 256);
    if (!base) ws.status = nullptr;
    return align_up(off, 256);
}

int batched_draft(const BatchedCall &c, cudaStream_t st, long long *launches) {
    const BatchedShape &sh = c.sh;
    const BatchedWs &ws = c.ws;
    const int B = c.B, K = c.K, d = sh.d;
    const int M0 = c.M0 > 1 ? c.M0 : 1;
    const bool ext = M0 > 1;                       // step 0 carries up to M0 extend rows per sequence
    int inject_gemm = c.inject == 2 ? 1 : 0, inject_attn = c.inject == 3 ? 1 : 0;      // self-test: one launch each
    const int qdim = sh.Hq * sh.dh, kvdim = sh.Hkv * sh.dh;
    // Argmax keys and the status word. A memset is a full dependency on the stream's earlier work, the one that makes it safe for
    // the call's kernels, which release each other at their first instruction, to read the call's inputs (hidden states,
    // lengths, block table, cached K/V, weights) before they wait for their predecessor: something of this kind has to stay first.
    cudaError_t e = cudaMemsetAsync(ws.keys, 0, ws.keys_bytes, st);
    if (e != cudaSuccess) return (int)e;

    // head rows in ascending id order (the debug logits keep the caller's order, so they skip this)
    const int32_t *head_ids = c.ids;
    if (c.ids && !c.out_logits) {
        const int n_words = (sh.V + 31) / 32;
        e = cudaMemsetAsync(ws.id_bitmap, 0, (size_t)n_words * 4, st);
        if (e != cudaSuccess) return (int)e;
        e = launch_chained(ids_mark_kernel, dim3((c.N + 255) / 256 < 1024 ? (c.N + 255) / 256 : 1024), dim3(256), 0, st, c.ids, c.N, sh.V,
                           ws.id_bitmap, ws.status);
        if (e == cudaSuccess) e = launch_chained(ids_compact_kernel, dim3(32), dim3(kCompactThreads), 0, st, ws.id_bitmap, n_words, ws.sorted_ids, c.N, c.ids, sh.V);
        *launches += 2;
        if (e != cudaSuccess) return (int)e;
        head_ids = ws.sorted_ids;
    }

    auto gemm = [&](GemmArgs &g, int rows, int n_rows, int Kdim, int lda, const bf16_t *x, int ldx) -> int {
        g.n_rows = n_rows; g.K = Kdim; g.lda = lda; g.x = x; g.ldx = ldx; g.NB = (2 * rows + 15) / 16 * 16; g.R = rows;
        g.status = ws.status;
        g.wait_limit_ns = c.wait_limit_ns;
        g.extra_arrivals = inject_gemm;
        inject_gemm = 0;
        pick_items(g, c.n_sm);
        g.partial = ws.partial; g.ldp = ws.ldp;
        ++*launches;
        return skinny_gemm_launch(g, c.n_sm, c.smem_optin, st, c.cache);
    };
    int rc = 0;

    // One pass of the MTP module (projection, decoder layer, final norm) over `rows` activation rows of the sequences
    // seq0 .. seq0 + rows / geo.M - 1 of the group. The final norm publishes into `xop_head` (the output head's operand),
    // hout and out_h, under the row's own index or, in an extend pass, under its sequence's.
    auto mtp_pass = [&](int step, int rows, int seq0, const RowGeo &geo, bf16_t *xop_head, int map_out) -> int {
        KvPtrs kv = c.kv;
        kv.block_table += (size_t)seq0 * kv.max_pages;
        kv.seq_lens += seq0;
        auto post = [&](int splits, int residual, int final, const bf16_t *gain) -> int {
            PostArgs a{};
            a.d = d; a.splits = splits; a.rows = rows; a.ldp = ws.ldp; a.ld = ws.ld0; a.residual = residual; a.final = final;
            a.K = K; a.step = step; a.eps = sh.eps; a.partial = ws.partial; a.x = ws.x; a.hout = ws.hout;
            a.out_h = c.out_h; a.gain = gain; a.xop = final ? xop_head : ws.xop0;
            a.map_out = final ? map_out : 0; a.seq0 = seq0; a.geo = geo;
            ++*launches;
            return launch_post(a, rows, st);
        };
        PrologueArgs pa{};
        pa.step = step; pa.K = K; pa.d = d; pa.V = sh.V; pa.ld = ws.ld0; pa.only_tokens = 0; pa.geo = geo;
        pa.eps = sh.eps; pa.h_last = c.h_last + (size_t)seq0 * M0 * d; pa.tok_last = c.tok_last + (size_t)seq0 * M0; pa.hout = ws.hout;
        pa.keys_prev = step > 0 ? ws.keys + (size_t)(step - 1) * kBatchRows : nullptr;
        pa.out_drafts = c.out_drafts; pa.embed = c.embed; pa.g_h = c.g_hnorm; pa.g_e = c.g_enorm;
        pa.xop = ws.xop0; pa.status = ws.status; pa.user_status = c.user_status;
        ++*launches;
        int rc = 0;
        if ((rc = launch_prologue(pa, rows, st))) return rc;
        GemmArgs g{};
        // x = W_p [rms(h); rms(e)]
        g.a[0] = c.w_proj; g.a_rows[0] = d; g.n_seg = 1; g.epi = EPI_PARTIAL;
        if ((rc = gemm(g, rows, d, 2 * d, 2 * d, ws.xop0, ws.ld0))) return rc;
        if ((rc = post(g.splits, 0, 0, c.layer.g_in))) return rc;
        // q, k, v
        g = GemmArgs{};
        g.a[0] = c.layer.wq; g.a[1] = c.layer.wk; g.a[2] = c.layer.wv;
        g.a_rows[0] = qdim; g.a_rows[1] = kvdim; g.a_rows[2] = kvdim; g.n_seg = 3; g.epi = EPI_PARTIAL;
        if ((rc = gemm(g, rows, qdim + 2 * kvdim, d, d, ws.xop0, ws.ld0))) return rc;
        {
            QkvArgs a{};
            a.qdim = qdim; a.kvdim = kvdim; a.dh = sh.dh; a.Hq = sh.Hq; a.Hkv = sh.Hkv; a.splits = g.splits; a.rows = rows;
            a.ldp = ws.ldp; a.page = sh.page; a.max_ctx = sh.max_ctx; a.geo = geo; a.partial = ws.partial; a.q = ws.q;
            a.kv = kv; a.rope_cos = c.rope_cos; a.rope_sin = c.rope_sin; a.status = ws.status;
            ++*launches;
            if ((rc = (int)launch_chained(qkv_finish_kernel, dim3(sh.Hq + 2 * sh.Hkv, rows), dim3(sh.dh / 2), 0, st, a))) return rc;
        }
        if ((rc = attention(sh, ws, kv, geo, rows, c.n_sm, c.wait_limit_ns, inject_attn, c.cache, st, launches))) return rc;
        inject_attn = 0;
        // x += W_o o
        g = GemmArgs{};
        g.a[0] = c.layer.wo; g.a_rows[0] = d; g.n_seg = 1; g.epi = EPI_PARTIAL;
        g.ahead[0] = c.layer.w_gate; g.ahead[1] = c.layer.w_up; g.ahead_rows = sh.F; g.ahead_ld = d; g.ahead_limit = gemm_ahead_limit(c.ahead_budget, sh.F);
        if ((rc = gemm(g, rows, d, qdim, qdim, ws.xop0, ws.ld0))) return rc;
        if ((rc = post(g.splits, 1, 0, c.layer.g_post))) return rc;
        // act = silu(W_gate n) * (W_up n), written as the down projection's operand
        g = GemmArgs{};
        g.a[0] = c.layer.w_gate; g.a_up = c.layer.w_up; g.a_rows[0] = sh.F; g.n_seg = 1; g.epi = EPI_SWIGLU;
        g.xop_out = ws.xopF; g.ld_out = ws.ldF;
        if ((rc = gemm(g, rows, sh.F, d, d, ws.xop0, ws.ld0))) return rc;
        // x += W_down act; h_out = rms(x; g_final)
        g = GemmArgs{};
        g.a[0] = c.layer.w_down; g.a_rows[0] = d; g.n_seg = 1; g.epi = EPI_PARTIAL;
        if ((rc = gemm(g, rows, d, sh.F, sh.F, ws.xopF, ws.ldF))) return rc;
        return post(g.splits, 1, 1, c.g_final);
    };

    for (int step = 0; step < K; ++step) {
        const bf16_t *xop_head = ws.xop0;
        if (step == 0 && ext) {
            // extend rows: whole sequences in passes of up to 64 rows; each pass streams the module's weights once and
            // publishes its sequences' last rows into the head's operand, so the output head runs once for the group
            const int Gs = kBatchRows / M0;
            for (int s0 = 0; s0 < B; s0 += Gs) {
                const int Bs = B - s0 < Gs ? B - s0 : Gs;
                const RowGeo geo{M0, M0, 0, c.n_ext ? c.n_ext + s0 : nullptr};
                if ((rc = mtp_pass(0, Bs * M0, s0, geo, ws.xopH, 1))) return rc;
            }
            xop_head = ws.xopH;
        } else {
            const RowGeo geo{1, M0, step, c.n_ext};
            if ((rc = mtp_pass(step, B, 0, geo, ws.xop0, 0))) return rc;
        }
        // compressed head + argmax (Eq. 3)
        GemmArgs g{};
        g.a[0] = c.lm_head; g.a_rows[0] = c.N; g.n_seg = 1; g.epi = EPI_ARGMAX;
        g.row_ids = head_ids; g.V = sh.V;
        g.keys = ws.keys + (size_t)step * kBatchRows;
        g.logits = c.out_logits ? c.out_logits + (size_t)step * c.N : nullptr;
        g.logits_stride = (long long)K * c.N;
        if ((rc = gemm(g, B, c.N, d, d, xop_head, ws.ld0))) return rc;
    }
    // the last step's argmax keys -> draft tokens; status word -> caller
    PrologueArgs pa{};
    pa.step = K; pa.K = K; pa.d = d; pa.V = sh.V; pa.ld = ws.ld0; pa.only_tokens = 1; pa.geo = RowGeo{1, M0, K, c.n_ext};
    pa.eps = sh.eps; pa.keys_prev = ws.keys + (size_t)(K - 1) * kBatchRows;
    pa.out_drafts = c.out_drafts; pa.status = ws.status; pa.user_status = c.user_status;
    ++*launches;
    return launch_prologue(pa, B, st);
}

int batched_target(const BatchedTargetCall &c, cudaStream_t st, long long *launches) {
    const BatchedShape &sh = c.sh;
    const BatchedWs &ws = c.ws;
    const int R = c.B * c.M, d = sh.d;
    const int qdim = sh.Hq * sh.dh, kvdim = sh.Hkv * sh.dh;
    const int NB = (2 * R + 15) / 16 * 16;
    const RowGeo geo{c.M, c.M, 0, nullptr};       // M rows per sequence at positions L .. L+M-1, all of them real
    // argmax keys and the status word; also the full dependency that the reads ahead of a wait rely on (see batched_draft)
    cudaError_t e = cudaMemsetAsync(ws.keys, 0, ws.keys_bytes, st);
    if (e != cudaSuccess) return (int)e;
    auto gemm = [&](GemmArgs &g, int n_rows, int Kdim, int lda, const bf16_t *x, int ldx) -> int {
        g.n_rows = n_rows; g.K = Kdim; g.lda = lda; g.x = x; g.ldx = ldx; g.NB = NB; g.R = R;
        g.status = ws.status;
        g.wait_limit_ns = c.wait_limit_ns;
        pick_items(g, c.n_sm);
        g.partial = ws.partial; g.ldp = ws.ldp;
        ++*launches;
        return skinny_gemm_launch(g, c.n_sm, c.smem_optin, st, c.cache);
    };
    auto post = [&](int splits, int final, const bf16_t *gain) -> int {
        PostArgs a{};
        a.d = d; a.splits = splits; a.rows = R; a.ldp = ws.ldp; a.ld = ws.ld0; a.residual = 1; a.final = final;
        a.K = 1; a.step = 0; a.eps = sh.eps; a.partial = ws.partial; a.x = ws.x; a.hout = ws.hout;
        a.out_h = c.out_h; a.gain = gain; a.xop = ws.xop0;
        ++*launches;
        return launch_post(a, R, st);
    };
    int rc = 0;

    // x = Emb(tokens); operand of the first layer = rms(x; g_in)
    ++*launches;
    if ((rc = (int)launch_chained(embed_kernel, dim3(R), dim3(kRowThreads), 0, st, c.tokens, c.embed, d, sh.V, ws.x, ws.status))) return rc;
    if ((rc = post(0, 0, c.layers[0].g_in))) return rc;
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerPtrs &L = c.layers[l];
        const KvPtrs &kv = c.kvs[l];
        GemmArgs g{};
        g.a[0] = L.wq; g.a[1] = L.wk; g.a[2] = L.wv;
        g.a_rows[0] = qdim; g.a_rows[1] = kvdim; g.a_rows[2] = kvdim; g.n_seg = 3; g.epi = EPI_PARTIAL;
        if ((rc = gemm(g, qdim + 2 * kvdim, d, d, ws.xop0, ws.ld0))) return rc;
        {
            QkvArgs a{};
            a.qdim = qdim; a.kvdim = kvdim; a.dh = sh.dh; a.Hq = sh.Hq; a.Hkv = sh.Hkv; a.splits = g.splits; a.rows = R;
            a.ldp = ws.ldp; a.page = sh.page; a.max_ctx = sh.max_ctx; a.geo = geo; a.partial = ws.partial; a.q = ws.q;
            a.kv = kv; a.rope_cos = c.rope_cos; a.rope_sin = c.rope_sin; a.status = ws.status;
            ++*launches;
            if ((rc = (int)launch_chained(qkv_finish_kernel, dim3(sh.Hq + 2 * sh.Hkv, R), dim3(sh.dh / 2), 0, st, a))) return rc;
        }
        if ((rc = attention(sh, ws, kv, geo, R, c.n_sm, c.wait_limit_ns, 0, c.cache, st, launches))) return rc;
        g = GemmArgs{};
        g.a[0] = L.wo; g.a_rows[0] = d; g.n_seg = 1; g.epi = EPI_PARTIAL;
        g.ahead[0] = L.w_gate; g.ahead[1] = L.w_up; g.ahead_rows = sh.F; g.ahead_ld = d; g.ahead_limit = gemm_ahead_limit(c.ahead_budget, sh.F);
        if ((rc = gemm(g, d, qdim, qdim, ws.xop0, ws.ld0))) return rc;
        if ((rc = post(g.splits, 0, L.g_post))) return rc;
        g = GemmArgs{};
        g.a[0] = L.w_gate; g.a_up = L.w_up; g.a_rows[0] = sh.F; g.n_seg = 1; g.epi = EPI_SWIGLU;
        g.xop_out = ws.xopF; g.ld_out = ws.ldF;
        if ((rc = gemm(g, sh.F, d, d, ws.xop0, ws.ld0))) return rc;
        g = GemmArgs{};
        g.a[0] = L.w_down; g.a_rows[0] = d; g.n_seg = 1; g.epi = EPI_PARTIAL;
        if ((rc = gemm(g, d, sh.F, sh.F, ws.xopF, ws.ldF))) return rc;
        const bool last = l + 1 == c.n_layers;
        if ((rc = post(g.splits, last ? 1 : 0, last ? c.g_final : c.layers[l + 1].g_in))) return rc;
    }
    if (c.out_logits || c.out_argmax) {
        // full output head; the greedy choice is made on the bf16-rounded logits a caller would see
        GemmArgs g{};
        g.a[0] = c.lm_head; g.a_rows[0] = sh.V; g.n_seg = 1; g.epi = EPI_ARGMAX; g.V = sh.V;
        g.keys = c.out_argmax ? ws.keys : nullptr;
        g.round_bf16 = 1; g.logits_bf16 = c.out_logits; g.logits_stride = sh.V;
        if ((rc = gemm(g, sh.V, d, d, ws.xop0, ws.ld0))) return rc;
    }
    // argmax keys -> token ids (if asked for), status word -> caller
    PrologueArgs pa{};
    pa.step = 1; pa.K = 1; pa.d = d; pa.V = sh.V; pa.ld = ws.ld0; pa.only_tokens = 1; pa.eps = sh.eps;
    pa.geo = geo;
    pa.keys_prev = ws.keys; pa.out_drafts = c.out_argmax; pa.status = ws.status; pa.user_status = c.user_status;
    ++*launches;
    return launch_prologue(pa, R, st);
}

}  // namespace fmtp
