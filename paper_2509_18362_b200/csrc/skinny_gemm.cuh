// Weight-streaming GEMM for 5..64 activation rows on the sm_100a tensor cores (tcgen05 + TMEM).
//
//   D[m, n] = sum_k A[m, k] * X[n, k]      m: weight rows (128 per tile, the MMA's M)
//                                          n: activation columns (NB = 16..128, the MMA's N)
//
// The weight matrix is read exactly once from HBM; the activation operand X (bf16, row n = 2r is
// the high part of activation row r and n = 2r + 1 the low part, so the pair carries an fp32
// value) is small and re-read from L2 for every item. One CTA per SM walks a static list of work
// items (row range, K range). Roles: warps 0-3 epilogue (TMEM -> registers -> global), warp 4 issues
// the MMAs, warp 5 the TMA tile copies of X, warp 14 see GemmArgs::ahead, warps 6-13 copy A with 16-byte cp.async, laid out as the MMA's
// 128-byte-swizzled K-major tiles (64 K elements wide). Accumulators are double buffered in TMEM so the epilogue of one
// item overlaps the MMAs of the next; in the epilogue of the last item the copy warps help.
//
// What bounds it: HBM, plus the wait for the first X block and the last item's epilogue of every launch (3584-wide layer:
// gate/up 40 us at 4 rows, 46 at 64 for 272 MB, 41.5 us at a plain copy's rate; down 20 and 23 for 136 MB). At 64 activation
// rows it was the weight bytes in flight: with A and X in one ring, half of the memory held X and 96 KB of weights were
// requested ahead per SM (gate/up 59 us). So A and X have rings of their own (128-160 KB for A; 56 us), an item of gate/up
// or of the output head has two tiles that share every X block, and the epilogue is cut short (see there). The split-K
// matrices have too few rows for two tiles.
// A stage is KA K blocks: four while three weight stages of that size fit, else two. Finer stages lose: a wait on a barrier
// costs the MMA thread 200 cycles even when it is over, the four MMAs of a K block 190-260.
// Weights by TMA lose too: the copy engine takes 47 GB/s per SM, and 128-byte pieces of rows 38 KB apart are slow at HBM
// (down 28 -> 35 us); four gathered rows per copy cost 27 ns (head of 16384 ids 29 -> 80 us).
//
// A stage's barrier counts one asynchronous arrival per copy thread (cp.async.mbarrier.arrive), so a
// stage is published the moment its bytes have landed.
//
// Every wait is time-bounded; on expiry the CTA raises the timeout flag, drains and returns.
#pragma once
#include "umma.cuh"
#include "batched.cuh"
#include "ahead.cuh"
#include <cuda.h>
#include <cstring>

namespace fmtp {

constexpr int kGemmProducers = 256;          // eight copy warps
constexpr int kGemmThreads = 192 + kGemmProducers + 32;     // warp 14 asks for a later GEMM's weights
constexpr int kGemmBK = 64;                 // K elements per swizzled block: one 128-byte row
constexpr int kGemmTileM = 128;
constexpr int kGemmTileBytes = kGemmTileM * 128;    // a tile's 64-wide block
constexpr int kGemmMaxStages = 6;
constexpr int kGemmMaxXStages = 4;

enum GemmEpilogue {
    EPI_PARTIAL = 0,   // fp32 partial sums  partial[split][r][m] = D[m,2r] + D[m,2r+1]
    EPI_SWIGLU = 1,    // tile 0 holds gate rows, tile 1 the up rows of the same indices: act = silu(g) * u, written as the
                       // hi/lo operand of the next GEMM
    EPI_ARGMAX = 2,    // per activation row the maximum of (logit, row id) as a packed key (atomicMax), optional fp32 logits
};

struct GemmArgs {
    const bf16_t *a[3];          // up to three matrices whose rows are concatenated (q, k, v); [rows][lda] bf16
    int a_rows[3];
    int n_seg;
    const bf16_t *a_up;          // EPI_SWIGLU: the up matrix (a[0] is the gate matrix, same shape)
    const int32_t *row_ids;      // optional: GEMM row m reads a[0][row_ids[m]] (compressed output head)
    int V;                       // rows of a[0] when row_ids is used (ids outside are clamped and flagged)
    int n_rows, K, lda;          // output rows (EPI_SWIGLU: ffn indices); K % 8 == 0
    const bf16_t *x;             // [NB][ldx] bf16
    int ldx, NB, R;              // NB % 16 == 0, 2R <= NB <= 128
    int item_rows, n_ranges;     // output rows of an item (at most 128, EPI_ARGMAX 256) and number of such row ranges
    int splits, kb_per_split;    // K is cut into `splits` ranges of kb_per_split 64-wide blocks
    int epi;
    float *partial;              // [splits][R][ldp]
    int ldp;
    bf16_t *xop_out;             // EPI_SWIGLU: [>= 2R][ld_out]
    int ld_out;
    unsigned long long *keys;    // EPI_ARGMAX: [R]
    float *logits;               // EPI_ARGMAX, optional: row r at logits + r*logits_stride, column m
    long long logits_stride;
    bf16_t *logits_bf16;         // EPI_ARGMAX with round_bf16, optional: the logits as bf16, same indexing
    int round_bf16;              // 1: the argmax is decided on the logits rounded to bf16 (the values a caller sees)
    uint32_t *status;
    int n_stages, n_xstages;
    unsigned long long wait_limit_ns;   // every wait of the kernel gives up after this long
    int extra_arrivals;          // self-test only: arrivals a ring stage expects beyond the copies that are made
    // Two row-major matrices [ahead_rows][ahead_ld] that a later GEMM streams by tiles of 128 rows: while this one runs, its CTAs ask for the
    // first kAheadTileRows rows of each to be brought into L2 (ahead.cuh), until their own last MMA is done: a GEMM of few tiles, and so few
    // CTAs, gets no further than its first tiles. Used by W_o for gate/up: its own weights are in the ring when attention
    // ends, and until gate/up starts (merge, W_o, post: 15 us) HBM has nothing else to do. Then every stage of gate/up is part
    // L2 hit, part HBM, and the copy path takes in both at once. 7B shape, none / 8 / 16 / 32 / 48 / 64 rows of 128, us: four ragged
    // sequences, five steps 727 / 715 / 706 / 703 / 703 / 703, 16 sequences with extend rows 556 / 554 / 552 / 552 / 552 / 552. At 64 rows it
    // gives nothing (64 ragged sequences 909 -> 907, 16 x 4 rows of 28 layers 4182 -> 4194): there the activation block's re-reads
    // fill the path between L2 and the SMs. So only with four-block stages.
    const bf16_t *ahead[2];
    int ahead_rows, ahead_ld;
    uint32_t ahead_limit;        // bytes a CTA may ask for per tile (gemm_ahead_limit)
};
constexpr uint32_t kAheadPieceNs = 600;     // from a request to the next one

struct GemmSmem {
    uint64_t full[kGemmMaxStages], empty[kGemmMaxStages];
    uint64_t xfull[kGemmMaxXStages], xempty[kGemmMaxXStages];
    uint64_t tfull[2], tempty[2], drain;
    uint32_t tmem_base, abort_flag;
    unsigned long long kmax[4][64];
};

__device__ __forceinline__ bool gemm_wait(GemmSmem *sm, uint64_t *bar, uint32_t parity, unsigned long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    uint32_t polls = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++polls & 63u) == 0) {
            if (*reinterpret_cast<volatile uint32_t *>(&sm->abort_flag)) return false;
            if (global_timer_ns() - t0 > limit_ns) {
                *reinterpret_cast<volatile uint32_t *>(&sm->abort_flag) = 1u;
                return false;
            }
        }
    }
    return true;
}

// After a timeout perhaps nobody has waited for the last copies of a ring (the next one would go to slot `pos` in phase
// `phase`): wait for them, with a limit, before the CTA exits. Normally the MMA thread has seen all of them.
__device__ __forceinline__ void gemm_drain(GemmSmem *sm, uint64_t *full, int n, int pos, uint32_t phase) {
    const unsigned long long t0 = global_timer_ns();
    for (int s = 0; s < n && *reinterpret_cast<volatile uint32_t *>(&sm->abort_flag); ++s) {
        if (pos == 0) { pos = n; phase ^= 1u; }
        --pos;
        while (!mbar_try_wait(&full[pos], phase) && global_timer_ns() - t0 < 1000000ull) { }
    }
}

// Work items of a CTA: items (row range, K range) are dealt round-robin over the CTAs. Ranges do not cross the
// matrices of a concatenation.
struct GemmItem { int row0, row_end, split, seg, src0; };       // output rows; matrix and its row of row0
__device__ __forceinline__ int gemm_my_items(int n_items) {
    return (int)blockIdx.x < n_items ? (n_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
}
__device__ __forceinline__ GemmItem gemm_my_item(const GemmArgs &g, int i) {
    GemmItem it;
    const int item = (int)blockIdx.x + i * (int)gridDim.x;
    int rng = item / g.splits, first = 0;
    it.split = item - rng * g.splits;
    it.seg = 0;
    int rows = g.n_rows;
    if (g.n_seg > 1) {
        rows = g.a_rows[0];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int n = (g.a_rows[s] + g.item_rows - 1) / g.item_rows;
            if (it.seg == s && s + 1 < g.n_seg && rng >= n) { rng -= n; first += g.a_rows[s]; it.seg = s + 1; rows = g.a_rows[s + 1]; }
        }
    }
    it.src0 = rng * g.item_rows;
    it.row0 = first + it.src0;
    it.row_end = first + min(it.src0 + g.item_rows, rows);
    return it;
}

// True on all 128 epilogue threads (warps 0-3) if `flag` is set on any of them.
__device__ __forceinline__ bool epi_any(bool flag) {
    uint32_t out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 2, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"(flag ? 1u : 0u)
        : "memory");
    return out != 0;
}

// One TMA tile copy global -> shared (2-D tensor map, element coordinates x, y); its bytes are counted on `bar`.
// x * element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst_smem), "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// The same for a 3-D tensor map, with an L2 eviction policy.
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst_smem, const CUtensorMap *map, int x, int y, int z, uint64_t *bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst_smem), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
// One contiguous copy global -> shared; both addresses and the size are multiples of 16 bytes.
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_smem), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

template <int KA>
__global__ void __launch_bounds__(kGemmThreads, 1) skinny_gemm_kernel(const __grid_constant__ GemmArgs g, const __grid_constant__ CUtensorMap xmap) {
    extern __shared__ __align__(1024) unsigned char ring[];
    const int S = g.n_stages, SX = g.n_xstages;
    constexpr int kStage = KA * kGemmTileBytes;             // one tile, KA K blocks
    const int xblock = g.NB * 128, xstage = KA * xblock;
    unsigned char *xring = ring + (size_t)S * kStage;
    GemmSmem *sm = reinterpret_cast<GemmSmem *>(xring + (size_t)SX * xstage);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool two = g.epi != EPI_PARTIAL;                  // items may have two tiles

    const int sub_cols = (g.NB + 31) & ~31;                 // TMEM columns of one tile's accumulator
    const int buf_cols = two ? 2 * sub_cols : sub_cols;     // and of one accumulator buffer
    uint32_t alloc_cols = 32;
    while ((int)alloc_cols < 2 * buf_cols) alloc_cols <<= 1;

    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(&sm->full[s], kGemmProducers + g.extra_arrivals); mbar_init(&sm->empty[s], 1); }
        for (int s = 0; s < SX; ++s) { mbar_init(&sm->xfull[s], 1); mbar_init(&sm->xempty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&sm->tfull[b], 1); mbar_init(&sm->tempty[b], 128); }
        mbar_init(&sm->drain, 1);
        sm->abort_flag = (smem_u32(ring) & 1023u) != 0u;    // swizzled tiles need the alignment: nothing runs without it
        mbar_fence_init();
    }
    if (warp == 4) {
        tmem_alloc(&sm->tmem_base, alloc_cols);
        tmem_relinquish();
        tc_fence_before_sync();
    }
    chain_release();         // the next kernel of the stream may start its own set-up
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(&sm->tmem_base);

    const int n_items = *reinterpret_cast<volatile uint32_t *>(&sm->abort_flag) ? 0 : g.n_ranges * g.splits;
    const int n_kb = (g.K + kGemmBK - 1) / kGemmBK;
    const int n_my = gemm_my_items(n_items);
    auto tiles_of = [&](const GemmItem &gi) -> int { return g.epi == EPI_SWIGLU || gi.row_end - gi.row0 > kGemmTileM ? 2 : 1; };

    if (warp == 14) {
        // ================= a later GEMM's weights into L2, one thread, until this CTA's last MMA is done
        if (KA == 4 && lane == 0 && g.ahead[0]) {
            uint32_t left = g.ahead_limit * (uint32_t)gemm_ahead_tiles((int)blockIdx.x, g.ahead_rows, (int)gridDim.x);
            const int end = 2 * ((g.ahead_rows + kAheadTile - 1) / kAheadTile);
            unsigned long long due = 0;
            bool go = true;
            for (int t = 2 * (int)blockIdx.x; t < end && left && go; t = gemm_ahead_next(t, (int)gridDim.x)) {
                const AheadReq r = gemm_ahead_share(t, g.ahead_rows, g.ahead_ld, left);
                left -= r.bytes;
                const unsigned char *src = reinterpret_cast<const unsigned char *>(g.ahead[r.mat] + r.at);
                for (uint32_t at = 0; at < r.bytes && go; at += kAheadPiece) {
                    while (go && global_timer_ns() < due) {
                        go = !mbar_test(&sm->drain, 0);
                        __nanosleep(100);
                    }
                    if (!go) break;
                    prefetch_l2(src + at, min(kAheadPiece, r.bytes - at));
                    due = global_timer_ns() + kAheadPieceNs;
                }
            }
        }
        __syncwarp();
    } else if (warp >= 6) {
        // ================= weight copies: thread pt copies 16-byte column c of rows r0, r0 + 32, ... of a tile, KA K blocks at a
        // time: the blocks are immediate offsets on the source, so a pointer register is rewritten only once per stage (a
        // cp.async reads its address when it leaves the queue; rewriting it waits for that)
        const int pt = tid - 192;
        const int c = pt & 7, r0 = pt >> 3;
        const uint32_t dst0 = smem_u32(ring) + (uint32_t)(r0 * 128 + ((c ^ (r0 & 7)) << 4));
        const uint64_t policy = l2_evict_first();
        int stage = 0;
        uint32_t phase = 0;
        bool ok_run = true;
        // The gathered head reads its row ids, which a kernel earlier in the same call wrote: that is a real
        // dependency, so those GEMMs wait for the chain first. Plain weights depend on nothing in the stream, so
        // these warps never wait for a predecessor.
        if (g.row_ids) chain_wait();
        for (int i = 0; i < n_my && ok_run; ++i) {
            const GemmItem gi = gemm_my_item(g, i);
            const int kb0 = gi.split * g.kb_per_split, kb1 = min(kb0 + g.kb_per_split, n_kb), n_tiles = tiles_of(gi);
            const bf16_t *ap[2][4];
            uint32_t valid[2] = {0u, 0u};                   // bit q: row r0 + 32 q of the tile exists (the others stay stale: their
#pragma unroll                                              // results are not used)
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int first = g.epi == EPI_SWIGLU ? 0 : u * kGemmTileM;
                    int r = first + r0 + 32 * q;
                    if (gi.row0 + r < gi.row_end) valid[u] |= 1u << q;
                    else r = gi.row_end - gi.row0 - 1;
                    int row = gi.src0 + r;
                    if (g.row_ids) {
                        row = g.row_ids[row];
                        if ((unsigned)row >= (unsigned)g.V) { atomicOr(g.status, 0x1u); row = 0; }
                    }
                    ap[u][q] = (u == 1 && g.epi == EPI_SWIGLU ? g.a_up : g.a[gi.seg]) + (size_t)row * g.lda + (size_t)kb0 * kGemmBK + c * 8;
                }
            for (int kb = kb0; kb < kb1 && ok_run; kb += KA) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u >= n_tiles) break;
                    if (!gemm_wait(sm, &sm->empty[stage], phase ^ 1u, g.wait_limit_ns)) { ok_run = false; break; }
                    const uint32_t d = dst0 + (uint32_t)stage * kStage;
                    if ((kb + KA) * kGemmBK <= g.K && kb + KA <= kb1 && valid[u] == 15u) {      // the common case: plain 16-byte copies
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            cp_async16_full_hint<0>(d + (uint32_t)(q * 4096), ap[u][q], policy);
                            cp_async16_full_hint<128>(d + (uint32_t)(q * 4096 + kGemmTileBytes), ap[u][q], policy);
                            if (KA == 4) {
                                cp_async16_full_hint<256>(d + (uint32_t)(q * 4096 + 2 * kGemmTileBytes), ap[u][q], policy);
                                cp_async16_full_hint<384>(d + (uint32_t)(q * 4096 + 3 * kGemmTileBytes), ap[u][q], policy);
                            }
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int j = 0; j < KA; ++j) {
                                if ((valid[u] >> q & 1u) && kb + j < kb1) {
                                    // a column beyond K is filled with zeros, nothing is read
                                    const uint32_t n = (kb + j) * kGemmBK + c * 8 < g.K ? 16u : 0u;
                                    cp_async16_off_hint<0>(d + (uint32_t)(q * 4096 + j * kGemmTileBytes), n ? ap[u][q] + j * kGemmBK : g.a[0], n, policy);
                                }
                            }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) ap[u][q] += KA * kGemmBK;
                    // this thread's arrival on the stage's barrier fires when its copies above have landed
                    cp_async_arrive(&sm->full[stage]);
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                }
            }
        }
        cp_async_wait_all();
    } else if (warp == 5) {
        // ================= X copies: one thread, one tile copy (64 K elements x NB columns) per K block, KA of them a stage
        chain_wait();
        if (lane == 0) {
            int xs = 0;
            uint32_t xphase = 0;
            bool ok_run = true;
            for (int i = 0; i < n_my && ok_run; ++i) {
                const int kb0 = gemm_my_item(g, i).split * g.kb_per_split, kb1 = min(kb0 + g.kb_per_split, n_kb);
                for (int kb = kb0; kb < kb1; kb += KA) {
                    if (!gemm_wait(sm, &sm->xempty[xs], xphase ^ 1u, g.wait_limit_ns)) { ok_run = false; break; }
                    const int nj = min(KA, kb1 - kb);
                    mbar_arrive_expect_tx(&sm->xfull[xs], (uint32_t)(nj * xblock));
                    for (int j = 0; j < nj; ++j)
                        tma_load_2d(smem_u32(xring) + (uint32_t)(xs * xstage + j * xblock), &xmap, (kb + j) * kGemmBK, 0, &sm->xfull[xs]);
                    if (++xs == SX) { xs = 0; xphase ^= 1u; }
                }
            }
            gemm_drain(sm, sm->xfull, SX, xs, xphase);
        }
        __syncwarp();
    } else if (warp == 4) {
        // ================= MMA issue: one thread
        if (lane == 0) {
            const uint32_t idesc = umma_idesc_bf16(g.NB);
            int stage = 0, xs = 0, buf = 0;
            uint32_t phase = 0, xphase = 0, tphase[2] = {0, 0};
            bool ok_run = true;
            for (int i = 0; i < n_my && ok_run; ++i) {
                const GemmItem gi = gemm_my_item(g, i);
                const int kb0 = gi.split * g.kb_per_split, kb1 = min(kb0 + g.kb_per_split, n_kb), n_tiles = tiles_of(gi);
                if (!gemm_wait(sm, &sm->tempty[buf], tphase[buf] ^ 1u, g.wait_limit_ns)) break;
                tc_fence_after_sync();
                const uint32_t d0 = tmem_base + (uint32_t)(buf * buf_cols);
                for (int kb = kb0; kb < kb1 && ok_run; kb += KA) {
                    ok_run = gemm_wait(sm, &sm->xfull[xs], xphase, g.wait_limit_ns);
                    const uint32_t sb = umma_desc_lo(smem_u32(xring) + (uint32_t)(xs * xstage));
                    for (int u = 0; u < n_tiles && ok_run; ++u) {
                        if (!gemm_wait(sm, &sm->full[stage], phase, g.wait_limit_ns)) { ok_run = false; break; }
                        fence_proxy_async();          // the copies' shared-memory writes, before the tensor core reads them
                        tc_fence_after_sync();
                        const uint32_t sa = umma_desc_lo(smem_u32(ring) + (uint32_t)stage * kStage);
#pragma unroll
                        for (int j = 0; j < KA; ++j)
                            if (kb + j < kb1)
                                umma_kblock(d0 + (uint32_t)(u * sub_cols), sa + (uint32_t)(j * (kGemmTileBytes >> 4)), sb + (uint32_t)(j * (xblock >> 4)),
                                            idesc, kb + j > kb0);
                        umma_commit(&sm->empty[stage]);
                        if (++stage == S) { stage = 0; phase ^= 1u; }
                    }
                    if (!ok_run) break;
                    umma_commit(&sm->xempty[xs]);
                    if (++xs == SX) { xs = 0; xphase ^= 1u; }
                }
                if (!ok_run) break;
                umma_commit(&sm->tfull[buf]);
                tphase[buf] ^= 1u;
                buf ^= 1;
            }
            // every MMA issued above has completed once this arrival lands
            umma_commit(&sm->drain);
            gemm_wait(sm, &sm->drain, 0, g.wait_limit_ns);
        }
        __syncwarp();
    }
    unsigned long long (*last_max)[64] = reinterpret_cast<unsigned long long (*)[64]>(ring);     // EPI_ARGMAX: maxima of the last item, per warp quarter
    if (warp < 4 || (warp >= 6 && warp < 14)) {
        // ================= epilogue: thread = one row of a tile (TMEM lane 32*(warp % 4) + lane), eight activation rows at a time.
        // One warp per scheduler would be a chain of latencies (64 rows, 3584-wide layer: 7 us of divides in gate/up, 18 us of
        // warp maxima in the output head when the rows went one after the other, 5 and 5 us by eights), and after the last item
        // nothing hides it. So the copy warps, which have nothing left to copy by then, take two thirds of the last item's rows.
        chain_wait();
        const int q = warp & 3, worker = warp < 4 ? 0 : 1 + ((warp - 6) >> 2), tr = q * 32 + lane;
        for (int i = worker == 0 || n_my == 0 ? 0 : n_my - 1; i < n_my; ++i) {
            const bool last = i == n_my - 1;
            const int first = last ? worker * 8 : 0, step = last ? 24 : 8, buf = i & 1;
            const GemmItem gi = gemm_my_item(g, i);
            // the copy warps come for the last item only: `drain` completes once, behind its MMAs (tfull's phase is no answer there,
            // the parity also fits two items earlier, which a CTA whose ring holds its last items may not have begun). It
            // completes after a timeout too, so they look at the flag as well
            const bool late = worker == 0 ? !gemm_wait(sm, &sm->tfull[buf], (uint32_t)(i >> 1) & 1u, g.wait_limit_ns)
                                          : !gemm_wait(sm, &sm->drain, 0, g.wait_limit_ns) || *reinterpret_cast<volatile uint32_t *>(&sm->abort_flag);
            // before another item the 128 epilogue threads agree on the outcome; after the last one there is no barrier but the CTA's
            if (last ? __any_sync(0xffffffffu, late) : epi_any(late)) break;
            tc_fence_after_sync();
            const uint32_t t0 = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * buf_cols);
            const int m0 = gi.row0 + tr;
            const bool m_ok = m0 < gi.row_end;
            if (g.epi == EPI_PARTIAL) {
                for (int r0 = first; r0 < g.R; r0 += step) {
                    uint32_t v[16];
                    tmem_ld16_issue(t0 + 2 * r0, v);
                    tmem_ld_wait();
                    float *out = g.partial + (size_t)(gi.split * g.R + r0) * g.ldp + m0;
                    if (m_ok) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (r0 + j < g.R) out[(size_t)j * g.ldp] = __uint_as_float(v[2 * j]) + __uint_as_float(v[2 * j + 1]);
                    }
                    __syncwarp();
                }
            } else if (g.epi == EPI_SWIGLU) {
                for (int r0 = first; r0 < g.R; r0 += step) {
                    uint32_t v[16], u[16];
                    tmem_ld16_issue(t0 + 2 * r0, v);
                    tmem_ld16_issue(t0 + sub_cols + 2 * r0, u);
                    tmem_ld_wait();
                    float gv[8], e[8], act[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        gv[j] = __uint_as_float(v[2 * j]) + __uint_as_float(v[2 * j + 1]);
                        e[j] = 1.0f + expf(-gv[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) act[j] = gv[j] / e[j] * (__uint_as_float(u[2 * j]) + __uint_as_float(u[2 * j + 1]));
                    bf16_t *out = g.xop_out + (size_t)(2 * r0) * g.ld_out + m0;
                    if (m_ok) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (r0 + j < g.R) {
                                uint16_t hi, lo;
                                split_bf16(act[j], hi, lo);
                                out[(size_t)(2 * j) * g.ld_out] = hi;
                                out[(size_t)(2 * j + 1) * g.ld_out] = lo;
                            }
                    }
                    __syncwarp();
                }
            } else {
                unsigned long long *best = last ? last_max[q] : sm->kmax[q];
                const int n_tiles = tiles_of(gi);
                for (int u = 0; u < n_tiles; ++u) {
                    const int m = m0 + u * kGemmTileM;
                    const bool in = m < gi.row_end;
                    uint32_t row_id = (uint32_t)m;
                    if (g.row_ids && in) {
                        int id = g.row_ids[m];
                        row_id = ((unsigned)id >= (unsigned)g.V) ? 0u : (uint32_t)id;
                    }
                    for (int r0 = first; r0 < g.R; r0 += step) {        // rows beyond R of the eight are not used
                        uint32_t v[16];
                        tmem_ld16_issue(t0 + u * sub_cols + 2 * r0, v);
                        tmem_ld_wait();
                        float x[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = __uint_as_float(v[2 * j]) + __uint_as_float(v[2 * j + 1]);
                        if (in && g.logits) {
                            float *out = g.logits + (size_t)r0 * g.logits_stride + m;
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                if (r0 + j < g.R) out[(size_t)j * g.logits_stride] = x[j];
                        }
                        if (g.round_bf16) {
                            uint16_t b[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) { b[j] = f32_bf16bits(x[j]); x[j] = bf16bits_f32(b[j]); }
                            if (in && g.logits_bf16) {
                                bf16_t *out = g.logits_bf16 + (size_t)r0 * g.logits_stride + m;
#pragma unroll
                                for (int j = 0; j < 8; ++j)
                                    if (r0 + j < g.R) out[(size_t)j * g.logits_stride] = b[j];
                            }
                        }
                        // the warp's maximum value, then the lowest id that has it (0: no value, never wins); lane j keeps row r0 + j
                        uint32_t top = 0u, top_id = 0u;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const uint32_t key = in ? float_order_key(x[j]) : 0u;
                            const uint32_t k = __reduce_max_sync(0xffffffffu, key);
                            const uint32_t id = __reduce_min_sync(0xffffffffu, in && key == k ? row_id : 0xffffffffu);
                            if (lane == j) { top = k; top_id = id; }
                        }
                        if (lane < 8 && r0 + lane < g.R) {
                            const unsigned long long k = ((unsigned long long)top << 32) | (0xffffffffu - top_id);
                            if (u == 0 || k > best[r0 + lane]) best[r0 + lane] = k;
                        }
                        __syncwarp();
                    }
                }
            }
            tc_fence_before_sync();
            if (last) break;
            mbar_arrive(&sm->tempty[buf]);
            if (g.epi == EPI_ARGMAX) {
                bar_sync(1, 128);
                if (tid < g.R && g.keys) {
                    unsigned long long k = sm->kmax[0][tid];
#pragma unroll
                    for (int w = 1; w < 4; ++w) k = sm->kmax[w][tid] > k ? sm->kmax[w][tid] : k;
                    atomicMax(&g.keys[tid], k);
                }
                bar_sync(1, 128);
            }
        }
    }
    __syncthreads();
    const bool aborted = *reinterpret_cast<volatile uint32_t *>(&sm->abort_flag) != 0u;
    if (tid == 0 && aborted) atomicOr(g.status, 0x8u);
    if (g.epi == EPI_ARGMAX && n_my > 0 && !aborted && tid < g.R && g.keys) {
        unsigned long long k = last_max[0][tid];
#pragma unroll
        for (int w = 1; w < 4; ++w) k = last_max[w][tid] > k ? last_max[w][tid] : k;
        atomicMax(&g.keys[tid], k);
    }
    if (warp == 4) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, alloc_cols);
    }
}

typedef CUresult (*TmapEncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                 const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
// The driver's tensor-map encoder (a host computation, no device work). Returns 0 or a cudaError_t.
inline int tmap_encoder(TmapEncodeFn *out) {
    static TmapEncodeFn encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qr;
        cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr);
        if (e != cudaSuccess) return (int)e;
        if (!fn || qr != cudaDriverEntryPointSuccess) return (int)cudaErrorNotSupported;
        encode = reinterpret_cast<TmapEncodeFn>(fn);
    }
    *out = encode;
    return 0;
}

// Tensor map of a row-major bf16 matrix [rows][ld] for copies of 64 K elements x box_rows rows, 128-byte swizzle (the
// layout the MMA reads), zeros beyond K. Returns 0 or a cudaError_t.
inline int gemm_encode_map(CUtensorMap *map, const bf16_t *p, long long rows, int ld, int K, int box_rows) {
    TmapEncodeFn encode;
    if (int rc = tmap_encoder(&encode)) return rc;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kGemmBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16_t *>(p), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : (int)cudaErrorInvalidValue;
}

// Launches the GEMM on `stream` with one CTA per SM (fewer when there are fewer work items).
// Returns the cudaError_t of the launch.
inline int skinny_gemm_launch(GemmArgs g, int n_sm, int smem_optin, cudaStream_t stream, TmapCache *cache) {
    const int avail = smem_optin - (int)sizeof(GemmSmem);
    // K blocks per stage: four where a ring of three weight stages then still fits; X in flight for the latency of L2
    // under a full HBM stream, the rest of the memory for the weights
    const int ka = g.NB <= 32 ? 4 : 2, xstage = ka * g.NB * 128, wstage = ka * kGemmTileBytes;
    const int want = ((g.epi == EPI_PARTIAL ? 96 : 64) * 1024 + xstage - 1) / xstage;
    g.n_xstages = ka == 4 ? 2 : want < 2 ? 2 : want > kGemmMaxXStages ? kGemmMaxXStages : want;
    int stages = (avail - g.n_xstages * xstage) / wstage;
    if (stages > kGemmMaxStages) stages = kGemmMaxStages;
    if (stages < 3) return (int)cudaErrorInvalidConfiguration;
    g.n_stages = stages;
    void (*kern)(const GemmArgs, const CUtensorMap) = ka == 4 ? skinny_gemm_kernel<4> : skinny_gemm_kernel<2>;
    bool &raised = cache->gemm_raised[ka == 4];
    const size_t smem = (size_t)stages * wstage + (size_t)g.n_xstages * xstage + sizeof(GemmSmem);
    const int n_items = g.n_ranges * g.splits;
    const int grid = n_items < n_sm ? n_items : n_sm;
    if (!raised) {       // once per context, to the most there is: the limit is the device's, a lower one would take away from other contexts
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
        if (e != cudaSuccess) return (int)e;
        raised = true;
    }
    // the activation operand is the library's own: its map depends on (address, row pitch, K, rows) only: encoded once, then reused
    CUtensorMap xmap;
    static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
    TmapEntry *hit = nullptr;
    for (int i = 0; i < cache->n; ++i)
        if (cache->e[i].x == g.x && cache->e[i].ldx == g.ldx && cache->e[i].K == g.K && cache->e[i].NB == g.NB) { hit = &cache->e[i]; break; }
    if (hit) std::memcpy(&xmap, hit->map, sizeof(xmap));
    else {
        if (int rc = gemm_encode_map(&xmap, g.x, g.NB, g.ldx, g.K, g.NB)) return rc;
        const int cap = (int)(sizeof(cache->e) / sizeof(cache->e[0]));
        TmapEntry &dst = cache->e[cache->n < cap ? cache->n++ : (cache->next++ % cap)];
        dst.x = g.x; dst.ldx = g.ldx; dst.K = g.K; dst.NB = g.NB;
        std::memcpy(dst.map, &xmap, sizeof(xmap));
    }
    return (int)launch_chained(kern, dim3(grid), dim3(kGemmThreads), smem, stream, g, xmap);
}

}  // namespace fmtp
