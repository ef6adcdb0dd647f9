// Gate/up weights that are asked into L2 before their phase: which rows, in which order, and how many of them. Both kernels
// walk these lists. They are host code as well, so that the requests of every CTA can be looked over without a GPU.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fmtp {

// One request: matrix (0 gate, 1 up), first element, bytes (a multiple of 16: widths are multiples of 64).
struct AheadReq { int mat; long long at; uint32_t bytes; };

// All CTAs' requests of a layer together stay within 9/16 of L2 (75 MB): what is pushed out again before its tile comes is read
// twice. The 7B shape asks for 59 MB (persistent kernel) and 68 (batched path). Without the bound a layer of d = 8192 with ffn
// 28672 asked for 232 MB: drafts of three steps at 2048 and 16384 positions 1212 and 1359 us, with it 1166 and 1312, without
// any request 1171 and 1297; d = 5120 with ffn 27648 at 16384 919 / 900 / 894. Bounds of 32, 48, 64 and 80 MB are within 1.5 % of each other.
__host__ __device__ inline long long ahead_budget(long long l2_bytes) {
    const long long share = l2_bytes / 16 * 9, most = 1ll << 30;      // (32-bit counts below)
    return share < most ? share : most;
}

// ---- persistent kernel: the first kAheadRows of the gate and of the up rows of every tile but the CTA's first, whole rows, a
// request each. Rows v0 .. v1 of ffn are the CTA's, a tile has `cap` of them.
constexpr int kAheadRows = 4;
// Requests a CTA may make.
__host__ __device__ inline int mega_ahead_limit(long long budget, int grid, int d) {
    return (int)(budget / grid / (kAheadRows * 2 * d) / 2) * 2;
}
__host__ __device__ inline int mega_ahead_count(int v0, int v1, int cap, int limit) {
    const int n = 2 * ((v1 - v0 + cap - 1) / cap - 1);
    return n < 0 ? 0 : n < limit ? n : limit;
}
__host__ __device__ inline AheadReq mega_ahead_req(int v0, int v1, int cap, int d, int i) {
    const int row = v0 + (1 + (i >> 1)) * cap, rows = v1 - row < kAheadRows ? v1 - row : kAheadRows;
    return AheadReq{i & 1, (long long)row * d, (uint32_t)rows * (uint32_t)d * 2u};
}

// ---- batched path: the first kAheadTileRows rows of every tile of 128, gate then up, tiles dealt over the CTAs of the GEMM that
// asks, in pieces of kAheadPiece bytes. The budget goes by tiles: by CTAs, those with a second tile would leave it out, and the
// GEMM that streams it would wait for that one. A CTA spends it from its first tile on; spread over all of its tiles (fewer rows of each) it loses
// (d = 8192 with ffn 28672, sixteen sequences 1294 us without requests, 1300 and 1310; two at 16384 positions 1303, 1298 and 1315).
constexpr int kAheadTile = 128, kAheadTileRows = 32;
constexpr uint32_t kAheadPiece = 16384;
// Bytes that a CTA may ask for per tile that it has.
__host__ __device__ inline uint32_t gemm_ahead_limit(long long budget, int rows) {
    const long long per_tile = budget / ((rows + kAheadTile - 1) / kAheadTile) / 16 * 16, most = 2ll << 20;      // (32 rows of 16384 columns, twice)
    return (uint32_t)(per_tile < most ? per_tile : most);
}
__host__ __device__ inline int gemm_ahead_tiles(int cta, int rows, int grid) {
    const int tiles = (rows + kAheadTile - 1) / kAheadTile;
    return cta < tiles ? (tiles - cta + grid - 1) / grid : 0;
}
// What is asked for of matrix t & 1 of tile t >> 1 with `left` bytes left; CTA `cta` begins with t = 2 * cta and goes on with gemm_ahead_next.
__host__ __device__ inline AheadReq gemm_ahead_share(int t, int rows, int ld, uint32_t left) {
    const int row = (t >> 1) * kAheadTile;
    const uint32_t all = (uint32_t)(rows - row < kAheadTileRows ? rows - row : kAheadTileRows) * (uint32_t)ld * 2u;
    return AheadReq{t & 1, (long long)row * ld, all < left ? all : left};
}
__host__ __device__ inline int gemm_ahead_next(int t, int grid) { return t & 1 ? t + 2 * grid - 1 : t + 1; }

}  // namespace fmtp
