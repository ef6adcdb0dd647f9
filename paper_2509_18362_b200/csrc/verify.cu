// Greedy verification: full-vocabulary argmax of every target-logit row, then the longest
// accepted draft prefix and the bonus token (Sec. 2.3 "Verification phase" of the paper).
//
// HBM-bound read-once scan. A row is cut into slices from the 16-byte boundary at or below its start; a launch has up to two
// CTAs per SM and each takes a contiguous range of slices (so most of a CTA's slices belong to one row). A thread keeps
// NV independent 128-bit streaming loads in flight and requests the next slice's before it looks at the current one's.
// Only values are compared while scanning, two at a time (max.bf16x2, NaN never wins), and each thread remembers in which
// slice its maximum first appeared; the token id is looked up once per row and CTA, by the threads that hold the row's
// maximum, which read that slice again (it is in L2). Comparing (value, id) pairs element by element took 2.5
// instructions per byte and held 256 rows of 152064 (78 MB) to 24.0 us; now 17.5 us, of which
// 5 us are the launch, the last winners and the last CTA's tail.
// Slices are as long as still gives every resident CTA one (a long slice publishes fewer winners): one sequence of four
// rows of 152064 is 300 slices of 2048 elements instead of 40 of 16384 (6.7 us by
// itself; calls back to back 8.9 -> 4.7 us, with the chained launch and a lighter host side).
// The row's winner (highest value, then lowest token id) is published as one 64-bit key with atomicMax (an integer
// maximum: order independent, so the result is reproducible). The CTA that arrives last turns the per-row winners into
// accept_len / bonus and clears the scratch for the next call.
#include "mega.cuh"
#include "ptx.cuh"
#include "umma.cuh"

namespace fmtp {

namespace {

constexpr int kVThreads = 256;
constexpr int kVCtasPerSm = 2;                                    // resident CTAs per SM at this register footprint
constexpr int kVMaxRows = 4096;
constexpr int kNoIdx = 0x7fffffff;
template <int NV> __host__ __device__ constexpr int slice_elems() { return kVThreads * NV * 8; }     // NV 16-byte loads per thread and slice

// A slice of one row: whole 16-byte vectors at src + 8 * v, v in [v0, v1), and the single elements src[h0 .. h1) before the
// row's first whole vector (first slice only) and src[t0 .. t1) after its last one (last slice only), at most seven each.
// src is the 16-byte boundary at or below the row, `base` elements before it.
struct SliceRef { const bf16_t *src; int row, v0, v1, h0, h1, t0, t1, base; };

template <int NV>
__device__ __forceinline__ SliceRef slice_ref(const bf16_t *logits, int V, int slices_per_row, int item) {
    constexpr int E = slice_elems<NV>();
    const int row = item / slices_per_row, slice = item - row * slices_per_row;
    SliceRef r;
    const bf16_t *p = logits + (size_t)row * V;
    const int off = (int)((reinterpret_cast<uintptr_t>(p) & 15u) >> 1);
    r.row = row;
    r.src = p - off;
    r.base = off;
    const int lo = slice * E, hi = min(lo + E, V + off);
    const int first = (off + 7) >> 3, last = (V + off) >> 3;                  // whole vectors of the row: [first, last)
    r.v0 = max(lo >> 3, first);
    r.v1 = max(r.v0, min((lo + E) >> 3, last));
    r.h0 = r.h1 = r.t0 = r.t1 = 0;
    if (slice == 0) { r.h0 = off; r.h1 = min(first * 8, V + off); }
    if (lo < hi && hi == V + off) { r.t0 = max(last * 8, max(lo, r.h1)); r.t1 = hi; }
    return r;
}
template <int NV>
__device__ __forceinline__ void slice_load(const SliceRef &r, uint4 (&v)[NV]) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int vi = r.v0 + (int)threadIdx.x + j * kVThreads;
        v[j] = (vi < r.v1) ? ldnc128(r.src + (size_t)vi * 8) : make_uint4(0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu);   // NaN: never wins
    }
}
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

template <int NV>
__global__ void __launch_bounds__(kVThreads, kVCtasPerSm) verify_kernel(const bf16_t *__restrict__ logits,
                                                            const int32_t *__restrict__ drafts, int B, int K, int V,
                                                            int slices_per_row, int n_items, int32_t *accept_len, int32_t *bonus,
                                                            int32_t *out_argmax, unsigned long long *keys,
                                                            uint32_t *counter, uint32_t *status,
                                                            uint32_t *user_status) {
    chain_release();
    chain_wait();
    __shared__ uint32_t wmax[kVThreads / 32];
    __shared__ int s_idx, is_last;
    __shared__ int s_tok[kVMaxRows];
    const int tid = threadIdx.x;
    const int i0 = (int)(((long long)blockIdx.x * n_items) / gridDim.x);
    const int i1 = (int)(((long long)(blockIdx.x + 1) * n_items) / gridDim.x);
    // this thread's maximum in the current row: over whole vectors, with the slice it first appeared in (-1: no value yet),
    // and over single elements at the row's ends, with its index
    float best = -INFINITY, ebest = -INFINITY;
    int bslice = -1, eidx = kNoIdx;

    // publishes this CTA's winner of row `row`; every thread calls it
    auto flush = [&](int row) {
        uint32_t k = bslice >= 0 ? float_order_key(best + 0.0f) : 0u;         // + 0: -0 and +0 are one value
        if (eidx != kNoIdx) k = max(k, float_order_key(ebest + 0.0f));
        k = __reduce_max_sync(0xffffffffu, k);
        __syncthreads();                                                      // wmax, s_idx free again
        if ((tid & 31) == 0) wmax[tid >> 5] = k;
        if (tid == 0) s_idx = kNoIdx;
        __syncthreads();
        uint32_t m = wmax[0];
#pragma unroll
        for (int w = 1; w < kVThreads / 32; ++w) m = max(m, wmax[w]);
        if (m == 0u) return;                                                  // block-uniform: no value in this CTA's part of the row
        int idx = kNoIdx;
        if (bslice >= 0 && float_order_key(best + 0.0f) == m) {               // holds the maximum: where?
            const SliceRef r = slice_ref<NV>(logits, V, slices_per_row, bslice);
            uint4 v[NV];
            slice_load<NV>(r, v);
#pragma unroll
            for (int j = NV - 1; j >= 0; --j) {
                const int e0 = (r.v0 + tid + j * kVThreads) * 8 - r.base;
                const uint32_t w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
                for (int q = 3; q >= 0; --q) {
                    if (bf16hi_f32(w[q]) == best) idx = e0 + 2 * q + 1;
                    if (bf16lo_f32(w[q]) == best) idx = e0 + 2 * q;
                }
            }
        }
        if (eidx != kNoIdx && float_order_key(ebest + 0.0f) == m) idx = min(idx, eidx);
        if (idx != kNoIdx) atomicMin(&s_idx, idx);
        __syncthreads();
        if (tid == 0) atomicMax(keys + row, ((unsigned long long)m << 32) | (0xffffffffu - (uint32_t)s_idx));
    };

    uint4 cur[NV], nxt[NV];
    SliceRef rc = slice_ref<NV>(logits, V, slices_per_row, i0 < i1 ? i0 : 0), rn = rc;
    if (i0 < i1) slice_load<NV>(rc, cur);
    int cur_row = -1;
    for (int item = i0; item < i1; ++item) {
        if (item + 1 < i1) {                               // the next slice's loads go out before this one's values are used
            rn = slice_ref<NV>(logits, V, slices_per_row, item + 1);
            slice_load<NV>(rn, nxt);
        }
        if (rc.row != cur_row) {
            if (cur_row >= 0) flush(cur_row);
            best = ebest = -INFINITY; bslice = -1; eidx = kNoIdx; cur_row = rc.row;
        }
        uint32_t m = 0x7fff7fffu;
#pragma unroll
        for (int j = 0; j < NV; ++j) m = max_bf16x2(m, max_bf16x2(max_bf16x2(cur[j].x, cur[j].y), max_bf16x2(cur[j].z, cur[j].w)));
        const float a = bf16lo_f32(m), b = bf16hi_f32(m);
        const float v = a != a ? b : (b > a ? b : a);
        // strict '>' keeps the earliest slice; the second clause admits the first value even if it is -inf
        if (v > best || (bslice < 0 && v == v)) { best = v; bslice = item; }
        // single elements at the row's ends
        const int e = tid < 8 ? rc.h0 + tid : rc.t0 + tid - 8;
        if (tid < 16 && e < (tid < 8 ? rc.h1 : rc.t1)) {
            const float x = bf16bits_f32(rc.src[e]);
            if (x > ebest || (eidx == kNoIdx && x == x)) { ebest = x; eidx = e - rc.base; }
        }
        rc = rn;
#pragma unroll
        for (int j = 0; j < NV; ++j) cur[j] = nxt[j];
    }
    if (cur_row >= 0) flush(cur_row);
    if (tid == 0) {
        __threadfence();
        uint32_t old = atomicAdd(counter, 1u);
        is_last = (old == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last) return;

    // ---- last CTA: winners of all rows, then accept lengths
    __threadfence();
    const int M = K + 1, rows = B * M;
    for (int i = tid; i < rows; i += kVThreads) {
        const unsigned long long k = ldcg_u64(keys + i);
        const int b = i / M, j = i - b * M;
        const int want = j < K ? drafts[(size_t)b * K + j] : -1;
        int g = 0;
        if ((k >> 32) == 0ull) { atomicOr(status, 0x10u); if (user_status) atomicOr(user_status, 0x10u); }
        else g = (int)argmax_key_id(k);
        if (out_argmax) out_argmax[i] = g;
        s_tok[i] = (j < K && want == g) ? ~g : g;          // an accepted row is marked by its complement
        keys[i] = 0ull;
    }
    if (tid == 0) *counter = 0u;
    __syncthreads();
    for (int b = tid; b < B; b += kVThreads) {
        int n = 0;
        while (s_tok[b * M + n] < 0) ++n;                  // ends: the last row of a sequence has no draft
        accept_len[b] = n;
        bonus[b] = s_tok[b * M + n];
    }
}

// The acceptance rule alone, for callers that already hold the target's greedy token of every row
// (fastmtp_target_step's out_argmax): one thread per sequence walks its K drafts.
__global__ void accept_ids_kernel(const int32_t *__restrict__ target_argmax, const int32_t *__restrict__ drafts, int B, int K,
                                  int32_t *accept_len, int32_t *bonus) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int32_t *g = target_argmax + (size_t)b * (K + 1);
    int a = 0;
    while (a < K && drafts[(size_t)b * K + a] == g[a]) ++a;
    accept_len[b] = a;
    bonus[b] = g[a];
}

}  // namespace

int accept_ids_launch(const int32_t *target_argmax, const int32_t *drafts, int B, int K, int32_t *accept_len, int32_t *bonus,
                      cudaStream_t stream) {
    accept_ids_kernel<<<(B + 127) / 128, 128, 0, stream>>>(target_argmax, drafts, B, K, accept_len, bonus);
    return (int)cudaGetLastError();
}

int verify_launch(const bf16_t *logits, const int32_t *drafts, int B, int K, int V, int32_t *accept_len,
                  int32_t *bonus, int32_t *out_argmax, unsigned long long *keys, uint32_t *counter,
                  uint32_t *status, uint32_t *user_status, int n_sm, cudaStream_t stream) {
    if (n_sm <= 0) {                       // a caller without a context: ask the device (no allocation involved)
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return (int)e;
    }
    const long long rows = (long long)B * (K + 1), ctas = (long long)n_sm * kVCtasPerSm;
    auto per_row = [&](int nv) { const int e = kVThreads * nv * 8; return (V + 7 + e - 1) / e; };   // a row may start 7 elements after a 16-byte boundary
    int nv = 8;
    while (nv > 1 && rows * per_row(nv) < ctas) nv >>= 1;
    const int slices = per_row(nv);
    const long long items = rows * slices;
    const int grid = (int)(items < ctas ? items : ctas);
    auto kern = nv == 8 ? verify_kernel<8> : nv == 4 ? verify_kernel<4> : nv == 2 ? verify_kernel<2> : verify_kernel<1>;
    // (a chained launch: the kernel's scheduling overlaps a predecessor that lets it)
    return (int)launch_chained(kern, dim3(grid), dim3(kVThreads), 0, stream, logits, drafts, B, K, V, slices, (int)items, accept_len, bonus,
                               out_argmax, keys, counter, status, user_status);
}

}  // namespace fmtp
