// Diagnostic entry points. The first shows, without hanging or faulting anything, what the library's device
// waits do when the event they wait for never comes. A one-warp kernel waits on an mbarrier that
// nothing arrives on, with the same poll-and-check-the-clock loop the decoder kernel uses for its
// ring and grid barriers but a caller-chosen limit; when the limit passes it ORs FMTP_DEV_TIMEOUT
// into the status word and returns normally, so the context stays usable. The second lists the requests for weights ahead of
// their phase, from the functions that the kernels walk.
#include "../../include/fastmtp.h"
#include "mega.cuh"
#include "ahead.cuh"
#include "ptx.cuh"

namespace {

__global__ void wait_probe_kernel(uint32_t *status, unsigned long long limit_ns, unsigned long long *waited_ns) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        fmtp::mbar_init(&bar, 1);
        fmtp::mbar_fence_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long t0 = fmtp::global_timer_ns();
        bool done = false;
        unsigned long long now = t0;
        for (uint32_t n = 0; !done; ++n) {
            if (fmtp::mbar_try_wait(&bar, 0)) { done = true; break; }     // never: no one arrives
            if ((n & 255u) == 255u) {
                now = fmtp::global_timer_ns();
                if (now - t0 > limit_ns) break;
            }
        }
        if (!done) atomicOr(status, FMTP_DEV_TIMEOUT);
        if (waited_ns) *waited_ns = now - t0;
    }
}

}  // namespace

extern "C" int fmtp_selftest_wait_timeout(uint32_t *dev_status, int limit_ms, unsigned long long *dev_waited_ns, void *stream) {
    if (!dev_status) return FMTP_EINVAL;
    if (limit_ms < 1 || limit_ms > 1000) return FMTP_EINVAL;          // bounded on purpose
    wait_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(dev_status, (unsigned long long)limit_ms * 1000000ull,
                                                                        dev_waited_ns);
    return cudaGetLastError() == cudaSuccess ? FMTP_OK : FMTP_ECUDA;
}

extern "C" int fmtp_selftest_ahead(int batched, int ffn, int d, int grid, long long l2_bytes, int cta, int max_requests, int *mat,
                                   long long *at, unsigned int *bytes) {
    const int most = 1 << 22;                                         // keeps every product of the lists inside its type
    if (ffn < 1 || ffn > most || d < 1 || d > most || grid < 1 || grid > most || l2_bytes < 0 || cta < 0 || cta >= grid) return FMTP_EINVAL;
    if (max_requests < 0 || (max_requests > 0 && (!mat || !at || !bytes))) return FMTP_EINVAL;
    const long long budget = fmtp::ahead_budget(l2_bytes);
    int n = 0;
    auto put = [&](const fmtp::AheadReq &r) {
        if (n < max_requests) { mat[n] = r.mat; at[n] = r.at; bytes[n] = r.bytes; }
        ++n;
    };
    if (batched) {
        uint32_t left = fmtp::gemm_ahead_limit(budget, ffn) * (uint32_t)fmtp::gemm_ahead_tiles(cta, ffn, grid);
        const int end = 2 * ((ffn + fmtp::kAheadTile - 1) / fmtp::kAheadTile);
        for (int t = 2 * cta; t < end && left; t = fmtp::gemm_ahead_next(t, grid)) {
            const fmtp::AheadReq r = fmtp::gemm_ahead_share(t, ffn, d, left);
            left -= r.bytes;
            for (uint32_t at = 0; at < r.bytes; at += fmtp::kAheadPiece)
                put(fmtp::AheadReq{r.mat, r.at + at / 2, r.bytes - at < fmtp::kAheadPiece ? r.bytes - at : fmtp::kAheadPiece});
        }
    } else {
        const int v0 = fmtp::share_first(cta, ffn, grid), v1 = fmtp::share_first(cta + 1, ffn, grid), cap = fmtp::kTileRows / 2;
        const int count = fmtp::mega_ahead_count(v0, v1, cap, fmtp::mega_ahead_limit(budget, grid, d));
        for (int i = 0; i < count; ++i) put(fmtp::mega_ahead_req(v0, v1, cap, d, i));
    }
    return n;
}
