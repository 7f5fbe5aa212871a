// dd_stream.cpp -- continuous dedispersion of a long observation in chunks.
//
// The paper dedisperses one second of data per call with an input of t
// samples, t covering the delay at the highest trial DM (Section III-A). For
// a continuous stream the same holds chunk by chunk: chunk k of S new samples
// per channel, preceded by the previous M = max-delay samples, is exactly one
// plan input of T_in = S + M samples, and gives the S output samples
// [kS - M, (k+1)S - M) of the continuous stream (samples before the stream's
// start count as zeros). The stream keeps two device buffers in the plan's
// input layout and alternates between them: a push fills one with the last M
// samples of the other and the new chunk behind them, in one kernel, and runs
// the forward (two buffers, so no copy overlaps itself).
#include <algorithm>
#include <cstring>

#include "dd_internal.h"

struct dd_stream_s {
    dd_plan plan = nullptr;
    void *buf[2] = {nullptr, nullptr};
    int cur = 0;
    int64_t pushed = 0;
};

using namespace dd;

namespace {

constexpr int kFillThreads = 256, kFillAhead = 4;
constexpr long long kFillStep = 16ll * kFillThreads * kFillAhead;  // bytes a CTA fills per step

// Four bytes of memory at any byte address, from the aligned words around it.
// (An aligned word never leaves the 256-byte granule of the allocation that
// holds one of its bytes.)
__device__ __forceinline__ uint32_t word_at(const unsigned char *p) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~uintptr_t(3));
    const uint32_t sh = uint32_t(a & 3) * 8;
    return sh ? __funnelshift_r(w[0], w[1], sh) : w[0];
}

__device__ __forceinline__ uint4 load16(const unsigned char *p) {
    if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) return *reinterpret_cast<const uint4 *>(p);
    return make_uint4(word_at(p), word_at(p + 4), word_at(p + 8), word_at(p + 12));
}

// cur[row][0, m) = prev[row][s, s + m), cur[row][m, m + s) = chunk[row][0, s),
// in bytes; rows of `pitch` bytes (a multiple of 16), chunk rows of s bytes.
// CTA (row, segment) fills `seg` bytes of a row (a multiple of kFillStep), with
// kFillAhead independent 16-byte loads per thread and step whatever the
// alignment of m and s (words across a seam go byte by byte). Bound by memory
// where the launch fills the machine: long rows are cut so that few of them do
// too. What a push takes beyond its forward, against one CTA per row with one
// load in flight, and two pitched copies before and after the forward: 32 rows
// of 8.1 MB 117, 1156 and 197 us; 32 of 1.3 MB 15, 174 and 49; 512 of 13 KB 5.9,
// 6.2 and 12.5; 6144 of 17 KB 34, 35 and 115.
__global__ void __launch_bounds__(kFillThreads)
    dd_stream_fill_kernel(unsigned char *__restrict__ cur, const unsigned char *__restrict__ prev,
                          const unsigned char *__restrict__ chunk, long long pitch, long long m,
                          long long s, long long seg) {
    const long long row = blockIdx.x, first = blockIdx.y * seg, n = m + s;
    const long long last = min(n, first + seg);
    unsigned char *dst = cur + row * pitch;
    const unsigned char *hist = prev + row * pitch + s, *fresh = chunk + row * s - m;
    for (long long o0 = first + 16ll * threadIdx.x; o0 < last; o0 += kFillStep) {
        uint4 v[kFillAhead];
        bool whole[kFillAhead];
#pragma unroll
        for (int q = 0; q < kFillAhead; ++q) {
            const long long o = o0 + q * 16ll * kFillThreads;
            whole[q] = o < last && (o + 16 <= m || (o >= m && o + 16 <= n));
            if (whole[q]) v[q] = load16((o < m ? hist : fresh) + o);
        }
#pragma unroll
        for (int q = 0; q < kFillAhead; ++q) {
            const long long o = o0 + q * 16ll * kFillThreads;
            if (whole[q])
                *reinterpret_cast<uint4 *>(dst + o) = v[q];
            else
                for (long long i = o; i < o + 16 && i < last; ++i)
                    dst[i] = i < m ? hist[i] : fresh[i];
        }
    }
}

}  // namespace

extern "C" {

dd_status dd_stream_create(dd_stream *out, dd_plan plan) {
    if (!out || !plan) return fail(DD_ERR_ARG, "null argument");
    *out = nullptr;
    auto *s = new (std::nothrow) dd_stream_s;
    if (!s) return fail(DD_ERR_NOMEM, "host allocation");
    s->plan = plan;
    const size_t bytes = size_t(plan->B) * plan->C * plan->stride * elt_bytes(plan->dtype);
    for (int i = 0; i < 2; ++i) {
        cudaError_t e = cudaMalloc(&s->buf[i], bytes);
        if (e == cudaSuccess) e = cudaMemset(s->buf[i], 0, bytes);
        if (e != cudaSuccess) {
            dd_stream_destroy(s);
            return cuda_fail(e, "stream buffers");
        }
    }
    *out = s;
    return DD_OK;
}

dd_status dd_stream_reset(dd_stream s, void *stream) {
    if (!s) return fail(DD_ERR_ARG, "null stream");
    const dd_plan p = s->plan;
    const size_t bytes = size_t(p->B) * p->C * p->stride * elt_bytes(p->dtype);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    for (int i = 0; i < 2; ++i) {
        cudaError_t e = cudaMemsetAsync(s->buf[i], 0, bytes, st);
        if (e != cudaSuccess) return cuda_fail(e, "stream reset");
    }
    s->cur = 0;
    s->pushed = 0;
    return DD_OK;
}

dd_status dd_stream_push(dd_stream s, const void *d_chunk, const void *d_w, void *d_out,
                         void *stream) {
    if (!s || !d_chunk || !d_w || !d_out) return fail(DD_ERR_ARG, "null argument");
    if (!aligned16(d_w) || !aligned16(d_out))
        return fail(DD_ERR_ARG, "device pointers must be 16-byte aligned");
    const dd_plan p = s->plan;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long elt = elt_bytes(p->dtype);
    const auto *prev = static_cast<const unsigned char *>(s->buf[1 - s->cur]);
    auto *cur = static_cast<unsigned char *>(s->buf[s->cur]);
    // segments of whole steps, about eight CTAs per SM where the rows are long
    const long long rows = (long long)p->B * p->C, n = (p->S + p->max_shift) * elt;
    const long long steps = (n + kFillStep - 1) / kFillStep;
    const long long want = std::min(steps, std::max(1ll, 8ll * p->sm_count / rows));
    const long long per = (steps + want - 1) / want;
    const dim3 grid(unsigned(rows), unsigned((steps + per - 1) / per));
    dd_stream_fill_kernel<<<grid, kFillThreads, 0, st>>>(
        cur, prev, static_cast<const unsigned char *>(d_chunk), p->stride * elt,
        p->max_shift * elt, p->S * elt, per * kFillStep);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "stream chunk copy");
    const dd_status r = launch_forward(p, p->fwd, cur, d_w, d_out, st);
    if (r != DD_OK) return r;
    s->cur = 1 - s->cur;
    s->pushed += 1;
    return DD_OK;
}

int64_t dd_stream_latency(dd_stream s) { return s ? int64_t(s->plan->max_shift) : -1; }

void dd_stream_destroy(dd_stream s) {
    if (!s) return;
    for (int i = 0; i < 2; ++i)
        if (s->buf[i]) cudaFree(s->buf[i]);
    delete s;
}

}  // extern "C"
