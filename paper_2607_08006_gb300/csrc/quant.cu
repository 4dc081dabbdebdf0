// Reduced-precision float payloads for the sum all-reduce (a precision extension; the
// paper's reductions are inherited from OpenSHMEM 1.6, Sec. 6.3): per-128-element
// block scales, bf16 or OCP FP8 E4M3 codes, dequantised and accumulated in binary32
// with Neumaier compensated summation in team-rank order.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "quant_dev.cuh"

namespace shmemg {

constexpr int Q_THREADS = 256;

// ---------------------------------------------------------------- quantize
struct QArgs {
    uint8_t *heap;
    uint64_t H;
    int start, stride, size;
    uint64_t q_off, s_off, x_off;
    uint64_t n;
};

// The codes of four values, one or two words.
template <int FMT>
__device__ __forceinline__ uint2 q_encode(uint64_t lo, uint64_t hi) {
    if (FMT == SHMEMG_FMT_E4M3)
        return make_uint2((uint32_t)e4m3x2_encode(f2_lo(lo), f2_hi(lo)) | ((uint32_t)e4m3x2_encode(f2_lo(hi), f2_hi(hi)) << 16), 0u);
    return make_uint2((uint32_t)bf16_encode(f2_lo(lo)) | ((uint32_t)bf16_encode(f2_hi(lo)) << 16),
                      (uint32_t)bf16_encode(f2_lo(hi)) | ((uint32_t)bf16_encode(f2_hi(hi)) << 16));
}

// The codes of RN(x / s) for four x, by four divisions only where they decide.  With r = RN(1/s),
// y = RN(x * r) lies within 1.5 * 2^-23 (relative) of RN(x / s): 2^-24 of r, 2^-24 of y, 2^-24 of the
// quotient.  y moved by 2^-21 down and up (and by the two products' own 2^-24) therefore
// encloses the quotient, and encoding is monotonic: where both ends have the same code, that is
// the quotient's.  The ends differ for about one element in 2^16 (E4M3) or 2^12 (bf16).  `safe`: s and
// 1/s far from the ends of binary32's range, so that r is that exact.  Products near or below the
// normal range (2^-126) keep fewer bits than that.  E4M3's first code is far above them: both ends
// give zero, and so does the quotient.  bf16's is 2^-133: a non-zero product below 2^-120 takes
// the divisions (one that rounds to zero is below 2^-149, and its code zero either way; 32 PEs x
// 1 Mi bf16 33.1 us without that look, 33.6 with it).
template <int FMT>
__device__ __forceinline__ uint2 q_codes(const float (&v)[4], float s, float r, bool safe) {
    const uint64_t rr = f2(r, r), dn = f2(1.0f - 0x1p-21f, 1.0f - 0x1p-21f), up = f2(1.0f + 0x1p-21f, 1.0f + 0x1p-21f);
    const uint64_t y0 = f2_mul(f2(v[0], v[1]), rr), y1 = f2_mul(f2(v[2], v[3]), rr);
    const uint2 a = q_encode<FMT>(f2_mul(y0, dn), f2_mul(y1, dn)), b = q_encode<FMT>(f2_mul(y0, up), f2_mul(y1, up));
    safe = safe && a.x == b.x && a.y == b.y;
    if (FMT == SHMEMG_FMT_E4M3) {
        if (safe) return a;
    } else {
        const float least = fminf(fminf(fabsf(f2_lo(y0)), fabsf(f2_hi(y0))), fminf(fabsf(f2_lo(y1)), fabsf(f2_hi(y1))));
        if (safe && least >= 0x1p-120f) return a;
        auto low = [](float y) { return y != 0.0f && fabsf(y) < 0x1p-120f; };
        if (safe && !(low(f2_lo(y0)) || low(f2_hi(y0)) || low(f2_lo(y1)) || low(f2_hi(y1)))) return a;
    }
    return q_encode<FMT>(f2(__fdiv_rn(v[0], s), __fdiv_rn(v[1], s)), f2(__fdiv_rn(v[2], s), __fdiv_rn(v[3], s)));
}

// the codes of elements e0 .. e0 + 3, those below n
template <int FMT>
__device__ __forceinline__ void q_store(const QArgs &a, uint8_t *base, uint64_t e0, bool full, uint2 w) {
    if (FMT == SHMEMG_FMT_E4M3) {
        uint8_t *q = base + a.q_off;
        if (full && ((a.q_off & 3) == 0)) {
            *(uint32_t *)(q + e0) = w.x;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (e0 + j < a.n) q[e0 + j] = (uint8_t)(w.x >> (8 * j));
        }
    } else {
        uint16_t *q = (uint16_t *)(base + a.q_off);
        if (full && ((a.q_off & 7) == 0)) {
            *(uint2 *)(q + e0) = w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (e0 + j < a.n) q[e0 + j] = (uint16_t)((j < 2 ? w.x : w.y) >> (16 * (j & 1)));
        }
    }
}

// A warp takes Q_BLOCKS consecutive 128-element blocks of a member at a time, lane l their
// elements 4l..4l+3: all blocks' loads are in flight before the first is used.
// Bound by its instructions until the divisions went (106 of them per block with five IEEE
// divisions a lane: 35 us for 32 PEs x 1 Mi E4M3, 47.5 with one block at a time), by memory
// now (29.5 us, 168 MB).
constexpr int Q_BLOCKS = 4;
template <int FMT>
__global__ void __launch_bounds__(Q_THREADS) k_quantize(QArgs a) {
    stream_enter();
    const uint64_t nblk = (a.n + 127) / 128, ngrp = (nblk + Q_BLOCKS - 1) / Q_BLOCKS;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    const uint64_t wid = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const float R = FMT == SHMEMG_FMT_E4M3 ? 448.0f : 1.0f;
    const uint64_t total = ngrp * (uint64_t)a.size;
    const bool vec = (a.x_off & 15) == 0;
    for (uint64_t it = wid; it < total; it += warps) {
        const int r = (int)(it / ngrp);
        const uint64_t b0 = (it - (uint64_t)r * ngrp) * Q_BLOCKS;
        uint8_t *base = a.heap + (uint64_t)(a.start + r * a.stride) * a.H;
        const float *x = (const float *)(base + a.x_off);
        float v[Q_BLOCKS][4];
#pragma unroll
        for (int k = 0; k < Q_BLOCKS; k++) {
            const uint64_t e0 = (b0 + k) * 128 + (uint64_t)lane * 4;
            if (vec && (b0 + k + 1) * 128 <= a.n) {
                const float4 t = __ldcs((const float4 *)(x + e0));
                v[k][0] = t.x; v[k][1] = t.y; v[k][2] = t.z; v[k][3] = t.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++) v[k][j] = e0 + j < a.n ? x[e0 + j] : 0.0f;
            }
        }
#pragma unroll
        for (int k = 0; k < Q_BLOCKS; k++) {
            if (b0 + k >= nblk) break;
            const float am = fmaxf(fmaxf(fabsf(v[k][0]), fabsf(v[k][1])), fmaxf(fabsf(v[k][2]), fabsf(v[k][3])));
            const uint32_t amb = __reduce_max_sync(0xffffffffu, __float_as_uint(am));  // |x| bits order like values
            const float amax = __uint_as_float(amb);
            const float s = amax == 0.0f ? 1.0f : FMT == SHMEMG_FMT_E4M3 ? __fdiv_rn(amax, R) : amax;
            const bool safe = s >= 0x1p-100f && s <= 0x1p100f;
            if (lane == 0) ((float *)(base + a.s_off))[b0 + k] = s;
            q_store<FMT>(a, base, (b0 + k) * 128 + (uint64_t)lane * 4, (b0 + k + 1) * 128 <= a.n && vec,
                         q_codes<FMT>(v[k], s, __frcp_rn(s), safe));
        }
    }
}

struct QSumArgs {
    uint8_t *heap;
    uint64_t H;
    int start, stride, size, gstride;
    uint64_t d_off, q_off, s_off;
    uint64_t n;
    bool vec;   // 4-element vector path allowed
    bool wide;  // 16-byte code path allowed
};

// Full, aligned chunks of blockDim x E elements: each thread accumulates E elements
// (one 4- to 16-byte code load per member) into shared memory and thread 0 bulk-stores the
// chunk to every member (two chunk buffers, so one chunk's stores drain while the next
// is accumulated).  The ragged tail runs in 4-element steps.
template <int FMT, int E>
__global__ void __launch_bounds__(Q_THREADS) k_qsum(QSumArgs a) {
    stream_enter();
    constexpr int M = E == 4 ? 16 : 8;                         // members loaded ahead
    __shared__ __align__(128) float s_out[2][Q_THREADS * E];   // alternate chunk buffers
    const int pe0 = a.start + blockIdx.y * a.gstride;
    const uint64_t CH = (uint64_t)blockDim.x * E;
    const uint64_t nfull = a.wide ? a.n / CH : 0;
    int buf = 0;
    for (uint64_t ch = blockIdx.x; ch < nfull; ch += gridDim.x) {
        qsum_chunk_tma<FMT, M, E>(a.heap, a.H, pe0, a.stride, a.size, a.d_off, a.q_off, a.s_off, ch * CH, s_out[buf]);
        buf ^= 1;
    }
    // the tail: the last CTAs first (they have a chunk less where the chunks don't come out even)
    const uint64_t t0 = nfull * CH;
    for (uint64_t f = t0 + 4 * ((uint64_t)(gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x); f < a.n;
         f += 4 * (uint64_t)gridDim.x * blockDim.x)
        qsum4<FMT>(a.heap, a.H, pe0, a.stride, a.size, a.d_off, a.q_off, a.s_off, f, a.n, a.vec);
    if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Elements per thread: 4 -- the most chunks, and 16 members ahead -- until chunks of 8 give
// every resident CTA two or more.  Measured, quantise and sum together: E4M3 64 PEs x 20000
// elements 58 / 30 / 20 us with 16 / 8 / 4, 32 PEs x 1 Mi 72.5 / 67.8 / 67.0, 4 PEs x 4 M 39.2 /
// 37.4 / 39.5; bf16 41 PEs x 156928 36 / 27 with 8 / 4, 8 PEs x 4 M 71.4 / 73.9.
template <int FMT, int E>
static void launch_qsum_e(const QSumArgs &a, int ngroups, cudaStream_t s) {
    const uint64_t need = (a.n + Q_THREADS * E - 1) / (Q_THREADS * E);
    const uint64_t cap = (uint64_t)ctas_for((const void *)k_qsum<FMT, E>, Q_THREADS, 0);
    // a chunk per CTA while that is at most eight rounds of the resident ones (64 PEs x 1 M: 120
    // us with resident CTAs taking chunks in turn, 115 so)
    const uint64_t gx = need * (uint64_t)ngroups <= 8 * cap ? need : balanced_grid(need, cap, ngroups);
    dim3 grid((unsigned)gx, (unsigned)ngroups);
    launch_chained(k_qsum<FMT, E>, grid, Q_THREADS, 0, s, a);
}
template <int FMT>
static void launch_qsum(const QSumArgs &a, int ngroups, cudaStream_t s) {
    const uint64_t two = 2 * (uint64_t)ctas_for((const void *)k_qsum<FMT, 8>, Q_THREADS, 0);
    if (a.n / (Q_THREADS * 8) * (uint64_t)ngroups >= two) launch_qsum_e<FMT, 8>(a, ngroups, s);
    else launch_qsum_e<FMT, 4>(a, ngroups, s);
}

}  // namespace shmemg

using namespace shmemg;

extern "C" {

int shmemg_quantize(shmemg_team_t team, void *q, float *scales, const float *src, int fmt, uint64_t n, void *stream) {
    if (int rc = check_init()) return rc;
    HostTeam t;
    if (team_get(team, &t)) return SHMEMG_ERR_INVALID_ARG;
    if (fmt != SHMEMG_FMT_BF16 && fmt != SHMEMG_FMT_E4M3) return SHMEMG_ERR_INVALID_ARG;
    const uint64_t qs = fmt == SHMEMG_FMT_E4M3 ? 1 : 2, nb = (n + 127) / 128;
    uint64_t qo, so, xo;
    if (sym_offset(q, n * qs, &qo) || sym_offset(scales, nb * 4, &so) || sym_offset(src, n * 4, &xo))
        return SHMEMG_ERR_NOT_SYMMETRIC;
    if ((so & 3) || (xo & 3) || (qo % qs)) return SHMEMG_ERR_INVALID_ARG;
    if (n == 0) return SHMEMG_SUCCESS;
    State &S = st();
    QArgs a;
    a.heap = S.heap;
    a.H = S.H;
    a.q_off = qo;
    a.s_off = so;
    a.x_off = xo;
    a.n = n;
    a.stride = t.stride;
    a.size = t.size;
    const bool e4 = fmt == SHMEMG_FMT_E4M3;
    const uint64_t cap = (uint64_t)ctas_for(e4 ? (const void *)k_quantize<SHMEMG_FMT_E4M3> : (const void *)k_quantize<SHMEMG_FMT_BF16>, Q_THREADS, 0);
    for (int g = 0; g < t.ngroups; g++) {
        a.start = t.start + g * t.gstride;
        const uint64_t warps = (nb + Q_BLOCKS - 1) / Q_BLOCKS * (uint64_t)t.size;
        const uint64_t ctas = (warps + (Q_THREADS / 32) - 1) / (Q_THREADS / 32);
        const unsigned grid = (unsigned)(ctas <= 64 * cap ? ctas : balanced_grid(ctas, cap));
        if (e4) launch_chained(k_quantize<SHMEMG_FMT_E4M3>, grid, Q_THREADS, 0, to_stream(stream), a);
        else launch_chained(k_quantize<SHMEMG_FMT_BF16>, grid, Q_THREADS, 0, to_stream(stream), a);
    }
    return cuda_rc(cudaGetLastError());
}

int shmemg_qsum_reduce(shmemg_team_t team, float *dst, const void *q, const float *scales, int fmt, uint64_t n,
                       void *stream) {
    if (int rc = check_init()) return rc;
    HostTeam t;
    if (team_get(team, &t)) return SHMEMG_ERR_INVALID_ARG;
    if (fmt != SHMEMG_FMT_BF16 && fmt != SHMEMG_FMT_E4M3) return SHMEMG_ERR_INVALID_ARG;
    const uint64_t qs = fmt == SHMEMG_FMT_E4M3 ? 1 : 2, nb = (n + 127) / 128;
    uint64_t qo, so, d;
    if (sym_offset(q, n * qs, &qo) || sym_offset(scales, nb * 4, &so) || sym_offset(dst, n * 4, &d))
        return SHMEMG_ERR_NOT_SYMMETRIC;
    if ((so & 3) || (d & 3) || (qo % qs)) return SHMEMG_ERR_INVALID_ARG;
    // dst must not overlap the payload or the scales (they are read by other threads)
    if ((d < qo + n * qs && qo < d + n * 4) || (d < so + nb * 4 && so < d + n * 4)) return SHMEMG_ERR_INVALID_ARG;
    if (n == 0) return SHMEMG_SUCCESS;
    State &S = st();
    QSumArgs a;
    a.heap = S.heap;
    a.H = S.H;
    a.start = t.start;
    a.stride = t.stride;
    a.size = t.size;
    a.gstride = t.gstride;
    a.d_off = d;
    a.q_off = qo;
    a.s_off = so;
    a.n = n;
    a.vec = (d & 15) == 0 && (qo & (fmt == SHMEMG_FMT_E4M3 ? 3 : 7)) == 0;
    a.wide = (d & 15) == 0 && (qo & 15) == 0;
    if (fmt == SHMEMG_FMT_E4M3) launch_qsum<SHMEMG_FMT_E4M3>(a, t.ngroups, to_stream(stream));
    else launch_qsum<SHMEMG_FMT_BF16>(a, t.ngroups, to_stream(stream));
    return cuda_rc(cudaGetLastError());
}

}  // extern "C"
