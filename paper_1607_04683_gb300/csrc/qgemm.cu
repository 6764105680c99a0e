// qgemm.cu — eq. (1): 8-bit code products with 32-bit accumulators, offset terms and recovery.
//
// Datapath for a few rows of A. sm_103a accepts no 8-bit integer tcgen05 MMA, so the exact integer
// product runs on the warp-level integer tensor-core instruction mma.sync m16n8k32 (u8 x u8 ->
// s32), with both operands streamed straight from global memory into its fragments.
//
// Epilogue (fused): S = acc + zw*rsA[m] + za[m]*csW[n] + K*za*zw in 64-bit integers (eq. 1 with
// V'' = V' + round(Q Vmin)), then y = S / (Qa Qw) + bias (eq. 3 recovery and Fig. 1's bias), and
// optionally the raw accumulator.
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "qnn_device.cuh"
#include "qnn_host.h"

namespace qnn {
namespace {

constexpr int kWarps = 8, THREADS = 32 * kWarps;

__device__ __forceinline__ void mma_u8(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 16 codes at p of which the first `valid` lie inside the row (the rest read as 0, which adds nothing
// to the sums). AL is the alignment every row start of the matrix has (16, 4 or 1 bytes).
template <int AL, bool kStream>
__device__ __forceinline__ uint4 ld_codes16(const uint8_t *__restrict__ p, int valid) {
    uint4 v = make_uint4(0, 0, 0, 0);
    if (valid >= 16) {
        if constexpr (AL == 16) {
            if constexpr (kStream)
                asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                    : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                    : "l"(p));
            else
                v = __ldg(reinterpret_cast<const uint4 *>(p));
        } else if constexpr (AL == 4) {
            const uint32_t *w = reinterpret_cast<const uint32_t *>(p);
            v = make_uint4(__ldg(w), __ldg(w + 1), __ldg(w + 2), __ldg(w + 3));
        } else {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                w[i] = (uint32_t)__ldg(p + 4 * i) | (uint32_t)__ldg(p + 4 * i + 1) << 8 |
                       (uint32_t)__ldg(p + 4 * i + 2) << 16 | (uint32_t)__ldg(p + 4 * i + 3) << 24;
            v = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else if (valid > 0) {
        uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < valid) w[i >> 2] |= (uint32_t)__ldg(p + i) << (8 * (i & 3));
        v = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return v;
}

// The product for a few rows of A: 16 MT rows of W x 8 NT rows of A per block, K spread over the
// block's warps. W is the m16 side of mma.sync m16n8k32, so eight rows of A cost one instruction's
// columns and a single row wastes columns, not loads. Each warp takes every kWarps-th 64-code chunk
// of K: lane (g, tq) loads 16 consecutive codes (offset 16 tq) of rows g and g + 8 of W and of row g
// of A, and uses words 0-1 and 2-3 as the fragments of two MMAs. Both operands permute k the same way,
// so the sums are the same integers; nothing passes through shared memory but the warps' partial sums,
// which integer atomics add exactly in any order.
//
// Bound: the bytes of W once (N K), and at small sizes the latency of one load round, the reduction
// and the epilogue. Sixteen rows a block because tiles of 128 rows leave a 2048-row W on 16 of 152
// SMs with 32 serial k-steps. Event-timed, 128-row tiles against this split: M = 1, 2048 x 2048 84 ->
// 8.2 us; M = 100, 2000 x 500 (rows 4-byte aligned) 67 -> 14 us. M = 1, 8192 x 8192: 16.3 us a call,
// 4.1 TB/s (20.5 us with three blocks an SM, whose last wave is nearly empty; four chunks in flight
// a warp with four blocks an SM gain nothing more).
template <int NT, int MT, int AL>
__global__ void __launch_bounds__(THREADS, NT == 1 ? 4 : NT == 2 ? 3 : NT == 4 ? 2 : 1) qgemm_imma_kernel(
    const uint8_t *__restrict__ A, int64_t lda, const qnn_qparams *__restrict__ pa, int a_per_row,
    const int32_t *__restrict__ rsA, int64_t M, int K, const uint8_t *__restrict__ W, int64_t ldw,
    const qnn_qparams *__restrict__ pw, int64_t rows_per_block, const int32_t *__restrict__ csW, int64_t N,
    const float *__restrict__ bias, float *__restrict__ Y, int64_t ldy, int32_t *__restrict__ acc_out,
    unsigned n_tiles) {
    constexpr int ROWS = 16 * MT, COLS = 8 * NT;
    constexpr int U = NT == 4 ? 4 : 2;  // chunks of W in flight per warp
    __shared__ int s_acc[COLS][ROWS + 1];
    const int64_t n0 = (int64_t)(blockIdx.x % n_tiles) * ROWS, m0 = (int64_t)(blockIdx.x / n_tiles) * COLS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
    for (int i = threadIdx.x; i < COLS * (ROWS + 1); i += THREADS) s_acc[0][i] = 0;
    // the constants of this thread's first output, loaded ahead of the products
    const int e_r = threadIdx.x % ROWS;
    const int64_t e_n = n0 + e_r;
    int e_cs = 0;
    float e_bias = 0.0f;
    qnn_qparams e_w{};
    if (e_n < N) {
        e_cs = csW[e_n];
        e_w = pw[e_n / rows_per_block];
        if (bias) e_bias = bias[e_n];
    }

    int acc[MT][NT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0;
    // rows past the end repeat the last one (their sums are dropped), so that the loads of whole
    // chunks need no predicates
    const uint8_t *wr[MT][2], *ar[NT];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) wr[i][h] = W + min(n0 + 16 * i + 8 * h + g, N - 1) * ldw + 16 * tq;
#pragma unroll
    for (int j = 0; j < NT; ++j) ar[j] = A + min(m0 + 8 * j + g, M - 1) * lda + 16 * tq;
    auto multiply = [&](const uint4 (&w)[MT][2], int k, int valid) {
        uint4 a[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) a[j] = ld_codes16<AL, false>(ar[j] + k, valid);
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            const uint4 lo = w[i][0], hi = w[i][1];
            const uint32_t f0[4] = {lo.x, hi.x, lo.y, hi.y}, f1[4] = {lo.z, hi.z, lo.w, hi.w};
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                mma_u8(acc[i][j], f0, a[j].x, a[j].y);
                mma_u8(acc[i][j], f1, a[j].z, a[j].w);
            }
        }
    };
    auto load_w = [&](uint4 (&w)[MT][2], int k, int valid) {
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) w[i][h] = ld_codes16<AL, true>(wr[i][h] + k, valid);
    };
    // a round's U chunks are consecutive (256 bytes of a row) when every warp then has some, else
    // spread over the warps; the ragged last chunk goes to the warp after the one with the last whole one
    const int whole = K / 64;
    const bool wide = whole >= kWarps * U;
    const int cu = wide ? 1 : kWarps;
    for (int c0 = wide ? warp * U : warp; c0 < whole; c0 += kWarps * U) {
        uint4 w[U][MT][2];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (u == 0 || c0 + cu * u < whole) load_w(w[u], 64 * (c0 + cu * u), 16);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (u == 0 || c0 + cu * u < whole) multiply(w[u], 64 * (c0 + cu * u), 16);
    }
    const bool tail = whole * 64 < K && warp == whole % kWarps;
    if (tail) {
        uint4 w[MT][2];
        load_w(w, 64 * whole, K - 64 * whole - 16 * tq);
        multiply(w, 64 * whole, K - 64 * whole - 16 * tq);
    }
    __syncthreads();  // s_acc is clear
    if (warp < whole || tail) {
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int col = 8 * j + 2 * tq + (e & 1);
                    if (m0 + col < M) atomicAdd(&s_acc[col][16 * i + 8 * (e >> 1) + g], acc[i][j][e]);
                }
    }
    __syncthreads();

    // Epilogue: offsets, recovery, bias (THREADS is a multiple of ROWS: each thread keeps its W row).
    if (e_n >= N) return;
    for (int c = threadIdx.x / ROWS; c < COLS; c += THREADS / ROWS) {
        const int64_t m = m0 + c;
        if (m >= M) break;
        const qnn_qparams qa = pa[a_per_row ? m : 0];
        const int a = s_acc[c][e_r];
        const long long S = offset_product(a, qa.z, e_w.z, rsA[m], e_cs, K);
        float y = recover_product(S, qa.Q, e_w.Q);
        if (bias) y = __fadd_rn(y, e_bias);
        if (Y) Y[m * ldy + e_n] = y;
        if (acc_out) acc_out[m * N + e_n] = a;
    }
}

}  // namespace

qnn_status launch_qgemm_imma(const uint8_t *A, int64_t lda, const qnn_qparams *pa, int ga, const int32_t *rsA,
                             int64_t M, int64_t K, const uint8_t *W, int64_t ldw, const qnn_qparams *pw,
                             int64_t rows_per_block, const int32_t *csW, int64_t N, const float *bias, float *Y,
                             int64_t ldy, int32_t *acc_out, cudaStream_t st) {
    if (M == 0 || N == 0) return QNN_OK;
    const uintptr_t at = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(W) | (uintptr_t)lda | (uintptr_t)ldw;
    const int al = (at & 15) == 0 ? 16 : (at & 3) == 0 ? 4 : 1;
    ProfScope prof("qgemm_imma", st);
    auto run = [&](auto nt, auto mt) -> qnn_status {
        constexpr int NT = decltype(nt)::value, MT = decltype(mt)::value;
        const int64_t n_tiles = (N + 16 * MT - 1) / (16 * MT), m_tiles = (M + 8 * NT - 1) / (8 * NT);
        if (n_tiles * m_tiles > INT32_MAX) return QNN_FAIL(QNN_ERR_INVALID_ARG);
        auto kern = al == 16  ? qgemm_imma_kernel<NT, MT, 16>
                    : al == 4 ? qgemm_imma_kernel<NT, MT, 4>
                              : qgemm_imma_kernel<NT, MT, 1>;
        kern<<<(unsigned)(n_tiles * m_tiles), THREADS, 0, st>>>(A, lda, pa, ga == QNN_PER_ROW, rsA, M, (int)K, W, ldw, pw,
                                                               rows_per_block, csW, N, bias, Y, ldy, acc_out,
                                                               (unsigned)n_tiles);
        QNN_CUDA_TRY(cudaGetLastError());
        return QNN_OK;
    };
    using std::integral_constant;
    if (M <= 8) return run(integral_constant<int, 1>{}, integral_constant<int, 1>{});
    if (M <= 16) return run(integral_constant<int, 2>{}, integral_constant<int, 1>{});
    if (M <= 32) return run(integral_constant<int, 4>{}, integral_constant<int, 1>{});
    return run(integral_constant<int, 8>{}, integral_constant<int, 2>{});
}

// Datapath choice, between three kernels that differ in what they do to the operands first:
//   - the streaming integer MMA kernel, nothing at all: up to 32 rows of A (2048 x 2048: 8.3 us at M = 32 against
//     10.3 for the codes kernel), and up to 127 for K below 2048 while its blocks (64 rows of A, 32 of W) are one
//     wave (33 x 1000 x 1000: 12.4 against 14.4; but 64 x 2048 x 2048: 16.5 against 10.4; 127 x 4096 x 4096: 49.8
//     against 21.0);
//   - the codes kernel, converting on the way into shared memory: up to 127 rows beyond that (127 x 8000 x 500:
//     13.4 against 32.9), and from 128 on while its tiles of 128 x 128 are one wave (M = 256, 8192 x 8192: 72 against
//     88 us; at two waves M = 512: 161 against 108; 1536 x 2000 x 500: 31 against 25), and its rows lie on 128-byte
//     lines or are short (1100 x 2000 x 500: 15.6 against 16.5), or, on 16-byte boundaries, its tiles of 128 x 64 are
//     one wave (300 x 3004 x 3008: 23.8 against 30.8; 512 x 4096 x 4000: 46 against 39), or these are so few that two
//     blocks or more share each (600 x 600 x 3001: 22.6 against 28.8; but 1000 x 1000 x 3001, which do not: 32.5
//     against 30.8);
//   - the fp16 tensor-core product after a pass that centers both operands into scratch: the rest.
// QNN_QGEMM=imma, =codes or =tc forces one (tests compare them).
qnn_status launch_qgemm(const uint8_t *A, int64_t lda, const qnn_qparams *pa, int ga, const int32_t *rsA, int64_t M,
                        int64_t K, const uint8_t *W, int64_t ldw, const qnn_qparams *pw, int64_t rows_per_block,
                        const int32_t *csW, int64_t N, const float *bias, float *Y, int64_t ldy, int32_t *acc_out,
                        cudaStream_t st) {
    if (M == 0 || N == 0) return QNN_OK;
    const char *force = std::getenv("QNN_QGEMM");
    enum { kImma, kCodes, kTc } path = kTc;
    const int64_t sms = sm_count();
    if (M < 128) {  // (neither takes scratch)
        path = M <= 32 || (K < 2048 && (M + 63) / 64 * ((N + 31) / 32) <= sms) ? kImma : kCodes;
    } else if ((M + 127) / 128 * ((N + 127) / 128) <= sms) {
        const uintptr_t at = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(W) | (uintptr_t)lda | (uintptr_t)ldw;
        const int64_t tiles = (M + 63) / 64 * ((N + 127) / 128);  // of 128 x 64
        if (K <= 512 || at % 128 == 0 || (at % 16 == 0 && tiles <= sms) || 16 * tiles <= 7 * sms) path = kCodes;
    }
    if (force && std::strcmp(force, "imma") == 0) path = kImma;
    if (force && std::strcmp(force, "codes") == 0) path = kCodes;
    if (force && std::strcmp(force, "tc") == 0) path = kTc;
    // the codes kernel loads aligned 16-byte units, and each operand has to hold one
    if (path == kCodes && ((M - 1) * lda + K < 31 || (N - 1) * ldw + K < 31)) path = kTc;
    if (path == kCodes)
        return launch_qgemm_codes(A, lda, pa, ga, rsA, M, K, W, ldw, pw, rows_per_block, csW, N, bias, Y, ldy, acc_out, st);
    if (path == kTc) {
        Scratch ws;
        QNN_TRY(ws.take(tc_scratch_bytes(M, N, K), st));
        return launch_qgemm_tc(A, lda, pa, ga, rsA, M, K, W, ldw, pw, rows_per_block, csW, N, bias, Y, ldy, acc_out,
                               ws.ptr(), st);
    }
    return launch_qgemm_imma(A, lda, pa, ga, rsA, M, K, W, ldw, pw, rows_per_block, csW, N, bias, Y, ldy, acc_out, st);
}

}  // namespace qnn

using namespace qnn;

extern "C" qnn_status qnn_qmatmul(const uint8_t *A, int64_t lda, const qnn_qparams *pa, int ga, const int32_t *rsA,
                                  int64_t M, int64_t K, const uint8_t *W, int64_t ldw, const qnn_qparams *pw,
                                  int64_t n_blocks, const int32_t *csW, int64_t N, const float *bias, float *Y,
                                  int64_t ldy, int32_t *acc_out, void *stream) {
    if (M < 0 || N <= 0 || K <= 0 || lda < K || ldw < K || n_blocks <= 0 || N % n_blocks) return QNN_ERR_INVALID_ARG;
    if (ga != QNN_PER_MATRIX && ga != QNN_PER_ROW) return QNN_ERR_INVALID_ARG;
    if (K > QNN_K_MAX) return QNN_ERR_K_TOO_LARGE;
    if (Y && ldy < N) return QNN_ERR_INVALID_ARG;
    if (M == 0) return QNN_OK;
    if (!is_device_ptr(A) || !is_device_ptr(pa) || !is_device_ptr(rsA) || !is_device_ptr(W) || !is_device_ptr(pw) ||
        !is_device_ptr(csW) || (bias && !is_device_ptr(bias)) || (Y && !is_device_ptr(Y)) ||
        (acc_out && !is_device_ptr(acc_out)))
        return QNN_ERR_INVALID_ARG;
    return launch_qgemm(A, lda, pa, ga, rsA, M, K, W, ldw, pw, N / n_blocks, csW, N, bias, Y, ldy, acc_out,
                        as_stream(stream));
}
