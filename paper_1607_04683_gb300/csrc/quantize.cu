// quantize.cu — the on-the-fly activation quantizer (Sec. 3 "Quantizing", eq. 2) on sm_103a.
//
// Two passes over each unit: a range pass (exact fp32 min/max, warp shuffles; non-finite values
// flagged) and a code pass (eq. 2 with the unit's Q and z, four codes per 32-bit store, row code
// sums). Per-row units (one frame of one sequence) take one warp per row; aligned rows of up to 1024
// values, and any of up to 256, stay in the warp's registers between the passes (read once), longer
// ones are re-read from L1/L2. A per-matrix unit first reduces block partials into a small scratch array; the last
// block to finish folds them into the unit's parameters, then a second launch writes codes.
//
// Bound: HBM (5 bytes a value for rows, 9 for a matrix beyond L2). Per matrix 8192 x 8192: 118 us with one
// 16-byte load in flight a lane and both passes from HBM; 98.5 us with eight in flight and the code pass
// starting where the range pass ended, in rows that L2 still holds.
#include <algorithm>
#include <cfloat>
#include <cstdlib>

#include "qnn_device.cuh"
#include "qnn_host.h"

namespace qnn {

namespace {

constexpr int kRowWarps = 8;  // warps (rows) per block in the per-row kernels

constexpr int kFlight = 8;    // loads (of 16 bytes, or of one value where rows are not aligned) in flight per lane in the
                              // passes over rows of at least kMidRow values (22002 x 2727: 174 us with one, so 101);
constexpr int kMidRow = 512;  // shorter ones take one, and the registers of more rows at once (100000 x 60: range 28 us
                              // with eight, 21 with one)
// Matrix rows that are not aligned, a value a load: eight in flight from 128 values on, four from 64 (one, four and
// eight: 200000 x 65 57, 51 and 60 us, x 95 67, 57 and 65; 150000 x 129 60, 63 and 54, 256410 x 234 178, 133 and 108). The last kLooseRest values or fewer
// go one by one (100000 x 257 58.2 us with a second round of eight for one value, so 53.9). WHOLE: whole rounds take no
// tests, for rows of their own (7722 x 7770 109 us with a test a value, so 98; 40000 x 600 31 and 27) but not for matrices
// (22002 x 2727 103 us with tests, 116 without).
constexpr int kLooseRest = 64;
inline int loose_flight(int64_t cols) { return cols >= 128 ? kFlight : cols >= 64 ? 4 : 1; }

// Running range of values and whether one was not finite: v * 0 is NaN then, and so is the sum.
struct Range {
    float mn = FLT_MAX, mx = -FLT_MAX, bad = 0.0f;
    __device__ __forceinline__ void add(float v) {
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
        bad = __fmaf_rn(v, 0.0f, bad);
    }
    __device__ __forceinline__ void add(const float4 &v) { add(v.x), add(v.y), add(v.z), add(v.w); }
    __device__ __forceinline__ bool finite() const { return bad == 0.0f; }
};

// Range of one row held by one warp; returns false if a value is not finite.
template <bool kVec, int F, bool WHOLE = false>
__device__ __forceinline__ bool warp_row_range(const float *__restrict__ xr, int cols, float &mn, float &mx) {
    const int lane = threadIdx.x & 31;
    Range r;
    int done = 0;
    if (kVec) {
        const float4 *x4 = reinterpret_cast<const float4 *>(xr);
        const int n4 = cols >> 2;
        for (int i = lane; i < n4; i += 32 * F) {
            float4 v[F];
#pragma unroll
            for (int u = 0; u < F; ++u)
                if (i + 32 * u < n4) v[u] = __ldg(x4 + i + 32 * u);
#pragma unroll
            for (int u = 0; u < F; ++u)
                if (i + 32 * u < n4) r.add(v[u]);
        }
        done = n4 << 2;
    }
    if (!kVec && F > 1) {
        for (; WHOLE && done + 32 * F <= cols; done += 32 * F) {
            float v[F];
#pragma unroll
            for (int u = 0; u < F; ++u) v[u] = __ldg(xr + done + lane + 32 * u);
#pragma unroll
            for (int u = 0; u < F; ++u) r.add(v[u]);
        }
        for (; cols - done > kLooseRest; done += 32 * F) {
            float v[F];
            const int i = done + lane;
#pragma unroll
            for (int u = 0; u < F; ++u)
                if (i + 32 * u < cols) v[u] = __ldg(xr + i + 32 * u);
#pragma unroll
            for (int u = 0; u < F; ++u)
                if (i + 32 * u < cols) r.add(v[u]);
        }
    }
    for (int i = done + lane; i < cols; i += 32) r.add(__ldg(xr + i));
    mn = warp_min(r.mn);
    mx = warp_max(r.mx);
    return __all_sync(0xffffffffu, r.finite());
}

// Codes of one row (eq. 2) and their sum, one warp.
template <bool kVec, int F, bool WHOLE = false>
__device__ __forceinline__ int warp_row_codes(const float *__restrict__ xr, int cols, const UnitCoder &unit,
                                              uint8_t *__restrict__ cr) {
    const int lane = threadIdx.x & 31;
    int s = 0;
    if (kVec) {
        const float4 *x4 = reinterpret_cast<const float4 *>(xr);
        uint32_t *c4 = reinterpret_cast<uint32_t *>(cr);
        const int n4 = cols >> 2;
        for (int i = lane; i < n4; i += 32 * F) {
            float4 v[F];
#pragma unroll
            for (int u = 0; u < F; ++u)
                if (i + 32 * u < n4) v[u] = __ldg(x4 + i + 32 * u);
#pragma unroll
            for (int u = 0; u < F; ++u) {
                if (i + 32 * u >= n4) break;
                const uint32_t a = unit.code(v[u].x), b = unit.code(v[u].y), c = unit.code(v[u].z),
                               d = unit.code(v[u].w);
                s += (int)(a + b + c + d);
                c4[i + 32 * u] = a | (b << 8) | (c << 16) | (d << 24);
            }
        }
        for (int i = (n4 << 2) + lane; i < cols; i += 32) {
            uint32_t a = unit.code(__ldg(xr + i));
            s += (int)a;
            cr[i] = (uint8_t)a;
        }
    } else {
        int done = 0;
        for (; WHOLE && F > 1 && done + 32 * F <= cols; done += 32 * F) {
            float v[F];
#pragma unroll
            for (int u = 0; u < F; ++u) v[u] = __ldg(xr + done + lane + 32 * u);
#pragma unroll
            for (int u = 0; u < F; ++u) {
                const uint32_t a = unit.code(v[u]);
                s += (int)a;
                cr[done + lane + 32 * u] = (uint8_t)a;
            }
        }
        for (; F > 1 && cols - done > kLooseRest; done += 32 * F) {
            float v[F];
            const int i = done + lane;
#pragma unroll
            for (int u = 0; u < F; ++u)
                if (i + 32 * u < cols) v[u] = __ldg(xr + i + 32 * u);
#pragma unroll
            for (int u = 0; u < F; ++u) {
                if (i + 32 * u >= cols) break;
                const uint32_t a = unit.code(v[u]);
                s += (int)a;
                cr[i + 32 * u] = (uint8_t)a;
            }
        }
        for (int i = done + lane; i < cols; i += 32) {
            const uint32_t a = unit.code(__ldg(xr + i));
            s += (int)a;
            cr[i] = (uint8_t)a;
        }
    }
    return warp_sum(s);
}

// Per-row units of at most 32 N values, a warp a row, N values a lane in registers: short rows of any alignment, and
// those of up to 256 values that are not aligned. (200000 x 40 by the passes of the kernel below 46 us, so 32; 100000 x 201
// 31 and 28; aligned, by the kernel after it with one float4 a lane, x 32 49 us, so 29, x 128 44 and 41.)
template <int N>
__global__ void __launch_bounds__(kRowWarps * 32) quantize_short_rows_kernel(const float *__restrict__ x, int64_t rows, int cols,
                                                                            int64_t ldx, uint8_t *__restrict__ codes, int64_t ldc,
                                                                            qnn_qparams *__restrict__ params,
                                                                            int32_t *__restrict__ sums, int *status) {
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    if (row >= rows) return;
    const float *xr = x + row * ldx + lane;
    float v[N];
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (lane + 32 * i < cols) v[i] = __ldg(xr + 32 * i);
    Range r;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (lane + 32 * i < cols) r.add(v[i]);
    float mn = warp_min(r.mn), mx = warp_max(r.mx);
    if (!__all_sync(0xffffffffu, r.finite())) {
        if (lane == 0) record_status(status, QNN_ERR_NONFINITE);
        mn = 0.0f;
        mx = 0.0f;
    }
    const qnn_qparams p = params_from_range(mn, mx);
    const UnitCoder unit(p.Q, p.z);
    uint8_t *cr = codes + row * ldc + lane;
    int s = 0;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (lane + 32 * i < cols) {
            const uint32_t a = unit.code(v[i]);
            s += (int)a;
            cr[32 * i] = (uint8_t)a;
        }
    s = warp_sum(s);
    if (lane == 0) {
        params[row] = p;
        if (sums) sums[row] = s;
    }
}

template <bool kVec, int F>
__global__ void __launch_bounds__(kRowWarps * 32) quantize_rows_kernel(const float *__restrict__ x, int64_t rows,
                                                                      int cols, int64_t ldx, uint8_t *__restrict__ codes,
                                                                      int64_t ldc, qnn_qparams *__restrict__ params,
                                                                      int32_t *__restrict__ sums, int *status) {
    const int64_t row = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    if (row >= rows) return;
    const float *xr = x + row * ldx;
    float mn, mx;
    bool ok = warp_row_range<kVec, F, true>(xr, cols, mn, mx);
    if (!ok) {
        if ((threadIdx.x & 31) == 0) record_status(status, QNN_ERR_NONFINITE);
        mn = 0.0f;
        mx = 0.0f;
    }
    qnn_qparams p = params_from_range(mn, mx);
    int s = warp_row_codes<kVec, F, true>(xr, cols, UnitCoder(p.Q, p.z), codes + row * ldc);
    if ((threadIdx.x & 31) == 0) {
        params[row] = p;
        if (sums) sums[row] = s;
    }
}

// Per-row units of 129 to 1024 values (16-byte aligned input rows): the warp holds its row in
// registers, NV float4 per lane, so the row is read once and the code pass needs no second read. A warp
// takes every gridDim kRowWarps-th row, and rows of at most 512 values are loaded while the row before is
// reduced and coded: the loads of one row alone leave memory idle through its reductions (128000 x 500:
// 72.0 us, 4.5 TB/s, with a row a warp; 55.3 us, 5.8 TB/s, so).
template <int NV>
__device__ __forceinline__ void load_row(float4 (&v)[NV], const float *__restrict__ xr, int cols) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int k = 4 * (lane + 32 * i);
        if (k + 4 <= cols) {
            v[i] = __ldg(reinterpret_cast<const float4 *>(xr + k));
        } else {  // ragged end of the row
            v[i].x = k < cols ? __ldg(xr + k) : 0.0f;
            v[i].y = k + 1 < cols ? __ldg(xr + k + 1) : 0.0f;
            v[i].z = k + 2 < cols ? __ldg(xr + k + 2) : 0.0f;
            v[i].w = k + 3 < cols ? __ldg(xr + k + 3) : 0.0f;
        }
    }
}

// Blocks per SM the registers leave room for.
constexpr int rows_reg_blocks(int NV) { return NV <= 2 ? 5 : NV <= 4 ? 4 : 3; }

template <int NV>
__global__ void __launch_bounds__(kRowWarps * 32, rows_reg_blocks(NV))
    quantize_rows_reg_kernel(const float *__restrict__ x, int64_t rows, int cols, int64_t ldx, uint8_t *__restrict__ codes,
                             int64_t ldc, qnn_qparams *__restrict__ params, int32_t *__restrict__ sums, int *status,
                             bool pack) {
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * kRowWarps;
    int64_t row = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    if (row >= rows) return;
    float4 v[NV];
    load_row<NV>(v, x + row * ldx, cols);
    while (true) {
        constexpr bool kAhead = NV <= 4;
        float4 w[kAhead ? NV : 1];
        const int64_t next = row + step;
        if constexpr (kAhead)
            if (next < rows) load_row<NV>(w, x + next * ldx, cols);
        Range r;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int k = 4 * (lane + 32 * i);
            if (k + 4 <= cols) {
                r.add(v[i]);
            } else {
                const float e[3] = {v[i].x, v[i].y, v[i].z};
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if (k + j < cols) r.add(e[j]);
            }
        }
        float mn = warp_min(r.mn), mx = warp_max(r.mx);
        if (!__all_sync(0xffffffffu, r.finite())) {
            if (lane == 0) record_status(status, QNN_ERR_NONFINITE);
            mn = 0.0f;
            mx = 0.0f;
        }
        const qnn_qparams p = params_from_range(mn, mx);
        const UnitCoder unit(p.Q, p.z);
        uint8_t *cr = codes + row * ldc;
        int s = 0;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int k = 4 * (lane + 32 * i);
            if (k >= cols) continue;
            const uint32_t a = unit.code(v[i].x), b = unit.code(v[i].y),
                           c = unit.code(v[i].z), d = unit.code(v[i].w);
            if (pack && k + 4 <= cols) {  // 4-byte aligned code rows: one store for four codes
                s += (int)(a + b + c + d);
                *reinterpret_cast<uint32_t *>(cr + k) = a | (b << 8) | (c << 16) | (d << 24);
            } else {
                const uint32_t q4[4] = {a, b, c, d};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (k + j < cols) {
                        s += (int)q4[j];
                        cr[k + j] = (uint8_t)q4[j];
                    }
            }
        }
        s = warp_sum(s);
        if (lane == 0) {
            params[row] = p;
            if (sums) sums[row] = s;
        }
        if (next >= rows) return;
        row = next;
        if constexpr (kAhead) {
#pragma unroll
            for (int i = 0; i < NV; ++i) v[i] = w[i];
        } else {
            load_row<NV>(v, x + row * ldx, cols);
        }
    }
}

// Per-matrix pass 1: block partial ranges; the last block folds them into params[0]. The warps take segments
// of at most kSegment values of the rows in turn, a row's all of one length (whole rows leave a last, nearly empty
// round).
constexpr int kSegment = 2048;
template <bool kVec, int F>
__global__ void __launch_bounds__(kRowWarps * 32) matrix_range_kernel(const float *__restrict__ x, int64_t rows,
                                                                     int cols, int64_t ldx, float *__restrict__ partials,
                                                                     unsigned *__restrict__ counter,
                                                                     qnn_qparams *__restrict__ params, int *status) {
    __shared__ float s_mn[kRowWarps], s_mx[kRowWarps];
    __shared__ int s_bad;
    __shared__ bool s_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    float mn = FLT_MAX, mx = -FLT_MAX;
    grid_dependents_launch();
    const int segs = (cols - 1) / kSegment + 1, seg = ((cols + segs - 1) / segs + 3) & ~3;
    auto add = [&](const float *xs, int n) {
        float a, b;
        if (!warp_row_range<kVec, F>(xs, n, a, b)) {
            if (lane == 0) s_bad = 1;
        } else {
            mn = fminf(mn, a);
            mx = fmaxf(mx, b);
        }
    };
    const int64_t first = (int64_t)blockIdx.x * kRowWarps + warp, step = (int64_t)gridDim.x * kRowWarps;
    if (segs == 1) {
        for (int64_t row = first; row < rows; row += step) add(x + row * ldx, cols);
    } else {
        for (int64_t i = first; i < rows * segs; i += step) {
            const int64_t row = i / segs;
            const int k0 = (int)(i - row * segs) * seg;
            add(x + row * ldx + k0, min(seg, cols - k0));
        }
    }
    if (lane == 0) {
        s_mn[warp] = mn;
        s_mx[warp] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kRowWarps; ++w) {
            mn = fminf(mn, s_mn[w]);
            mx = fmaxf(mx, s_mx[w]);
        }
        if (s_bad) record_status(status, QNN_ERR_NONFINITE);
        partials[2 * blockIdx.x] = mn;
        partials[2 * blockIdx.x + 1] = mx;
        __threadfence();
        unsigned done = atomicAdd(counter, 1u);
        s_last = (done == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (warp == 0) {
        mn = FLT_MAX;
        mx = -FLT_MAX;
        for (unsigned b = lane; b < gridDim.x; b += 32) {
            mn = fminf(mn, __ldcg(partials + 2 * b));
            mx = fmaxf(mx, __ldcg(partials + 2 * b + 1));
        }
        mn = warp_min(mn);
        mx = warp_max(mx);
        if (mn > mx) {  // every value was non-finite
            mn = 0.0f;
            mx = 0.0f;
        }
        if (lane == 0) {
            params[0] = params_from_range(mn, mx);
            *counter = 0u;  // ready for the next call on this scratch
        }
    }
}

// Per-matrix pass 2: codes and row sums with the single unit's parameters. Rows of at least kLongRow values
// take a block each (contiguous parts of the row by warp), shorter ones a warp (16384 x 2048: 45 us by warps, 83 by
// blocks; 10000 x 6200 85 and 91; but 4096 x 8192 49 and 48, 100 x 100000 59 and 27; not aligned, a value a load, 20000 x
// 2050 70 and 127, 1000 x 20001 72 and 40). Last rows first: the range pass read them last, so about an L2 of them is
// still there.
constexpr int kLongRow = 8192;
template <bool kVec>
__global__ void __launch_bounds__(kRowWarps * 32) matrix_long_rows_kernel(const float *__restrict__ x, int cols, int64_t ldx,
                                                                         uint8_t *__restrict__ codes, int64_t ldc,
                                                                         const qnn_qparams *__restrict__ params,
                                                                         int32_t *__restrict__ sums) {
    __shared__ int s_sum[kRowWarps];
    const int64_t row = gridDim.x - 1 - blockIdx.x;
    const int warp = threadIdx.x >> 5, part = ((cols + kRowWarps - 1) / kRowWarps + 3) & ~3, k0 = warp * part;
    grid_dependency_wait();
    const UnitCoder unit(__ldcg(&params[0].Q), __ldcg(&params[0].z));
    const int s = k0 < cols ? warp_row_codes<kVec, kFlight>(x + row * ldx + k0, min(part, cols - k0), unit, codes + row * ldc + k0) : 0;
    if (!sums) return;
    if ((threadIdx.x & 31) == 0) s_sum[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) t += s_sum[w];
        sums[row] = t;
    }
}

template <bool kVec, int F>
__global__ void __launch_bounds__(kRowWarps * 32) matrix_codes_kernel(const float *__restrict__ x, int64_t rows,
                                                                     int cols, int64_t ldx, uint8_t *__restrict__ codes,
                                                                     int64_t ldc, const qnn_qparams *__restrict__ params,
                                                                     int32_t *__restrict__ sums) {
    const int64_t groups = (rows + kRowWarps - 1) / kRowWarps;
    // once a block, of a grid of one wave: in blocks of eight short rows the wait took most of the time (197307 x 57:
    // 87 us, so 31). Two waves from 48 blocks an SM on, where one leaves warps idle at its end (67556 x 118 of 121 apart
    // 36.7 us a call, so 34.5; but 20000 x 300 18.5 and 21.7)
    grid_dependency_wait();
    const UnitCoder unit(__ldcg(&params[0].Q), __ldcg(&params[0].z));
    for (int64_t b = blockIdx.x; b < groups; b += gridDim.x) {
        const int64_t row = (groups - 1 - b) * kRowWarps + (threadIdx.x >> 5);
        if (row >= rows) continue;
        const int s = warp_row_codes<kVec, F>(x + row * ldx, cols, unit, codes + row * ldc);
        if (sums && (threadIdx.x & 31) == 0) sums[row] = s;
    }
}

inline bool vec_ok(const float *x, int64_t ldx, const uint8_t *codes, int64_t ldc) {
    return ((reinterpret_cast<uintptr_t>(x) & 15) == 0) && (ldx % 4 == 0) &&
           ((reinterpret_cast<uintptr_t>(codes) & 3) == 0) && (ldc % 4 == 0);
}

}  // namespace

qnn_status launch_quantize_rows(const float *x, int64_t rows, int64_t cols, int64_t ldx, uint8_t *codes, int64_t ldc,
                                qnn_qparams *params, int32_t *sums, cudaStream_t st) {
    if (rows == 0) return QNN_OK;
    int *status = nullptr;
    QNN_TRY(status_word(&status));
    dim3 grid((unsigned)((rows + kRowWarps - 1) / kRowWarps));
    ProfScope prof("quantize_rows", st);
    const int nv = (int)((cols + 127) / 128);  // float4 per lane for a register-resident row
    const bool x_ok = ((reinterpret_cast<uintptr_t>(x) & 15) == 0) && (ldx % 4 == 0);
    if (cols <= 128 || (!x_ok && cols <= 256)) {
        const auto kern = cols <= 32    ? quantize_short_rows_kernel<1>
                          : cols <= 64  ? quantize_short_rows_kernel<2>
                          : cols <= 128 ? quantize_short_rows_kernel<4>
                                        : quantize_short_rows_kernel<8>;
        kern<<<grid, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, codes, ldc, params, sums, status);
    } else if (x_ok && nv <= 8) {
        const bool pack = ((reinterpret_cast<uintptr_t>(codes) & 3) == 0) && (ldc % 4 == 0);
        const int r = nv <= 2 ? 2 : nv <= 4 ? 4 : 8;
        grid.x = std::min<unsigned>(grid.x, (unsigned)(sm_count() * rows_reg_blocks(r)));  // one wave
        switch (r) {
            case 2: quantize_rows_reg_kernel<2><<<grid, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, codes, ldc, params, sums, status, pack); break;
            case 4: quantize_rows_reg_kernel<4><<<grid, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, codes, ldc, params, sums, status, pack); break;
            default: quantize_rows_reg_kernel<8><<<grid, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, codes, ldc, params, sums, status, pack); break;
        }
    } else if (vec_ok(x, ldx, codes, ldc))
        quantize_rows_kernel<true, kFlight><<<grid, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, codes, ldc, params, sums, status);
    else
        quantize_rows_kernel<false, kFlight><<<grid, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, codes, ldc, params, sums, status);
    QNN_CUDA_TRY(cudaGetLastError());
    return QNN_OK;
}

qnn_status launch_quantize_matrix(const float *x, int64_t rows, int64_t cols, int64_t ldx, uint8_t *codes, int64_t ldc,
                                  qnn_qparams *params, int32_t *sums, float *partials, unsigned *counter,
                                  int max_blocks, cudaStream_t st) {
    int *status = nullptr;
    QNN_TRY(status_word(&status));
    const int64_t want = (rows + kRowWarps - 1) / kRowWarps;
    const int64_t range = (rows * ((cols - 1) / kSegment + 1) + kRowWarps - 1) / kRowWarps;
    const unsigned nb = (unsigned)(range < max_blocks ? range : max_blocks);
    const bool v = vec_ok(x, ldx, codes, ldc);
    const int f = !v ? loose_flight(cols) : cols >= kMidRow ? kFlight : 1;
    {
    ProfScope prof("quantize_matrix_range", st);
    const auto kern = v ? (f == kFlight ? matrix_range_kernel<true, kFlight> : matrix_range_kernel<true, 1>)
                        : (f == kFlight ? matrix_range_kernel<false, kFlight>
                           : f == 4     ? matrix_range_kernel<false, 4>
                                        : matrix_range_kernel<false, 1>);
    kern<<<nb, kRowWarps * 32, 0, st>>>(x, rows, (int)cols, ldx, partials, counter, params, status);
    QNN_CUDA_TRY(cudaGetLastError());
    }
    ProfScope prof("quantize_matrix_codes", st);
    // programmatic dependent launch: the blocks are set up while the range pass ends (they wait for it)
    cudaLaunchConfig_t cfg = {};
    const bool long_rows = cols >= kLongRow && rows <= INT32_MAX;
    cfg.gridDim = dim3((unsigned)(long_rows ? rows : std::min<int64_t>(want, (want >= 48 * (int64_t)sm_count() ? 16 : 8) * (int64_t)sm_count())));
    cfg.blockDim = dim3(kRowWarps * 32);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (long_rows)
        QNN_CUDA_TRY(cudaLaunchKernelEx(&cfg, v ? matrix_long_rows_kernel<true> : matrix_long_rows_kernel<false>, x, (int)cols, ldx,
                                        codes, ldc, (const qnn_qparams *)params, sums));
    else
        QNN_CUDA_TRY(cudaLaunchKernelEx(&cfg,
                                        v ? (f == kFlight ? matrix_codes_kernel<true, kFlight> : matrix_codes_kernel<true, 1>)
                                          : (f == kFlight ? matrix_codes_kernel<false, kFlight>
                                             : f == 4     ? matrix_codes_kernel<false, 4>
                                                          : matrix_codes_kernel<false, 1>),
                                        x, rows, (int)cols, ldx, codes, ldc, (const qnn_qparams *)params, sums));
    return QNN_OK;
}

}  // namespace qnn

using namespace qnn;

extern "C" qnn_status qnn_quantize(const float *x, int64_t rows, int64_t cols, int64_t ldx, int granularity,
                                   uint8_t *codes, int64_t ldc, qnn_qparams *params, int32_t *code_sums,
                                   void *stream) {
    if (rows < 0 || cols <= 0 || ldx < cols || ldc < cols || cols > INT32_MAX) return QNN_ERR_INVALID_ARG;
    if (granularity != QNN_PER_MATRIX && granularity != QNN_PER_ROW) return QNN_ERR_INVALID_ARG;
    if (rows == 0) return granularity == QNN_PER_MATRIX ? QNN_ERR_INVALID_ARG : QNN_OK;
    if (!is_device_ptr(x) || !is_device_ptr(codes) || !is_device_ptr(params) ||
        (code_sums && !is_device_ptr(code_sums)))
        return QNN_ERR_INVALID_ARG;
    cudaStream_t st = as_stream(stream);
    if (granularity == QNN_PER_ROW) return launch_quantize_rows(x, rows, cols, ldx, codes, ldc, params, code_sums, st);
    Scratch ws;
    QNN_TRY(ws.take_reduce(st));
    return launch_quantize_matrix(x, rows, cols, ldx, codes, ldc, params, code_sums, ws.partials(), ws.counter(),
                                  kReduceBlocks * sm_count(), st);
}
