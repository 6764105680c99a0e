// qgemm_codes.cu — eq. (1) on the sm_103a tcgen05 tensor cores straight from the 8-bit codes, for
// products too small to pay for a centered fp16 copy of their operands.
//
// The arithmetic is that of the centered product (codes as c - 128 in fp16, exact fp32 sums of at most
// 1024 terms drained into int32), but the operands are converted on their way into shared memory: sixteen
// warps load 16 codes a lane, two stages of two k-blocks ahead in registers, and store them as 32 bytes of the swizzled
// fp16 tile; one thread of another warp issues the MMAs. The same sixteen warps drain the accumulators (two
// in tensor memory, alternating by 1024-term chunk, a chunk one stage after its last) and recover.
// Rows of any alignment: a lane loads the aligned 16-byte unit below its codes and takes the rest of them
// from its neighbour's, so every load is one instruction.
//
// Tile: 128 rows of W on the tensor-memory lanes x BN rows of A on the columns, so that a warp's outputs
// of one row of A are 32 consecutive floats. BN = 64 while those tiles are one wave, else 128.
//
// Few tiles share their reductions: a cluster of up to 8 blocks takes a tile, each its part of K, and adds the
// parts through distributed shared memory (128 x 2048 x 2048 17.8 us by 32 blocks, 10.8 by 128; 256 x 1024 x
// 8192 51.8 and 19.6; 129 x 64 x 8192 52 and 12.3).
//
// Bound: the shared-memory port (a 128 x 128 k-block loads 16 KB of codes, stores 32 KB and has the MMAs read
// 32 KB: 640 clk at 128 bytes a clk) and the latencies around it. M = 256, 8192 x 8192: 72 us, 1050 clk a
// k-block; 132 us with eight converting warps and k-blocks one by one (each then waits, converts and loads in
// turn), 148 us when a test of the matrix's ends stood before every load (nothing stayed in flight). The
// centering pass and the fp16 product take 37 + 54 us there. M = 256, 2048 x 2048: 20.6 us, so 17.8.
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>

#include "qnn_device.cuh"
#include "qnn_host.h"
#include "tc_gemm.h"
#include "tc_ptx.cuh"

namespace qnn {
namespace {

constexpr int kRowsW = 128, kBK = 64, kKps = 2;  // W rows of a tile, codes of a k-block, k-blocks of a stage
constexpr int kChunk = 1024 / (kKps * kBK);      // stages of a chunk
constexpr int kConv = 16, kThreads = 32 * (kConv + 4);  // (three warps only complete the issuing warpgroup)
constexpr int kStages = 3;
constexpr unsigned long long kWaitNs = 2000000000ull;

struct CodeArgs {
    const uint8_t *A;
    int64_t lda;
    const qnn_qparams *pa;
    int a_per_row;
    const int32_t *rsA;
    int64_t M;
    int K;
    const uint8_t *W;
    int64_t ldw;
    const qnn_qparams *pw;
    int64_t rows_per_block;
    const int32_t *csW;
    int64_t N;
    const float *bias;
    float *Y;
    int64_t ldy;
    int32_t *acc_out;
    int *status;
    unsigned tiles_m;
    int splits, per;  // blocks of a cluster, which share a tile's reduction, and the stages of each
};

struct RowConst {  // constants of one row of A
    int ra, za, amax;  // code sum, zero point, largest |a' + za|
    float Qa;
};

// The bytes of a code matrix and its first and last aligned 16-byte units (it has one inside).
struct Extent {
    const uint8_t *lo, *hi, *first, *last;
    __device__ __forceinline__ Extent(const uint8_t *p, int64_t bytes) : lo(p), hi(p + bytes) {
        first = p + ((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15);
        last = hi - (reinterpret_cast<uintptr_t>(hi) & 15) - 16;
    }
};

// A lane's unit of every k-block of one row: p + 64 kb, held to the k-blocks in which it lies inside the
// matrix (another unit of the matrix if it never does), so that loads need no branch and stay in flight.
struct Units {
    const uint8_t *p;
    int k0, k1;
    __device__ __forceinline__ Units() {}
    __device__ __forceinline__ Units(const uint8_t *unit, const Extent &e) : p(unit) {
        k0 = unit < e.first ? 1 : 0;
        k1 = e.last < unit ? -1 : (int)min((e.last - unit) / kBK, (int64_t)INT_MAX);
        if (k1 < k0) p = e.first, k0 = k1 = 0;
    }
    __device__ __forceinline__ uint4 load(int kb) const {
        return __ldg(reinterpret_cast<const uint4 *>(p + (int64_t)kBK * max(k0, min(kb, k1))));
    }
};
// A unit that lies across an end of its matrix, byte by byte (0 outside).
__device__ __noinline__ uint4 edge_unit(const uint8_t *p, const uint8_t *lo, const uint8_t *hi) {
    uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (p + i >= lo && p + i < hi) w[i >> 2] |= (uint32_t)__ldg(p + i) << (8 * (i & 3));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

template <int BN>
struct CodesTile {
    static constexpr int THREADS = kThreads;
    // 96 registers a thread at launch; the issuing warpgroup leaves its to the four converting ones, which spill
    // at 96 (M = 256, 8192 x 8192: 83 us, so 72)
    static constexpr int MAX_REGS = 96, REGS_CONV = 112, REGS_ISSUE = 32;
    static constexpr int SUB = (kRowsW + BN) * kBK * 2, STAGE = kKps * SUB;  // bytes of a k-block and a stage
    static constexpr size_t SMEM = (size_t)kStages * STAGE + 1024;
};

template <int BN, bool SHIFT, bool SPLITK>
__global__ void __launch_bounds__((CodesTile<BN>::THREADS)) __maxnreg__((CodesTile<BN>::MAX_REGS))
    qgemm_codes_kernel(const CodeArgs a) {
    constexpr int kSub = CodesTile<BN>::SUB, kStage = CodesTile<BN>::STAGE;
    constexpr int kCols = BN / 4;                // accumulator columns a warp drains
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t bars[2 * kStages + 4];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    __shared__ RowConst s_row[BN];
    const uint32_t full0 = su32(bars), empty0 = su32(bars + kStages), chunk0 = su32(bars + 2 * kStages),
                   drained0 = su32(bars + 2 * kStages + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = a.K, KB = (K + kBK - 1) / kBK;
    const unsigned tile = SPLITK ? blockIdx.x / a.splits : blockIdx.x;
    const int64_t m0 = (int64_t)(tile % a.tiles_m) * BN, n0 = (int64_t)(tile / a.tiles_m) * kRowsW;
    // this block's stages of the reduction: st0 .. st0 + steps - 1 of `all`
    const int all = (KB + kKps - 1) / kKps, rank = SPLITK ? (int)cluster_rank() : 0;
    const int st0 = SPLITK ? rank * a.per : 0, steps = SPLITK ? min(a.per, all - st0) : all;
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int i = 0; i < kStages; ++i) {
            mb_init(full0 + 8 * i, kConv);
            mb_init(empty0 + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mb_init(chunk0 + 8 * i, 1);
            mb_init(drained0 + 8 * i, kConv);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kConv) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_slot)), "n"(2 * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    grid_dependency_wait();
    grid_dependents_launch();
    for (int i = threadIdx.x; i < BN; i += kThreads) {
        const int64_t m = min(m0 + i, a.M - 1);
        const qnn_qparams qa = a.pa[a.a_per_row ? m : 0];
        s_row[i] = RowConst{a.rsA[m], qa.z, max(abs(qa.z), abs(qa.z + 255)), qa.Q};
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_slot;
    // waits are bounded; after one gave up the block's other loops end too
    auto wait = [&](uint32_t bar, unsigned parity) {
        return mbar_try(bar, parity) ||
               (!*reinterpret_cast<volatile int *>(&s_abort) && mbar_wait_bounded(bar, parity, a.status, kWaitNs));
    };

    if (warp >= kConv) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(CodesTile<BN>::REGS_ISSUE));
        if (warp == kConv && lane == 0) {
            constexpr uint32_t idesc = mma_idesc_f16(kRowsW, BN);
            const uint32_t desc0 = smem_desc_lo(su32(smem));
            uint32_t d = desc0, bar = full0, tmem_d = tmem_base;
            unsigned parity = 0;
            for (int st = 0; st < steps; ++st) {
                const int c = st / kChunk;
                const bool fresh = st % kChunk == 0;
                if (fresh) {
                    tmem_d = tmem_base + (c & 1) * BN;
                    if (c >= 2 && !wait(drained0 + 8 * (c & 1), ((c >> 1) - 1) & 1)) {
                        s_abort = 1;
                        break;
                    }
                }
                if (!wait(bar, parity)) {
                    s_abort = 1;
                    break;
                }
                // the converters' stores before the MMAs' reads; here, where no loads are in flight for it to wait for
                fence_async_smem();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int v = 0; v < kKps; ++v) {
                    if (v > 0 && kKps * (st0 + st) + v >= KB) break;
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k) {
                        const uint32_t w = d + ((v * kSub + 32 * k) >> 4), x = w + ((kRowsW * kBK * 2) >> 4);
                        mma_f16_lo(tmem_d, w, x, idesc, v == 0 && k == 0 && fresh ? 0u : 1u);
                    }
                }
                mma_commit(bar + 8 * kStages);
                if (st % kChunk == kChunk - 1 || st == steps - 1) mma_commit(chunk0 + 8 * (c & 1));
                d += kStage >> 4, bar += 8;
                if (bar == full0 + 8 * kStages) d = desc0, bar = full0, parity ^= 1u;
            }
        }
        __syncwarp();
        if constexpr (SPLITK) cluster_sync(), cluster_sync();  // (the converting warps' two)
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(CodesTile<BN>::REGS_CONV));
        // lane (r, c): codes 16 c .. 16 c + 15 of every k-block of row r of W and of A; rows past the end repeat
        // the last one (their sums are dropped)
        const int r = threadIdx.x >> 2, c = threadIdx.x & 3;
        const bool both = r < BN;  // (uniform in a warp)
        const Extent ew(a.W, (a.N - 1) * a.ldw + K), ea(a.A, (a.M - 1) * a.lda + K);
        auto unit = [&](int i, int &s) {  // the unit of k-block 0, and how far below the lane's codes it starts
            const uint8_t *row = i == 0 ? a.W + min(n0 + r, a.N - 1) * a.ldw : a.A + min(m0 + r, a.M - 1) * a.lda;
            s = SHIFT ? (int)(reinterpret_cast<uintptr_t>(row) & 15) : 0;
            return row - s + 16 * c;
        };
        Units src[2];
        int sh[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint8_t *u = unit(i, sh[i]);
            src[i] = Units(u, i == 0 ? ew : ea);
        }
        struct Stage {
            uint4 v[kKps][2];
        };
        auto load = [&](Stage &g, int st) {
#pragma unroll
            for (int v = 0; v < kKps; ++v) {
                g.v[v][0] = src[0].load(kKps * (st0 + st) + v);
                if (both) g.v[v][1] = src[1].load(kKps * (st0 + st) + v);
            }
        };
        auto mend = [&](uint4 (&v)[2], int kb) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                int s;
                const uint8_t *u = unit(i, s) + (int64_t)kBK * kb;
                const Extent &e = i == 0 ? ew : ea;
                if (u < e.first || u > e.last) v[i] = edge_unit(u, e.lo, e.hi);
            }
        };
        int run[kCols];
#pragma unroll
        for (int i = 0; i < kCols; ++i) run[i] = 0;
        const int q = warp & 3, col0 = (warp >> 2) * kCols;
        const uint32_t taddr = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)col0;
        auto drain = [&](int ch) -> bool {
            if (!__all_sync(0xffffffffu, wait(chunk0 + 8 * (ch & 1), (ch >> 1) & 1))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int j = 0; j < kCols; j += 16) {
                uint32_t t[16];
                tmem_ld16(taddr + (uint32_t)((ch & 1) * BN + j), t);
#pragma unroll
                for (int i = 0; i < 16; ++i) run[j + i] += f32_integer_to_s32(__uint_as_float(t[i]));
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mb_arrive(drained0 + 8 * (ch & 1));
            return true;
        };

        uint8_t *const dst0 = smem + r * 128;
        const int u0 = ((2 * c) ^ (r & 7)) << 4, u1 = ((2 * c + 1) ^ (r & 7)) << 4;
        // one lane's 16 codes of k-block kb, from its unit and (with SHIFT) the one 16 bytes on
        auto put = [&](uint8_t *d, const uint4 &cur, const uint4 &next, int s, int valid) {
            uint32_t w[4] = {cur.x, cur.y, cur.z, cur.w};
            if constexpr (SHIFT) {
                const uint32_t g[4] = {c == 0 ? next.x : w[0], c == 0 ? next.y : w[1], c == 0 ? next.z : w[2],
                                       c == 0 ? next.w : w[3]};
                uint32_t e[8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    e[j] = w[j];
                    e[4 + j] = __shfl_sync(0xffffffffu, g[j], (lane & ~3) | ((c + 1) & 3));
                }
                // whole words first (by two, by one), then bytes
#pragma unroll
                for (int j = 0; j < 6; ++j) e[j] = s & 8 ? e[j + 2] : e[j];
#pragma unroll
                for (int j = 0; j < 5; ++j) e[j] = s & 4 ? e[j + 1] : e[j];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = __funnelshift_r(e[j], e[j + 1], 8 * (s & 3));
            }
            if (valid < 16) {  // 128 (a centered zero) past the row
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int n = valid - 4 * j;
                    const uint32_t in = n >= 4 ? 0xffffffffu : n <= 0 ? 0u : (1u << (8 * n)) - 1u;
                    w[j] = (w[j] & in) | (0x80808080u & ~in);
                }
            }
            *reinterpret_cast<uint4 *>(d + u0) =
                make_uint4(center2(w[0], 0x4140u), center2(w[0], 0x4342u), center2(w[1], 0x4140u), center2(w[1], 0x4342u));
            *reinterpret_cast<uint4 *>(d + u1) =
                make_uint4(center2(w[2], 0x4140u), center2(w[2], 0x4342u), center2(w[3], 0x4140u), center2(w[3], 0x4342u));
        };
        int slot = 0;
        unsigned free_parity = 1;
        bool ok = true, is_free = false;
        // stage st from the registers of its loads (and, with SHIFT, of the next stage's) into its slot
        auto convert = [&](Stage &cur, Stage &next, int st) -> bool {
            if (st >= kStages && !__all_sync(0xffffffffu, is_free || wait(empty0 + 8 * slot, free_parity))) return false;
            // units across an end of their matrix are in the first k-block, the last and (with SHIFT) the one after
            const int kb = kKps * (st0 + st);
            if (kb == 0) mend(cur.v[0], 0);
            if (st0 + st + 2 >= all) {
                mend(cur.v[0], kb), mend(cur.v[1], kb + 1);
                if (SHIFT) mend(next.v[0], kb + 2);
            }
#pragma unroll
            for (int v = 0; v < kKps; ++v) {
                const int valid = K - kBK * (kb + v) - 16 * c;  // codes of the chunk that lie inside the row
                uint8_t *const d = dst0 + slot * kStage + v * kSub;
                const uint4(&nx)[2] = v + 1 < kKps ? cur.v[(v + 1) % kKps] : next.v[0];
                put(d, cur.v[v][0], nx[0], sh[0], valid);
                if (both) put(d + kRowsW * 128, cur.v[v][1], nx[1], sh[1], valid);
            }
            __syncwarp();
            if (lane == 0) mb_arrive(full0 + 8 * slot);
            if (++slot == kStages) slot = 0, free_parity ^= 1u;
            is_free = mbar_try(empty0 + 8 * slot, free_parity);  // (answered while the loads are issued)
            load(cur, st + 2);
            // a chunk is drained a stage into the next one, when its MMAs have been issued
            return st % kChunk != 1 || st < kChunk || drain(st / kChunk - 1);
        };
        Stage g[2];
        load(g[0], 0);
        load(g[1], 1);
        for (int st = 0; st < steps && ok; st += 2) {
            ok = convert(g[0], g[1], st);
            if (ok && st + 1 < steps) ok = convert(g[1], g[0], st + 1);
        }
        // chunks not drained yet: the last, and the one before if the last has one stage
        const int chunks = (steps - 1) / kChunk + 1;
        if (ok && chunks > 1 && (steps - 1) % kChunk < 1) ok = drain(chunks - 2);
        if (ok) ok = drain(chunks - 1);
        if (!ok) *reinterpret_cast<volatile int *>(&s_abort) = 1;
        // Outputs of row n of W (P its sum with row i of the tile's rows of A):
        // S of eq. (1) = P + ra (128 + zw) + za (K zw + cs) + 128 cs - 128^2 K; while K |a' + za| |w' + zw|
        // stays below 2^31, wrapping 32-bit arithmetic gives it exactly
        auto outputs = [&](int64_t n, auto for_each) {
            const qnn_qparams qw = a.pw[n / a.rows_per_block];
            const int zw = qw.z, cs = a.csW[n];
            const float bias = a.bias ? a.bias[n] : 0.0f;
            const uint32_t z128 = (uint32_t)(128 + zw), kz = (uint32_t)K * (uint32_t)zw + (uint32_t)cs,
                           s0 = 128u * (uint32_t)cs - 16384u * (uint32_t)K;
            const int a_lim = (int)(INT_MAX / ((long long)K * max(abs(zw), abs(zw + 255))));
            for_each([&](int i, int P) {
                const RowConst rc = s_row[i];
                const int raw = (int)((uint32_t)P + 128u * (uint32_t)rc.ra + s0);  // raw code product
                if (a.acc_out) a.acc_out[(m0 + i) * a.N + n] = raw;
                if (!a.Y) return;
                const float den = __fmul_rn(rc.Qa, qw.Q);
                float v;
                if (rc.amax <= a_lim && den >= 0x1p-60f && den <= 0x1p60f) {
                    const int S = (int)((uint32_t)P + (uint32_t)rc.ra * z128 + (uint32_t)rc.za * kz + s0);
                    v = div_by_recip(__int2float_rn(S), den, rcp_rn(den));
                } else {
                    v = recover_product(offset_product(raw, rc.za, zw, rc.ra, cs, K), rc.Qa, qw.Q);
                }
                a.Y[(m0 + i) * a.ldy + n] = a.bias ? __fadd_rn(v, bias) : v;
            });
        };
        const int rows = (int)min((int64_t)BN, a.M - m0);
        if constexpr (!SPLITK) {
            const int64_t n = n0 + 32 * q + lane;
            if (ok && n < a.N)
                outputs(n, [&](auto put) {
#pragma unroll
                    for (int j = 0; j < kCols; ++j) {
                        if (col0 + j >= rows) break;
                        put(col0 + j, run[j]);
                    }
                });
        } else {
            // every block's sums into its own (no longer used) ring, [column][W row]; then each block adds the
            // cluster's sums of its share of the columns and writes their outputs
            int *const part = reinterpret_cast<int *>(smem);
#pragma unroll
            for (int j = 0; j < kCols; ++j) part[(col0 + j) * kRowsW + 32 * q + lane] = run[j];
            __syncwarp();
            cluster_sync();
            const int share = (BN + a.splits - 1) / a.splits, row = threadIdx.x & (kRowsW - 1);
            if (ok && n0 + row < a.N)
                outputs(n0 + row, [&](auto put) {
                    for (int i = rank * share + (threadIdx.x >> 7); i < min(rows, (rank + 1) * share); i += kConv / 4) {
                        int P = 0;
                        for (int b = 0; b < a.splits; ++b) {
                            int v;
                            asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_addr(su32(part + i * kRowsW + row), b)));
                            P += v;
                        }
                        put(i, P);
                    }
                });
            __syncwarp();
            cluster_sync();  // no block leaves while another reads its sums
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (s_abort && threadIdx.x == 0) {  // MMAs still in flight end before the tensor memory is freed (bounded)
        const unsigned long long t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 4000000ull) __nanosleep(1000);
    }
    __syncthreads();
    if (warp == kConv) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(2 * BN) : "memory");
    }
}

template <int BN, bool SHIFT, bool SPLITK>
qnn_status launch_codes_as(const CodeArgs &a, int64_t tiles, cudaStream_t st) {
    constexpr size_t smem = CodesTile<BN>::SMEM;
    static int configured = -1;
    int dev = 0;
    QNN_CUDA_TRY(cudaGetDevice(&dev));
    if (configured != dev) {
        QNN_CUDA_TRY(cudaFuncSetAttribute(qgemm_codes_kernel<BN, SHIFT, SPLITK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        configured = dev;
    }
    ProfScope prof(SPLITK ? "qgemm_codes_split" : "qgemm_codes", st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * a.splits));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.splits, attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = SPLITK ? 2 : 1;
    QNN_CUDA_TRY(cudaLaunchKernelEx(&cfg, qgemm_codes_kernel<BN, SHIFT, SPLITK>, a));
    return QNN_OK;
}

template <int BN, bool SHIFT>
qnn_status launch_codes(CodeArgs &a, cudaStream_t st) {
    const int64_t tm = (a.M + BN - 1) / BN, tiles = tm * ((a.N + kRowsW - 1) / kRowsW);
    if (tiles > INT32_MAX) return QNN_FAIL(QNN_ERR_INVALID_ARG);
    a.tiles_m = (unsigned)tm;
    // a tile's reduction over the blocks of a cluster, up to 8 of at least four stages, while they find SMs
    // (a cluster's blocks share a part of the chip, so an eighth of the SMs is left out; tiles of 128 rows of A, taken
    // when those of 64 are more than a wave, never do)
    if constexpr (BN == 64) {
        const int64_t steps = (a.K + kKps * kBK - 1) / (kKps * kBK);
        a.splits = (int)std::max<int64_t>(1, std::min<int64_t>({8, steps / 4, sm_count() * 7 / 8 / tiles}));
        a.per = (int)((steps + a.splits - 1) / a.splits);
        a.splits = (int)((steps + a.per - 1) / a.per);
        if (a.splits > 1) return launch_codes_as<BN, SHIFT, true>(a, tiles, st);
    }
    return launch_codes_as<BN, SHIFT, false>(a, tiles, st);
}

}  // namespace

qnn_status launch_qgemm_codes(const uint8_t *A, int64_t lda, const qnn_qparams *pa, int ga, const int32_t *rsA, int64_t M,
                              int64_t K, const uint8_t *W, int64_t ldw, const qnn_qparams *pw, int64_t rows_per_block,
                              const int32_t *csW, int64_t N, const float *bias, float *Y, int64_t ldy, int32_t *acc_out,
                              cudaStream_t st) {
    if (M == 0 || N == 0) return QNN_OK;
    CodeArgs a{A, lda, pa, ga == QNN_PER_ROW, rsA, M, (int)K, W, ldw, pw, rows_per_block, csW, N, bias, Y, ldy, acc_out,
               nullptr, 0, 1, 0};
    QNN_TRY(status_word(&a.status));
    const uintptr_t at = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(W) | (uintptr_t)lda | (uintptr_t)ldw;
    const bool wide = ((M + 63) / 64) * ((N + kRowsW - 1) / kRowsW) > (int64_t)sm_count();
    if ((at & 15) == 0) return wide ? launch_codes<128, false>(a, st) : launch_codes<64, false>(a, st);
    return wide ? launch_codes<128, true>(a, st) : launch_codes<64, true>(a, st);
}

}  // namespace qnn
