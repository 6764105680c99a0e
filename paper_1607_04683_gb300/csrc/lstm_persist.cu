// lstm_persist.cu — a whole unprojected LSTM stack for batches of up to 256 sequences in one
// persistent launch on the tcgen05 tensor cores, with every recurrent and input weight resident in
// shared memory.
//
// Roles. Layer l runs on G blocks (one per SM); block g of a layer owns the cells [CB g, CB g + CB),
// CB = 4 NC, and keeps the 16 NC gate columns of Wx and Wh for them in shared memory as centered fp16
// (the exact datapath of qgemm_tc.cu: sums of up to 1024 products are exact integers in the fp32
// accumulators). A block has 16 epilogue warps, a producer warp (TMA) and an MMA warp:
//   per frame t and row tile (128 sequences; one or two of them):
//   X  x_t's codes (the previous layer's h_t, or the quantized frames) against Wx into one
//      accumulator as soon as the previous layer has released frame t;
//   H  h_{t-1}'s codes against Wh into a second one as soon as every block of the layer has written
//      its cells of h_{t-1};
//   E  the epilogue warps, a lane per sequence, recover both sums (eq. 1, eq. 3), add the bias, apply
//      gates and cell update (c stays in registers) and publish the range of their cells of h_t, one
//      tagged 16-byte word per sequence; they gather the other blocks' words, so that every block
//      knows each row's unit (eq. 2), quantize their own cells, write the codes and release them.
// A row's unit spans the layer's blocks, so a frame costs two exchanges between them (ranges, codes);
// nothing else synchronises, and layers run one frame apart. The four row quarters of a tile (a
// tensor-memory lane quarter, 32 sequences each) go through E independently.
//
// Bound: the chain of one frame (operand stream of h_{t-1}, gate arithmetic, two exchanges). A step
// as launches of a quantizer and a gate kernel per layer takes two launches' latency and streams the
// weights again; the grid barriers of lstm_recurrent_kernel keep one layer at a time on the GPU. 5 x 500
// cells, 100 frames, this kernel alone (whole pass before): B = 16 593 us (5.5 ms), B = 64 995 us (2.3 ms);
// B = 256, 500 frames 7.6 ms (13.4 ms). A frame at B = 32 took about 15,000
// cycles while one row quarter's warps, all on one scheduler, did all its cells: h's operand stream and
// products 4,700, gates 5,000, range exchange 2,200, codes and release 2,700. With the cells spread over the
// four schedulers (SP = 4) a B = 16 pass went from 869 to 717 us; two quarters' over all four (SP = 2), 5 x
// 300, 40 frames, B = 48, from 376 to 350 us, 5 x 512 551 to 529, 1 x 128 231 to 224 (all before the register
// split below).
//
// Every wait is bounded in time: one that gives up records QNN_ERR_TIMEOUT and raises the abort
// flag, after which all waits return at once and the launch runs to its end with meaningless outputs.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <climits>
#include <cstdlib>
#include <type_traits>
#include <utility>
#include <vector>

#include "lstm_model.h"
#include "persist_plan.h"
#include "qnn_device.cuh"
#include "tc_gemm.h"
#include "tc_ptx.cuh"

namespace qnn {
namespace {

using namespace persist;

constexpr int kEpiWarps = 16;
constexpr int kThreads = 32 * (kEpiWarps + 4);  // (two warps only complete the last warpgroup)
// Registers a thread: 96 at launch (640 threads), of which the producer's warpgroup leaves its share to the
// four epilogue ones (4 x 112 + 32 = 5 x 96). With 96 their rows' constants and cells spill, and a reload
// misses the little L1 that the weights leave: 5 x 500 cells, B = 16 and 64, 100 frames 714 and 1435 us, B = 256,
// 500 frames 9.59 ms; so 630, 1352 us and 8.37 ms.
constexpr int kRegsEpi = 112, kRegsIssue = 32;
constexpr unsigned long long kWaitLimit = 2000000000ull;

__host__ __device__ inline int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

struct PersistLayer {
    const qnn_qparams *pwx, *pwh;  // [4] one unit per gate matrix
    const float2 *pairc;           // [pairs][kPairConsts] column constants
    const qnn_qparams *prm_x;      // [T B] units of the layer input rows, time-major
    const int32_t *rs_x;           // [T B] their code sums
    qnn_qparams *prm;              // [T B] units of h_t (the next layer's input)
    int32_t *rs;                   // [T B] code sums (zero at launch, summed by the blocks)
    __half *codes;                 // [T B][kh] centered codes of h_t
    float *out;                    // nullable: fp32 outputs, row b of frame t at out + t out_t + b out_b
    int kin, kbx;
};

struct PersistArgs {
    CUtensorMap mx[kMaxL], mh[kMaxL], mwx[kMaxL], mwh[kMaxL];
    CUtensorMap mh0;                // initial codes of every layer, [L B][kh]
    PersistLayer layer[kMaxL];
    const qnn_qparams *prm_h0;      // [L B]
    const int32_t *rs_h0;
    const float *c0;                // [L][B][H], nullable (zero)
    float *h_fin, *c_fin;           // [L][B][R], [L][B][H], nullable
    int64_t out_t, out_b;
    uint4 *mm;                      // [L][2][tiles][G][128] published ranges (tag 0 at launch)
    unsigned *ctr;                  // [L][2] row quarters whose codes are written (0 at launch)
    int *abort_flag, *status;
    int B, T, H, kh, kbh, G;
    int rows_box;                   // rows of an operand box (a multiple of 8)
    int kps, slots, slot_bytes;     // k-blocks per ring slot, ring slots
};

// ---- waits ----------------------------------------------------------------------------------------

__device__ __forceinline__ bool gave_up(const PersistArgs &a, unsigned long long t0) {
    if (*(volatile int *)a.abort_flag) return true;
    if (global_timer_ns() - t0 > kWaitLimit) {
        record_status(a.status, QNN_ERR_TIMEOUT);
        atomicExch(a.abort_flag, 1);
        return true;
    }
    return false;
}
__device__ __forceinline__ void wait_bar(const PersistArgs &a, uint32_t bar, unsigned parity) {
    uint32_t ok;
    unsigned long long t0 = 0;
    while (true) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspendNs)
            : "memory");
        if (ok) return;
        if (t0 == 0) t0 = global_timer_ns();
        if (gave_up(a, t0)) return;
    }
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void wait_counter(const PersistArgs &a, const unsigned *p, unsigned target) {
    if (ld_acquire(p) >= target) return;
    const unsigned long long t0 = global_timer_ns();
    for (int n = 1; ld_acquire(p) < target; ++n)
        if (n % 64 == 0 && gave_up(a, t0)) return;
}
__device__ __forceinline__ void red_release(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// 16-byte words written and read whole
__device__ __forceinline__ void st_word(uint4 *p, uint4 v) {
    const unsigned long long lo = v.x | (unsigned long long)v.y << 32, hi = v.z | (unsigned long long)v.w << 32;
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p), "l"(lo),
                 "l"(hi)
                 : "memory");
}
__device__ __forceinline__ uint4 ld_word(const uint4 *p) {
    unsigned long long lo, hi;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// fp32 order as signed integer order (finite values lie below INT_MAX, which marks a non-finite value)
__device__ __forceinline__ int order_key(float f) {
    const int b = __float_as_int(f);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_value(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// A quantized row's constants of eq. (1) and eq. (3) for the four gate matrices of one operand, kept in
// registers while the thread stays on its row.
struct RowTerms {
    float z128;               // 128 + z
    float d[4], r[4], rt[4];  // divisors, their reciprocals, constant parts of the sums
};

// The terms of a row with unit (Q, z) and code sum rs; false when the bounds of the fp32 form do not hold:
// with |rt| + |128 + z| 255 K < 2^24 the offset term rt + (128 + z) cs is an exact integer (cs <= 255 K),
// formed by one fused multiply-add; the tensor-core sum P is an exact integer too, so the one rounded
// addition P + (offset term) equals the correctly rounded S of eq. (1); the quotient S / (Qa Qw) from the
// divisor's reciprocal equals the IEEE quotient while the divisor lies within 2^-60 .. 2^60. Offsets beyond
// +-1023 (no fp32 form for K >= 57) are left to the general form so that rt fits 32 bits:
// |(128 + zw) rs| <= 1151 255 1024 and |K (z zw - 16384)| <= 1024 (2^20 + 2^14).
__device__ __forceinline__ bool row_terms(RowTerms &e, float Q, int z, int rs, const qnn_qparams *pw, int K) {
    bool ok = z >= -1023 && z <= 1023;
    e.z128 = (float)(128 + z);
    const int room = (1 << 24) - abs(128 + (ok ? z : 1023)) * (255 * K);
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float Qw = __ldg(&pw[g].Q);
        const int zw = __ldg(&pw[g].z);
        const int rt = (int)((uint32_t)(128 + zw) * (uint32_t)rs + (uint32_t)K * ((uint32_t)z * (uint32_t)zw - 16384u));
        e.d[g] = __fmul_rn(Q, Qw);
        e.r[g] = rcp_rn(e.d[g]);
        e.rt[g] = (float)rt;
        ok &= zw >= -1023 && zw <= 1023 && abs(rt) < room && e.d[g] >= 0x1p-60f && e.d[g] <= 0x1p60f;
    }
    return ok;
}

// One recovered sum the general way: the exact 64-bit S of eq. (1), rounded, and an IEEE divide.
__device__ __noinline__ float recover_general(float P, float Q, int z, int rs, float cs, const qnn_qparams *pw, int K) {
    const qnn_qparams w = *pw;
    const long long S = (long long)f32_integer_to_s32(P) + (long long)(128 + w.z) * rs +
                        (long long)K * ((long long)z * w.z - 16384) + (long long)(128 + z) * __float2int_rn(cs);
    return __fdiv_rn(s64_to_f32_rn(S), __fmul_rn(Q, w.Q));
}

// Column constants of a cell pair: [4 gates][3], the pair's biases, Wx row code sums and Wh row code sums
// (integers below 2^24, exact in fp32).
constexpr int kPairConsts = 12;

// Pre-activations of a pair of cells from its sums rx (x_t Wx) and rh (h_{t-1} Wh), rows in the fp32 form.
// (Paired instructions: 130 issue cycles a pair against 150 for scalar ones.)
template <bool kSmem>
__device__ __forceinline__ void pair_pre(float2 (&pre)[4], const uint32_t (&rx)[8], const uint32_t (&rh)[8], const RowTerms &X,
                                         const RowTerms &H, const float2 *cc, const float4 *sums) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float2 bias = __ldg(cc + 3 * g);
        float2 csx, csh;
        if (kSmem) {
            const float4 v = sums[g];
            csx = make_float2(v.x, v.y), csh = make_float2(v.z, v.w);
        } else {
            csx = __ldg(cc + 3 * g + 1), csh = __ldg(cc + 3 * g + 2);
        }
        const float2 ox = ffma2_rn(f2(X.z128), csx, f2(X.rt[g])), oh = ffma2_rn(f2(H.z128), csh, f2(H.rt[g]));
        const float2 vx = fadd2_rn(make_float2(__uint_as_float(rx[2 * g]), __uint_as_float(rx[2 * g + 1])), ox);
        const float2 vh = fadd2_rn(make_float2(__uint_as_float(rh[2 * g]), __uint_as_float(rh[2 * g + 1])), oh);
        pre[g] = fadd2_rn(fadd2_rn(div_by_recip2(vx, X.d[g], X.r[g]), bias), div_by_recip2(vh, H.d[g], H.r[g]));
    }
}

// The same for any row: (Qx, zx, rsx) the unit and code sum of x_t, (Qh, zh, rsh) of h_{t-1}; pwx and pwh the
// gate matrices' units for these cells, `stride` entries apart.
struct PairSums {
    uint32_t x[8], h[8];
};
struct PairPre {
    float2 g[4];
};
__device__ __noinline__ PairPre pair_pre_general(const PairSums s, float Qx, int zx, int rsx, const qnn_qparams *pwx, int Kx,
                                                 float Qh, int zh, int rsh, const qnn_qparams *pwh, int K, int stride,
                                                 const float2 *cc) {
    PairPre pre;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float2 bias = cc[3 * g], csx = cc[3 * g + 1], csh = cc[3 * g + 2];
        const qnn_qparams *wx = pwx + g * stride, *wh = pwh + g * stride;
        const float x0 = recover_general(__uint_as_float(s.x[2 * g]), Qx, zx, rsx, csx.x, wx, Kx);
        const float x1 = recover_general(__uint_as_float(s.x[2 * g + 1]), Qx, zx, rsx, csx.y, wx, Kx);
        const float h0 = recover_general(__uint_as_float(s.h[2 * g]), Qh, zh, rsh, csh.x, wh, K);
        const float h1 = recover_general(__uint_as_float(s.h[2 * g + 1]), Qh, zh, rsh, csh.y, wh, K);
        pre.g[g] = make_float2(__fadd_rn(__fadd_rn(x0, bias.x), h0), __fadd_rn(__fadd_rn(x1, bias.y), h1));
    }
    return pre;
}

// SP: with one (SP = 4) or two (SP = 2) row quarters in use, the warps of the other quarters, which cannot read
// those rows' tensor memory and would leave their schedulers idle, take SP - 1 of SP cell pairs: the warp that
// can hands it their sums through shared memory.
template <int NC, int MT, int SP>
struct Cfg {
    static_assert(SP == 1 || MT == 1, "two row tiles use every quarter");
    static constexpr int CB = 4 * NC, N = 16 * NC;           // cells and gate columns of a block
    static constexpr int SL = (MT == 1 ? 4 : 2) * SP;        // cell slices of a tile: a warp each per row quarter
    static constexpr int PAIRS = SP > 1 ? (2 * NC + SL - 1) / SL : MT == 1 ? NC / 2 : NC;  // cell pairs of a thread
    static constexpr bool ODD = SP == 1 && MT == 1 && (NC & 1);  // and one more cell
    static constexpr int GIVEN = SP > 1 ? 2 * NC - (2 * NC + SP - 1) / SP : 0;  // pairs handed over per row quarter
    static constexpr int TMEM_USED = tmem_used(NC, MT), TMEM_COLS = TMEM_USED <= 128 ? 128 : TMEM_USED <= 256 ? 256 : kTmemCols;
    static_assert(TMEM_USED <= kTmemCols, "the accumulators fit the tensor memory");
    static constexpr int KB_BYTES = N * 128;             // a k-block of weights
};

template <int NC, int MT, int SP>
__global__ void __launch_bounds__(kThreads, 1) lstm_persist_kernel(const __grid_constant__ PersistArgs a) {
    using C = Cfg<NC, MT, SP>;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l = blockIdx.x / a.G, blk = blockIdx.x % a.G;
    const PersistLayer &ly = a.layer[l];
    uint8_t *const wts = smem + a.slots * a.slot_bytes;
    const int kbw = ly.kbx + a.kbh;
    uint8_t *const misc = wts + kbw * C::KB_BYTES;
    const uint32_t full0 = su32(misc), empty0 = full0 + 8 * kMaxSlots, wfull = empty0 + 8 * kMaxSlots;
    const uint32_t acc0 = wfull + 8, drained0 = acc0 + 16, ready0 = drained0 + 16;
    uint32_t *const tmem_slot = reinterpret_cast<uint32_t *>(misc + 8 * (2 * kMaxSlots + 8));
    // per row: the block's range (its minimum later the code sum) and the gathered range
    int *const s_min = reinterpret_cast<int *>(tmem_slot + 4), *const s_max = s_min + MT * kTile;
    int *const g_min = MT == 1 ? s_max + kTile : s_min, *const g_max = MT == 1 ? g_min + kTile : s_max;  // (MT = 2: one pair for both)
    float4 *const s_sums = reinterpret_cast<float4 *>(s_min + 4 * kTile);  // MT = 1: [pair][gate] Wx and Wh code sums
    const int B = a.B, T = a.T, H = a.H;
    auto tile_rows = [&](int i) { return min(kTile, B - kTile * i); };
    auto quarters = [&](int i) { return (tile_rows(i) + 31) / 32; };

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.slots; ++i) {
            mb_init(full0 + 8 * i, 1);
            mb_init(empty0 + 8 * i, 1);
        }
        mb_init(wfull, 1);
        for (int i = 0; i < MT; ++i) {
            mb_init(acc0 + 8 * i, 1);
            mb_init(drained0 + 8 * i, C::SL / SP * quarters(i));  // the warps that read the accumulators
            mb_init(ready0 + 8 * i, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    for (int i = threadIdx.x; i < MT * kTile; i += kThreads)
        s_min[i] = g_min[i] = INT_MAX, s_max[i] = g_max[i] = INT_MIN;
    if (MT == 1)
        for (int i = threadIdx.x; i < 8 * NC; i += kThreads) {
            const float2 *c = ly.pairc + min(blk * 2 * NC + i / 4, (a.H + 1) / 2 - 1) * kPairConsts + 3 * (i % 4);
            s_sums[i] = make_float4(c[1].x, c[1].y, c[2].x, c[2].y);
        }
    if (warp == kEpiWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "n"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    // accumulators: x_t by frame parity and tile, then h_{t-1} by tile
    auto acc_x = [&](int t, int i) { return tmem + (uint32_t)(((t & 1) * MT + i) * C::N); };
    auto acc_h = [&](int i) { return tmem + (uint32_t)((2 * MT + i) * C::N); };

    if (warp >= kEpiWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
        if (warp == kEpiWarps) {
            // ---------------- producer ----------------
            if (lane == 0) {
                const uint32_t w0 = su32(wts);
                mb_expect(wfull, (uint32_t)(kbw * C::KB_BYTES));
                for (int kb = 0; kb < ly.kbx; ++kb) tma_load_2d(w0 + kb * C::KB_BYTES, &a.mwx[l], wfull, 64 * kb, blk * C::N);
                for (int kb = 0; kb < a.kbh; ++kb)
                    tma_load_2d(w0 + (ly.kbx + kb) * C::KB_BYTES, &a.mwh[l], wfull, 64 * kb, blk * C::N);
                // (one thread: its loop is on the critical path, so the ring advances by additions)
                const uint32_t ring = su32(smem), ring_end = ring + a.slots * a.slot_bytes, slot_bytes = a.slot_bytes;
                const int kps = a.kps;
                uint32_t dst = ring, bar = full0;
                unsigned parity = 1;  // a fresh slot's empty barrier passes with parity 1
                auto stream = [&](const CUtensorMap *map, int kbs, int row) {
                    for (int kb = 0; kb < kbs; kb += kps) {
                        wait_bar(a, bar + 8 * kMaxSlots, parity);
                        mb_expect(bar, slot_bytes);
                        tma_load_3d(dst, map, bar, 0, row, kb);  // k-blocks past the matrix read as zero
                        dst += slot_bytes, bar += 8;
                        if (dst == ring_end) dst = ring, bar = full0, parity ^= 1u;
                    }
                };
                for (int t = 0; t < T; ++t) {
#pragma unroll
                    for (int i = 0; i < MT; ++i) {
                        if (l > 0) {
                            wait_counter(a, a.ctr + 2 * (l - 1) + i, (unsigned)(quarters(i) * a.G * (t + 1)));
                            asm volatile("fence.proxy.async.global;" ::: "memory");
                        }
                        stream(&a.mx[l], ly.kbx, t * B + kTile * i);
                    }
#pragma unroll
                    for (int i = 0; i < MT; ++i) {
                        if (t > 0) wait_counter(a, a.ctr + 2 * l + i, (unsigned)(quarters(i) * a.G * t));
                        mb_arrive(ready0 + 8 * i);  // x_t and h_{t-1}: their units and code sums may be read
                        asm volatile("fence.proxy.async.global;" ::: "memory");
                        if (t > 0)
                            stream(&a.mh[l], a.kbh, (t - 1) * B + kTile * i);
                        else
                            stream(&a.mh0, a.kbh, l * B + kTile * i);
                    }
                }
            }
        } else if (warp == kEpiWarps + 1) {
            // ---------------- MMA issuer ----------------
            if (lane == 0) {
                constexpr uint32_t idesc = mma_idesc_f16(kTile, C::N);
                const uint32_t da0 = smem_desc_lo(su32(smem)), sub = (uint32_t)a.rows_box * 128 / 16, slot16 = a.slot_bytes / 16;
                const uint32_t bar_end = full0 + 8 * a.slots;
                const int kps = a.kps;
                uint32_t da = da0, bar = full0;
                unsigned parity = 0;
                wait_bar(a, wfull, 0);
                // d = the k-blocks of one operand against the weights at w; `done` (0: none) completes with them
                auto multiply = [&](uint32_t d, uint32_t w, int kbs, uint32_t done) {
                    uint32_t accumulate = 0;
                    for (int kb = 0; kb < kbs; kb += kps) {
                        wait_bar(a, bar, parity);
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const int nv = min(kps, kbs - kb);
                        uint32_t x = da;
#pragma unroll 2
                        for (int v = 0; v < nv; ++v) {
                            mma_f16_lo(d, x, w, idesc, accumulate);
                            accumulate = 1;
#pragma unroll
                            for (int k = 1; k < 4; ++k) mma_f16_lo(d, x + 2 * k, w + 2 * k, idesc, 1u);  // 16 fp16 = 32 bytes
                            x += sub, w += C::KB_BYTES / 16;
                        }
                        if (done && kb + kps >= kbs) mma_commit(done);  // (before the slot's: a commit takes 250 cycles)
                        mma_commit(bar + 8 * kMaxSlots);
                        da += slot16, bar += 8;
                        if (bar == bar_end) da = da0, bar = full0, parity ^= 1u;
                    }
                };
                const uint32_t wx = smem_desc_lo(su32(wts)), wh = wx + ly.kbx * (C::KB_BYTES / 16);
                for (int t = 0; t < T; ++t) {
#pragma unroll
                    for (int i = 0; i < MT; ++i) multiply(acc_x(t, i), wx, ly.kbx, 0);
#pragma unroll
                    for (int i = 0; i < MT; ++i) {
                        // both accumulators of frame t - 1 read out (and, one frame back, x's of this parity)
                        if (t > 0) wait_bar(a, drained0 + 8 * i, (unsigned)(t - 1) & 1);
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        multiply(acc_h(i), wh, a.kbh, acc0 + 8 * i);
                    }
                }
            }
        }
    } else {
        // ---------------- epilogue ----------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
        // row quarter q, slice e; `own`: this warp may read the quarter's tensor-memory lanes
        const int tile = MT == 2 ? warp >> 3 : 0, q = warp & (4 / SP - 1), rep = (warp & 3) / (4 / SP);
        const int e = SP > 1 ? (warp >> 2) * SP + rep : (warp >> 2) & (C::SL - 1);
        const bool own = SP == 1 || rep == 0;
        const int rows = tile_rows(tile);
        if (32 * q < rows) {
            constexpr int GT = 32 * C::SL;  // threads of a row quarter
            const int bar_id = 1 + 4 * tile + q;
            const int rl = 32 * q + lane, b = kTile * tile + rl;
            const bool bv = rl < rows;
            const int K = H, Kx = ly.kin;
            int *const my_min = s_min + tile * kTile + rl, *const my_max = s_max + tile * kTile + rl;
            int *const all_min = g_min + tile * kTile + rl, *const all_max = g_max + tile * kTile + rl;
            const uint32_t lane_base = (uint32_t)(32 * q) << 16;
            const int nsrc = (a.G - e + C::SL - 1) / C::SL;  // blocks whose ranges this warp gathers: e, e + SL, ..
            const int last_pair = (H + 1) / 2 - 1;  // (pairs past H repeat it: their results are dropped)
            const int j_blk = blk * C::CB;
            // cells of this thread: pairs e PAIRS .. of the block, and for odd NC one of pair 2 NC - 2 ..
            const int pair0 = e * C::PAIRS, pair_odd = 4 * C::PAIRS + (e >> 1), odd = e & 1;
            constexpr int CELLS = 2 * C::PAIRS + (C::ODD ? 1 : 0);
            float c[CELLS];
            // (SP > 1: pairs e, e + SL of the block; cells of no pair lie past every row)
            auto pair_of = [&](int k) { return SP > 1 ? e + C::SL * k : pair0 + k; };
            auto cell_of = [&](int k) {
                if (SP > 1) return pair_of(k / 2) < 2 * NC ? j_blk + 2 * pair_of(k / 2) + (k & 1) : 1 << 30;
                return j_blk + (k < 2 * C::PAIRS ? 2 * pair0 + k : 2 * pair_odd + odd);
            };
            // sums of a pair handed over: 16-byte words v = 0 .. 3 of each row
            float4 *const xch = reinterpret_cast<float4 *>(s_min + 4 * kTile) + (MT == 1 ? 8 * NC : 0);
            auto given = [&](int p, int v) { return xch + ((q * C::GIVEN + p - p / SP - 1) * 4 + v) * 32 + lane; };
#pragma unroll
            for (int k = 0; k < CELLS; ++k) {
                const int j = cell_of(k);
                c[k] = (a.c0 && bv && j < H) ? a.c0[((int64_t)l * B + b) * H + j] : 0.0f;
            }
            float Qh = 1.0f;
            int zh = 0;
            if (bv) {
                const qnn_qparams p = a.prm_h0[(int64_t)l * B + b];
                Qh = p.Q, zh = p.z;
            }
            for (int t = 0; t < T; ++t) {
                float h[CELLS];
                // ---- units and code sums of the row's x_t and h_{t-1} ----
                float Qx = 1.0f;
                int zx = 0, rsx = 0, rsh = 0;
                wait_bar(a, ready0 + 8 * tile, (unsigned)t & 1);
                if (bv) {
                    const int64_t r = (int64_t)t * B + b;
                    Qx = __ldcg(&ly.prm_x[r].Q), zx = __ldcg(&ly.prm_x[r].z), rsx = __ldcg(ly.rs_x + r);
                    rsh = t > 0 ? __ldcg(ly.rs + r - B) : a.rs_h0[(int64_t)l * B + b];
                }
                RowTerms X, Hh;
                const bool fast_x = row_terms(X, Qx, zx, rsx, ly.pwx, Kx);
                bool fast = row_terms(Hh, Qh, zh, rsh, ly.pwh, K) && fast_x;
                if (!bv) {  // no row: finite results of any kind, the short way
                    fast = true;
#pragma unroll
                    for (int g = 0; g < 4; ++g) X.r[g] = Hh.r[g] = 0.0f;
                }
                if (own) {
                    wait_bar(a, acc0 + 8 * tile, (unsigned)t & 1);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                // ---- gates and cells ----
                const uint32_t tx = acc_x(t, tile) + lane_base, th = acc_h(tile) + lane_base;
                int kmin = INT_MAX, kmax = INT_MIN;
                auto note = [&](float v, int j) {
                    if (j < H) {
                        const int k = isfinite(v) ? order_key(v) : INT_MAX;
                        kmin = min(kmin, k), kmax = max(kmax, k);
                    }
                };
                if constexpr (SP > 1) {
                    const int hand = 5 + 4 * q + (warp >> 2);  // barrier of a reading warp and those it hands sums to
                    if (own) {
#pragma unroll
                        for (int i = 0; i < C::PAIRS * (SP - 1); ++i) {
                            const int p = pair_of(i / (SP - 1)) + 1 + i % (SP - 1);
                            if (p >= 2 * NC) continue;
                            uint32_t x[8], y[8];
                            tmem_ld8_nowait(tx + 8 * p, x);
                            tmem_ld8_nowait(th + 8 * p, y);
                            tmem_wait_ld();
#pragma unroll
                            for (int v = 0; v < 2; ++v) {
                                *reinterpret_cast<uint4 *>(given(p, v)) = make_uint4(x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]);
                                *reinterpret_cast<uint4 *>(given(p, 2 + v)) = make_uint4(y[4 * v], y[4 * v + 1], y[4 * v + 2], y[4 * v + 3]);
                            }
                        }
                        asm volatile("bar.arrive %0, %1;" ::"r"(hand), "n"(32 * SP) : "memory");
                    } else {
                        bar_sync(hand, 32 * SP);
                    }
                }
                auto pre_of = [&](int p) {  // pre-activations of a pair of the block's cells
                    PairSums P;
                    if (own) {
                        tmem_ld8_nowait(tx + 8 * p, P.x);
                        tmem_ld8_nowait(th + 8 * p, P.h);
                        tmem_wait_ld();
                    } else {
#pragma unroll
                        for (int v = 0; v < 2; ++v) {
                            const uint4 x = *reinterpret_cast<const uint4 *>(given(p, v)),
                                        y = *reinterpret_cast<const uint4 *>(given(p, 2 + v));
                            P.x[4 * v] = x.x, P.x[4 * v + 1] = x.y, P.x[4 * v + 2] = x.z, P.x[4 * v + 3] = x.w;
                            P.h[4 * v] = y.x, P.h[4 * v + 1] = y.y, P.h[4 * v + 2] = y.z, P.h[4 * v + 3] = y.w;
                        }
                    }
                    const float2 *cc = ly.pairc + min(blk * 2 * NC + p, last_pair) * kPairConsts;
                    PairPre pre;
                    if (fast)
                        pair_pre<MT == 1>(pre.g, P.x, P.h, X, Hh, cc, s_sums + 4 * p);
                    else
                        pre = pair_pre_general(P, Qx, zx, rsx, ly.pwx, Kx, Qh, zh, rsh, ly.pwh, K, 1, cc);
                    return pre;
                };
#pragma unroll
                for (int p = 0; p < C::PAIRS; ++p) {
                    if (SP > 1 && pair_of(p) >= 2 * NC) continue;  // (uniform in the warp)
                    const PairPre pre = pre_of(pair_of(p));
                    float2 cv = make_float2(c[2 * p], c[2 * p + 1]);
                    const float2 m = lstm_cell2(pre.g[0], pre.g[1], pre.g[2], pre.g[3], cv);
                    c[2 * p] = cv.x, c[2 * p + 1] = cv.y;
                    h[2 * p] = m.x, h[2 * p + 1] = m.y;
                    note(m.x, cell_of(2 * p));
                    note(m.y, cell_of(2 * p + 1));
                }
                if constexpr (C::ODD) {
                    constexpr int k = 2 * C::PAIRS;
                    const PairPre pre = pre_of(pair_odd);
                    lstm_cell(odd ? pre.g[0].y : pre.g[0].x, odd ? pre.g[1].y : pre.g[1].x, odd ? pre.g[2].y : pre.g[2].x,
                              odd ? pre.g[3].y : pre.g[3].x, c[k], h[k]);
                    note(h[k], cell_of(k));
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (own && lane == 0) mb_arrive(drained0 + 8 * tile);
                // ---- the row's range over the layer's blocks ----
                atomicMin(my_min, kmin);
                atomicMax(my_max, kmax);
                uint4 *const mm = a.mm + ((int64_t)((l * 2 + (t & 1)) * MT + tile) * a.G) * kTile + rl;
                const unsigned tag = (unsigned)t + 1;
                bar_sync(bar_id, GT);
                if (e == 0) {
                    st_word(mm + (int64_t)blk * kTile, make_uint4((unsigned)*my_min, (unsigned)*my_max, tag, 0u));
                    *my_min = MT == 1 ? 0 : INT_MAX, *my_max = INT_MIN;  // (MT = 1: the code sum from here, ordered by the next barrier)
                }
                if (MT == 2) bar_sync(bar_id, GT);
                // outputs in fp32, and after the last frame the state
                if (bv) {
#pragma unroll
                    for (int k = 0; k < CELLS; ++k) {
                        const int j = cell_of(k);
                        if (j >= H) continue;
                        if (ly.out) ly.out[t * a.out_t + b * a.out_b + j] = h[k];
                        if (t == T - 1) {
                            if (a.h_fin) a.h_fin[((int64_t)l * B + b) * H + j] = h[k];
                            if (a.c_fin) a.c_fin[((int64_t)l * B + b) * H + j] = c[k];
                        }
                    }
                }
                // every lane reads its row's words until all carry this frame's tag
                kmin = INT_MAX, kmax = INT_MIN;
                const uint4 *const src = mm + (int64_t)e * kTile;
                for (int s0 = 0; s0 < nsrc; s0 += 8) {
                    const uint4 *p = src + (int64_t)s0 * C::SL * kTile;
                    uint4 w[8];
                    unsigned long long t0 = 0;
                    for (int n = 0;; ++n) {
                        bool ready = true;
#pragma unroll
                        for (int s = 0; s < 8; ++s)
                            if (s0 + s < nsrc) w[s] = ld_word(p + (int64_t)s * C::SL * kTile);
#pragma unroll
                        for (int s = 0; s < 8; ++s)
                            if (s0 + s < nsrc) ready &= w[s].z == tag;
                        if (__all_sync(0xffffffffu, ready)) break;
                        if (n == 0) t0 = global_timer_ns();
                        if (n % 64 == 63 && __any_sync(0xffffffffu, gave_up(a, t0))) break;
                    }
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (s0 + s < nsrc) kmin = min(kmin, (int)w[s].x), kmax = max(kmax, (int)w[s].y);
                }
                atomicMin(all_min, kmin);
                atomicMax(all_max, kmax);
                bar_sync(bar_id, GT);
                kmin = *all_min, kmax = *all_max;
                if (MT == 2) bar_sync(bar_id, GT);
                // ---- codes (eq. 2), the row's unit and code sum ----
                float mn = key_value(kmin), mx = key_value(kmax);
                if (kmax == INT_MAX) {  // some value of the row was not finite
                    if (bv && e == 0 && blk == 0) record_status(a.status, QNN_ERR_NONFINITE);
                    mn = 0.0f, mx = 0.0f;
                }
                const qnn_qparams p = params_from_range(mn, mx);
                Qh = p.Q, zh = p.z;
                const int64_t orow = (int64_t)t * B + b;
                __half *const crow = ly.codes + orow * a.kh;
                int sum = 0;
                if (bv) {
#pragma unroll
                    for (int k = 0; k < CELLS; k += 2) {
                        const int j = cell_of(k);
                        uint32_t w = 0;
                        if (j < H) {
                            const int v = (int)quant_code(h[k], p.Q, p.z);
                            sum += v;
                            w = __half_as_ushort(__int2half_rn(v - 128));
                        }
                        if (k + 1 < CELLS) {
                            if (j + 1 < H) {
                                const int v = (int)quant_code(h[k + 1], p.Q, p.z);
                                sum += v;
                                w |= (uint32_t)__half_as_ushort(__int2half_rn(v - 128)) << 16;
                            }
                            if (j < a.kh) *reinterpret_cast<uint32_t *>(crow + j) = w;  // (cells past H: zeros)
                        } else if (j < a.kh) {
                            *reinterpret_cast<unsigned short *>(crow + j) = (unsigned short)w;
                        }
                    }
                    if (blk == a.G - 1)  // zeros past the last block's cells
                        for (int j = a.G * C::CB + 2 * e; j < a.kh; j += 2 * C::SL) *reinterpret_cast<uint32_t *>(crow + j) = 0u;
                }
                if (MT == 1)
                    atomicAdd(my_min, sum);
                else if (e == 1)  // two slices: this one's sum, added by the other
                    *my_min = sum;
                bar_sync(bar_id, GT);
                if (e == 0) {
                    if (bv) {
                        atomicAdd(ly.rs + orow, MT == 1 ? *my_min : sum + *my_min);
                        if (blk == 0) ly.prm[orow] = p;
                    }
                    *my_min = *all_min = INT_MAX, *my_max = *all_max = INT_MIN;  // (before the release that the next frame follows)
                    // the quarter's codes, units and sums are ordered before this by its barriers and the
                    // release; the readers' producers put the proxy fence between their acquire and the
                    // TMA reads
                    __syncwarp();
                    if (lane == 0) red_release(a.ctr + 2 * l + tile, 1u);
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*(volatile int *)a.abort_flag && threadIdx.x == 0) {
        // let copies still in flight land before the block leaves (bounded)
        const unsigned long long t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 4000000ull) __nanosleep(1000);
    }
    __syncthreads();
    if (warp == kEpiWarps + 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(C::TMEM_COLS) : "memory");
    }
}

// Gate matrices (u8 codes, row g H + j) -> centered fp16 rows by cell pair: row 8 (j / 2) + 2 g + (j & 1) is
// gate g of cell j, so that a pair's eight sums are eight consecutive accumulator columns and a block's rows
// are contiguous for any number of cells per block; rows of cells >= H are zero.
__global__ void pair_rows_kernel(const uint8_t *__restrict__ codes, int64_t ld, int H, int K, int kp, int64_t rows,
                                 __half *__restrict__ out) {
    const int64_t total = rows * (kp / 8);
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t n = x / (kp / 8);
        const int k0 = (int)(x % (kp / 8)) * 8, g = (int)(n % 8) / 2;
        const int64_t j = 2 * (n / 8) + (n & 1);
        __align__(16) __half v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + i;
            v[i] = (j < H && k < K) ? __int2half_rn((int)codes[(g * (int64_t)H + j) * ld + k] - 128) : __int2half_rn(0);
        }
        *reinterpret_cast<uint4 *>(out + n * kp + k0) = *reinterpret_cast<const uint4 *>(v);
    }
}

// Column constants by cell pair: [pairs][4 gates][3] float2, bias, Wx and Wh row code sums (integers below
// 2^24, exact), zero past H.
__global__ void pair_constants_kernel(const float *__restrict__ bias, const int32_t *__restrict__ sx,
                                      const int32_t *__restrict__ sh, int H, int64_t pairs, float2 *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pairs * 4) return;
    const int64_t j = i / 4 * 2, n = i % 4 * H + j;
    float2 b = make_float2(0.0f, 0.0f), cx = b, ch = b;
    if (j < H) b.x = bias[n], cx.x = (float)sx[n], ch.x = (float)sh[n];
    if (j + 1 < H) b.y = bias[n + 1], cx.y = (float)sx[n + 1], ch.y = (float)sh[n + 1];
    out[3 * i] = b, out[3 * i + 1] = cx, out[3 * i + 2] = ch;
}

bool plan_of(const qnn_lstm_model *m, int64_t B, Plan *p) {
    if (m->P != 0 || m->S != 1) return false;
    int64_t kx = 0;
    for (int64_t l = 0; l < m->L; ++l) kx = std::max(kx, round_up(m->layers[l].kin, 64));
    return make_plan(m->L, m->H, kx, round_up(m->H, 64), B, sm_count(), p);
}

template <int NC, int MT, int SP>
qnn_status launch(const PersistArgs &a, const Plan &p, int64_t L, cudaStream_t st) {
    static std::atomic<int> configured{-1};
    int dev = 0;
    QNN_CUDA_TRY(cudaGetDevice(&dev));
    if (configured.load() != dev) {
        QNN_CUDA_TRY(cudaFuncSetAttribute(lstm_persist_kernel<NC, MT, SP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
        configured.store(dev);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L * p.G));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = coop_refused() ? cudaErrorCooperativeLaunchTooLarge
                                         : cudaLaunchKernelEx(&cfg, lstm_persist_kernel<NC, MT, SP>, a);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        return QNN_ERR_NO_COOP;
    }
    QNN_CUDA_TRY(e);
    return QNN_OK;
}

// The stack's weights in the layout above (once per model), and the 8-bit output layer's.
qnn_status prepare(qnn_lstm_model *m) {
    if (m->pw) return QNN_OK;
    const int64_t H = m->H, L = m->L, kh = round_up(H, 64), pairs = (H + 1) / 2, rows = 8 * pairs;
    const bool quant_out = m->C > 0 && m->d.output_mode == QNN_OUT_QUANT;
    const int64_t const_bytes = round_up(pairs * kPairConsts * (int64_t)sizeof(float2), 256);
    size_t bytes = quant_out ? m->C * kh * 2 : 0;
    for (int64_t l = 0; l < L; ++l) bytes += rows * (round_up(m->layers[l].kin, 64) + kh) * 2 + const_bytes;
    void *buf = nullptr;
    QNN_TRY(model_alloc(m, &buf, bytes, true));
    char *w = reinterpret_cast<char *>(buf);
    qnn_status s = QNN_OK;
    std::vector<PersistWeights> pl((size_t)L);
    auto grid = [](int64_t n) { return (unsigned)((n + 255) / 256); };
    for (int64_t l = 0; l < L && s == QNN_OK; ++l) {
        const LayerDev &ly = m->layers[l];
        PersistWeights &o = pl[(size_t)l];
        const int64_t kx = round_up(ly.kin, 64);
        o.wx16 = reinterpret_cast<__half *>(w), w += rows * kx * 2;
        o.wh16 = reinterpret_cast<__half *>(w), w += rows * kh * 2;
        o.pairc = reinterpret_cast<float2 *>(w), w += const_bytes;
        pair_rows_kernel<<<grid(rows * (kx / 8)), 256>>>(ly.wx.codes, ly.wx.ld, (int)H, (int)ly.kin, (int)kx, rows, o.wx16);
        pair_rows_kernel<<<grid(rows * (kh / 8)), 256>>>(ly.wh.codes, ly.wh.ld, (int)H, (int)H, (int)kh, rows, o.wh16);
        pair_constants_kernel<<<grid(pairs * 4), 256>>>(ly.bias, ly.wx.sums, ly.wh.sums, (int)H, pairs, o.pairc);
        if (cudaGetLastError() != cudaSuccess) s = QNN_FAIL(QNN_ERR_CUDA);
    }
    __half *wo = nullptr;
    if (quant_out && s == QNN_OK) {
        wo = reinterpret_cast<__half *>(w);
        s = launch_center_fp16(m->wo.codes, m->C, H, m->wo.ld, wo, kh, nullptr);
    }
    if (s == QNN_OK && cudaDeviceSynchronize() != cudaSuccess) s = QNN_FAIL(QNN_ERR_CUDA);
    if (s != QNN_OK) {
        cudaFree(buf);
        return s;
    }
    m->pw = buf, m->pw_bytes = bytes, m->pw_wo16 = wo, m->pw_layers = std::move(pl);
    return QNN_OK;
}

}  // namespace

void persist_release(qnn_lstm_model *m) {
    cudaDeviceSynchronize();
    cudaFree(m->pw);
    cudaFree(m->pws);
    m->pw = m->pws = nullptr, m->pw_bytes = m->pws_bytes = 0;
    m->pw_wo16 = nullptr, m->pw_layers.clear();
}

// Where the launch-per-step recurrences keep a stack that qualifies. Stacks gain from layers running side
// by side in one launch (40 frames, this against the best other path, us: 5 x 500 B = 64 486 : 950, B = 256
// 912 : 1184; 2 x 128 B = 256 356 : 459). A single layer is one chain either way, and two row tiles or long
// reductions share one block's operand stream there, while the tensor-core recurrence spreads a step over every
// SM: it keeps single layers from its smallest batch on (1 x 500 B = 64 292 : 354, B = 128 362 : 361, B = 256 480
// : 393). With a few rows of a wide layer the layerwise kernel is as good (1 x 1024 B = 1 383 : 369, B = 5 383 :
// 391). Posteriors in pinned host memory cross the link during the wavefront's recurrence but only after this
// one, which counts where there are many (5 x 500 B = 256, 500 frames, end to end ms, 2000 classes 13.4 : 14.5,
// 4000 classes 19.1 : 17.0).
bool persist_preferred(const qnn_lstm_model *m, int64_t B, bool host_posteriors) {
    const bool tc = tc_recurrence_supported(m) && B >= kTcMinBatch;
    if (m->L == 1) return !tc && (m->H <= 512 || B > 4);
    return !(host_posteriors && B > kTile && m->C > 2048 && tc && tc_stack_supported(m));
}

qnn_status persist_path_forward(qnn_lstm_model *m, const float *x, int64_t B, int64_t T, float *y, float *logits,
                                float *h_state, float *c_state, float *h_all, cudaStream_t st, bool *used) {
    *used = false;
    Plan p;
    if (!plan_of(m, B, &p) || B * T > INT32_MAX / 2 || T >= (1 << 24)) return QNN_OK;
    QNN_TRY(prepare(m));
    const int64_t L = m->L, I = m->I, H = m->H, C = m->C, R = m->R, rows = B * T;
    const int64_t kh = round_up(H, 64), kx0 = round_up(I, 64);
    const bool quant_out = C > 0 && m->d.output_mode == QNN_OUT_QUANT;
    const bool x_dev = is_device_ptr(x), y_dev = is_device_ptr(y);
    const bool hs_dev = h_state && is_device_ptr(h_state), cs_dev = c_state && is_device_ptr(c_state);
    const bool ha_dev = h_all && is_device_ptr(h_all);
    float *const y_map = (!y_dev && C > 0) ? static_cast<float *>(host_mapped_ptr(y)) : nullptr;
    const int64_t ycols = C > 0 ? C : R;
    size_t need = 0;
    auto acct = [&](size_t n) {
        const size_t at = (size_t)round_up((int64_t)need, 256);
        need = at + n;
        return at;
    };
    // zeroed at every call: counters, abort flag, range words, code sums
    const size_t o_ctr = acct(sizeof(unsigned) * 2 * kMaxL), o_abort = acct(4);
    const size_t o_mm = acct(sizeof(uint4) * L * 2 * p.MT * p.G * kTile);
    const size_t o_rs = acct(4 * L * rows);
    const size_t zeroed = need;
    const size_t o_codes = acct(2 * L * rows * kh), o_prm = acct(sizeof(qnn_qparams) * L * rows);
    const size_t o_h016 = acct(2 * L * B * kh), o_h0p = acct(sizeof(qnn_qparams) * L * B), o_h0s = acct(4 * L * B);
    const size_t o_x16 = acct(2 * rows * kx0), o_xp = acct(sizeof(qnn_qparams) * rows), o_xs = acct(4 * rows);
    const size_t o_h = acct(4 * L * B * R), o_c = acct(4 * L * B * H);
    const size_t o_x = x_dev ? 0 : acct(4 * rows * I);
    // fp32 outputs: every layer's with h_all, else the top layer's where they are read
    const bool top_out = C == 0 || m->d.output_mode == QNN_OUT_FLOAT;
    const size_t o_top = (top_out && !h_all && !(C == 0 && y_dev)) ? acct(4 * rows * R) : 0;
    const size_t o_ha = (h_all && !ha_dev) ? acct(4 * L * rows * R) : 0;
    const size_t o_lg = C > 0 ? acct(4 * rows * C) : 0;
    const size_t o_y = (y_dev || y_map || C == 0) ? 0 : acct(4 * rows * ycols);
    // logits in the caller's row order: written there, or staged for one copy to pageable memory
    float *const lg_to = !logits || !quant_out ? nullptr : is_device_ptr(logits) ? logits : static_cast<float *>(host_mapped_ptr(logits));
    const size_t o_ls = (logits && quant_out && !lg_to) ? acct(4 * rows * C) : 0;
    if (need > m->pws_bytes) {
        if (m->pws) {
            QNN_CUDA_TRY(cudaStreamSynchronize(st));
            QNN_CUDA_TRY(cudaFree(m->pws));
            m->pws = nullptr, m->pws_bytes = 0;
        }
        QNN_TRY(model_alloc(m, &m->pws, need, true));
        m->pws_bytes = need;
    }
    char *const ws = reinterpret_cast<char *>(m->pws);
    auto at = [&](size_t o) { return reinterpret_cast<float *>(ws + o); };
    int *status = nullptr;
    QNN_TRY(status_word(&status));
    QNN_CUDA_TRY(cudaMemsetAsync(ws, 0, zeroed, st));
    const float *xd = x;
    if (!x_dev) {
        QNN_CUDA_TRY(cudaMemcpyAsync(at(o_x), x, 4 * rows * I, cudaMemcpyHostToDevice, st));
        xd = at(o_x);
    }
    const float *h0 = at(o_h), *c0 = nullptr;
    if (hs_dev)
        h0 = h_state;
    else if (h_state)
        QNN_CUDA_TRY(cudaMemcpyAsync(at(o_h), h_state, 4 * L * B * R, cudaMemcpyHostToDevice, st));
    else
        QNN_CUDA_TRY(cudaMemsetAsync(at(o_h), 0, 4 * L * B * R, st));
    if (cs_dev)
        c0 = c_state;
    else if (c_state) {
        QNN_CUDA_TRY(cudaMemcpyAsync(at(o_c), c_state, 4 * L * B * H, cudaMemcpyHostToDevice, st));
        c0 = at(o_c);
    }
    __half *const x16 = reinterpret_cast<__half *>(ws + o_x16), *const h016 = reinterpret_cast<__half *>(ws + o_h016);
    qnn_qparams *const xp = reinterpret_cast<qnn_qparams *>(ws + o_xp), *const h0p = reinterpret_cast<qnn_qparams *>(ws + o_h0p);
    int32_t *const xs = reinterpret_cast<int32_t *>(ws + o_xs), *const h0s = reinterpret_cast<int32_t *>(ws + o_h0s);
    QNN_TRY(quantize_rows_f16(xd, I, rows, I, kx0, x16, xp, xs, status, st, T, B));
    QNN_TRY(quantize_rows_f16(h0, R, L * B, R, kh, h016, h0p, h0s, status, st, 0, 0));

    PersistArgs a{};
    a.prm_h0 = h0p, a.rs_h0 = h0s, a.c0 = c0;
    a.h_fin = h_state ? (hs_dev ? h_state : at(o_h)) : nullptr;
    a.c_fin = c_state ? (cs_dev ? c_state : at(o_c)) : nullptr;
    a.out_t = R, a.out_b = T * R;
    a.mm = reinterpret_cast<uint4 *>(ws + o_mm);
    a.ctr = reinterpret_cast<unsigned *>(ws + o_ctr);
    a.abort_flag = reinterpret_cast<int *>(ws + o_abort);
    a.status = status;
    a.B = (int)B, a.T = (int)T, a.H = (int)H, a.kh = (int)kh, a.kbh = (int)(kh / 64), a.G = p.G;
    a.rows_box = p.rows_box, a.kps = p.kps, a.slots = p.slots, a.slot_bytes = p.slot_bytes;
    QNN_TRY(tc_map_kblocks(&a.mh0, h016, L * B, kh, p.rows_box, p.kps));
    __half *const codes = reinterpret_cast<__half *>(ws + o_codes);
    qnn_qparams *const prm = reinterpret_cast<qnn_qparams *>(ws + o_prm);
    int32_t *const rs = reinterpret_cast<int32_t *>(ws + o_rs);
    float *const all = h_all ? (ha_dev ? h_all : at(o_ha)) : nullptr;
    float *const top = !top_out ? nullptr : all ? all + (L - 1) * rows * R : (C == 0 && y_dev) ? y : at(o_top);
    for (int64_t l = 0; l < L; ++l) {
        const LayerDev &ly = m->layers[l];
        const PersistWeights &pw = m->pw_layers[(size_t)l];
        const int64_t kx = round_up(ly.kin, 64), wrows = 4 * round_up(H, 2);  // (rows past them load as zero)
        PersistLayer &d = a.layer[l];
        d.pwx = ly.wx.params, d.pwh = ly.wh.params, d.pairc = pw.pairc;
        d.prm_x = l == 0 ? xp : prm + (l - 1) * rows, d.rs_x = l == 0 ? xs : rs + (l - 1) * rows;
        d.prm = prm + l * rows, d.rs = rs + l * rows, d.codes = codes + l * rows * kh;
        d.out = all ? all + l * rows * R : l == L - 1 ? top : nullptr;
        d.kin = (int)ly.kin, d.kbx = (int)(kx / 64);
        QNN_TRY(tc_map_kblocks(&a.mx[l], l == 0 ? x16 : codes + (l - 1) * rows * kh, rows, kx, p.rows_box, p.kps));
        QNN_TRY(tc_map_kblocks(&a.mh[l], d.codes, rows, kh, p.rows_box, p.kps));
        QNN_TRY(tc_map_f16(&a.mwx[l], pw.wx16, wrows, kx, 16 * p.NC));
        QNN_TRY(tc_map_f16(&a.mwh[l], pw.wh16, wrows, kh, 16 * p.NC));
    }
    {
        ProfScope prof("lstm_persist", st);
        auto run = [&](auto nc) -> qnn_status {
            constexpr int NC = decltype(nc)::value;
            if (p.MT == 2) {
                if constexpr (tmem_used(NC, 2) <= kTmemCols)
                    return launch<NC, 2, 1>(a, p, L, st);
                else
                    return QNN_FAIL(QNN_ERR_INVALID_ARG);  // (no plan asks for it)
            }
            return p.SP == 4 ? launch<NC, 1, 4>(a, p, L, st) : p.SP == 2 ? launch<NC, 1, 2>(a, p, L, st) : launch<NC, 1, 1>(a, p, L, st);
        };
        using std::integral_constant;
        QNN_TRY(p.NC == 2   ? run(integral_constant<int, 2>{})
                : p.NC == 4 ? run(integral_constant<int, 4>{})
                : p.NC == 5 ? run(integral_constant<int, 5>{})
                            : run(integral_constant<int, 6>{}));
    }
    float *const lg = C > 0 ? at(o_lg) : nullptr;
    float *const yd = y_dev ? y : y_map ? y_map : at(o_y);
    if (quant_out) {
        // the top layer's codes are the output product's operand, time-major; so are its logits
        TcOperands op;
        QNN_TRY(tc_operands(&op, codes + (L - 1) * rows * kh, rows, m->pw_wo16, C, kh, tc_pick_bn(rows, C, kh)));
        QNN_TRY(tc_linear(op, prm + (L - 1) * rows, 1, rs + (L - 1) * rows, R, m->wo.params, C, m->wo.sums, m->bo, lg, C,
                          nullptr, st));
        if (logits) {
            QNN_TRY(launch_rows_to_sequences(lg, B, T, C, lg_to ? lg_to : at(o_ls), st));
            if (!lg_to) QNN_CUDA_TRY(cudaMemcpyAsync(logits, at(o_ls), 4 * rows * C, cudaMemcpyDeviceToHost, st));
        }
        QNN_TRY(launch_softmax_rows(lg, rows, C, yd, st, B, T, 0));
    } else if (C > 0) {
        QNN_TRY(launch_float_linear(top, rows, R, m->wo_f, C, m->bo, lg, st));
        if (logits) QNN_CUDA_TRY(cudaMemcpyAsync(logits, lg, rows * C * 4, cudaMemcpyDefault, st));
        QNN_TRY(launch_softmax_rows(lg, rows, C, yd, st));
    } else if (top != y) {
        QNN_CUDA_TRY(cudaMemcpyAsync(y, top, rows * R * 4, cudaMemcpyDefault, st));
    }
    if (C > 0 && !y_dev && !y_map) QNN_CUDA_TRY(cudaMemcpyAsync(y, yd, rows * C * 4, cudaMemcpyDeviceToHost, st));
    if (h_all && !ha_dev) QNN_CUDA_TRY(cudaMemcpyAsync(h_all, all, 4 * L * rows * R, cudaMemcpyDeviceToHost, st));
    if (h_state && !hs_dev) QNN_CUDA_TRY(cudaMemcpyAsync(h_state, at(o_h), 4 * L * B * R, cudaMemcpyDeviceToHost, st));
    if (c_state && !cs_dev) QNN_CUDA_TRY(cudaMemcpyAsync(c_state, at(o_c), 4 * L * B * H, cudaMemcpyDeviceToHost, st));
    *used = true;
    return QNN_OK;
}

}  // namespace qnn
