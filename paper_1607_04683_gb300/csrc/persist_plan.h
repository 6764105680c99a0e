// persist_plan.h — how the persistent stack kernel (lstm_persist.cu) lays a model and a batch out on the
// SMs: plain host arithmetic without CUDA, so that it can be checked over its whole range on the CPU.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace qnn {
namespace persist {

constexpr int kMaxL = 8;               // layers of a launch (tensor maps are kernel arguments)
constexpr int kMaxSlots = 4;           // operand ring slots
constexpr int kSlotBytes = 32 * 1024;  // at most (two k-blocks of 128 rows)
constexpr int kTile = 128;             // rows (sequences) of a tile
constexpr int kSmemMax = 227 * 1024;
constexpr int kTmemCols = 512;         // tensor-memory columns of an SM

// Tensor-memory columns of a block of 4 NC cells: per row tile two accumulators for x_t (by frame parity) and
// one for h_{t-1}, 16 NC gate columns each.
constexpr int tmem_used(int NC, int MT) { return 3 * MT * 16 * NC; }

// Shared memory beside the ring and the weights: barriers, ranges, (MT = 1) the pairs' code sums, and the sums
// handed over, [quarter][pair][16 words][32 rows].
constexpr int misc_bytes(int NC, int MT, int SP) {
    return 8 * (2 * kMaxSlots + 8) + 16 + 4 * kTile * 4 + (MT == 1 ? 2 * NC * 64 : 0) +
           (SP > 1 ? (2 * NC - (2 * NC + SP - 1) / SP) * (4 / SP) * 64 * 32 : 0);
}

struct Plan {
    int NC = 0, MT = 1, SP = 1, G = 0;  // cells of a block / 4, row tiles, quarters a pair's warps share, blocks a layer
    int rows_box = 0, kps = 0, slots = 0, slot_bytes = 0;
    size_t smem = 0;
};

// The smallest cell count per block for which the blocks of a stack of L layers of H cells (reductions of kx
// and kh, rounded up to 64) fit the SMs one each, their accumulators the tensor memory, and the widest layer's
// weights leave room for the operand ring; false if there is none.
inline bool make_plan(int64_t L, int64_t H, int64_t kx, int64_t kh, int64_t B, int64_t sms, Plan *p) {
    if (L > kMaxL || B < 1 || B > 2 * kTile || kh > 1024 || kx > 1024) return false;
    p->MT = B > kTile ? 2 : 1;
    p->rows_box = (int)std::min<int64_t>(kTile, (B + 7) / 8 * 8);
    p->SP = B <= 32 ? 4 : B <= 64 ? 2 : 1;
    for (int NC : {2, 4, 5, 6}) {
        const int64_t G = (H + 4 * NC - 1) / (4 * NC);
        if (G * L > sms || tmem_used(NC, p->MT) > kTmemCols) continue;
        const int64_t weights = (kx + kh) / 64 * NC * 2048;
        // (by the widest slots, so that a model's layout does not depend on the batch)
        const int64_t left = kSmemMax - weights - misc_bytes(NC, p->MT, p->SP);
        if (kSmemMax - weights - std::max(misc_bytes(NC, 1, 1), misc_bytes(NC, 2, 1)) < 2 * kSlotBytes) continue;
        // (handed-over sums take up to 24 KB: where two whole slots don't fit beside them, two halves do)
        p->kps = std::max(1, std::min(8, (left >= 2 * kSlotBytes ? kSlotBytes : kSlotBytes / 2) / (p->rows_box * 128)));
        p->slot_bytes = p->kps * p->rows_box * 128;
        const int64_t slots = std::min<int64_t>(kMaxSlots, left / p->slot_bytes);
        p->NC = NC, p->G = (int)G, p->slots = (int)slots;
        // an operand box of fewer than 128 rows is multiplied as 128: its last slot's reads stay inside
        const int64_t used = slots * p->slot_bytes + weights + misc_bytes(NC, p->MT, p->SP);
        p->smem = (size_t)std::min<int64_t>(kSmemMax, std::max(used, slots * p->slot_bytes + kTile * 128));
        return (int64_t)p->smem >= slots * p->slot_bytes + kTile * 128;
    }
    return false;
}

}  // namespace persist
}  // namespace qnn
