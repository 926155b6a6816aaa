// Which forward and backward calls are replayed from graphs: host bookkeeping only (stage.cu captures and launches).
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

#include <vector>

namespace ast {

// One forward or backward call as a graph: the kernels of a call depend on the slot and on the caller's two buffers only.
struct Replay {
    bool bwd;
    int slot;
    const void *a, *b;                             // x and y, or dy and dx
    uint64_t used;                                 // round in which it was last asked for
    int seen;                                      // direct calls so far; -1: cannot be captured
    uint64_t launches;
    cudaGraphExec_t exec;
};
// At most MAX_REPLAYS calls of a stage are kept.  A round asks for two calls a micro-batch in the same order every time, so a full table must not
// make room for the newest call: from 33 micro-batches on each entry would go just before it comes round again, and nothing would ever be replayed.
// An entry goes when it was not asked for in the last REPLAY_ROUNDS rounds; until then the calls beyond the table are launched directly.
// A sixth of MobileNetV2 at batch 4, us a micro-batch with 32, 33, 40 and 64 of them a round: 203, 204, 216, 236; with the least recently used
// entry making room for the newest call 203, 238, 238, 238.
constexpr size_t MAX_REPLAYS = 64;
constexpr uint64_t REPLAY_ROUNDS = 64;

// The entry of a call in round `round`; nullptr: the table is full and the call is not in it.  *dropped: the graph of the entry that made room, or null.
inline Replay* replay_entry(std::vector<Replay>& table, bool bwd, int slot, const void* a, const void* b, uint64_t round, cudaGraphExec_t* dropped) {
    *dropped = nullptr;
    Replay* oldest = nullptr;
    for (Replay& q : table) {
        if (q.bwd == bwd && q.slot == slot && q.a == a && q.b == b) {
            q.used = round;
            return &q;
        }
        if (!oldest || q.used < oldest->used) oldest = &q;
    }
    const Replay fresh{bwd, slot, a, b, round, 0, 0, nullptr};
    if (table.size() < MAX_REPLAYS) {
        table.push_back(fresh);
        return &table.back();
    }
    if (round - oldest->used <= REPLAY_ROUNDS) return nullptr;
    *dropped = oldest->exec;
    *oldest = fresh;
    return oldest;
}

}  // namespace ast
