// Internal declarations of the resuming launch that spreads one shot over a cluster of blocks
// (relay_split.cu), shared with the host API.
#pragma once

#include "qldpc_internal.h"

namespace qldpc {

constexpr int kSplit = 4;                   // blocks of a cluster
constexpr uint32_t kNoSlot = 0xffffffffu;   // past a fault's degree

// The graph split over the blocks of a cluster: block b holds checks row0[b] .. row0[b+1]-1
// (row0 even; the rows laid out as in FusedGraph, by their index in the block) and up to
// threads * vpt faults.
struct SplitGraph {
    int N, cor_words, min_deg;
    int row0[kSplit + 1];
    int msg_bytes;             // a block's message array
    int rows;                  // rows of a block's message array (even)
    int pad_stride;            // words of pad_mask a block
    const uint8_t *chk_deg;    // [Mp]
    const int32_t *fault;      // [kSplit][threads * vpt] fault of each fault slot, -1: none
    const uint4 *slots;        // [kSplit][threads * vpt] the fault's messages, increasing check
                               // order: block << 24 | byte offset there, kNoSlot past its degree
    const uint32_t *pad_mask;  // [kSplit][pad_stride] binary16 only (see FusedGraph)
    const float *w;            // [N]
    const float *gamma;        // [(R+1)][N]
};

struct SplitKernel {
    int msg_fp16, threads, vpt, dv;
    const void *fn;
    cudaError_t (*launch)(int clusters, size_t smem, cudaStream_t st, const SplitGraph &g,
                          const DevParams &p, const uint64_t *syn, DecodeOut out,
                          unsigned int *counter, ShotMap map, TailCont tc, int most);
};
void split_table(const SplitKernel **out, int *n);

inline size_t split_smem_bytes(const SplitGraph &g) {
    return (size_t)g.msg_bytes + 8 * (size_t)g.rows;  // messages, decision bytes
}

}  // namespace qldpc
