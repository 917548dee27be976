// Batched execution of the many tiny contractions near the leaves of a tree.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace tn {

constexpr int64_t MICRO_MAX = 4096;  // entries (all items) of every tensor of a micro node
constexpr int MICRO_BETA = 1024;     // batch items a micro kernel handles
constexpr int MICRO_THREADS = 1024;      // at most (fewer where no level has that many outputs)
constexpr int MICRO_OTAB = 256;          // outputs per item / summed entries with offset tables
constexpr int MICRO_KTAB = 64;
constexpr int MICRO_BLOB = 144 * 1024;   // bytes of a subtree's records at most
constexpr int MICRO_SMEM = 200 * 1024;   // records, staged values and maxima
constexpr int MICRO_MAXIMA = 2048;       // staged maxima at most

// Lanes that share one output's summed space (a power of two): enough to keep
// the serial part short where the outputs alone leave most lanes idle.
inline int micro_lanes(int64_t elems, double K) {
    int kl = 1;
    while (kl < 32 && K >= 8.0 * kl && elems * kl * 2 <= 1024) kl *= 2;
    return kl;
}
// Warp steps of a node: its tasks (32 lanes each) times summed entries per lane.
inline double micro_cost(int64_t elems, double K) {
    const int kl = micro_lanes(elems, K);
    return (double)((elems * kl + 31) / 32) * ((K + kl - 1) / kl);
}

// One tiny pairwise contraction, offsets relative to the program arena
// (elements) and to the maxima / argmax buffers, and positions of the staged
// copies in shared memory (elements / slots; -1: not staged).  otab / ktab:
// byte position in the records of the {A, B} offsets (16 bits each) of every
// output of an item / summed index; -1: decoded from the int4 {size, shift,
// stride A, stride B} of the output and the summed dimensions after the head.
struct alignas(16) MicroHead {
    int32_t nout, nk, klog, flags;       // flags 1: power-of-two sizes, 2: one task and one item
    int32_t nout_total, ktotal, nbeta, elems;
    int32_t sA, sB, sC, otab;
    int32_t smxa, smxb, smxc, ktab;
    int16_t bsa, bsb, mxa_bs, mxb_bs;
    int64_t offA, offB, offC, amoff;     // amoff: argmax offset (-1: none)
    int64_t mxa, mxb, mxc;               // maximum slots (-1: none)
};

// A subtree: its records at byte `off` of the buffer, `bytes` long (a multiple
// of 16), then nin uint32 arena offsets of the staged inputs and nmx uint32
// maximum slots (bit 31: the subtree's own, written back at the end; else read
// at the start).  Records: first task of each level (nlevels + 1 int32), the
// tasks (uint32: position of the node's head in 16-byte units << 16 | index of
// the task in the node) at byte `tasks`, then the heads with their dimensions
// and the offset tables.
// Shared memory: records, nmx maxima, staged values (inputs first).
struct MicroSub {
    int64_t off;
    int32_t bytes, nlevels, tasks, nin, nmx, pad;
};

template <typename T>
void launch_micro(const unsigned char *blob, const MicroSub *subs, int nsub, int smem, int semiring,
                  int threads, T *arena, unsigned long long *mx, int32_t *am, cudaStream_t st);

}  // namespace tn
