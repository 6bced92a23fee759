// The coarse end of a cycle in one launch (m1_tail.cu): its interface, and the rule
// for where it begins.
#pragma once
#include <cstddef>
#include <cuda_runtime.h>

#include "m1_device.cuh"

namespace m1 {

// Blocks of the largest cluster, clusters of that size in a launch, cluster sizes (16, 8,
// 4, 2, 1), levels, and the dynamic shared memory a block may take.
constexpr int kTailBlocks = 16, kTailClusters = 36, kTailSizes = 5, kTailLevels = 20;
constexpr int kTailSmem = 220 * 1024;
// The tail begins at the first coarse FP64 level of at most this many cells, which is
// about what 16 blocks hold with the levels below.  With the line at 2048 cells a step of
// 320 x 208 (a level of 4160) took 112.8 ms, at 8192 106.2; the paper's beam at 512^2
// (64^2) 23.4 and 23.6; ten small instances, whose clusters no longer all run at once,
// 85.1 and 89.5.
constexpr int kTailCells = 8192;

// Operations of a tail's program, one byte each: the operation + 8 x the level
// counted from the tail's first.  FIRST: the FAS right-hand side and the first
// pseudo-time step of a fresh visit; PSEUDO: one more step; RESID: the residual;
// RESTRICT: from the level above into this one; PROLONG: from the level below onto
// this one.  The FP32 tail forms the FAS right-hand side in an operation of its own
// (FAS) before FIRST.
enum TailOp { TAIL_FIRST = 0, TAIL_PSEUDO = 1, TAIL_RESID = 2, TAIL_RESTRICT = 3, TAIL_PROLONG = 4,
              TAIL_FAS = 5 };

// Cells per block of a level of n cells over nb blocks: equal shares, but no
// fewer than make a block's work worth a cluster barrier.
__host__ __device__ inline int tail_per(int n, int nb)
{
    int p = (n + nb - 1) / nb;
    const int least = 64;
    const int cap = n < least ? n : least;
    p = p < cap ? cap : p;
    return (p + 3) & ~3;
}

// Blocks an instance's cluster should have when `count` instances step together, so that
// all of them run at once (the device holds 9 clusters of 16 of these blocks, 18 of 8).
// V-cycles of 64^2 instances, ms a cycle, always 16 blocks and by this rule: 10 instances
// 0.393 and 0.253, 32 0.92 and 0.36, 128 3.59 and 1.05 (a launch per coarse operation: 0.53,
// 0.89, 2.73); 128^2, whose tails need 8 blocks: 32 1.36 and 1.39 (2.26).
inline int tail_blocks_for(int count)
{
    return count <= 9 ? 16 : count <= 18 ? 8 : count <= 36 ? 4 : count <= 74 ? 2 : 1;
}

// Dynamic shared memory of a block for a tail of nlev levels, the first of n0 cells.
size_t tail_smem(int n0, int nb, int dim, int nlev);

// The kernel's attributes on the current device (once per engine).
cudaError_t tail_prepare();

// items of wl: (instance, first tail level); progs[first level]: (offset, length)
// in prog; a cluster of `blocks` each.
cudaError_t launch_tail(const Level<double>* lv, int cap, int nlev, WorkList wl, Ctl* ctls,
                        const unsigned char* prog, const int2* progs, size_t smem, int blocks,
                        cudaStream_t s);

// ---- the FP32 hierarchy's (m1_tail32.cu) -----------------------------------------
// Its levels give the same bits in the tail and in launches of their own, so where it
// begins may depend on the company: with more instances each gets a smaller cluster
// (all of them then run at once) and a tail of fewer cells.
// A 1024^2 mixed step took 263.0 ms with at most 1024 cells a block (128^2 in 16), 269.5
// with 256 (64^2).
constexpr int kTail32Smem = 216 * 1024, kTail32Cells = 1024;   // a block's; cells a block at most

__host__ __device__ inline int tail32_per(int n, int nb)
{
    int p = (n + nb - 1) / nb;
    const int least = 128;
    const int cap = n < least ? n : least;
    p = p < cap ? cap : p;
    return (p + 3) & ~3;
}

// Blocks of an instance's cluster when `count` instances step together.
inline int tail32_blocks(int count)
{
    return count <= 8 ? 16 : count <= 18 ? 8 : count <= 36 ? 4 : count <= 74 ? 2 : 1;
}

size_t tail32_smem(int n0, int nb, int dim, int nlev);
cudaError_t tail32_prepare();
// ring: bit l set where the sweeps of level l are those of the cp.async strips.
cudaError_t launch_tail32(const Level<float>* lv, int cap, int nlev, WorkList wl, Ctl* ctls,
                          const unsigned char* prog, const int2* progs, unsigned ring, size_t smem,
                          int blocks, cudaStream_t s);

}  // namespace m1
