// batch_fast.h -- the persistent batched kernel for plans of the specialised
// FP32 sizes (batch_fast_f32.cu).
#pragma once
#include "batch.h"
#include "fast.h"

namespace fsp {

// One solve of a batch: the argument blocks of its five passes and its size.
struct FastBatchSolve {
    fast::RowArgs r1, r5;
    fast::ColArgs c2, c3, c4;
    int N;
};

// A work item: consecutive tiles of one pass of one solve.
struct FastBatchItem {
    int seg;    // BatchSeg with the item's solve, pass and dependency
    int tile0;  // first tile
};

struct FastBatchLaunch {
    const FastBatchSolve *solves;
    const BatchSeg *segs;
    const FastBatchItem *items;
    int total;
    BatchCtl *ctl;
    unsigned long long timeout_ns;
    unsigned grid;
    size_t smem;
};

bool fast_batch_has(int N);
// tiles of each pass, and tiles per item of each pass
void fast_batch_tiles(int N, int ntiles[5], int group[5]);
size_t fast_batch_smem(int N);
int fast_batch_blocks_per_sm(size_t smem);
cudaError_t launch_fast_batch(const FastBatchLaunch &L, cudaStream_t s);

}  // namespace fsp
