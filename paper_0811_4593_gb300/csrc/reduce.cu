// reduce.cu -- final folds of the per-block partial sums.
#include "reduce.cuh"

namespace lbm {

// Two-level fold of one lattice: block g folds rows g FOLD_ROWS .. of the partial sums
// into row nblocks + g, and the block that finishes last folds those rows into out. One
// block did all of it before: 16.8 MB of partial sums through one SM's FP64 pipe on a
// 512^3 lattice (524,288 rows), about 0.6 ms.
__global__ void __launch_bounds__(FOLD_THREADS)
    final_reduce_kernel(double* partials, uint32_t nblocks, double* out, uint32_t* ticket) {
  const uint32_t first = blockIdx.x * FOLD_ROWS;
  const uint32_t count = nblocks - first < FOLD_ROWS ? nblocks - first : FOLD_ROWS;
  if (gridDim.x == 1) {
    fold_rows(partials, count, out);
    return;
  }
  double* group = partials + 4ull * nblocks;
  fold_rows(partials + 4ull * first, count, group + 4ull * blockIdx.x);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();  // the group's row (written by this warp) before the ticket
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  fold_rows(group, gridDim.x, out);
  if (threadIdx.x == 0) *ticket = 0;  // ready for the next fold
}

cudaError_t launch_final_reduce(double* partials, uint32_t nblocks, double* out, uint32_t* ticket, cudaStream_t s) {
  final_reduce_kernel<<<fold_groups(nblocks), FOLD_THREADS, 0, s>>>(partials, nblocks, out, ticket);
  return cudaGetLastError();
}

// Final reduction of every lattice of a batch: block i folds entry i's partials, group
// after group as above, into results[slot][4]; blocks past the entries in use return at
// once.
__global__ void __launch_bounds__(FOLD_THREADS)
    batch_final_reduce_kernel(const BatchHeader* __restrict__ hdr, const BatchEntry* __restrict__ ents,
                              double* __restrict__ results) {
  if (blockIdx.x >= hdr->nentries) return;
  const BatchEntry& e = ents[blockIdx.x];
  double* partials = e.a.partials;
  double* out = results + 4ull * e.slot;
  const uint32_t nblocks = e.nblocks, groups = fold_groups(nblocks);
  if (groups == 1) {
    fold_rows(partials, nblocks, out);
    return;
  }
  double* group = partials + 4ull * nblocks;
  for (uint32_t g = 0; g < groups; ++g) {
    const uint32_t first = g * FOLD_ROWS;
    const uint32_t count = nblocks - first < FOLD_ROWS ? nblocks - first : FOLD_ROWS;
    fold_rows(partials + 4ull * first, count, group + 4ull * g);
  }
  __threadfence_block();
  fold_rows(group, groups, out);
}

cudaError_t launch_batch_final_reduce(const BatchHeader* hdr, const BatchEntry* ents, int capacity, double* results,
                                      cudaStream_t s) {
  batch_final_reduce_kernel<<<capacity, FOLD_THREADS, 0, s>>>(hdr, ents, results);
  return cudaGetLastError();
}

}  // namespace lbm
