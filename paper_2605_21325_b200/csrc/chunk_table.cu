// Chunk table of a packed batch, built on the device.
//
// The sequence offsets (host memory) travel as kernel parameters, a few hundred sequences per
// launch, so no host-to-device copy, staging buffer or synchronisation is involved: the table is
// ready in stream order before the kernel that reads it.
#include "common.cuh"

namespace tri_inv {
namespace {

constexpr int kSeqsPerLaunch = 960;

struct SeqBatch {
  int32_t cu[kSeqsPerLaunch + 1];  // offsets of the sequences of this launch
  int32_t n_seqs;
  int32_t first_chunk;             // index of this batch's first table entry
  int32_t C;
};

// A warp per sequence: its lanes sum the chunks of the sequences before it and write its entries.  A thread per sequence did both one by
// one, with a division for each sequence before its own: a packed fused call on 960 / 500 sequences of up to 20 / 60 tokens took 86 / 70 us,
// 57 / 54 so; 64 sequences of up to 2048 tokens 242 and 238; with a few sequences there is no difference.
constexpr int kWarps = 8;
__global__ void __launch_bounds__(kWarps * 32) chunk_table_kernel(ChunkEntry* tab, const __grid_constant__ SeqBatch b) {
  __shared__ int32_t cu[kSeqsPerLaunch + 1];   // indexed by lane below, which kernel parameters serve one address at a time
  const int lane = threadIdx.x & 31, s = blockIdx.x * kWarps + (threadIdx.x >> 5), shift = 31 - __clz(b.C);   // C: a power of two
  const int last = min((int)(blockIdx.x + 1) * kWarps, b.n_seqs);   // offsets 0 .. last are all that the block reads
  for (int q = threadIdx.x; q <= last; q += kWarps * 32) cu[q] = b.cu[q];
  __syncthreads();
  let_successor_start();
  wait_for_predecessor();
  if (s >= b.n_seqs) return;
  int before = 0;
  for (int q = lane; q < s; q += 32) before += (cu[q + 1] - cu[q] + b.C - 1) >> shift;
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) before += __shfl_xor_sync(0xffffffffu, before, m);
  const int beg = cu[s], len = cu[s + 1] - beg;
  for (int c = lane; c << shift < len; c += 32) tab[b.first_chunk + before + c] = ChunkEntry{beg + (c << shift), min(b.C, len - (c << shift))};
}

}  // namespace

cudaError_t launch_chunk_table(ChunkEntry* dev_tab, const tri_inv_desc* d, cudaStream_t stream) {
  int first_chunk = 0;
  for (int s0 = 0; s0 < d->n_seqs; s0 += kSeqsPerLaunch) {
    SeqBatch b;
    b.n_seqs = d->n_seqs - s0 < kSeqsPerLaunch ? d->n_seqs - s0 : kSeqsPerLaunch;
    b.first_chunk = first_chunk;
    b.C = d->C;
    for (int q = 0; q <= b.n_seqs; ++q) b.cu[q] = d->cu_seqlens[s0 + q];
    for (int q = 0; q < b.n_seqs; ++q) first_chunk += (b.cu[q + 1] - b.cu[q] + d->C - 1) / d->C;
    const cudaError_t e = launch_early(chunk_table_kernel, dim3((b.n_seqs + kWarps - 1) / kWarps), kWarps * 32, 0, stream, dev_tab, b);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace tri_inv
