// Internal interface of the FNV-1a-64 digest kernels (wt_fnv.cu) for the host library
// (wt_host.cpp, wt_noalloc.cu).  Not part of the public C ABI (include/wt.h).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace wt {

// ---------------------------------------------------------------- FNV-1a-64
constexpr uint64_t kLeafBytes = 4096;
// Largest buffer a digest call accepts (1 TiB, above any device's memory): bounds the leaf and
// chunk counts so that no size the caller passes can wrap them.
constexpr uint64_t kMaxFnvBufferBytes = 1ull << 40;

// The tree digest's second level is a serial FNV chain over 8 bytes per leaf.  It runs in
// chunks of kTreeChunk bytes, one thread each, combined exactly (see the kernels).
constexpr uint32_t kTreeChunk = 256;
constexpr uint32_t kChunkLeaves = kTreeChunk / 8;

// The buffers of one batch, as a kernel parameter.  24 bytes each, so that the largest
// batch just fits the 32,764-byte parameter space.
template <int N>
struct FnvTab {
  static constexpr int kMax = N;
  uint32_t n;
  uint32_t chunk;       // bytes of a chunk of the serial stream
  uint64_t chunk_pow;   // p^chunk mod 2^64
  uint64_t *out;        // device address of the first buffer's digest (contiguous)
  const uint8_t *ptr[N];
  uint64_t nbytes[N];
  uint32_t leaf_prefix[N + 1];   // first leaf of buffer i in the batch; [n] = total
  uint32_t chunk_prefix[N + 1];  // first chunk of buffer i in the batch; [n] = total
};
constexpr int kMaxFnv = 1344;  // buffers per batch
using FnvBatch = FnvTab<kMaxFnv>;

// Device scratch per chunk beyond the leaf digests: a transition table, the starting low byte
// and the chunk's sum.
constexpr size_t kChunkScratchBytes = 4 + 4 + 8;

// Fills b with the leading buffers of the list (*taken of them, at least one) and returns the
// device scratch bytes that launch_fnv_tree, or with `plain` launch_fnv_plain, needs for them
// (0 for literal digests where no buffer has more than 64 KiB and the batch no more than 32 MiB).
// Digest i goes to out[i].
size_t fnv_fill_batch(FnvBatch &b, const void *const *ptr, const uint64_t *nbytes, uint64_t *out, size_t n, bool plain,
                      size_t *taken);

// Kernel launches of launch_fnv_tree for the batch.
int fnv_tree_launches(const FnvBatch &b);

cudaError_t launch_fnv_tree(const FnvBatch &b, void *scratch, cudaStream_t s);

// The literal digests.  With the scratch that fnv_fill_batch asked for the chains run in chunks;
// where there is none to be had, every buffer of the batch in one thread.
int fnv_plain_launches(const FnvBatch &b, bool scratch);
cudaError_t launch_fnv_plain(const FnvBatch &b, void *scratch, cudaStream_t s);

}  // namespace wt
