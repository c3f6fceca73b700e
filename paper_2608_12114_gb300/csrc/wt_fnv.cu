// sm_103a kernels of the per-buffer FNV-1a-64 digests that prove ingested bytes equal the
// file's: the literal serial digest, and the tree digest (FNV-1a-64 of each 4 KiB leaf,
// then FNV-1a-64 over the buffer's length and its leaf digests).  The second level of the
// tree runs in parallel chunks, with the exact result of the serial chain.
#include <algorithm>
#include <cstring>

#include "wt_device.cuh"
#include "wt_fnv.h"
#include "wt_kernels.h"

namespace wt {

namespace {

// ------------------------------------------------------------------ FNV-1a-64
// The 64-bit state is held as two 32-bit words.  With p = 2^40 + 0x1b3 and x = lo ^ b,
//   (hi 2^32 + x) p mod 2^64 = (hi 0x1b3 + (x << 8) + high32(x 0x1b3)) 2^32 + low32(x 0x1b3),
// since hi 2^72 vanishes and x 2^40 keeps only (x << 8) in the high word.  The serial chain
// through a byte is then an xor and one 32 x 32 multiply on the low word; the high word is a
// multiply-add beside it.  The constants are FNV-1a-64's offset basis and prime.
constexpr uint32_t kFnvOffLo = 0x84222325u, kFnvOffHi = 0xcbf29ce4u;
constexpr uint32_t kFnvP = 0x1b3u;

struct Fnv {
  uint32_t lo = kFnvOffLo, hi = kFnvOffHi;
  __device__ __forceinline__ void byte(uint32_t b) {
    const uint32_t x = lo ^ b;
    const uint64_t w = (uint64_t)x * kFnvP;
    lo = (uint32_t)w;
    hi = hi * kFnvP + ((uint32_t)(w >> 32) + (x << 8));
  }
  // A word's four bytes, little-endian: the low word's chain first (the byte xored into the
  // low byte, one 32 x 32 -> 64 multiply), then the high word's four multiply-adds in one
  // Horner run, since hi' = hi p + t with t from the low word's step alone.  The masked xor
  // is one lop3 (a ^ (b & c), truth table 0x78) on the shifted word.  Measured on GB300 over
  // 1 GiB of leaves: 3.89 TB/s byte at a time, 4.28 TB/s this way, 4.40 TB/s with the
  // 64-byte slices of 8-warp blocks below.
  __device__ __forceinline__ void word(uint32_t v) {
    uint32_t t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint32_t x;
      asm("lop3.b32 %0, %1, %2, 0xff, 0x78;" : "=r"(x) : "r"(lo), "r"(v >> (8 * k)));
      const uint64_t w = (uint64_t)x * kFnvP;
      lo = (uint32_t)w;
      t[k] = (uint32_t)(w >> 32) + (x << 8);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) hi = hi * kFnvP + t[k];
  }
  __device__ __forceinline__ void vec(const uint4 &v) {
    word(v.x);
    word(v.y);
    word(v.z);
    word(v.w);
  }
  __device__ __forceinline__ void le64(uint64_t v) {
    word((uint32_t)v);
    word((uint32_t)(v >> 32));
  }
  __device__ __forceinline__ uint64_t value() const { return ((uint64_t)hi << 32) | lo; }
};

// The buffer that holds entry i of a prefix array (uniform over a warp unless it straddles two).
__device__ __forceinline__ uint32_t find_in(const uint32_t *prefix, uint32_t n, uint32_t i) {
  uint32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One thread per 4 KiB leaf.  A warp stages 64-byte slices of its 32 leaves in shared
// memory with coalesced asynchronous 16-byte copies (four lanes per leaf slice, eight
// leaves per warp instruction), double-buffered: slice s + 1 is in flight while each lane
// hashes its own row of slice s.  Rows are padded to 80 bytes, so the lanes that read at
// once use distinct banks.  A warp whose 32 leaves are whole, 16-byte aligned and from one
// buffer (every warp inside a large tensor) computes the copy addresses directly; other
// warps fetch each leaf's pointer and length from its lane.  Blocks of 8 warps hold 40 KB of
// staging; 64-byte slices in 8-warp blocks measured 4.40 TB/s against 4.28 with 128-byte
// slices in 4-warp blocks and 4.00 with 256-byte slices (1 GiB of leaves, GB300).
constexpr int kFnvWarps = 8;
constexpr int kSlice = 64;
constexpr int kSliceStride = kSlice + 16;
constexpr int kLanesPerLeaf = kSlice / 16;
constexpr int kLeavesPerRound = 32 / kLanesPerLeaf;

__device__ __forceinline__ void fnv_stage_fast(uint8_t (*dst)[kSliceStride], const uint8_t *wbase, uint32_t pitch,
                                               uint32_t s0, int lane) {
  const int sub = lane / kLanesPerLeaf, q = lane % kLanesPerLeaf;
  const uint8_t *src = wbase + (size_t)sub * pitch + s0 + q * 16;
#pragma unroll
  for (int r = 0; r < 32; r += kLeavesPerRound)
    cp_async16(smem_u32(&dst[r + sub][q * 16]), src + (size_t)r * pitch);
  cp_async_commit();
}

__device__ __forceinline__ void fnv_stage(uint8_t (*dst)[kSliceStride], const uint8_t *lp, uint32_t llen,
                                          uint32_t s0, int lane) {
  const int sub = lane / kLanesPerLeaf, q = lane % kLanesPerLeaf;
#pragma unroll 2
  for (int r = 0; r < 32; r += kLeavesPerRound) {
    const int src = r + sub;
    const uint8_t *p = reinterpret_cast<const uint8_t *>(__shfl_sync(0xffffffffu, (unsigned long long)lp, src));
    const uint32_t n = __shfl_sync(0xffffffffu, llen, src);
    const uint32_t o = s0 + q * 16;
    uint8_t *d = &dst[src][q * 16];
    if (p != nullptr && o < n) {
      if (o + 16 <= n && ((reinterpret_cast<uintptr_t>(p) + o) & 15) == 0) {
        cp_async16(smem_u32(d), p + o);
      } else {
        for (uint32_t k = 0; k < 16 && o + k < n; ++k) d[k] = p[o + k];
      }
    }
  }
  cp_async_commit();
}

// Runs h over this lane's llen bytes at lp, the warp staging slices of its 32 rows together
// (buf is the warp's own).  fast (warp-uniform): row r starts at wbase + r * pitch, 16-byte
// aligned, and its bytes up to the longest row's length may be read.
template <class H>
__device__ __forceinline__ void run_rows(H &h, uint8_t (*buf)[32][kSliceStride], const uint8_t *lp, uint32_t llen,
                                         bool fast, const uint8_t *wbase, uint32_t pitch, int lane) {
  // slices the longest row of the warp needs (warp-uniform)
  const uint32_t nsl = (__reduce_max_sync(0xffffffffu, llen) + kSlice - 1) / kSlice;
  if (nsl) {
    if (fast) fnv_stage_fast(buf[0], wbase, pitch, 0, lane);
    else fnv_stage(buf[0], lp, llen, 0, lane);
  }
  for (uint32_t si = 0; si < nsl; ++si) {
    if (si + 1 < nsl) {
      if (fast) fnv_stage_fast(buf[(si + 1) & 1], wbase, pitch, (si + 1) * kSlice, lane);
      else fnv_stage(buf[(si + 1) & 1], lp, llen, (si + 1) * kSlice, lane);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const uint32_t s0 = si * kSlice;
    if (s0 < llen) {
      const uint32_t m = min((uint32_t)kSlice, llen - s0);
      const uint8_t *row = buf[si & 1][lane];
      uint32_t k = 0;
      for (; k + 16 <= m; k += 16) h.vec(*reinterpret_cast<const uint4 *>(row + k));
      for (; k < m; ++k) h.byte(row[k]);
    }
    __syncwarp();  // every lane is done with this buffer before it is refilled
  }
}

// Device scratch of one batch.
struct FnvScratch {
  uint64_t *leaves;  // tree: leaf digests, buffer t's from word chunk_prefix[t] * kChunkLeaves on
  uint32_t *tab;     // [chunks] transition table of the chunk
  uint32_t *lstart;  // [chunks] low byte of the state at the chunk's start
  uint64_t *sum;     // [chunks] the chunk's part of the state (D below)
};

template <class Tab>
__global__ void __launch_bounds__(kFnvWarps * 32) fnv_leaf_kernel(const __grid_constant__ Tab b, uint64_t *leaves) {
  __shared__ __align__(16) uint8_t buf[kFnvWarps][2][32][kSliceStride];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t total = b.leaf_prefix[b.n];
  const uint64_t nwarps = (uint64_t)gridDim.x * kFnvWarps;
  for (uint64_t base = ((uint64_t)blockIdx.x * kFnvWarps + warp) * 32; base < total; base += nwarps * 32) {
    const uint64_t leaf = base + lane;
    const bool mine = leaf < total;
    const uint8_t *lp = nullptr;
    uint32_t llen = 0, t = 0xffffffffu;
    uint64_t slot = 0;
    if (mine) {
      t = find_in(b.leaf_prefix, b.n, (uint32_t)leaf);
      const uint64_t i = leaf - b.leaf_prefix[t];
      lp = b.ptr[t] + i * kLeafBytes;
      llen = (uint32_t)min(kLeafBytes, b.nbytes[t] - i * kLeafBytes);
      slot = (uint64_t)b.chunk_prefix[t] * kChunkLeaves + i;
    }
    const uint32_t t0 = __shfl_sync(0xffffffffu, t, 0);
    const bool fast = __all_sync(0xffffffffu, mine && t == t0 && llen == kLeafBytes &&
                                                   (reinterpret_cast<uintptr_t>(lp) & 15) == 0);
    const uint8_t *wbase = reinterpret_cast<const uint8_t *>(__shfl_sync(0xffffffffu, (unsigned long long)lp, 0));
    Fnv h;
    run_rows(h, buf[warp], lp, llen, fast, wbase, (uint32_t)kLeafBytes, lane);
    if (mine) leaves[slot] = h.value();
  }
}

// ---- a long serial chain in parallel chunks
//
// The chain costs one dependent xor and 32 x 32 multiply per byte (10 to 12 cycles), so the
// second level of a 1 GB tensor, 2 MB of leaf digests, takes 11 ms in one thread.  It is cut
// into chunks, one thread each, and combined exactly, from two facts about one FNV step
// h' = (h ^ b) p mod 2^64:
//  1. the low k bits of h evolve on their own, by a permutation of 2^k states whose top bit is
//     free: starting from s ^ 2^(k-1) instead of s flips bit k-1 at the end and nothing else
//     (p is odd).  So 8 starts describe what a chunk does to the low nibble, and, once the low
//     nibble at its start is known, 8 starts what it does to the high nibble of the low byte;
//  2. h ^ b = h + d with d = (l ^ b) - l, l the low byte of h, so over a chunk of m bytes
//     h_end = p^m h_start + D, where D depends only on the chunk's bytes and the low byte l at
//     its start: running the chain from h = l alone gives D = h_end - p^m l.
// Passes: (1) every chunk's low-nibble table; (2) per buffer, the chunks' low nibbles through
// those tables; (3) every chunk's high-nibble table; (4) as (2); (5) every chunk's D; (6) per
// buffer, h from its start and the D.  The result equals the serial chain bit for bit.
// Per byte (1) and (3) take 14 operations and (5) one run, where tables of the whole low byte
// take 320 and separate runs for the low and the high word of h two.  Every buffer of more than
// one chunk goes this way: 256-byte chunks keep the passes at a few microseconds each.
// Measured on GB300 (whole calls, leaves included): 2.97 GB with two 1 GB tensors 1332 -> 814
// us, 1253 tensors of 8 KiB to 8 MiB (1.56 GB) 1261 -> 457 us, against whole-byte tables over
// 4096-byte chunks for buffers above 16 MiB and one thread per buffer below; 797 and 443 us
// with short streams in one block each and the tables of long ones loaded ahead.  The literal
// digest of eight 16 MiB tensors, one thread each before: 276 ms -> 0.19 ms.

// p^e mod 2^64 by square and multiply
__host__ __device__ __forceinline__ uint64_t fnv_pow(uint64_t q, uint32_t e) {
  uint64_t r = 1;
  for (; e; e >>= 1, q *= q)
    if (e & 1) r *= q;
  return r;
}
constexpr uint64_t kFnvPrime = 0x100000001b3ull;

// Byte k of v in every byte, or in bytes 0 and 2.
template <int k>
__device__ __forceinline__ uint32_t bytes4(uint32_t v) { return __byte_perm(v, 0, 0x1111u * k); }
template <int k>
__device__ __forceinline__ uint32_t bytes2(uint32_t v) { return __byte_perm(v, 0, 0x4040u | k | k << 8); }

// The low nibble from starts 0..7, eight-bit lanes in two registers: (u 3) < 2^8 for u < 16
// and 3 = p mod 16, so one multiply advances four starts and no lane carries into the next.
// The mask of one step merges with the xor of the next.
struct LowNibble {
  uint32_t r0 = 0x03020100u, r1 = 0x07060504u;
  __device__ __forceinline__ void step(uint32_t bb) {
    r0 = ((r0 ^ bb) & 0x0f0f0f0fu) * 3u;
    r1 = ((r1 ^ bb) & 0x0f0f0f0fu) * 3u;
  }
  __device__ __forceinline__ void byte(uint32_t b) { step(bytes4<0>(b)); }
  __device__ __forceinline__ void word(uint32_t v) {
    step(bytes4<0>(v));
    step(bytes4<1>(v));
    step(bytes4<2>(v));
    step(bytes4<3>(v));
  }
  __device__ __forceinline__ void vec(const uint4 &v) { word(v.x), word(v.y), word(v.z), word(v.w); }
  // the low nibble at the end for start j in bits 4j .. 4j + 3
  __device__ __forceinline__ uint32_t table() const {
    uint32_t t = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) t |= (r0 >> (8 * j) & 15u) << (4 * j) | (r1 >> (8 * j) & 15u) << (16 + 4 * j);
    return t;
  }
};

// The low byte from starts nib + 16 j (j = 0..7), sixteen-bit lanes in four registers:
// (u 0xb3) < 2^16 for u < 256 and 0xb3 = p mod 256.
struct HighNibble {
  uint32_t r[4];
  __device__ __forceinline__ explicit HighNibble(uint32_t nib) {
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = (nib | 0x100000u) + (nib << 16) + 0x200020u * i;
  }
  __device__ __forceinline__ void step(uint32_t bb) {
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = ((r[i] & 0x00ff00ffu) ^ bb) * 0xb3u;
  }
  __device__ __forceinline__ void byte(uint32_t b) { step(bytes2<0>(b)); }
  __device__ __forceinline__ void word(uint32_t v) {
    step(bytes2<0>(v));
    step(bytes2<1>(v));
    step(bytes2<2>(v));
    step(bytes2<3>(v));
  }
  __device__ __forceinline__ void vec(const uint4 &v) { word(v.x), word(v.y), word(v.z), word(v.w); }
  __device__ __forceinline__ uint32_t table() const {
    uint32_t t = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) t |= (r[i] >> 4 & 15u) << (8 * i) | (r[i] >> 20 & 15u) << (8 * i + 4);
    return t;
  }
};

// One entry of a table of 8 starts: start s < 16, the upper 8 from the lower by fact 1.
__device__ __forceinline__ uint32_t through(uint32_t table, uint32_t s) {
  return (table >> ((s & 7u) << 2) & 15u) ^ (s & 8u);
}
// The table of `a` followed by `b`.
__device__ __forceinline__ uint32_t then(uint32_t a, uint32_t b) {
  uint32_t t = a & 0x88888888u;
#pragma unroll
  for (int j = 0; j < 8; ++j) t ^= (b >> ((a >> (4 * j) & 7u) << 2) & 15u) << (4 * j);
  return t;
}
constexpr uint32_t kIdentity = 0x76543210u;

// The state before this lane's table when the lanes' tables follow one another from s.
__device__ __forceinline__ uint32_t walk_lanes(uint32_t g, uint32_t s, int lane) {
  uint32_t mine = 0;
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    if (k == lane) mine = s;
    s = through(__shfl_sync(0xffffffffu, g, k), s);
  }
  return mine;
}

// Walks n tables f[0..n) from start s with one warp: start[k] becomes the state before table k.
__device__ __forceinline__ void walk_tables(const uint32_t *f, uint32_t *start, uint32_t n, uint32_t s, int lane) {
  const uint32_t per = (n + 31) / 32;
  const uint32_t a = min(n, lane * per), e = min(n, a + per);
  uint32_t g = kIdentity;
  for (uint32_t k = a; k < e; ++k) g = then(g, f[k]);
  uint32_t mine = walk_lanes(g, s, lane);
  for (uint32_t k = a; k < e; ++k) {
    start[k] = mine;
    mine = through(f[k], mine);
  }
}

// A buffer's serial stream: its own bytes from FNV's offset basis (PLAIN, the literal digest),
// or the leaf digests from the state after LE64(nbytes) (the tree digest's second level).
template <bool PLAIN, class Tab>
__device__ __forceinline__ uint64_t stream_head(const Tab &b, uint32_t t) {
  Fnv h;
  if constexpr (!PLAIN) h.le64(b.nbytes[t]);
  return h.value();
}
template <bool PLAIN, class Tab>
__device__ __forceinline__ uint64_t stream_bytes(const Tab &b, uint32_t t) {
  if constexpr (PLAIN) return b.nbytes[t];
  return 8ull * (b.leaf_prefix[t + 1] - b.leaf_prefix[t]);
}

// Passes 1, 3 and 5 (PASS 0, 1, 2): one thread per chunk.  Blocks of two warps spread a few
// thousand chunks over the SMs.  The leaf digests of a batch lie in whole chunks one after
// another (and up to a whole warp's), so every row may be read to its end; a caller's bytes
// take the coalesced copies where a warp's 32 chunks are whole, aligned and of one buffer.
constexpr int kChunkWarps = 2;
template <bool PLAIN, class Tab, int PASS>
__global__ void __launch_bounds__(kChunkWarps * 32) fnv_chunk_kernel(const __grid_constant__ Tab b, FnvScratch sc) {
  __shared__ __align__(16) uint8_t buf[kChunkWarps][2][32][kSliceStride];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t first = (blockIdx.x * kChunkWarps + warp) * 32, c = first + lane;
  const uint32_t total = b.chunk_prefix[b.n];
  if (first >= total) return;
  uint32_t len = 0, nchunk = 0, t = 0;
  if (c < total) {
    t = find_in(b.chunk_prefix, b.n, c);
    nchunk = b.chunk_prefix[t + 1] - b.chunk_prefix[t];
    len = (uint32_t)min((uint64_t)b.chunk, stream_bytes<PLAIN>(b, t) - (uint64_t)(c - b.chunk_prefix[t]) * b.chunk);
  }
  // a buffer of one chunk starts from a known state: it needs no table
  const bool mine = PASS == 2 ? nchunk > 0 : nchunk > 1;
  if (!mine) len = 0;
  const uint8_t *wbase, *lp = nullptr;
  bool fast = true;
  if constexpr (PLAIN) {
    if (mine) lp = b.ptr[t] + (uint64_t)(c - b.chunk_prefix[t]) * b.chunk;
    wbase = reinterpret_cast<const uint8_t *>(__shfl_sync(0xffffffffu, (unsigned long long)lp, 0));
    const uint32_t t0 = __shfl_sync(0xffffffffu, t, 0);
    fast = __all_sync(0xffffffffu, mine && t == t0 && len == b.chunk && (reinterpret_cast<uintptr_t>(lp) & 15) == 0);
  } else {
    wbase = reinterpret_cast<const uint8_t *>(sc.leaves) + (uint64_t)first * b.chunk;
    lp = wbase + (uint64_t)lane * b.chunk;
  }
  if constexpr (PASS == 0) {
    LowNibble h;
    run_rows(h, buf[warp], lp, len, fast, wbase, b.chunk, lane);
    if (mine) sc.tab[c] = h.table();
  } else if constexpr (PASS == 1) {
    HighNibble h(mine ? sc.lstart[c] : 0);
    run_rows(h, buf[warp], lp, len, fast, wbase, b.chunk, lane);
    if (mine) sc.tab[c] = h.table();
  } else {
    uint32_t l = 0;
    if (mine) l = nchunk > 1 ? sc.lstart[c] : (uint32_t)stream_head<PLAIN>(b, t) & 0xffu;
    Fnv h;
    h.lo = l;
    h.hi = 0;
    run_rows(h, buf[warp], lp, len, fast, wbase, b.chunk, lane);
    if (mine) sc.sum[c] = h.value() - (len == b.chunk ? b.chunk_pow : fnv_pow(kFnvPrime, len)) * l;
  }
}

// Passes 2 and 4 (HIGH): one block per buffer.  Each thread composes the tables of a run of
// chunks, warp 0 walks the threads' tables, and each thread walks its run.  The run's tables
// are loaded eight at a time: loaded one by one by 256 threads, the L2 round trips made this
// pass 21 us (ncu, cold, 8018 chunks) where it now takes 14.
constexpr int kWalkThreads = 1024;
template <bool PLAIN, class Tab, bool HIGH>
__global__ void __launch_bounds__(kWalkThreads) fnv_walk_kernel(const __grid_constant__ Tab b, FnvScratch sc) {
  __shared__ uint32_t f[kWalkThreads];
  __shared__ uint32_t start[kWalkThreads];
  constexpr uint32_t kAhead = 8;
  const uint32_t t = blockIdx.x, i = threadIdx.x;
  const uint32_t c0 = b.chunk_prefix[t], nc = b.chunk_prefix[t + 1] - c0;
  if (nc <= 1) return;
  const uint32_t run = (nc + kWalkThreads - 1) / kWalkThreads;
  const uint32_t a = min(nc, i * run), e = min(nc, a + run);
  const uint32_t *tab = sc.tab + c0;
  uint32_t *ls = sc.lstart + c0;
  uint32_t g = kIdentity;
  for (uint32_t k = a; k < e; k += kAhead) {
    uint32_t v[kAhead];
#pragma unroll
    for (uint32_t j = 0; j < kAhead; ++j) v[j] = k + j < e ? tab[k + j] : kIdentity;
#pragma unroll
    for (uint32_t j = 0; j < kAhead; ++j) g = then(g, v[j]);
  }
  f[i] = g;
  __syncthreads();
  if (i < 32) walk_tables(f, start, (nc + run - 1) / run, (uint32_t)stream_head<PLAIN>(b, t) >> (HIGH ? 4 : 0) & 15u, i);
  __syncthreads();
  if (a >= e) return;
  uint32_t s = start[i];
  for (uint32_t k = a; k < e; k += kAhead) {
    uint32_t v[kAhead], l[kAhead];
#pragma unroll
    for (uint32_t j = 0; j < kAhead; ++j) {
      v[j] = k + j < e ? tab[k + j] : kIdentity;
      l[j] = HIGH && k + j < e ? ls[k + j] : 0;
    }
#pragma unroll
    for (uint32_t j = 0; j < kAhead; ++j) {
      if (k + j < e) ls[k + j] = HIGH ? l[j] | s << 4 : s;
      s = through(v[j], s);
    }
  }
}

// Pass 6: one block per buffer folds h = p^m h + D over its chunks: each thread its run of whole
// chunks by Horner's rule, moved to the end of the whole chunks by a power of p^m; the sum of
// those; then the last chunk.
constexpr int kFoldThreads = 256;
template <bool PLAIN, class Tab>
__global__ void __launch_bounds__(kFoldThreads) fnv_fold_kernel(const __grid_constant__ Tab b, FnvScratch sc) {
  __shared__ uint64_t part[kFoldThreads / 32];
  const uint32_t t = blockIdx.x, i = threadIdx.x;
  const uint32_t c0 = b.chunk_prefix[t], nc = b.chunk_prefix[t + 1] - c0;
  const uint32_t whole = nc ? nc - 1 : 0;
  uint64_t h = 0;
  if (whole) {
    const uint32_t run = (whole + kFoldThreads - 1) / kFoldThreads;
    const uint32_t a = min(whole, i * run), e = min(whole, a + run);
    constexpr uint32_t kAhead = 8;
    for (uint32_t k = a; k < e; k += kAhead) {
      uint64_t v[kAhead];
#pragma unroll
      for (uint32_t j = 0; j < kAhead; ++j) v[j] = k + j < e ? sc.sum[c0 + k + j] : 0;
#pragma unroll
      for (uint32_t j = 0; j < kAhead; ++j)
        if (k + j < e) h = h * b.chunk_pow + v[j];
    }
    if (a < e) h *= fnv_pow(b.chunk_pow, whole - e);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    if ((i & 31) == 0) part[i >> 5] = h;
    __syncthreads();
  }
  if (i != 0) return;
  h = stream_head<PLAIN>(b, t);
  if (whole) {
    h *= fnv_pow(b.chunk_pow, whole);
    for (int w = 0; w < kFoldThreads / 32; ++w) h += part[w];
  }
  if (nc) {
    const uint32_t len = (uint32_t)(stream_bytes<PLAIN>(b, t) - (uint64_t)whole * b.chunk);
    h = h * fnv_pow(kFnvPrime, len) + sc.sum[c0 + whole];
  }
  b.out[t] = h;
}

// All six passes of a buffer of at most kBlockChunks chunks in one block: the stream is copied
// to shared memory once, rows padded by 16 bytes so that the threads' reads of their own rows
// fall in different banks, and each thread runs its chunk three times from there.
constexpr uint32_t kBlockChunks = 256;
constexpr uint32_t kRowPitch = kTreeChunk + 16;

template <class H>
__device__ __forceinline__ void run_row(H &h, const uint8_t *row, uint32_t len) {
  uint32_t k = 0;
  for (; k + 16 <= len; k += 16) h.vec(*reinterpret_cast<const uint4 *>(row + k));
  for (; k < len; ++k) h.byte(row[k]);
}

template <bool PLAIN, class Tab>
__global__ void __launch_bounds__(kBlockChunks) fnv_block_kernel(const __grid_constant__ Tab b, const uint64_t *leaves) {
  extern __shared__ __align__(16) uint8_t rows[];
  __shared__ uint32_t f[kBlockChunks], low[kBlockChunks], high[kBlockChunks];
  __shared__ uint64_t part[kBlockChunks / 32];
  const uint32_t t = blockIdx.x, i = threadIdx.x;
  const uint32_t c0 = b.chunk_prefix[t], nc = b.chunk_prefix[t + 1] - c0;
  const uint64_t head = stream_head<PLAIN>(b, t);
  if (nc == 0) {
    if (i == 0) b.out[t] = head;
    return;
  }
  const uint32_t n = (uint32_t)stream_bytes<PLAIN>(b, t);
  const uint8_t *src = PLAIN ? b.ptr[t] : reinterpret_cast<const uint8_t *>(leaves) + (uint64_t)c0 * kTreeChunk;
  uint32_t k = 0;
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    for (k = i * 16; k + 16 <= n; k += blockDim.x * 16)
      *reinterpret_cast<uint4 *>(rows + k / kTreeChunk * kRowPitch + k % kTreeChunk) =
          *reinterpret_cast<const uint4 *>(src + k);
    k = n & ~15u;
  }
  for (k += i; k < n; k += blockDim.x) rows[k / kTreeChunk * kRowPitch + k % kTreeChunk] = src[k];
  __syncthreads();
  const uint8_t *row = rows + i * kRowPitch;
  const uint32_t len = i < nc ? min(kTreeChunk, n - i * kTreeChunk) : 0;
  uint32_t l = (uint32_t)head & 0xffu;
  if (nc > 1) {
    if (i < nc) {
      LowNibble h;
      run_row(h, row, len);
      f[i] = h.table();
    }
    __syncthreads();
    if (i < 32) walk_tables(f, low, nc, l & 15u, i);
    __syncthreads();
    if (i < nc) {
      HighNibble h(low[i]);
      run_row(h, row, len);
      f[i] = h.table();
    }
    __syncthreads();
    if (i < 32) walk_tables(f, high, nc, l >> 4, i);
    __syncthreads();
    if (i < nc) l = low[i] | high[i] << 4;
  }
  uint64_t sum = 0, last = 0;
  if (i < nc) {
    Fnv h;
    h.lo = l;
    h.hi = 0;
    run_row(h, row, len);
    const bool final_chunk = i == nc - 1;
    sum = h.value() - (len == kTreeChunk ? b.chunk_pow : fnv_pow(kFnvPrime, len)) * l;
    if (final_chunk) {
      last = sum;
      sum = 0;
    } else {
      sum *= fnv_pow(b.chunk_pow, nc - 2 - i);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((i & 31) == 0) part[i >> 5] = sum;
  __syncthreads();
  if (i == nc - 1) {
    uint64_t h = head * fnv_pow(b.chunk_pow, nc - 1);
    for (uint32_t w = 0; w < blockDim.x / 32; ++w) h += part[w];
    b.out[t] = h * fnv_pow(kFnvPrime, len) + last;
  }
}

// The leaves of a call that does not fill the GPU, one warp per leaf: a lane runs 128 bytes three
// times (the passes above, within the warp).  One thread takes 53 us for a leaf, whatever the
// number of leaves up to a few thousand; a warp takes 5 us, at 3.5 times the operations.
constexpr int kSplitWarps = 4;
constexpr uint32_t kSplitChunk = (uint32_t)kLeafBytes / 32;
template <class Tab>
__global__ void __launch_bounds__(kSplitWarps * 32) fnv_leaf_split_kernel(const __grid_constant__ Tab b, uint64_t *leaves) {
  __shared__ __align__(16) uint8_t buf[kSplitWarps][32][kSplitChunk + 16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t(*rows)[kSplitChunk + 16] = buf[warp];
  const uint32_t total = b.leaf_prefix[b.n], step = gridDim.x * kSplitWarps;
  const uint64_t head = Fnv().value(), whole = fnv_pow(kFnvPrime, kSplitChunk);
  for (uint32_t leaf = blockIdx.x * kSplitWarps + warp; leaf < total; leaf += step) {
    const uint32_t t = find_in(b.leaf_prefix, b.n, leaf);
    const uint64_t first = leaf - b.leaf_prefix[t];
    const uint8_t *src = b.ptr[t] + first * kLeafBytes;
    const uint32_t n = (uint32_t)min(kLeafBytes, b.nbytes[t] - first * kLeafBytes);
    __syncwarp();  // every lane is done with the last leaf's rows
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
#pragma unroll
      for (uint32_t j = 0; j < kLeafBytes / 512; ++j) {
        const uint32_t k = j * 512 + lane * 16;
        if (k + 16 <= n)
          *reinterpret_cast<uint4 *>(&rows[k / kSplitChunk][k % kSplitChunk]) =
              __ldg(reinterpret_cast<const uint4 *>(src + k));
        else
          for (uint32_t i = k; i < n; ++i) rows[i / kSplitChunk][i % kSplitChunk] = src[i];
      }
    } else {
      for (uint32_t k = lane; k < n; k += 32) rows[k / kSplitChunk][k % kSplitChunk] = src[k];
    }
    __syncwarp();
    const uint8_t *row = rows[lane];
    const uint32_t at = lane * kSplitChunk, len = at < n ? min(kSplitChunk, n - at) : 0;
    LowNibble lw;
    run_row(lw, row, len);
    const uint32_t low = walk_lanes(lw.table(), (uint32_t)head & 15u, lane);
    HighNibble hg(low);
    run_row(hg, row, len);
    const uint32_t l = low | walk_lanes(hg.table(), (uint32_t)head >> 4 & 15u, lane) << 4;
    Fnv h;
    h.lo = l;
    h.hi = 0;
    run_row(h, row, len);
    uint64_t sum = (h.value() - (len == kSplitChunk ? whole : fnv_pow(kFnvPrime, len)) * l) * fnv_pow(kFnvPrime, n - (at + len));
    if (len == 0) sum = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) leaves[(uint64_t)b.chunk_prefix[t] * kChunkLeaves + first] = head * fnv_pow(kFnvPrime, n) + sum;
  }
}

// One thread per buffer: the literal serial FNV-1a-64, for short buffers and without scratch.
template <class Tab>
__global__ void fnv_plain_kernel(const __grid_constant__ Tab b) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= b.n) return;
  const uint8_t *p = b.ptr[t];
  const uint64_t n = b.nbytes[t];
  Fnv h;
  uint64_t i = 0;
  // bytes up to the first 16-byte boundary, then vectors, then the tail
  while (i < n && ((reinterpret_cast<uintptr_t>(p) + i) & 15) != 0) h.byte(p[i++]);
  const uint4 *v = reinterpret_cast<const uint4 *>(p + i);
  const uint64_t nv = (n - i) >> 4;
  for (uint64_t k = 0; k < nv; ++k) h.vec(v[k]);
  for (i += nv << 4; i < n; ++i) h.byte(p[i]);
  b.out[t] = h.value();
}

}  // namespace

// Chunks a literal digest aims at: enough threads to fill the GPU, few enough that one block
// per buffer composes their tables quickly.
constexpr uint64_t kPlainChunks = 1 << 17;
// A literal digest of buffers up to this length runs one thread per buffer: 6 us of call at 256
// bytes, 10 at 512 and 16 at 1024, where a block takes 12 from 1 to 4 KiB and 17 at 64 KiB.
constexpr uint64_t kSerialBytes = 640;

// Calls of up to this many leaves take a warp per leaf (four buffers, whole calls, against a
// thread per leaf: 16 leaves 18 us against 63, 1024 28 / 71, 4096 42 / 73, 8192 59 / 74, 16384
// 99 / 75).
constexpr uint64_t kSplitLeaves = 8192;

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// Scratch layout of one batch: the tree digest's leaf digests (whole chunks, up to a whole
// warp's), then the per-chunk arrays, each 256-byte aligned.
static FnvScratch fnv_layout(const FnvBatch &b, bool plain, void *base, size_t *bytes) {
  const size_t C = b.chunk_prefix[b.n];
  constexpr int kParts = 4;
  const size_t len[kParts] = {plain ? 0 : ((C + 31) & ~(size_t)31) * kTreeChunk, C * 4, C * 4, C * 8};
  size_t off[kParts];
  size_t o = 0;
  for (int i = 0; i < kParts; ++i) {
    off[i] = o;
    o = align256(o + len[i]);
  }
  if (bytes) *bytes = o;
  FnvScratch sc;
  const uintptr_t p = reinterpret_cast<uintptr_t>(base);
  sc.leaves = reinterpret_cast<uint64_t *>(p + off[0]);
  sc.tab = reinterpret_cast<uint32_t *>(p + off[1]);
  sc.lstart = reinterpret_cast<uint32_t *>(p + off[2]);
  sc.sum = reinterpret_cast<uint64_t *>(p + off[3]);
  return sc;
}

// Chunks of the batch's longest stream.
static uint32_t longest_stream(const FnvBatch &b) {
  uint32_t m = 0;
  for (uint32_t t = 0; t < b.n; ++t) m = std::max(m, b.chunk_prefix[t + 1] - b.chunk_prefix[t]);
  return m;
}
// One block takes a stream of up to kBlockChunks chunks of kTreeChunk bytes: a call of 12 to 17
// us (64 KiB) where six launches take 32.  Longer streams need more than one SM.
static bool in_blocks(const FnvBatch &b, uint32_t longest) { return longest <= kBlockChunks && b.chunk == kTreeChunk; }

size_t fnv_fill_batch(FnvBatch &b, const void *const *ptr, const uint64_t *nbytes, uint64_t *out, size_t n, bool plain,
                      size_t *taken) {
  uint64_t leaves = 0, chunks = 0, bytes = 0;
  size_t k = 0;
  for (; k < n && k < (size_t)kMaxFnv; ++k) {
    const uint64_t l = (nbytes[k] + kLeafBytes - 1) / kLeafBytes;
    if (k && leaves + l > 1ull << 31) break;
    leaves += l;
    bytes += nbytes[k];
  }
  b.n = (uint32_t)k;
  b.out = out;
  b.chunk = kTreeChunk;
  if (plain)  // about kPlainChunks chunks a call, of 256 to 4096 bytes
    while (b.chunk < kLeafBytes && bytes / b.chunk > kPlainChunks) b.chunk *= 2;
  b.chunk_pow = fnv_pow(kFnvPrime, b.chunk);
  leaves = 0;
  for (size_t i = 0; i < k; ++i) {
    const uint64_t l = (nbytes[i] + kLeafBytes - 1) / kLeafBytes;
    b.leaf_prefix[i] = (uint32_t)leaves;
    b.chunk_prefix[i] = (uint32_t)chunks;
    b.ptr[i] = static_cast<const uint8_t *>(ptr[i]);
    b.nbytes[i] = nbytes[i];
    leaves += l;
    chunks += plain ? (nbytes[i] + b.chunk - 1) / b.chunk : (l + kChunkLeaves - 1) / kChunkLeaves;
  }
  b.leaf_prefix[k] = (uint32_t)leaves;
  b.chunk_prefix[k] = (uint32_t)chunks;
  *taken = k;
  size_t need = 0;
  if (!plain || !in_blocks(b, longest_stream(b))) fnv_layout(b, plain, nullptr, &need);
  return need;
}

int fnv_tree_launches(const FnvBatch &b) {
  if (b.n == 0) return 0;
  return (b.chunk_prefix[b.n] ? 1 : 0) + (in_blocks(b, longest_stream(b)) ? 1 : 6);
}

// The serial streams of a batch (passes 1 to 6).
template <bool PLAIN, class Tab>
static cudaError_t run_fnv_streams(const Tab &b, const FnvScratch &sc, bool blocks_do, uint32_t longest, cudaStream_t s) {
  if (blocks_do) {
    const uint32_t threads = std::max(32u, (longest + 31) / 32 * 32);
    const size_t smem = (size_t)longest * kRowPitch;
    const cudaError_t e = cudaFuncSetAttribute(fnv_block_kernel<PLAIN, Tab>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(kBlockChunks * kRowPitch));
    if (e != cudaSuccess) return e;
    fnv_block_kernel<PLAIN, Tab><<<b.n, threads, smem, s>>>(b, sc.leaves);
    return cudaGetLastError();
  }
  const uint32_t blocks = (b.chunk_prefix[b.n] + kChunkWarps * 32 - 1) / (kChunkWarps * 32);
  fnv_chunk_kernel<PLAIN, Tab, 0><<<blocks, kChunkWarps * 32, 0, s>>>(b, sc);
  fnv_walk_kernel<PLAIN, Tab, false><<<b.n, kWalkThreads, 0, s>>>(b, sc);
  fnv_chunk_kernel<PLAIN, Tab, 1><<<blocks, kChunkWarps * 32, 0, s>>>(b, sc);
  fnv_walk_kernel<PLAIN, Tab, true><<<b.n, kWalkThreads, 0, s>>>(b, sc);
  fnv_chunk_kernel<PLAIN, Tab, 2><<<blocks, kChunkWarps * 32, 0, s>>>(b, sc);
  fnv_fold_kernel<PLAIN, Tab><<<b.n, kFoldThreads, 0, s>>>(b, sc);
  return cudaGetLastError();
}

template <class Tab>
static cudaError_t run_fnv_tree(const Tab &b, const FnvScratch &sc, bool blocks_do, uint32_t longest, cudaStream_t s) {
  const uint64_t total = b.leaf_prefix[b.n];
  if (total > 0 && total <= kSplitLeaves) {
    const uint64_t want = (total + kSplitWarps - 1) / kSplitWarps, cap = (uint64_t)num_sms() * 12;
    fnv_leaf_split_kernel<Tab><<<(int)(want < cap ? want : cap), kSplitWarps * 32, 0, s>>>(b, sc.leaves);
  } else if (total > 0) {
    const uint64_t warps = (total + 31) / 32;
    const uint64_t want = (warps + kFnvWarps - 1) / kFnvWarps;
    const uint64_t cap = (uint64_t)num_sms() * 24;
    fnv_leaf_kernel<Tab><<<(int)(want < cap ? want : cap), kFnvWarps * 32, 0, s>>>(b, sc.leaves);
  }
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : run_fnv_streams<false>(b, sc, blocks_do, longest, s);
}

template <class Tab>
static cudaError_t run_fnv_serial(const Tab &b, cudaStream_t s) {
  fnv_plain_kernel<Tab><<<(b.n + 63) / 64, 64, 0, s>>>(b);
  return cudaGetLastError();
}

// The same batch with a table of `Tab`'s size: a call of few buffers passes a small parameter.
template <class Tab>
static Tab shrink(const FnvBatch &b) {
  Tab t;
  t.n = b.n;
  t.chunk = b.chunk;
  t.chunk_pow = b.chunk_pow;
  t.out = b.out;
  memcpy(t.ptr, b.ptr, b.n * sizeof b.ptr[0]);
  memcpy(t.nbytes, b.nbytes, b.n * sizeof b.nbytes[0]);
  memcpy(t.leaf_prefix, b.leaf_prefix, (b.n + 1) * sizeof b.leaf_prefix[0]);
  memcpy(t.chunk_prefix, b.chunk_prefix, (b.n + 1) * sizeof b.chunk_prefix[0]);
  return t;
}

using FnvSmall = FnvTab<32>;

cudaError_t launch_fnv_tree(const FnvBatch &b, void *scratch, cudaStream_t s) {
  if (b.n == 0) return cudaSuccess;
  const FnvScratch sc = fnv_layout(b, false, scratch, nullptr);
  const uint32_t longest = longest_stream(b);
  if (b.n <= (uint32_t)FnvSmall::kMax) return run_fnv_tree(shrink<FnvSmall>(b), sc, in_blocks(b, longest), longest, s);
  return run_fnv_tree(b, sc, in_blocks(b, longest), longest, s);
}

// How a literal digest runs: serially (0), in blocks (1), or with all six passes (2).
static int plain_way(const FnvBatch &b, bool scratch) {
  if (in_blocks(b, longest_stream(b))) {
    for (uint32_t t = 0; t < b.n; ++t)
      if (b.nbytes[t] > kSerialBytes) return 1;
    return 0;
  }
  return scratch ? 2 : 0;
}

int fnv_plain_launches(const FnvBatch &b, bool scratch) { return b.n == 0 ? 0 : plain_way(b, scratch) == 2 ? 6 : 1; }

cudaError_t launch_fnv_plain(const FnvBatch &b, void *scratch, cudaStream_t s) {
  if (b.n == 0) return cudaSuccess;
  const int way = plain_way(b, scratch != nullptr);
  const uint32_t longest = longest_stream(b);
  FnvScratch sc{};
  if (way == 2) sc = fnv_layout(b, true, scratch, nullptr);
  if (b.n <= (uint32_t)FnvSmall::kMax) {
    const FnvSmall t = shrink<FnvSmall>(b);
    return way ? run_fnv_streams<true>(t, sc, way == 1, longest, s) : run_fnv_serial(t, s);
  }
  return way ? run_fnv_streams<true>(b, sc, way == 1, longest, s) : run_fnv_serial(b, s);
}

}  // namespace wt
