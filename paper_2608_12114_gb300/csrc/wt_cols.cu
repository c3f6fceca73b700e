// Multi-column GEMV: Y[t, :] = diag(s) W X[t, :] for t < T <= 16 activation columns, every
// weight read once per pass and reused by all T columns (the paper's multi-column packed-int8
// kernel and its T-sweep, Sec. 4.3 / Sec. 6; speculative batches reuse each weight read).
//
// W streams HBM -> shared memory on an mbarrier ring of 2-D TMA tensor copies: one copy per
// stage brings a tile of 16 rows x vc 16-byte vectors (a box of the matrix seen as
// [M, 2V] 8-byte elements; rows and vectors past the end arrive as zeros).  Per-row 1-D
// copies of 1.5 KB were issue-bound near 3.4 TB/s; one box per 16 rows is not.  The row
// pitch vc * 16 is 64 bytes past a multiple of 128, so the two rows a quarter-warp reads
// fall in different banks.  Eight consumer warps split each tile
// along K and multiply on the tensor cores with warp-level m16n8k16 MMAs (fp32 accumulate):
//
//   A (16 x 16)  16 weight rows, decoded in registers (int8 -> exact f16; bf16/f16 as is)
//   B (16 x 8)   8 activation columns (two MMAs per A for T > 8)
//
// The sum over k does not depend on the order of k, so each thread's four k values of one
// MMA are four consecutive elements of one 16-byte weight vector, and its B values are the
// same four k of X: A and B fragments come straight from whole vector loads, and an int8
// word decodes into exactly the two f16x2 registers a fragment needs.
//
// Four 16-row tiles (two where T > 8 runs two CTAs per SM) form a super block whose X registers
// are loaded once per K chunk.  At the end of a super block the warps' partial tiles meet in
// shared memory and are summed in pairs, in a fixed order (deterministic; rows never depend on
// the partition across CTAs).
//
// Ragged operands (RAG: rows of W or X that are no whole number of 16-byte vectors, or W or X
// off a 16-byte boundary): no tensor map can describe such rows, so each lane of the producer
// warp brings one row's share of a chunk by a 1-D copy, and every weight and X vector is put
// together from the two 16-byte vectors that hold it.  These calls had fp32 FMAs before, one warp
// per row, and the tensor cores truncate what they accumulate.  So the MMAs of each half of a vector
// start from zero and meet in ordinary additions, and these the fp32 sums (bf16, 801 and 2731
// columns, T = 8: FMAs 6.7e-8 and 8.5e-8, whole vectors 7.0e-8 and 8.3e-8, halves 6.8e-8 and 8.1e-8);
// and in kRaggedKept every MMA has a second one that brings back what the first dropped
// (mma16816_kept).  The host's cols_kept takes it where the error against 64 bits would be larger
// than with FMAs.  Eight 16384 x 2731 matrices at T = 8 / 16, with FMAs / in halves / kept: bf16 1924, 4011 /
// 199, 375 / 217, 448 us, int8 1532, 3097 / 145, 321 / 192, 433 us (bf16 T = 8: 3600 GB/s, two CTAs per
// SM, bound by the latencies of putting vectors together; 16 columns kept on one CTA per SM with
// twice the registers 594 and 495 us).
//
// Why warp-level MMAs and not tcgen05: the A operand is decoded from int8 in registers and
// goes to the MMA from there; tcgen05 takes A only from shared or tensor memory, which would
// add a store and a fence per decoded tile, and for T <= 16 the tensor rate is far from the
// bound either way (2 * 16 flops per weight byte at most).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "wt_device.cuh"
#include "wt_kernels.h"

namespace wt {

namespace {

constexpr int kColWarps = 8;  // consumer warps
constexpr int kColConsumers = kColWarps * 32;
constexpr int kColThreads = kColConsumers + 32;  // + one producer warp
constexpr int kColRows = kColTileRows;           // rows of one stage (one MMA tile)
constexpr int kColGroups = (kColVecMax / 4 + kColWarps - 1) / kColWarps;  // 4-vector groups per warp
// a ragged row's chunk sits at its 16-byte phase: the pitch is this many vectors past the chunk
// (a multiple of 8: still 64 bytes past a multiple of 128)
constexpr uint32_t kColRagPad = 8;
static_assert(kColRagPad == kColVecMax - kColVecMaxRagged, "a padded chunk fills a stage row");
constexpr uint32_t kColStageBytes = kColRows * kColVecMax * 16;
static_assert(kColVecMax % 8 == 4, "row pitch 64 bytes past a multiple of 128");
static_assert(kColStageBytes % 128 == 0, "stages stay 128-byte aligned for the tensor copies");

// Where a partial sum of (column, row) sits among its tile's: a pair of columns takes 32 floats,
// turned by 8 per pair, so that neither the stores of a fragment (rows g of the columns 2t; in
// plain order the four shared a bank) nor the sums over a pair meet in a bank.
__device__ __forceinline__ uint32_t red_at(uint32_t col, uint32_t row) {
  return (col >> 1) * 32 + ((((col & 1) << 4) + row + 8 * (col >> 1)) & 31);
}

// Per-launch geometry: NT = 8-column MMA tiles (T <= 8: 1, else 2).  int8 weights and
// ragged operands run two CTAs per SM with half the ring each (the same bytes in flight per SM,
// twice the warps; those paths are latency-bound on decoding and on shifting).  The cross-warp
// partials of one 16-row tile take 16 x 8 NT floats per warp, in two alternating halves.
// So do, in kAlignedTwo, 2-byte weights with 16 columns in launches that are mostly of few short chunks
// (the host's cols_two_ctas): there the waits for X and for the other warps' partials are a large
// part of a super block, and the second CTA fills them (T = 16, bf16, 1 GiB of 16384-row matrices, us
// with one / two: K = 768 259 / 207, 1024 210 / 188, 1536 196 / 177; but 2048 173 / 177, 8192 165 /
// 168).  The sums are the same in either.
enum ColMode : int { kAligned = 0, kAlignedTwo = 1, kRagged = 2, kRaggedKept = 3 };
template <int DT, int NT, int MODE = kAligned>
struct ColGeo {
  static constexpr bool RAG = MODE >= kRagged, KEEP = MODE == kRaggedKept;
  static constexpr int kCtasPerSm = DT == 3 || MODE != kAligned ? 2 : 1;
  static constexpr int kStages = kCtasPerSm == 2 ? 3 : 6;
  // 16-row tiles per super block (X registers are loaded once per super block and chunk):
  // four, or two for int8 with 16 columns, which then fits two CTAs per SM (registers and
  // partial buffers halve; X is reloaded every 32 rows instead of 64)
  static constexpr int kBlocks = kCtasPerSm == 2 && NT == 2 ? 2 : 4;
  // accumulator sets per tile (even / odd k16 steps: shorter MMA chains; ragged operands: even /
  // odd vectors, or the sums and what they lost); int8 and ragged f16 with 16 columns have one,
  // their two column tiles already give two independent chains per A (ragged bf16 needs the second
  // for precision, at 10 % more time)
  static constexpr int kAcc = NT == 2 && !KEEP && (DT == 3 || (RAG && DT == 2)) ? 1 : 2;
  static constexpr int kSuper = kColRows * kBlocks;
  static constexpr uint32_t kRedStride = 128 * NT;  // floats per (tile, warp)
  static constexpr size_t kRedFloats = (size_t)kBlocks * kColWarps * kRedStride;  // one half
  static constexpr size_t kRedOff = (size_t)kStages * kColStageBytes;
  static constexpr size_t kBarOff = kRedOff + 2 * kRedFloats * sizeof(float);
  static constexpr size_t kFlagOff = kBarOff + 2 * kStages * sizeof(uint64_t);
  static constexpr size_t kSmem = kFlagOff + 16;
};
static_assert(ColGeo<1, 2>::kSmem <= 232448 && 2 * (ColGeo<3, 1>::kSmem + 1024) <= 233472 &&
                  2 * (ColGeo<3, 2>::kSmem + 1024) <= 233472 && 2 * (ColGeo<1, 1, kRagged>::kSmem + 1024) <= 233472 &&
                  2 * (ColGeo<1, 2, kRagged>::kSmem + 1024) <= 233472 && 2 * (ColGeo<1, 2, kAlignedTwo>::kSmem + 1024) <= 233472,
              "multi-column shared memory");

// 32-bit words of X per weight vector: 16 fp16 activations for an int8 vector, else 8.
template <int DT>
struct ColX {
  static constexpr int W = DT == 3 ? 8 : 4;
};

template <int DT>
__device__ __forceinline__ float col_scale(const uint8_t *s, uint64_t row) {
  if constexpr (DT == 3) return __half2float(reinterpret_cast<const __half *>(s)[row]);
  return 1.f;
}

// The activations of weight vector `vec` (global vector index col * V + v) of one column.
template <int DT>
__device__ __forceinline__ void load_xvec(const uint8_t *X, uint64_t vec, bool ok, uint32_t (&xr)[ColX<DT>::W]) {
  const uint4 *p = reinterpret_cast<const uint4 *>(X) + (DT == 3 ? 2 * vec : vec);
  const uint4 a = ok ? __ldg(p) : make_uint4(0, 0, 0, 0);
  xr[0] = a.x;
  xr[1] = a.y;
  xr[2] = a.z;
  xr[3] = a.w;
  if constexpr (DT == 3) {
    const uint4 b = ok ? __ldg(p + 1) : make_uint4(0, 0, 0, 0);
    xr[4] = b.x;
    xr[5] = b.y;
    xr[6] = b.z;
    xr[7] = b.w;
  }
}

// Bytes [o, o + 16) of X, which has `total` bytes at any address, those from `end` on zero.
__device__ __forceinline__ uint4 ldg_shifted(const uint8_t *X, uint64_t o, uint64_t end, uint64_t total) {
  if (o >= end) return make_uint4(0, 0, 0, 0);
  const uint64_t a = reinterpret_cast<uint64_t>(X) + o, x0 = reinterpret_cast<uint64_t>(X);
  const uint32_t ph = (uint32_t)a & 15u;
  uint4 r;
  if (a - ph >= x0 && a - ph + (ph ? 32 : 16) <= x0 + total) {
    const uint4 *p = reinterpret_cast<const uint4 *>(a - ph);
    const uint4 lo = __ldg(p), hi = ph ? __ldg(p + 1) : lo;
    r = shift_bytes(lo, hi, ph);
  } else {  // the first or last vector of X
    uint64_t lo = 0, hi = 0;
#pragma unroll 1
    for (int i = 15; i >= 0; --i) {
      hi = (hi << 8) | (lo >> 56);
      lo = (lo << 8) | (o + i < total ? __ldg(X + o + i) : 0);
    }
    r = make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
  }
  return o + 16 <= end ? r : and4(r, byte_mask(0, (int)(end - o)));
}

// load_xvec for ragged operands: weight vector v (of the whole row) of column `col`.
template <int DT>
__device__ __forceinline__ void load_xvec_ragged(const MatDesc &md, uint32_t col, uint32_t v, bool ok,
                                                 uint32_t (&xr)[ColX<DT>::W]) {
  constexpr uint32_t kXB = DT == 3 ? 32 : 16;  // X bytes of a weight vector
  const uint64_t xp = (uint64_t)md.rb * (kXB / 16);
  const uint64_t o = col * xp + (uint64_t)v * kXB, end = (col + 1) * xp, total = md.G * xp;
#pragma unroll
  for (uint32_t k = 0; k < kXB / 16; ++k) {
    const uint4 a = ldg_shifted(md.x, o + 16 * k, ok ? end : 0, total);
    xr[4 * k] = a.x, xr[4 * k + 1] = a.y, xr[4 * k + 2] = a.z, xr[4 * k + 3] = a.w;
  }
}

// 2-D tensor copy of one box into this CTA's shared memory, completion counted on `bar`.
// x (in 8-byte elements) is always a multiple of 2: 16-byte aligned.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *tmap, int32_t x, int32_t y, uint32_t bar,
                                            uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(tmap), "r"(x), "r"(y), "r"(bar), "l"(pol)
      : "memory");
}

// One stage: rows g and g + 8 of the tile against this warp's vectors of the chunk.
// Thread (g, t) takes vector (q * warps + warp) * 4 + t of group q.
// The box holds vc vectors per row at pitch vc * 16, nv of them the row's; rows and vectors past
// the matrix are zeros, so only whole groups past nv are skipped (at K = 1024 the 17th group of
// a chunk is padding, and was warp 0's third).
// RAG: row g starts ph0 bytes past its pitch's start, row g + 8 ph1 bytes; of vector v only the
// row's own bytes count (left: those from the chunk's start on; an int8 neighbour meets a zero
// of X and is a finite number, so only the 2-byte types mask it).
template <int DT, int NT, int H, int MODE>
__device__ __forceinline__ void cols_stage(uint32_t tile, uint32_t vc, uint32_t nv, int warp, uint32_t g, uint32_t t,
                                           const uint32_t (&xr)[kColGroups][NT][ColX<DT>::W], float (&acc)[H][NT][4],
                                           uint32_t ph0, uint32_t ph1, uint32_t left) {
  constexpr bool RAG = MODE >= kRagged, KEEP = MODE == kRaggedKept;
  const uint32_t pitch = RAG ? (vc + kColRagPad) * 16 : vc * 16;
#pragma unroll
  for (int q = 0; q < kColGroups; ++q) {
    const uint32_t v0 = (uint32_t)(q * kColWarps + warp) * 4;
    if (v0 >= nv) continue;  // warp-uniform: the row ends before this group
    const uint32_t v = v0 + t;
    uint4 w0, w1;
    if constexpr (RAG) {
      w0 = lds_shifted(tile + g * pitch + ph0 + v * 16);
      w1 = lds_shifted(tile + (g + 8) * pitch + ph1 + v * 16);
      if (DT != 3 && left < vc * 16) {  // uniform: the row's last chunk
        const uint4 m = byte_mask(0, (int)left - (int)(v * 16));
        w0 = and4(w0, m);
        w1 = and4(w1, m);
      }
    } else {
      w0 = lds128(tile + g * pitch + v * 16);
      w1 = lds128(tile + (g + 8) * pitch + v * 16);
    }
    const uint32_t ra[4] = {w0.x, w0.y, w0.z, w0.w};
    const uint32_t rb[4] = {w1.x, w1.y, w1.z, w1.w};
    float part[2][NT][4];  // kRagged: the products of the vector's two halves
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int n = 0; n < NT; ++n) part[h][n][0] = part[h][n][1] = part[h][n][2] = part[h][n][3] = 0.f;
    if constexpr (DT == 3) {
      // word j = weights k 4j..4j+3 of the vector; its activations are x words 2j, 2j+1
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t u0 = ra[j] ^ 0x80808080u, u1 = rb[j] ^ 0x80808080u;
        const uint32_t a0 = i8x2_to_f16x2(u0, 0x4140u), a2 = i8x2_to_f16x2(u0, 0x4342u);
        const uint32_t a1 = i8x2_to_f16x2(u1, 0x4140u), a3 = i8x2_to_f16x2(u1, 0x4342u);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if constexpr (KEEP)
            mma16816_kept<2>(acc[0][n], acc[1][n], a0, a1, a2, a3, xr[q][n][2 * j], xr[q][n][2 * j + 1]);
          else
            mma16816<2>(RAG ? part[j / 2][n] : acc[(j & 1) % H][n], a0, a1, a2, a3, xr[q][n][2 * j], xr[q][n][2 * j + 1]);
        }
      }
    } else {
      // words 2s, 2s+1 = elements 4s..4s+3 of the vector
#pragma unroll
      for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if constexpr (KEEP)
            mma16816_kept<DT>(acc[0][n], acc[1][n], ra[2 * s], rb[2 * s], ra[2 * s + 1], rb[2 * s + 1], xr[q][n][2 * s],
                              xr[q][n][2 * s + 1]);
          else
            mma16816<DT>(RAG ? part[s][n] : acc[s % H][n], ra[2 * s], rb[2 * s], ra[2 * s + 1], rb[2 * s + 1],
                         xr[q][n][2 * s], xr[q][n][2 * s + 1]);
        }
      }
    }
    if constexpr (RAG && !KEEP) {
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[q % H][n][i] += part[0][n][i] + part[1][n][i];
    }
  }
}

struct Ring {
  uint32_t stage0, full0, empty0;
  volatile int *abort_flag;
  int *status;
};

// Consumer side of one piece (rows [r0, r1) of one matrix), NT = 8-column MMA tiles.
template <int DT, int NT, int MODE>
__device__ __forceinline__ void cols_piece(const MatDesc &md, const Piece &pc, const Ring &R, float *red_base,
                                           uint32_t &it, uint32_t &par, int warp, int lane) {
  const uint32_t V = md.V, vc = md.vc, T = md.G;
  // vectors from one column of X to the next: the whole row of a column segment; int8 has no
  // segments (96 registers: the second length cost its T = 16 kernel 12 %)
  const uint32_t xpitch = DT == 3 ? V : md.rs;
  const uint32_t nchunk = (V + vc - 1) / vc;
  const uint32_t g = lane >> 2, t = lane & 3;
  const int ct = threadIdx.x;
  constexpr bool RAG = ColGeo<DT, NT, MODE>::RAG, KEEP = ColGeo<DT, NT, MODE>::KEEP;
  constexpr int kColBlocks = ColGeo<DT, NT, MODE>::kBlocks;
  constexpr int kColSuper = ColGeo<DT, NT, MODE>::kSuper;
  for (uint32_t sb = pc.r0; sb < pc.r1; sb += kColSuper) {
    const uint32_t rows = min((uint32_t)kColSuper, pc.r1 - sb);
    const uint32_t nrb = (rows + kColRows - 1) / kColRows;
    constexpr int H = ColGeo<DT, NT, MODE>::kAcc;
    float acc[kColBlocks][H][NT][4];
#pragma unroll
    for (int b = 0; b < kColBlocks; ++b)
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int n = 0; n < NT; ++n) acc[b][h][n][0] = acc[b][h][n][1] = acc[b][h][n][2] = acc[b][h][n][3] = 0.f;
    for (uint32_t c = 0; c < nchunk; ++c) {
      const uint32_t nv = min(vc, V - c * vc);
      uint32_t xr[kColGroups][NT][ColX<DT>::W];
#pragma unroll
      for (int q = 0; q < kColGroups; ++q) {
        const uint32_t v = (uint32_t)(q * kColWarps + warp) * 4 + t;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint32_t col = g + 8 * n;
          if constexpr (RAG) load_xvec_ragged<DT>(md, col, c * vc + v, v < nv && col < T, xr[q][n]);
          else load_xvec<DT>(md.x, (uint64_t)col * xpitch + (uint64_t)c * vc + v, v < nv && col < T, xr[q][n]);
        }
      }
#pragma unroll
      for (int b = 0; b < kColBlocks; ++b) {
        if ((uint32_t)b < nrb) {
          const uint32_t s = it % ColGeo<DT, NT, MODE>::kStages;
          bounded_wait(R.full0 + 8 * s, (it / ColGeo<DT, NT, MODE>::kStages) & 1, R.abort_flag, R.status);
          const uint64_t row = reinterpret_cast<uint64_t>(md.W) + (uint64_t)(sb + b * kColRows + g) * md.rb;
          cols_stage<DT, NT, H, MODE>(R.stage0 + s * kColStageBytes, vc, nv, warp, g, t, xr, acc[b], (uint32_t)row & 15u,
                                     (uint32_t)(row + 8ull * md.rb) & 15u, md.rb - c * vc * 16);
          __syncwarp();
          if (lane == 0) mbar_arrive(R.empty0 + 8 * s);
          ++it;
        }
      }
    }
    // warp partials -> red[b][warp][col][row]; C fragment: (g, 2t), (g, 2t+1), (g+8, 2t), (g+8, 2t+1).
    // Two halves alternate, so one barrier per super block suffices: a half is rewritten
    // only after every thread has passed the next super block's barrier.
    constexpr uint32_t kStride = ColGeo<DT, NT, MODE>::kRedStride;
    float *red = red_base + par * ColGeo<DT, NT, MODE>::kRedFloats;
    par ^= 1;
#pragma unroll
    for (int b = 0; b < kColBlocks; ++b) {
      if ((uint32_t)b < nrb) {
        float *r = red + (b * kColWarps + warp) * kStride;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint32_t c0 = 2 * t + 8 * n;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float a0 = acc[b][0][n][i], a1 = H == 2 ? acc[b][H - 1][n][i] : 0.f;
            r[red_at(c0 + (i & 1), g + 8 * (i >> 1))] = KEEP ? kept_sum(a0, a1) : a0 + a1;
          }
        }
      }
    }
    named_bar(1, kColConsumers);
    for (uint32_t o = ct; o < nrb * kStride; o += kColConsumers) {
      const uint32_t b = o / kStride, e = o % kStride, col = e >> 4, row = b * kColRows + (e & 15);
      if (col < T && row < rows) {
        const float *r = red + b * kColWarps * kStride + red_at(col, e & 15);
        float p[kColWarps];
#pragma unroll
        for (int w = 0; w < kColWarps; ++w) p[w] = r[w * kStride];
#pragma unroll
        for (int h = kColWarps / 2; h > 0; h /= 2)  // in pairs: three roundings, not seven
#pragma unroll
          for (int w = 0; w < h; ++w) p[w] += p[w + h];
        md.y[(uint64_t)col * md.M + sb + row] = p[0] * col_scale<DT>(md.s, sb + row);
      }
    }
  }
}

template <int DT, int NT, int MODE>
__global__ void __launch_bounds__(kColThreads, (ColGeo<DT, NT, MODE>::kCtasPerSm))
    gemm_cols_kernel(const MatDesc *__restrict__ mats, const Piece *__restrict__ pieces,
                     const uint32_t *__restrict__ begin, int *status, const uint8_t *__restrict__ maps) {
  using Geo = ColGeo<DT, NT, MODE>;
  constexpr bool RAG = Geo::RAG;
  constexpr int kColStages = Geo::kStages;
  extern __shared__ __align__(128) uint8_t smem[];
  Ring R;
  R.stage0 = smem_u32(smem);
  R.full0 = smem_u32(smem + Geo::kBarOff);
  R.empty0 = R.full0 + kColStages * 8;
  R.abort_flag = reinterpret_cast<volatile int *>(smem + Geo::kFlagOff);
  R.status = status;
  float *red = reinterpret_cast<float *>(smem + Geo::kRedOff);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t p0 = begin[blockIdx.x];
  const uint32_t p1 = begin[blockIdx.x + 1];

  if (threadIdx.x == 0) {
    for (int s = 0; s < kColStages; ++s) {
      mbar_init(R.full0 + 8 * s, 1);
      mbar_init(R.empty0 + 8 * s, kColWarps);
    }
    *R.abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();

  if (warp == kColWarps) {
    // ---------------- producer: one thread issues every tensor copy of the CTA (ragged rows:
    // sixteen threads a row's copy each)
    if (RAG || lane == 0) {
      const uint64_t pol = l2_evict_first_policy();
      uint32_t it = 0;
      bool live = true;
      for (uint32_t pi = p0; pi < p1 && live; ++pi) {
        const Piece pc = pieces[pi];
        const MatDesc md = mats[pc.mat];
        const uint8_t *tmap = maps + (size_t)pc.mat * kTensorMapBytes;
        const uint32_t nchunk = (md.V + md.vc - 1) / md.vc;
        for (uint32_t sb = pc.r0; sb < pc.r1 && live; sb += Geo::kSuper) {
          const uint32_t rows = min((uint32_t)Geo::kSuper, pc.r1 - sb);
          const uint32_t nrb = (rows + kColRows - 1) / kColRows;
          for (uint32_t c = 0; c < nchunk && live; ++c) {
            for (uint32_t b = 0; b < nrb; ++b) {
              const uint32_t s = it % kColStages;
              if (it >= kColStages &&
                  !bounded_wait(R.empty0 + 8 * s, ((it / kColStages) - 1) & 1, R.abort_flag, status))
                live = false;
              if (RAG) live = __all_sync(0xffffffffu, live);
              if (!live) break;
              const uint32_t bar = R.full0 + 8 * s;
              if constexpr (RAG) {
                const uint32_t row0 = sb + b * kColRows;
                ragged_rows(md, row0, min((uint32_t)kColRows, pc.r1 - row0), c * md.vc * 16,
                            min(md.vc * 16, md.rb - c * md.vc * 16), R.stage0 + s * kColStageBytes,
                            (md.vc + kColRagPad) * 16, bar, pol, lane);
                ++it;
                continue;
              }
              mbar_expect_tx(bar, kColRows * md.vc * 16);  // the whole box, zero fill included
              tma_load_2d(R.stage0 + s * kColStageBytes, tmap, (int32_t)(2 * c * md.vc),
                          (int32_t)(sb + b * kColRows), bar, pol);
              ++it;
            }
          }
        }
      }
      if ((!live || *R.abort_flag) && lane == 0) {
        // drain: the copies of the last (up to kColStages) issued stages may still be in flight
        const uint32_t first = it > (uint32_t)kColStages ? it - kColStages : 0;
        for (uint32_t j = first; j < it; ++j) {
          const long long t0 = clock64();
          while (!mbar_try_wait(R.full0 + 8 * (j % kColStages), (j / kColStages) & 1) &&
                 clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------- consumers: 8 warps (every matrix of the launch has T <= 8 NT)
    uint32_t it = 0, par = 0;
    for (uint32_t pi = p0; pi < p1; ++pi) {
      const Piece pc = pieces[pi];
      const MatDesc md = mats[pc.mat];
      cols_piece<DT, NT, MODE>(md, pc, R, red, it, par, warp, lane);
    }
  }
  __syncthreads();
}

}  // namespace

int gemm_cols_ctas_per_sm(int dtype, bool ragged, bool two) { return dtype == 3 || ragged || two ? 2 : 1; }

template <int DT, int NT, int MODE>
static cudaError_t cols_attr() {
  return cudaFuncSetAttribute(gemm_cols_kernel<DT, NT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)ColGeo<DT, NT, MODE>::kSmem);
}

// The modes that some types do without: f16 never keeps (the host's cols_kept).
template <int DT>
constexpr int kKept = DT == 2 ? kRagged : kRaggedKept;
template <int DT, int NT>
constexpr int kTwo = DT != 3 && NT == 2 ? kAlignedTwo : kAligned;

// Every variant of one dtype.
template <int DT>
static cudaError_t cols_attrs() {
  cudaError_t e;
  if ((e = cols_attr<DT, 1, kAligned>()) != cudaSuccess || (e = cols_attr<DT, 2, kAligned>()) != cudaSuccess ||
      (e = cols_attr<DT, 1, kRagged>()) != cudaSuccess || (e = cols_attr<DT, 2, kRagged>()) != cudaSuccess ||
      (e = cols_attr<DT, 1, kKept<DT>>()) != cudaSuccess || (e = cols_attr<DT, 2, kKept<DT>>()) != cudaSuccess)
    return e;
  return cols_attr<DT, 2, kTwo<DT, 2>>();
}

cudaError_t gemm_cols_prepare() {
  cudaError_t e;
  if ((e = cols_attrs<1>()) != cudaSuccess || (e = cols_attrs<2>()) != cudaSuccess) return e;
  return cols_attrs<3>();
}

template <int DT, int NT, int MODE>
static void cols_go(const GemvLaunch &L, cudaStream_t s) {
  gemm_cols_kernel<DT, NT, MODE>
      <<<L.grid, kColThreads, ColGeo<DT, NT, MODE>::kSmem, s>>>(L.mats, L.pieces, L.begin, L.status, L.maps);
}

template <int DT, int NT>
static void cols_launch(const GemvLaunch &L, cudaStream_t s) {
  if (L.ragged && L.keep) cols_go<DT, NT, kKept<DT>>(L, s);
  else if (L.ragged) cols_go<DT, NT, kRagged>(L, s);
  else if (L.two) cols_go<DT, NT, kTwo<DT, NT>>(L, s);
  else cols_go<DT, NT, kAligned>(L, s);
}

cudaError_t launch_gemm_cols(const GemvLaunch &L, cudaStream_t s) {
  if ((L.maps == nullptr && !L.ragged) || (L.nt != 1 && L.nt != 2)) return cudaErrorInvalidValue;
  switch (L.dtype * 4 + L.nt) {
    case 1 * 4 + 1: cols_launch<1, 1>(L, s); break;
    case 1 * 4 + 2: cols_launch<1, 2>(L, s); break;
    case 2 * 4 + 1: cols_launch<2, 1>(L, s); break;
    case 2 * 4 + 2: cols_launch<2, 2>(L, s); break;
    case 3 * 4 + 1: cols_launch<3, 1>(L, s); break;
    case 3 * 4 + 2: cols_launch<3, 2>(L, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace wt
