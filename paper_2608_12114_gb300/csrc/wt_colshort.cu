// Multi-column GEMV Y[t] = diag(s) W X[t], t < T <= 16, for short rows (at most short_row_bytes),
// and the one-column GEMV of int8 weights with such rows.
//
// The kernels for longer rows bring a box of 16 or 128 rows by a fixed share of K per stage; of
// rows shorter than the box little of a stage is left (1 KB of 24 KB at K = 32), and the wait
// for the next stage sets the pace: the many-small set (1253 matrices of 32 to 2048 columns,
// 1.6 GB) took 3607 us at T = 8, bf16.  Here a stage is filled with whole rows, in one 1-D copy,
// and X [T, K] of the matrix is laid out in shared memory once per piece:
//
//   producer warp   per stage one bulk copy of as many rows as fit 32 KB; ragged rows (no whole
//                   number of 16-byte vectors, or W off a 16-byte boundary) arrive the same way
//   8 MMA warps     take 32-row groups of the stages in turn, each over all of K: thread (g, t)
//                   reads vector 4q + t of rows g, g + 8, g + 16, g + 24 and of columns g, g + 8
//                   of X, and multiplies them with m16n8k16 MMAs whose four k per thread are
//                   four consecutive elements of its vectors (wt_cols.cu has the argument)
//
// The tensor cores truncate what they accumulate.  Whole vectors: every MMA starts from zero, the
// two (int8: four) of 64 bytes meet in ordinary additions, and these the row's fp32 sums, one of the
// even and one of the odd 64 bytes (error against 64 bits at T = 8, here / on the kernel that had
// these rows before: 32 columns bf16 3.7e-8 / 3.7e-8, f16 5.5e-8 / 5.5e-8, int8 4.1e-8 / 4.2e-8; 512
// columns 7.0e-8 / 7.3e-8, 8.3e-8 / 9.3e-8, 6.8e-8 / 7.5e-8).  Ragged rows, which had fp32 FMAs
// before, keep what the truncation drops (mma16816_kept; 33 columns 2.8e-8 / 3.2e-8, 3.8e-8 / 5.6e-8,
// 3.5e-8 / 3.8e-8; 333 columns 3.0e-8 / 5.8e-8, 3.8e-8 / 8.0e-8, 3.8e-8 / 6.2e-8), at 3 to 14 % more
// time for T <= 8 and 14 to 45 % for T = 16.  A row's result depends on its matrix alone.  HBM
// bounds the kernel where rows have 256 bytes and more; below that, the loads of shared memory and
// the stores of Y.
#include <cuda_fp16.h>

#include "wt_device.cuh"
#include "wt_kernels.h"

namespace wt {

namespace {

constexpr int kSWarps = 8;
constexpr int kSConsumers = kSWarps * 32;
constexpr int kSThreads = kSConsumers + 32;  // + one producer warp
constexpr int kSStages = 5;
constexpr uint32_t kSTiles = 2;                  // 16-row MMA tiles of a group (share the X loads)
constexpr uint32_t kSGroup = 16 * kSTiles;
// a column of X: its elements (int8 weights: two bytes for each of W's), 64 bytes past a
// multiple of 128 (int8: 16), so that the columns g and g + 1 a quarter-warp reads lie in
// different banks
__host__ __device__ constexpr uint32_t short_xpitch(int dt, uint32_t nq) {
  const uint32_t n = nq * (dt == 3 ? 128 : 64);
  return (n + 127) / 128 * 128 + (dt == 3 ? 16 : 64);
}
constexpr size_t kSXOff = (size_t)kSStages * kStageBytes;
constexpr size_t kSXBytes = 16 * (size_t)short_xpitch(1, short_row_bytes(1) / 64);
constexpr size_t kSBarOff = kSXOff + kSXBytes;
constexpr size_t kSFlagOff = kSBarOff + 2 * kSStages * sizeof(uint64_t);
constexpr size_t kSSmem = kSFlagOff + 16;
static_assert(kSSmem <= 232448 && kSBarOff % 8 == 0, "short-row shared memory");
static_assert(16 * (size_t)short_xpitch(3, short_row_bytes(3) / 64) <= kSXBytes, "X of int8 weights");

// X of the matrix to shared memory: 8 NT columns of nq 64-byte (int8: 128-byte) groups, zeros
// past column T and past a column's end; all consumers.
template <int DT, int NT>
__device__ __forceinline__ void stage_cols(uint32_t xs, const MatDesc &md, uint32_t row_bytes, uint32_t nq, int ct) {
  const uint32_t xb = DT == 3 ? 2 * row_bytes : row_bytes;  // bytes of a column
  const uint32_t vecs = nq * (DT == 3 ? 8 : 4), pitch = short_xpitch(DT, nq);
  for (uint32_t i = ct; i < vecs * 8 * NT; i += kSConsumers) {
    const uint32_t col = i / vecs, o = i % vecs * 16;
    const uint8_t *p = md.x + (uint64_t)col * xb + o;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (col < md.G && o < xb) {
      if (o + 16 <= xb && (reinterpret_cast<uint64_t>(p) & 15) == 0) {
        v = __ldg(reinterpret_cast<const uint4 *>(p));
      } else {
        uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
        for (uint32_t b = 0; b < 16; ++b)
          if (o + b < xb) w[b / 4] |= (uint32_t)__ldg(p + b) << (8 * (b % 4));
        v = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(xs + col * pitch + o), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w)
                 : "memory");
  }
}

// Step j of a vector's MMAs: to p, each from zero and added in fp32, or with KEEP to the row's
// sums s, and what they lost to m.
template <int DT, bool KEEP>
__device__ __forceinline__ void mma_step(float (&s)[4], float (&m)[4], float (&p)[4], int j, uint32_t a0, uint32_t a1,
                                         uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  if constexpr (KEEP) {
    mma16816_kept<DT>(s, m, a0, a1, a2, a3, b0, b1);
  } else {
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    if (j == 0) {
      mma16816<DT>(p, a0, a1, a2, a3, b0, b1);
    } else {
      mma16816<DT>(z, a0, a1, a2, a3, b0, b1);
      add_x2(p[0], p[1], z[0], z[1]);
      add_x2(p[2], p[3], z[2], z[3]);
    }
  }
}

template <int DT, int NT, bool RAG>
__global__ void __launch_bounds__(kSThreads, 1)
    gemm_short_kernel(const MatDesc *__restrict__ mats, const Piece *__restrict__ pieces,
                      const uint32_t *__restrict__ begin, int *status) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t stage0 = smem_u32(smem), xs = stage0 + (uint32_t)kSXOff;
  const uint32_t full0 = stage0 + (uint32_t)kSBarOff, empty0 = full0 + kSStages * 8;
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kSFlagOff);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t p0 = begin[blockIdx.x], p1 = begin[blockIdx.x + 1];

  if (threadIdx.x == 0) {
    for (int s = 0; s < kSStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, kSWarps);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();

  if (warp == kSWarps) {
    // ---------------- producer
    if (RAG || lane == 0) {
      const uint64_t pol = l2_evict_first_policy();
      uint32_t it = 0;
      bool live = true;
      for (uint32_t pi = p0; pi < p1 && live; ++pi) {
        const Piece pc = pieces[pi];
        const MatDesc md = mats[pc.mat];
        for (uint32_t r = pc.r0; r < pc.r1; r += md.rt) {
          const uint32_t nr = min(md.rt, pc.r1 - r);
          const uint32_t s = it % kSStages;
          if (it >= kSStages && !bounded_wait(empty0 + 8 * s, ((it / kSStages) - 1) & 1, abort_flag, status)) live = false;
          if (RAG) live = __all_sync(0xffffffffu, live);
          if (!live) break;
          const uint32_t dst = stage0 + s * kStageBytes, bar = full0 + 8 * s;
          if constexpr (RAG) {
            ragged_rows(md, r, 1, 0, nr * md.rb, dst, 0, bar, pol, lane);
          } else {
            mbar_expect_tx(bar, nr * md.V * 16);
            bulk_g2s(dst, md.W + (uint64_t)r * md.V * 16, nr * md.V * 16, bar, pol);
          }
          ++it;
        }
      }
      if (lane == 0 && (!live || *abort_flag)) {
        // drain: the copies of the last (up to kSStages) issued stages may still be in flight
        const uint32_t first = it > (uint32_t)kSStages ? it - kSStages : 0;
        for (uint32_t j = first; j < it; ++j) {
          const long long t0 = clock64();
          while (!mbar_try_wait(full0 + 8 * (j % kSStages), (j / kSStages) & 1) && clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------- MMA warps
    const int ct = threadIdx.x;
    const uint32_t g = lane >> 2, t = lane & 3;
    uint32_t it = 0, turn = 0;  // stages; groups of all stages so far (mod 8)
    for (uint32_t pi = p0; pi < p1; ++pi) {
      const Piece pc = pieces[pi];
      const MatDesc md = mats[pc.mat];
      const uint32_t rowb = RAG ? md.rb : md.V * 16;
      const uint32_t nq = (md.V + 3) / 4, xpitch = short_xpitch(DT, nq);
      named_bar(1, kSConsumers);  // every warp has done with the last matrix's X
      stage_cols<DT, NT>(xs, md, rowb, nq, ct);
      named_bar(1, kSConsumers);
      const uint32_t xl = xs + g * xpitch + t * (DT == 3 ? 32 : 16);
      // of the last 64 bytes' vectors: the bytes that are the row's
      const uint4 tail = byte_mask(0, (int)rowb - (int)(16 * (4 * (nq - 1) + t)));
      const bool whole = rowb % 64 == 0;
      for (uint32_t r = pc.r0; r < pc.r1; r += md.rt) {
        const uint32_t nr = min(md.rt, pc.r1 - r);
        const uint32_t s = it % kSStages;
        bounded_wait(full0 + 8 * s, (it / kSStages) & 1, abort_flag, status);
        const uint32_t tile =
            stage0 + s * kStageBytes + (RAG ? (uint32_t)(reinterpret_cast<uint64_t>(md.W) + (uint64_t)r * rowb) & 15u : 0);
        const uint32_t ng = (nr + kSGroup - 1) / kSGroup;
        for (uint32_t gi = (warp - turn) & (kSWarps - 1); gi < ng; gi += kSWarps) {
          const uint32_t q0 = gi * kSGroup;
          uint32_t a[2 * kSTiles];  // this thread's rows; those past the tile read row 0
#pragma unroll
          for (uint32_t k = 0; k < 2 * kSTiles; ++k) {
            const uint32_t row = q0 + 8 * k + g;
            a[k] = tile + (row < nr ? row : 0) * rowb + t * 16;
          }
          // sums of the even and of the odd 64 bytes; RAG: the sums and what they lost
          float acc[kSTiles][NT][4], more[kSTiles][NT][4];
#pragma unroll
          for (uint32_t k = 0; k < kSTiles; ++k)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
              for (int i = 0; i < 4; ++i) acc[k][n][i] = more[k][n][i] = 0.f;
#pragma unroll 2
          for (uint32_t q = 0; q < nq; ++q) {
            uint32_t xr[NT][DT == 3 ? 8 : 4];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
              const uint32_t xa = xl + 8 * n * xpitch + q * (DT == 3 ? 128 : 64);
              const uint4 x0 = lds128(xa);
              xr[n][0] = x0.x, xr[n][1] = x0.y, xr[n][2] = x0.z, xr[n][3] = x0.w;
              if constexpr (DT == 3) {
                const uint4 x1 = lds128(xa + 16);
                xr[n][4] = x1.x, xr[n][5] = x1.y, xr[n][6] = x1.z, xr[n][7] = x1.w;
              }
            }
            uint4 w[2 * kSTiles];
#pragma unroll
            for (uint32_t k = 0; k < 2 * kSTiles; ++k) w[k] = RAG ? lds_shifted(a[k] + q * 64) : lds128(a[k] + q * 64);
            if (!whole && q + 1 == nq) {
#pragma unroll
              for (uint32_t k = 0; k < 2 * kSTiles; ++k) w[k] = and4(w[k], tail);
            }
#pragma unroll
            for (uint32_t k = 0; k < kSTiles; ++k) {
              const uint4 &u = w[2 * k], &v = w[2 * k + 1];
              const uint32_t ra[4] = {u.x, u.y, u.z, u.w}, rb[4] = {v.x, v.y, v.z, v.w};
              float part[NT][4];
#pragma unroll
              for (int n = 0; n < NT; ++n) part[n][0] = part[n][1] = part[n][2] = part[n][3] = 0.f;
              if constexpr (DT == 3) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const uint32_t u0 = ra[j] ^ 0x80808080u, u1 = rb[j] ^ 0x80808080u;
                  const uint32_t a0 = i8x2_to_f16x2(u0, 0x4140u), a2 = i8x2_to_f16x2(u0, 0x4342u);
                  const uint32_t a1 = i8x2_to_f16x2(u1, 0x4140u), a3 = i8x2_to_f16x2(u1, 0x4342u);
#pragma unroll
                  for (int n = 0; n < NT; ++n)
                    mma_step<2, RAG>(acc[k][n], more[k][n], part[n], j, a0, a1, a2, a3, xr[n][2 * j], xr[n][2 * j + 1]);
                }
              } else {
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                  for (int n = 0; n < NT; ++n)
                    mma_step<DT, RAG>(acc[k][n], more[k][n], part[n], j, ra[2 * j], rb[2 * j], ra[2 * j + 1],
                                      rb[2 * j + 1], xr[n][2 * j], xr[n][2 * j + 1]);
              }
              if constexpr (!RAG) {
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    const float o = acc[k][n][i] + part[n][i];  // the two sets change places
                    acc[k][n][i] = more[k][n][i];
                    more[k][n][i] = o;
                  }
              }
            }
          }
#pragma unroll
          for (uint32_t k = 0; k < kSTiles; ++k)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
              for (int i = 0; i < 4; ++i)
                acc[k][n][i] = RAG ? kept_sum(acc[k][n][i], more[k][n][i]) : acc[k][n][i] + more[k][n][i];
          // C fragment: (g, 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1) of each 8-column tile
#pragma unroll
          for (uint32_t k = 0; k < 2 * kSTiles; ++k) {
            const uint32_t row = q0 + 8 * k + g;
            if (row < nr) {
              const float sc = DT == 3 ? __half2float(reinterpret_cast<const __half *>(md.s)[r + row]) : 1.f;
#pragma unroll
              for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                  const uint32_t col = 2 * t + i + 8 * n;
                  const float y = acc[k / 2][n][2 * (k & 1) + i];
                  if (col < md.G) md.y[(uint64_t)col * md.M + r + row] = DT == 3 ? y * sc : y;
                }
            }
          }
        }
        turn = (turn + ng) & (kSWarps - 1);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8 * s);
        ++it;
      }
    }
  }
  __syncthreads();
}

template <int DT, int NT>
cudaError_t short_attr() {
  const cudaError_t e = cudaFuncSetAttribute(gemm_short_kernel<DT, NT, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(gemm_short_kernel<DT, NT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmem);
}

template <int DT, int NT>
void short_launch(const GemvLaunch &L, cudaStream_t s) {
  if (L.ragged) gemm_short_kernel<DT, NT, true><<<L.grid, kSThreads, kSSmem, s>>>(L.mats, L.pieces, L.begin, L.status);
  else gemm_short_kernel<DT, NT, false><<<L.grid, kSThreads, kSSmem, s>>>(L.mats, L.pieces, L.begin, L.status);
}

}  // namespace

cudaError_t gemm_short_prepare() {
  cudaError_t e;
  if ((e = short_attr<1, 1>()) != cudaSuccess || (e = short_attr<1, 2>()) != cudaSuccess ||
      (e = short_attr<2, 1>()) != cudaSuccess || (e = short_attr<2, 2>()) != cudaSuccess ||
      (e = short_attr<3, 1>()) != cudaSuccess)
    return e;
  return short_attr<3, 2>();
}

cudaError_t launch_gemm_short(const GemvLaunch &L, cudaStream_t s) {
  if (L.grid <= 0) return cudaSuccess;
  if (L.nt != 1 && L.nt != 2) return cudaErrorInvalidValue;
  switch (L.dtype * 4 + L.nt) {
    case 1 * 4 + 1: short_launch<1, 1>(L, s); break;
    case 1 * 4 + 2: short_launch<1, 2>(L, s); break;
    case 2 * 4 + 1: short_launch<2, 1>(L, s); break;
    case 2 * 4 + 2: short_launch<2, 2>(L, s); break;
    case 3 * 4 + 1: short_launch<3, 1>(L, s); break;
    case 3 * 4 + 2: short_launch<3, 2>(L, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace wt
