// Device-side helpers shared by the sm_103a kernel files: mbarrier ring
// primitives, 1-D TMA bulk copies, bounded waits, shared-memory loads.
// Internal to the library (each translation unit gets its own copies).
#pragma once

#include <cmath>
#include <cstdint>

#include "wt_kernels.h"

namespace wt {
namespace {

constexpr int kStatusTimedOut = -7;  // WT_ETIMEDOUT
constexpr long long kWaitCycles = 1ll << 31;  // ~1 s at 2 GHz

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

// Raises the transaction count alone, without the arrival.
__device__ __forceinline__ void mbar_expect_only(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// 1-D bulk copy global -> this CTA's shared memory, completion counted on `bar`.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes,
                                         uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}

__device__ __forceinline__ void named_bar(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Bounded wait.  Returns false (and raises the CTA's abort flag on a timeout)
// instead of spinning forever.
__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                             int *status) {
  if (*abort_flag) return false;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > kWaitCycles) {
      *abort_flag = 1;
      if (status) atomicCAS(status, 0, kStatusTimedOut);
      return false;
    }
  }
  return true;
}

// Programmatic dependent launch (launch attribute cudaLaunchAttributeProgrammaticStreamSerialization):
// griddep_wait blocks until the grid this one depends on in its stream has completed and its
// memory is visible (a no-op when the launch had no such dependency); griddep_launch lets the
// next grid of the stream be launched, its CTAs taking SMs as this grid's CTAs leave them.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The global nanosecond timer (comparable across the SMs of one GPU) and the SM this thread
// runs on; read by the stamping instantiation of the one-column kernel only.
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t sm_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return r;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr));
  return v;
}


__device__ __forceinline__ uint4 lds_or_zero(uint32_t addr, bool ok) {
  return ok ? lds128(addr) : make_uint4(0, 0, 0, 0);
}

__device__ __forceinline__ void sts8(uint32_t addr, uint8_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"((uint32_t)v) : "memory");
}

// The 16 bytes from byte `ph` (0..15) of the 32 bytes lo, hi on: two word selects and four
// funnel shifts.
__device__ __forceinline__ uint4 shift_bytes(const uint4 &lo, const uint4 &hi, uint32_t ph) {
  uint32_t q0 = lo.x, q1 = lo.y, q2 = lo.z, q3 = lo.w, q4 = hi.x, q5 = hi.y;
  if (ph & 8) q0 = lo.z, q1 = lo.w, q2 = hi.x, q3 = hi.y, q4 = hi.z, q5 = hi.w;
  if (ph & 4) q0 = q1, q1 = q2, q2 = q3, q3 = q4, q4 = q5;
  const uint32_t b = (ph & 3) * 8;
  return make_uint4(__funnelshift_r(q0, q1, b), __funnelshift_r(q1, q2, b), __funnelshift_r(q2, q3, b),
                    __funnelshift_r(q3, q4, b));
}

// 16 bytes of shared memory from any address: the two vectors that hold them.  Bytes past the
// caller's data may be read (from the vector that holds its last byte, or the next).
__device__ __forceinline__ uint4 lds_shifted(uint32_t addr) {
  const uint32_t ph = addr & 15u;
  const uint4 lo = lds128(addr - ph);
  const uint4 hi = lds128(addr - ph + (ph ? 16 : 0));
  return shift_bytes(lo, hi, ph);
}

// The mask of a vector's bytes [lo, hi).
__device__ __forceinline__ uint4 byte_mask(int lo, int hi) {
  uint32_t m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = min(max(lo - 4 * i, 0), 4), b = min(max(hi - 4 * i, 0), 4);
    m[i] = a >= b ? 0u : (0xffffffffu >> (32 - 8 * (b - a))) << (8 * a);
  }
  return make_uint4(m[0], m[1], m[2], m[3]);
}

__device__ __forceinline__ uint4 and4(const uint4 &a, const uint4 &b) {
  return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w);
}

// Bytes [off, off + len) of rows [r, r + n) of a ragged matrix to its stage, by the whole
// producer warp (lane q takes rows q, q + 32, ...: one thread's address arithmetic alone held
// such copies to 3.5 TB/s).  Row q arrives with its byte src at dst + q * pitch + (src & 15): a
// bulk copy brings the whole 16-byte vectors that hold the range and lie inside the matrix;
// bytes of the matrix's first or last vector that no such vector holds go one by one.
__device__ __forceinline__ void ragged_rows(const MatDesc &md, uint32_t r, uint32_t n, uint32_t off, uint32_t len,
                                            uint32_t dst, uint32_t pitch, uint32_t bar, uint64_t pol, int lane) {
  const uint64_t w0 = reinterpret_cast<uint64_t>(md.W), wend = w0 + (uint64_t)(md.M - 1) * md.rs + md.rb;
  const uint64_t wlo = (w0 + 15) & ~(uint64_t)15, whi = wend & ~(uint64_t)15;
  for (uint32_t q0 = 0; q0 < n; q0 += 32) {
    const uint32_t q = q0 + lane;
    const uint64_t src = w0 + (uint64_t)(r + q) * md.rs + off, a = src & ~(uint64_t)15, end = src + len;
    uint64_t lo = max(a, wlo), hi = min((end + 15) & ~(uint64_t)15, whi);
    const uint32_t d = dst + q * pitch;
    uint32_t bulk = 0;
    if (q < n) {
      if (hi > lo) bulk = (uint32_t)(hi - lo);
      else lo = hi = end;
      if (src < lo || hi < end) {
        for (uint64_t p = src; p < lo; ++p) sts8(d + (uint32_t)(p - a), *reinterpret_cast<const uint8_t *>(p));
        for (uint64_t p = max(hi, src); p < end; ++p)
          sts8(d + (uint32_t)(p - a), *reinterpret_cast<const uint8_t *>(p));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
    }
    const uint32_t tx = __reduce_add_sync(0xffffffffu, bulk);
    __syncwarp();
    // the stage's one arrival comes with its last bytes announced, after every lane's stores
    if (lane == 0) {
      if (q0 + 32 < n) mbar_expect_only(bar, tx);
      else mbar_expect_tx(bar, tx);
    }
    __syncwarp();
    if (bulk) bulk_g2s(d + (uint32_t)(lo - a), reinterpret_cast<const void *>(lo), bulk, bar, pol);
  }
}

// Two int8 weights as exact f16x2.  With u = b ^ 0x80 (0..255) in the low byte and 0x64 in
// the high byte, a half holds 1024 + u (f16 has unit spacing on [1024, 2048)); subtracting
// 1152 = 1024 + 128 leaves b, an integer in [-128, 127], exactly.
__device__ __forceinline__ uint32_t i8x2_to_f16x2(uint32_t u, uint32_t sel) {
  uint32_t h;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(__byte_perm(u, 0x64646464u, sel)), "r"(0x64806480u));
  return h;
}

// d += A B on one 16x8x16 tile; bf16 operands for DT 1, f16 otherwise.
template <int DT>
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  if constexpr (DT == 1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  } else {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
}

// Two fp32 differences or sums in one instruction.
__device__ __forceinline__ void sub_x2(float &d0, float &d1, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 x, y;\n\t"
      "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "sub.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ void add_x2(float &d0, float &d1, float b0, float b1) {
  asm("{\n\t.reg .b64 x, y;\n\t"
      "mov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\t"
      "add.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "+f"(d0), "+f"(d1)
      : "f"(b0), "f"(b1));
}

// s + c += A B, s the running sum and c what it lost.  The tensor cores truncate their sum to
// fp32; a second MMA from the step s took backwards, A B - (s' - s), gives what they dropped,
// because they align the products with a few bits more than a result keeps (16 random products,
// 2-norm error of A B against 64 bits: f16 4.7e-8, with the second MMA 2.1e-8, rounded to nearest
// 2.5e-8; bf16 2.5e-8, 3.9e-9, 1.8e-8; int8 2.1e-8, 2.9e-9, 1.5e-8).
template <int DT>
__device__ __forceinline__ void mma16816_kept(float (&s)[4], float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                              uint32_t a3, uint32_t b0, uint32_t b1) {
  float t[4], r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) t[i] = s[i];
  mma16816<DT>(t, a0, a1, a2, a3, b0, b1);
  sub_x2(r[0], r[1], s[0], s[1], t[0], t[1]);
  sub_x2(r[2], r[3], s[2], s[3], t[2], t[3]);
  mma16816<DT>(r, a0, a1, a2, a3, b0, b1);
  add_x2(c[0], c[1], r[0], r[1]);
  add_x2(c[2], c[3], r[2], r[3]);
#pragma unroll
  for (int i = 0; i < 4; ++i) s[i] = t[i];
}
// The sum: beside an infinite s, c means nothing.
__device__ __forceinline__ float kept_sum(float s, float c) { return fabsf(s) < INFINITY ? s + c : s; }

}  // namespace
}  // namespace wt
