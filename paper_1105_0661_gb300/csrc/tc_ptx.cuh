// PTX wrappers shared by the tensor-core beam formers (bf_tc.cu, bf_split.cu): mbarriers with
// bounded waits, tcgen05 MMA with the A operand in tensor memory and B in shared memory, tensor
// memory loads and stores.  Both kernels use one MMA shape: M = 128 rows (64 beams x re|im), N = 128
// columns (two 64-column swizzle atoms of 2 pols x 32 spectra), K = 16.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include "lbf_internal.cuh"

namespace lbf {
namespace tc {

constexpr int kRows = 128;                  // UMMA M
constexpr int kSpec = 32;                   // spectra per 64-column atom (2 pols side by side)
constexpr int kCols = 4 * kSpec;            // UMMA N: two atoms
constexpr int kMaxKpad = 128;               // S <= 64
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kWaitIters = 1u << 20;   // polls before a wait gives up

enum ErrCode { ERR_NONE = 0, ERR_PRODUCER = 1, ERR_MMA = 2, ERR_EPILOGUE = 3 };

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Bounded wait for the phase with the given parity; false on expiry or when another role aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  for (uint32_t i = 0; i < kWaitIters; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (*abort_flag) return false;
    if (i > 64) __nanosleep(64);
  }
  return false;
}

// The same with the thread suspended by the hardware between polls (up to `kSuspendNs` at a time):
// a warp that polls in a loop takes issue slots from the working warps of its scheduler.  Bounded by
// the clock, since the number of polls says nothing here.
constexpr uint32_t kSuspendNs = 20000;
constexpr long long kWaitCycles = 1ll << 28;   // ~0.14 s
__device__ __forceinline__ bool mbar_wait_suspended(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  long long t0 = 0;
  for (uint32_t i = 0;; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(kSuspendNs)
        : "memory");
    if (done) return true;
    if (*abort_flag) return false;
    if (i == 0) t0 = clock64();
    else if (clock64() - t0 > kWaitCycles) return false;
  }
}

// The waits of a whole warp: one answer for all lanes, which have converged again when it returns.  A
// lane still polling while lane 0 went on and arrived elsewhere could miss its phase (the parity comes
// back two phases later), and the .sync.aligned tensor-memory instructions need the whole warp.  The
// vote sits in the loop: behind the loops above it cost the epilogue registers (spills, 5-14 %).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  for (uint32_t i = 0; i < kWaitIters; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (__all_sync(0xffffffffu, done)) return true;
    if (__any_sync(0xffffffffu, *abort_flag)) return false;
    if (i > 64) __nanosleep(64);
  }
  return false;
}
__device__ __forceinline__ bool warp_wait_suspended(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  return __all_sync(0xffffffffu, mbar_wait_suspended(bar, parity, abort_flag));
}

__device__ __forceinline__ void fail(volatile int *abort_flag, int *err, int code) {
  *abort_flag = 1;
  atomicCAS(err, 0, code);
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
      : "memory");
}

// UMMA shared-memory descriptor of the MN-major B operand with the 128-byte swizzle: atoms of 8 K
// rows x 128 bytes; the next 8 K rows are 1024 bytes on (stride offset), the next 64 columns
// `lbo` bytes on (leading offset).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;                       // descriptor version
  d |= (uint64_t)2 << 61;                       // SWIZZLE_128B
  return d;
}

// Instruction descriptor: kind::f16, D = F32, A = B = F16, A K-major, B MN-major, M = 128, N = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 16) | ((uint32_t)(kCols >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);

// D[tmem] (+)= A[tmem] B[smem]
__device__ __forceinline__ void umma(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(kIdesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_half2(float lo_k, float hi_k) {
  const __half2 h = __floats2half2_rn(lo_k, hi_k);   // .x (low 16 bits) is the lower K index
  return *reinterpret_cast<const uint32_t *>(&h);
}

// Output of short integration windows.  The lanes of an epilogue warp hold rows of windows (a row
// per beam for I, a row per lane for IQUV: ro 0 holds I and Q, ro 1 U and V, in two buffers), but
// each lane's row lies megabytes from the next in the output.  A warp therefore collects kW windows
// of every row in its own piece of shared memory, the window index XORed so that neither walk meets
// a bank twice, and writes runs of kW windows.
template <int NS, int kW>
struct ShortRows {
  static constexpr int kRowsPer = 32 / kW;                        // rows per store instruction
  static constexpr int kBuf = (NS == 1 ? 16 : 32) * kW;           // floats of one buffer
  static constexpr int kBytes = (NS == 1 ? 1 : 2) * kBuf * 4;     // per warp
  __device__ static int index(int row, int w) {
    if (NS == 1) return row * kW + (w ^ ((2 * (row / kRowsPer)) & (kW - 1)));
    return row * kW + (w ^ ((row / kRowsPer) & (kW - 1)));
  }
  // parameters of window w: NS 1, r0 = I (both lanes of a beam hold it); NS 4, (I, Q) or (U, V)
  __device__ static void put(float *stage, int lane, int w, float r0, float r1) {
    if (NS == 1) {
      if ((w & 1) == (lane & 1)) stage[index(lane >> 1, w)] = r0;
    } else {
      stage[index(lane, w)] = r0;
      stage[kBuf + index(lane, w)] = r1;
    }
  }
  // windows w0 .. w0 + kW - 1 of the warp's first `nbeams` beams; row0: parameter I of the first one
  __device__ static void flush(const float *stage, int lane, int nbeams, int w0, int Mq, float *row0, long long bstride,
                               long long pstride) {
    const int w = lane % kW, rl = lane / kW;
    const int nb = w0 + w < Mq ? nbeams : 0;
    float *dst = row0 + (long long)(NS == 1 ? rl : rl >> 1) * bstride + (NS == 1 ? 0 : (rl & 1) * 2 * pstride) + w0 + w;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < (NS == 1 ? 16 : 32) / kRowsPer; ++k) {
      const int row = k * kRowsPer + rl;
      const int jq = NS == 1 ? row : row >> 1;
      // one row a store: addresses formed per row (stepping them took 1.93 ms for 1.80, 127 beams IQUV)
      float *const d = NS == 4 && kRowsPer == 1 ? row0 + (long long)jq * bstride + w0 + w + (row & 1) * 2 * pstride : dst;
      if (jq < nb) {
        d[0] = stage[index(row, w)];
        if (NS == 4) d[pstride] = stage[kBuf + index(row, w)];
      }
      if (NS == 1) dst += kRowsPer * bstride;
      else dst += kRowsPer / 2 * bstride;
    }
    __syncwarp();   // the rows are rewritten by the next chunk
  }
};

}  // namespace tc
}  // namespace lbf
