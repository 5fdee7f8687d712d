// FP32 tied-array beam former (Section 4.3) on the tensor cores: the FP32 corner-turned block and
// the weights are cut into FP16 slices, six slice products run as tcgen05 MMAs, and the result is no
// further from the 64-bit value than that of the FP32 FMA kernels of beamform.cu.  Fused with the
// Stokes I / IQUV integration epilogue (Sections 4.5, 5.1) or writing the beam voltages.
//
// Why: the beam former of B beams does 16 B flop per station-sample.  In FP32 FMAs that is bound by
// the FMA pipe from about 10 beams on (80 TFLOP/s: 58 ms for the 127-beam LOFAR block), while the
// block could be read in 5.4 ms and its six FP16 products take 15 ms at the measured tensor-core rate.
//
// The slices.  The tensor cores add FP16 products exactly but truncate the FP32 accumulator toward
// zero as they go; that bias does not average out over an integration window, and is why the
// three-product form of bf_tc.cu stays at 1e-6.  Here the leading product is exact instead (the
// error-free transformation of Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59, 2012):
//  * a column of the block (one spectrum and polarisation, all stations) is scaled by the power of
//    two that puts its largest component in [2^9, 2^10); y1 is the scaled value rounded to an
//    integer, y2 the rest rounded to a multiple of 2^-11 and y3 what then remains in FP16, good to
//    2^-33 of the peak: a station 500 times weaker than the strongest keeps its 24 bits;
//  * 128 w = w1 + w2 + w3 with w1 an integer, w2 and w3 FP16 (exact to 2^-29);
//  * D1 = W1 Y1 never rounds: |w1| < 2^7.01 and |y1| <= 2^10.5 keep a station's term below 2^17.51 and
//    the sum of 64 stations in phase below 2^23.51; D2 = W2 Y1 + W3 Y1 + W1 Y2 + W2 Y2 + W1 Y3
//    accumulates apart from it, 2^7 smaller and more, so that its truncation is below the result's
//    last bit; the products left out are below 2^-28 of the peak;
//  * V = (D1 + D2) 2^-e in FP32.
// What remains is the rounding of V and of the FP32 weights, where the FMA kernels round the
// accumulator at every station.  RMS error of the voltages against 64 bits for a given block, FMA
// kernel and this one: 8 stations 7.5e-8 and 3.7e-8, 24 stations 1.2e-7 and 3.6e-8, 64 stations 2.0e-7
// and 3.6e-8; 48 stations with the first 30 times stronger 2.4e-7 and 3.7e-8, with the last 5.6e-8 and
// 4.0e-8.  (Two slices of y and w12 = fp16(128 w) in the place of the last three products are off by
// 1.2e-7 to 1.5e-7 for equal stations, but by 4.4e-7 in the last two cases: 127 beams of 30 subbands
// took 2.0 ms so, 2.5 with three slices.)  Columns that hold an infinity, or nothing but numbers
// below 2^-118, are recomputed at the end of their work item with FP32 FMAs (fix_item).
//
// Work.  A persistent CTA per SM walks the work items (f, c, span of spectra, block of 64 beams)
// with a stride of the grid; the beam blocks of one (f, c) run together and share its block in L2.
// An item is one UMMA M tile of 128 rows (64 beams x re|im) by the span's tiles of 64 spectra x 2
// pols (N = 128), K = 2 stations x S padded to 16.  Warpgroup 0 holds the MMA issuer and three
// evaluators of the next item's weights; then
//  * converter warps (8, two groups of four; a group owns one 32-spectrum half of each tile): each
//    thread loads four adjacent spectra of one polarisation of every eighth station (one 32-byte load
//    where rows allow it), the column maxima meet in shared memory across a barrier of the group, and
//    the three slices go to the stage ring in the swizzled layout the MMA reads (64-bit stores, a whole
//    128-byte row per half-warp: no bank conflicts).  The loads of the next tile are issued as the
//    registers of the current one are consumed; the MMA thread prefetches the tiles after it into L2
//    (one tensor box per tile: a row at a time from the converters, the prefetches took 2700 cycles
//    per tile).  Sixteen warps of two spectra per thread: 10 % slower (twice the loop overhead).
//  * epilogue warps (8): warp w serves TMEM lane quadrant w % 4 and one 32-spectrum half.  They take
//    D2 into registers while the MMAs fill D1, and D1 while the MMAs fill the next tile's D2, so
//    that one accumulator of each suffices (256 TMEM columns, next to 3 x 64 of weight slices).
// What bounds it: the issue slots (ncu, 8 subbands of the LOFAR block: 56 % of them used, 9000 warp
// instructions per tile of 64 beams, most of them the converters') and the latency of the converters'
// chain; the MMAs (64 cycles each) take 57 % of a tile's 4000 cycles.  127 beams of the LOFAR block: 86.2
// ms in FP32 FMAs, 20.5 here; 37 beams of 30 subbands: 5.5 ms and 1.29; voltages of 127 beams, 16 subbands:
// 5.7 ms and 1.87.  The ring holds two stages up to 56 stations and one beyond (64 stations, 127 beams, 8
// subbands: 1.20 ms against 0.74 for 56).  Measured and dropped: stages of two slices that share a third
// one (64 stations 1.20 -> 1.10 ms, 48 stations 0.67 -> 0.71: registers), stages released by halves (an
// MMA of 64 columns takes as long as one of 128: 48 stations 0.67 -> 1.08).
// Every mbarrier wait is bounded: on expiry the kernel records an error code, stops issuing work,
// waits (bounded) for its MMAs in flight, frees TMEM and returns.  The MMA thread, the evaluators and
// the converters wait suspended; the epilogue polls (suspended waits cost it up to 70 % on short
// items).
#include <atomic>

#include "tc_ptx.cuh"

namespace lbf {
namespace {

using namespace tc;

constexpr int kItemBeams = kRows / 2;       // 64 beams per work item
constexpr int kTileSpec = 2 * kSpec;        // 64 spectra per tile
constexpr int kEpiWarps = 8, kConvWarps = 8;
constexpr int kGroup = kConvWarps / 2;      // converter warps per half tile
constexpr int kThreads = 128 + 32 * (kEpiWarps + kConvWarps);   // warpgroup 0: MMA issuer and 3 weight evaluators
// a third and fourth stage gain nothing and take the L1 cache from the voltage rows (24 stations, 61 beams,
// 16 subbands: 0.90 ms with four, 0.78 with two)
constexpr int kMaxStages = 2;
constexpr int kBarBytes = 1024;
constexpr int kSlots = 8;                   // column-scale ring: more than the stages + 3 tiles in flight
constexpr int kScaleBytes = kSlots * kCols * 4;
constexpr int kColmaxBytes = 2 * 3 * 64 * 4;   // [group][3][column]
constexpr int kSmemLimit = (int)kCtaSharedBytes;
// shared memory: barriers and flags, column scales, column maxima, stage ring (1024-byte aligned),
// output staging, weight stage
constexpr int kScaleOff = kBarBytes, kColmaxOff = kScaleOff + kScaleBytes;
constexpr int kNonfOff = 256;               // in the barrier page: [kSlots][group] flags
constexpr int kGfailOff = 232, kAbortOff = 228;
constexpr int kRingOff = (kColmaxOff + kColmaxBytes + 1023) / 1024 * 1024;
constexpr int kFixed = 1024 /* alignment slack */ + kRingOff;
constexpr int kMinSmem = 120 * 1024;        // one CTA per SM: each allocates all of TMEM
constexpr uint32_t kD1 = 0, kD2 = kCols, kW0 = 2 * kCols;   // TMEM columns: D1, D2, three weight slices
constexpr uint32_t kWPlane = 64;
constexpr float kWUnit = 128.f;
constexpr float kMagic = 12582912.f;        // 1.5 * 2^23: x + kMagic rounds x to an integer
constexpr float kMagic2 = 6144.f;           // 1.5 * 2^12: x + kMagic2 rounds x to a multiple of 2^-11
constexpr int kPrefetch = 4;                // tiles an L2 prefetch runs ahead of the loads
// Registers per thread after the split of what the CTA is launched with (640 x 96 = 61440): 128 x 40 +
// 256 x 112 (epilogue) + 256 x 104 (converters) = 60416.  The compiler allocates each section by its own
// share: with 120 and 96 all kernels spilled 300 bytes and more a thread, so up to 90.  (The voltage
// epilogue of 24 stations gains 3 % from 120, but 64 stations lose 40 % with 96 for the converters.)
constexpr int kLaunchRegs = 96;

struct SpParams {
  int S, F, B, M, Kpad, ntiles, ipf;        // ipf: beam blocks per (f, c)
  int tpc, chunks;                          // tiles per item, items along the spectra
  int items, first_item;
  int stage_bytes;                          // 3 slices x 2 atoms x Kpad rows x 128 bytes
  int vec, align;                           // output rows 16-byte aligned; bytes the input rows are aligned to
  const int *phase0;
  const float *step;
  const float2 *ct;
  float *out;
  int *err;
};

// map[i]: tensor map of plan i's block for the L2 prefetches (rows 16-byte aligned)
constexpr int kMaxPlans = 32;
struct SpLaunch {
  CUtensorMap map[kMaxPlans];
  SpParams plan[kMaxPlans];
  int nplans, items, nstages, stage_max;
};

__device__ __forceinline__ int plan_of(const SpLaunch &L, int item) {
  int i = 0;
  while (i + 1 < L.nplans && L.plan[i + 1].first_item <= item) ++i;
  return i;
}

// Coordinates of a work item: beam block fastest, then the span of spectra, then (f, c).
struct Item {
  int fc, bb, t0, t1;
};
__device__ __forceinline__ Item item_of(const SpParams &p, int item) {
  Item it;
  const int li = item - p.first_item;
  const int r = li / p.ipf;
  it.bb = li - r * p.ipf;
  it.fc = r / p.chunks;
  it.t0 = (r - it.fc * p.chunks) * p.tpc;
  it.t1 = min(p.ntiles, it.t0 + p.tpc);
  return it;
}

__device__ __forceinline__ float2 weight_of(const SpParams &p, int f, int c, int b, int s) {
  const long long bs = (long long)b * p.S + s;
  return fixed_phasor(weight_phase(__ldg(&p.phase0[(long long)f * p.B * p.S + bs]), __ldg(&p.step[bs]),
                                   (float)(c - kN / 2)));
}

// The weights of an item go through the weight stage [S][64 beams] float2 in shared memory.  The
// evaluator warps fill it while the item before runs; the epilogue warps slice them on their way to
// TMEM (put_weights) as soon as that item's last MMA is done.  (Sliced by the evaluators, the stage is
// half as large again, and IQUV of 52 to 56 stations keeps one ring stage: 8 subbands, 127 beams 1.14 ms
// against 0.79.)
constexpr int kEvalWarps = 3;
constexpr int weight_stage_bytes(int Kpad) { return (Kpad / 2) * kItemBeams * 8; }

// exp(2 pi i phi) of two phases in 2^-32 cycle, as packed operations: reduced to the nearest quarter
// cycle in integers, then the Taylor polynomials of sine (degree 9) and cosine (degree 10), whose
// remainders at an eighth of a cycle are 2e-9 and 1e-10 (twice as fast as two general sincos).
__device__ __forceinline__ void two_phasors(int phi0, int phi1, float2 &w0, float2 &w1) {
  const int q0 = (int)((unsigned)phi0 + (1u << 29)) >> 30, q1 = (int)((unsigned)phi1 + (1u << 29)) >> 30;
  const int r0 = (int)((unsigned)phi0 - ((unsigned)q0 << 30)), r1 = (int)((unsigned)phi1 - ((unsigned)q1 << 30));
  auto both = [](float a) { return make_float2(a, a); };
  const float2 x = __fmul2_rn(make_float2((float)r0, (float)r1), both(1.4629180792671596e-9f));   // radians
  const float2 x2 = __fmul2_rn(x, x);
  float2 s = __ffma2_rn(x2, both(2.7557319e-6f), both(-1.98412698e-4f));
  s = __ffma2_rn(x2, s, both(8.3333333e-3f));
  s = __ffma2_rn(x2, s, both(-1.66666667e-1f));
  s = __ffma2_rn(__fmul2_rn(x2, s), x, x);
  float2 c = __ffma2_rn(x2, both(-2.7557319e-7f), both(2.48015873e-5f));
  c = __ffma2_rn(x2, c, both(-1.38888889e-3f));
  c = __ffma2_rn(x2, c, both(4.16666667e-2f));
  c = __ffma2_rn(x2, c, both(-0.5f));
  c = __ffma2_rn(x2, c, both(1.f));
  auto turn = [](int q, float s, float c) {
    const float a = (q & 1) ? -s : c, b = (q & 1) ? c : s;
    return (q & 2) ? make_float2(-a, -b) : make_float2(a, b);
  };
  w0 = turn(q0, s.x, c.x);
  w1 = turn(q1, s.y, c.y);
}

// slices of (cos, sin), each a half2
__device__ __forceinline__ void slice_weight(float2 w, uint32_t &w1, uint32_t &w2, uint32_t &w3) {
  const float2 u = make_float2(kWUnit, kWUnit), mg = make_float2(kMagic, kMagic), m1 = make_float2(-1.f, -1.f);
  const float2 h = __ffma2_rn(__ffma2_rn(w, u, mg), m1, mg);    // minus the integer part
  const float2 rest = __ffma2_rn(w, u, h);
  const __half2 second = __floats2half2_rn(rest.x, rest.y);
  const float2 third = __ffma2_rn(__half22float2(second), m1, rest);
  w1 = pack_half2(-h.x, -h.y);
  w2 = *reinterpret_cast<const uint32_t *>(&second);
  w3 = pack_half2(third.x, third.y);
}

// Beams fastest over the lanes of a warp, so that the stage is written without bank conflicts; a
// lane keeps one beam and walks the stations.
__device__ __forceinline__ void eval_weights(const SpParams &p, float2 *stage, const Item &it, int ew, int lane) {
  const int f = it.fc / kN, S2 = p.Kpad / 2;
  const float dc = (float)(it.fc - f * kN - kN / 2);
#pragma unroll 1
  for (int u = ew; u < S2 / 2; u += kEvalWarps) {          // 4 stations of half the beams
    const int s0 = (u >> 1) * 4, bl = (u & 1) * 32 + lane, b = it.bb * kItemBeams + bl;
    const int *ph = p.phase0 + ((long long)f * p.B + b) * p.S;
    const float *st = p.step + (long long)b * p.S;
    int phi[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      phi[k] = b < p.B && s0 + k < p.S ? weight_phase(__ldg(ph + s0 + k), __ldg(st + s0 + k), dc) : 0;
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      float2 w[2];
      two_phasors(phi[k], phi[k + 1], w[0], w[1]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int s = s0 + k + e;
        if (b >= p.B || s >= p.S) w[e] = make_float2(0.f, 0.f);
        stage[s * kItemBeams + bl] = w[e];
      }
    }
  }
}

// Column s of a slice in TMEM holds (Re w, -Im w) for a Re row (ro = 0) and (Im w, Re w) for an Im
// row; warp `half` of a lane quadrant moves every second group of 8 stations.  bl: beam of the row.
__device__ __forceinline__ void put_weights(const SpParams &p, const float2 *stage, uint32_t ta, int bl, int ro,
                                            int half) {
  const uint32_t sel = ro ? 0x1032u : 0x3210u, flip = ro ? 0u : 0x80000000u;
#pragma unroll 1
  for (int g8 = half; g8 < p.Kpad / 16; g8 += 2) {
    const float2 *d = stage + g8 * 8 * kItemBeams + bl;
    const uint32_t t = ta + (uint32_t)(g8 * 8);
    uint32_t a[3][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      slice_weight(d[j * kItemBeams], a[0][j], a[1][j], a[2][j]);
#pragma unroll
      for (int k = 0; k < 3; ++k) a[k][j] = __byte_perm(a[k][j], 0, sel) ^ flip;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) tmem_st8(t + k * kWPlane, a[k]);
  }
  tmem_wait_st();
}

// Output staging for windows of 8 spectra and more: 8 consecutive windows of every (beam, Stokes
// parameter) row of a lane quadrant meet in shared memory and leave as whole 32-byte sectors.  A
// quadrant's buffer: 16 beams x NS parameters x 8 windows, the 16-byte chunks of a beam
// XOR-swizzled by the beam; two buffers alternate.  Shorter windows and voltages go through 4 KB per
// warp.
constexpr int kVStageBytes = 8 * 2 * kSpec * 8;   // 8 beams x 2 pols x 32 spectra, cf32
template <int NS, int Q>
struct Stage {
  static constexpr bool kOn = NS != 0 && Q >= 8;
  static constexpr int kPeriod = Q >= 8 ? Q / 8 : 1;           // tiles per flush
  static constexpr int kRow = NS * 8;                          // floats per beam
  static constexpr int kBuf = 16 * kRow;                       // floats per quadrant buffer
  static constexpr int kBytes = kOn ? 4 * 2 * kBuf * 4 : kEpiWarps * kVStageBytes;
  __device__ static int index(int jq, int param, int wl) {     // float index within a beam's row
    const int chunk = (param * 2 + (wl >> 2)) ^ (jq & (2 * NS - 1));
    return chunk * 4 + (wl & 3);
  }
};

// Write a quadrant's staged windows wbase .. wbase + 7 (the quadrant's 64 threads, tq their index).
template <int NS, int Q>
__device__ __forceinline__ void flush_stage(const SpParams &p, const float *buf, int tq, int quad, int bb, int f,
                                            int c, int wbase) {
  const int Mq = p.M / Q;
#pragma unroll
  for (int k = 0; k < (NS * 32 + 63) / 64; ++k) {
    const int i = tq + 64 * k;
    const int part = i & 1, param = (i >> 1) % NS, jq = (i >> 1) / NS;
    const int b = bb * kItemBeams + quad * 16 + jq;
    const int w0 = wbase + part * 4;
    if (i >= NS * 32 || b >= p.B || w0 >= Mq) continue;
    const float4 v = *reinterpret_cast<const float4 *>(buf + jq * Stage<NS, Q>::kRow +
                                                       ((param * 2 + part) ^ (jq & (2 * NS - 1))) * 4);
    float *dst = p.out + ((((long long)b * NS + param) * p.F + f) * kN + c) * Mq + w0;
    if (p.vec && w0 + 3 < Mq) {
      *reinterpret_cast<float4 *>(dst) = v;
    } else {
      const float e[4] = {v.x, v.y, v.z, v.w};
      for (int q = 0; q < 4 && w0 + q < Mq; ++q) dst[q] = e[q];
    }
  }
}

// Windows of a half tile for the short rows (Q 2 and 4).
template <int Q>
struct Short {
  static constexpr int kW = Q <= 4 ? kSpec / Q : 8;
};

// Stokes parameters of one 32-spectrum half tile (spectra m0 .. m0 + 31) from this lane's voltage
// component (Re rows ro = 0, Im rows ro = 1): vx, vy hold pairs of spectra of pol X and Y.  Windows of
// Q >= 8 spectra go to the staging row `srow`, shorter ones through `wstage` to the output rows (row0:
// parameter I of the warp's first beam, of which `nbeams` exist).
template <int NS, int Q>
__device__ __forceinline__ void stokes_half(const float2 (&vx)[16], const float2 (&vy)[16], int m0, int lane, int nbeams,
                                            int M, float *row0, long long bstride, long long pstride, float *srow,
                                            float *wstage, int wbase) {
  constexpr int kW = Q >= 16 ? 1 : 16 / Q;     // windows that end in 16 spectra
  const int ro = lane & 1, jq = lane >> 1;
  const int Mq = M / Q;
  if constexpr (Q == 1) {
    // Every spectrum is a window: the parameters replace the voltages, and a whole half tile leaves as
    // 128-byte rows, the second parameter of each lane after the first (Stokes I, 40 beams of 2
    // stations, 4 subbands of 768 spectra: 316 us through 16-window short rows, 131 here).
    float p0[kSpec], p1[kSpec];
#pragma unroll
    for (int i = 0; i < kSpec; ++i) {
      const float x = i & 1 ? vx[i >> 1].y : vx[i >> 1].x, y = i & 1 ? vy[i >> 1].y : vy[i >> 1].x;
      if (NS == 1) {
        const float own = x * x + y * y;
        p0[i] = own + __shfl_xor_sync(0xffffffffu, own, 1);
      } else {
        const float yp = __shfl_xor_sync(0xffffffffu, y, 1);   // the partner lane's Y component
        const float xx = x * x, yy = y * y, v = x * yp;
        const float i_own = xx + yy, q_own = xx - yy, u_own = x * y, v_own = ro ? v : -v;
        float k0 = ro ? u_own : i_own, k1 = ro ? v_own : q_own;
        k0 += __shfl_xor_sync(0xffffffffu, ro ? i_own : u_own, 1);
        k1 += __shfl_xor_sync(0xffffffffu, ro ? q_own : v_own, 1);
        p0[i] = ro ? 2.f * k0 : k0;
        p1[i] = ro ? 2.f * k1 : k1;
      }
    }
#pragma unroll
    for (int pass = 0; pass < (NS == 4 ? 2 : 1); ++pass) {
      if (NS == 1) {
#pragma unroll
        for (int i = 0; i < kSpec / 2; ++i) wstage[jq * kSpec + ((2 * i + ro) ^ (2 * jq))] = ro ? p0[2 * i + 1] : p0[2 * i];
      } else {
#pragma unroll
        for (int i = 0; i < kSpec; ++i) wstage[lane * kSpec + (i ^ lane)] = pass ? p1[i] : p0[i];
      }
      __syncwarp();
      float *dst = row0 + pass * pstride + m0 + lane;
      const int nb = m0 + lane < M ? nbeams : 0;
#pragma unroll 8
      for (int b = 0; b < 16; ++b, dst += bstride)
        if (b < nb) {
          if (NS == 1) {
            dst[0] = wstage[b * kSpec + (lane ^ (2 * b))];
          } else {
            dst[0] = wstage[2 * b * kSpec + (lane ^ (2 * b))];
            dst[2 * pstride] = wstage[(2 * b + 1) * kSpec + (lane ^ (2 * b + 1))];
          }
        }
      __syncwarp();   // the rows are rewritten by the next pass
    }
    return;
  }
  float2 pxx = make_float2(0.f, 0.f), pyy = pxx, pxy = pxx, pv = pxx;
#pragma unroll
  for (int ch = 0; ch < 2; ++ch) {
    const int w0 = (m0 + 16 * ch) / Q;         // first window of this chunk
    auto finish = [&](int w, float sxx, float syy, float sxy, float sv) {   // window sums -> parameters
      float r0, r1 = 0.f;
      if (NS == 1) {
        const float own = sxx + syy;
        r0 = own + __shfl_xor_sync(0xffffffffu, own, 1);
      } else {
        // lane ro 0 ends with (I, Q), lane ro 1 with (U, V): each sends what its partner keeps
        const float i_own = sxx + syy, q_own = sxx - syy, u_own = sxy, v_own = ro ? sv : -sv;
        float k0 = ro ? u_own : i_own, k1 = ro ? v_own : q_own;
        const float s0 = ro ? i_own : u_own, s1 = ro ? q_own : v_own;
        k0 += __shfl_xor_sync(0xffffffffu, s0, 1);
        k1 += __shfl_xor_sync(0xffffffffu, s1, 1);
        r0 = ro ? 2.f * k0 : k0;
        r1 = ro ? 2.f * k1 : k1;
      }
      if constexpr (Stage<NS, Q>::kOn) {
        if (w0 + w < Mq && jq < nbeams) {
          if (NS == 1) {
            if (ro == 0) srow[Stage<NS, Q>::index(jq, 0, w0 + w - wbase)] = r0;
          } else {
            srow[Stage<NS, Q>::index(jq, ro ? 2 : 0, w0 + w - wbase)] = r0;
            srow[Stage<NS, Q>::index(jq, ro ? 3 : 1, w0 + w - wbase)] = r1;
          }
        }
      } else {
        ShortRows<NS, Short<Q>::kW>::put(wstage, lane, ch * kW + w, r0, r1);
      }
    };
#pragma unroll
    for (int i = 0; i < 8; ++i) {              // pairs of spectra
      const float2 x = vx[ch * 8 + i], y = vy[ch * 8 + i];
      float2 yp = make_float2(0.f, 0.f);       // the partner lane's Y component
      if (NS == 4) yp = make_float2(__shfl_xor_sync(0xffffffffu, y.x, 1), __shfl_xor_sync(0xffffffffu, y.y, 1));
      {
        pxx = __ffma2_rn(x, x, pxx);
        pyy = __ffma2_rn(y, y, pyy);
        if (NS == 4) {
          pxy = __ffma2_rn(x, y, pxy);
          pv = __ffma2_rn(x, yp, pv);
        }
        if ((ch * 16 + 2 * i + 2) % Q == 0) {
          finish(Q >= 16 ? 0 : (2 * i + 2) / Q - 1, pxx.x + pxx.y, pyy.x + pyy.y, pxy.x + pxy.y, pv.x + pv.y);
          pxx = pyy = pxy = pv = make_float2(0.f, 0.f);
        }
      }
    }
    if constexpr (!Stage<NS, Q>::kOn)
      if (ch == 1) ShortRows<NS, Short<Q>::kW>::flush(wstage, lane, nbeams, m0 / Q, Mq, row0, bstride, pstride);
  }
}

// One 32-spectrum half tile as beam voltages (vol [B][F][N][P][M] cf32; `vrow0` the pol-X row of the
// warp's first beam, of which `nbeams` exist, beams `bstride` apart), one polarisation at a time
// through the warp's 4 KB: a row of 32 complex values per beam, the spectrum XORed by the beam so that
// the 32 lanes (16 beams x re|im) write 32 banks, then out as whole 256-byte rows.
__device__ __forceinline__ void voltage_half(const float2 (&vx)[16], const float2 (&vy)[16], int m0, int lane, int nbeams,
                                             int M, float2 *vrow0, long long bstride, float *stage) {
  const int ro = lane & 1, jq = lane >> 1, m = m0 + lane;
  float *const mine = stage + jq * 64 + ro;
#pragma unroll
  for (int pol = 0; pol < 2; ++pol) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float2 v = pol ? vy[i] : vx[i];
      mine[2 * ((2 * i) ^ jq)] = v.x;
      mine[2 * ((2 * i + 1) ^ jq)] = v.y;
    }
    __syncwarp();
    float2 *dst = vrow0 + (long long)pol * M + m;
#pragma unroll 8
    for (int b = 0; b < 16; ++b, dst += bstride)
      if (b < nbeams && m < M) *dst = *reinterpret_cast<const float2 *>(stage + b * 64 + 2 * (lane ^ b));
    __syncwarp();
  }
}

// Recompute an item that has a column with an infinity or too small to scale with FP32 FMAs, station by
// station, as the FMA kernels do (an infinite sample times a weight slice would turn into a NaN
// otherwise).
template <int NS, int Q>
__device__ __noinline__ void fix_item(const SpParams &p, const Item &it, int et) {
  constexpr int kG = NS == 0 ? 4 : (Q < 4 ? 4 : Q);     // spectra per thread and step
  constexpr int kWin = NS == 0 ? 1 : Q;
  const int f = it.fc / kN, c = it.fc - f * kN;
  const float2 *y = p.ct + (long long)it.fc * p.S * kP * p.M;
  const int ma = it.t0 * kTileSpec, mb = min(p.M, it.t1 * kTileSpec);
  const int steps = (mb - ma + kG - 1) / kG;
  for (int idx = et; idx < kItemBeams * steps; idx += 32 * kEpiWarps) {
    const int b = it.bb * kItemBeams + idx % kItemBeams;
    const int mg = ma + (idx / kItemBeams) * kG;
    if (b >= p.B) continue;
    float wxx = 0.f, wyy = 0.f, wre = 0.f, wim = 0.f;
    for (int m4 = mg; m4 < min(mb, mg + kG); m4 += 4) {
      float2 X[4], Y[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) X[q] = Y[q] = make_float2(0.f, 0.f);
      for (int s = 0; s < p.S; ++s) {
        const float2 w = weight_of(p, f, c, b, s);
        const float2 *rx = y + (long long)(s * kP) * p.M, *ry = rx + p.M;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (m4 + q >= mb) continue;
          const float2 a = rx[m4 + q], d = ry[m4 + q];
          X[q] = make_float2(fmaf(-w.y, a.y, fmaf(w.x, a.x, X[q].x)), fmaf(w.y, a.x, fmaf(w.x, a.y, X[q].y)));
          Y[q] = make_float2(fmaf(-w.y, d.y, fmaf(w.x, d.x, Y[q].x)), fmaf(w.y, d.x, fmaf(w.x, d.y, Y[q].y)));
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = m4 + q;
        if (m >= mb) continue;
        if (NS == 0) {
          float2 *v = reinterpret_cast<float2 *>(p.out) + (((long long)b * p.F + f) * kN + c) * kP * p.M;
          v[m] = X[q];
          v[p.M + m] = Y[q];
          continue;
        }
        wxx += fmaf(X[q].x, X[q].x, X[q].y * X[q].y);
        wyy += fmaf(Y[q].x, Y[q].x, Y[q].y * Y[q].y);
        wre += fmaf(X[q].x, Y[q].x, X[q].y * Y[q].y);
        wim += fmaf(X[q].y, Y[q].x, -X[q].x * Y[q].y);
        if ((m + 1) % kWin == 0) {
          const int Mq = p.M / kWin;
          float *o = p.out + (((long long)b * NS * p.F + f) * kN + c) * Mq + m / kWin;
          const long long ps = (long long)p.F * kN * Mq;
          o[0] = wxx + wyy;
          if (NS == 4) {
            o[ps] = wxx - wyy;
            o[2 * ps] = 2.f * wre;
            o[3 * ps] = 2.f * wim;
          }
          wxx = wyy = wre = wim = 0.f;
        }
      }
    }
  }
}

// Barrier of `n` threads under named barrier `id`; whether any of them passed `pred`.
__device__ __forceinline__ bool group_sync_any(uint32_t id, uint32_t n, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

// Four consecutive spectra (32 bytes) of a corner-turned row into v, which keeps its value where
// nothing is loaded: n spectra exist from p on.  kAl: bytes the rows are aligned to.
template <int kAl>
__device__ __forceinline__ void load_quad(float (&v)[8], const float2 *p, int n) {
  if constexpr (kAl == 32) {   // four spectra or none
    asm volatile(
        "{\n\t.reg .pred a;\n\tsetp.gt.s32 a, %9, 0;\n\t"
        "@a ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
        : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7])
        : "l"(p), "r"(n));
  } else if constexpr (kAl == 16) {   // an even number
    asm volatile(
        "{\n\t.reg .pred a, b;\n\tsetp.gt.s32 a, %9, 0;\n\tsetp.gt.s32 b, %9, 2;\n\t"
        "@a ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%8];\n\t"
        "@b ld.global.nc.v4.f32 {%4, %5, %6, %7}, [%8+16];\n\t}"
        : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7])
        : "l"(p), "r"(n));
  } else {
    asm volatile(
        "{\n\t.reg .pred a, b, c, d;\n\tsetp.gt.s32 a, %9, 0;\n\tsetp.gt.s32 b, %9, 1;\n\t"
        "setp.gt.s32 c, %9, 2;\n\tsetp.gt.s32 d, %9, 3;\n\t"
        "@a ld.global.nc.v2.f32 {%0, %1}, [%8];\n\t@b ld.global.nc.v2.f32 {%2, %3}, [%8+8];\n\t"
        "@c ld.global.nc.v2.f32 {%4, %5}, [%8+16];\n\t@d ld.global.nc.v2.f32 {%6, %7}, [%8+24];\n\t}"
        : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7])
        : "l"(p), "r"(n));
  }
}

// The converter role.  NLD: stations per thread (at least Kpad / 16), so that a tile's loads are
// straight-line code: behind a branch per station they ran one after the other (7000 cycles per tile).
template <int NLD, int kAl, bool kMulti>
__device__ __forceinline__ void convert(const SpLaunch &L, unsigned char *const sbase, int cw, int lane) {
  const uint32_t bar0 = smem_u32(sbase);
  float *const scales = reinterpret_cast<float *>(sbase + kScaleOff);
  uint32_t *const colmax = reinterpret_cast<uint32_t *>(sbase + kColmaxOff);
  volatile int *const gfail = reinterpret_cast<volatile int *>(sbase + kGfailOff);
  volatile int *const nonfinite = reinterpret_cast<volatile int *>(sbase + kNonfOff);
  volatile int *const abort_flag = reinterpret_cast<volatile int *>(sbase + kAbortOff);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 64u + 8u * s; };
  const int grp = cw / kGroup, wg = cw % kGroup;
  const int s0 = 2 * wg + (lane >> 4);       // station within a step of 2 kGroup
  const int pol = (lane >> 3) & 1, j = lane & 7;
  const int col = grp * kSpec + 4 * j;       // first spectrum of the thread within a tile
  const int cc = pol * kSpec + 4 * j;        // its first column within the half tile
  float r[NLD][8];                            // four spectra of every eighth station
  int item = blockIdx.x, t = 0, t1 = 0, pi = 0;
  const float2 *ptr = nullptr;                // row of station s0, at this thread's spectra of the tile
  auto plan = [&]() -> const SpParams & { return L.plan[kMulti ? pi : 0]; };
  auto enter = [&]() {
    if (kMulti) pi = plan_of(L, item);
    const SpParams &p = plan();
    const Item w = item_of(p, item);
    t = w.t0;
    t1 = w.t1;
    ptr = p.ct + (((long long)w.fc * p.S + s0) * kP + pol) * p.M + t * kTileSpec + col;
  };
  // Station s0 + 8 i of the first S.  Pad stations keep finite values, which meet weights of zero;
  // columns past M keep what they held and are never stored.
  auto load_tile = [&](int i, int S, int M) {
    load_quad<kAl>(r[i], ptr + (long long)(i * 2 * kGroup * kP) * M, s0 + 2 * kGroup * i < S ? M - (t * kTileSpec + col) : 0);
  };
  auto clear = [&](int i) {
#pragma unroll
    for (int e = 0; e < 8; ++e) r[i][e] = 0.f;
  };
#pragma unroll
  for (int i = 0; i < NLD; ++i) clear(i);
  enter();
  {
    const int S = plan().S, M = plan().M;
#pragma unroll
    for (int i = 0; i < NLD; ++i) load_tile(i, S, M);
  }
  uint32_t *const cm0 = colmax + grp * 3 * 64;
  if (wg == 0) cm0[2 * lane] = cm0[2 * lane + 1] = 0;   // n = 0
  group_sync_any(1 + grp, 32 * kGroup, false);
  int s = 0, slot = 0, n = 0;
  uint32_t ph = 0;
  int b3 = 0;
  bool failed = false, more = true;
  while (more) {
    const int Kpad = plan().Kpad;
    float mx[4] = {0.f, 0.f, 0.f, 0.f};       // largest component of the four columns (NaNs ignored)
#pragma unroll
    for (int i = 0; i < NLD; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) mx[e] = fmaxf(mx[e], fmaxf(fabsf(r[i][2 * e]), fabsf(r[i][2 * e + 1])));
    // three rotating maxima per column: tile n's, tile n + 1's cleared before the barrier (its
    // readers, of tile n - 2, passed the barrier of tile n - 1)
    uint32_t *cm = cm0 + b3 * 64 + pol * 8 + j;   // [4 columns of a thread][16 threads]
    b3 = b3 == 2 ? 0 : b3 + 1;
#pragma unroll
    for (int e = 0; e < 4; ++e) atomicMax(cm + 16 * e, __float_as_uint(mx[e]));
    if (wg == 0) *reinterpret_cast<uint2 *>(cm0 + b3 * 64 + 2 * lane) = make_uint2(0, 0);
    if (failed) gfail[grp * 2 + (n & 1)] = 1;
    const bool inf = group_sync_any(1 + grp, 32 * kGroup,
                                    fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) > 3.402823466e38f);
    if (gfail[grp * 2 + (n & 1)]) break;      // the whole group leaves together
    // scale 2^(136 - E) for a peak in [2^(E - 127), 2^(E - 126)), E >= 9: the peak lands in
    // [2^9, 2^10); its inverse, with the weights' 2^7, is 2^(E - 127) 2^-16
    auto scale_of = [](uint32_t cb, float &inv) {
      const uint32_t e = max(cb & 0x7f800000u, 9u << 23);
      inv = __uint_as_float(e) * 1.52587890625e-5f;
      return __uint_as_float((263u << 23) - e);
    };
    float4 inv;
    const uint4 peak = make_uint4(cm[0], cm[16], cm[32], cm[48]);
    const float sc[4] = {scale_of(peak.x, inv.x), scale_of(peak.y, inv.y), scale_of(peak.z, inv.z),
                         scale_of(peak.w, inv.w)};
    // columns too small to scale (a peak below 2^-118, yet not zero) are left to the FMAs as well
    auto tiny = [](uint32_t cb) { return cb - 1u < (9u << 23) - 1u; };
    bool fix = inf;
    if (wg == 0)   // the lanes of a warp cover the columns of the half tile
      fix = __any_sync(0xffffffffu, inf || tiny(peak.x) || tiny(peak.y) || tiny(peak.z) || tiny(peak.w));
    if (!warp_wait_suspended(empty_bar(s), ph ^ 1u, abort_flag)) { fail(abort_flag, plan().err, ERR_PRODUCER); failed = true; }
    // row k of a slice's atom: 128 bytes [pol X | pol Y][32 spectra], 16-byte chunks XOR (k & 7);
    // station s0 + 8 i holds rows k = 2 s0 + 16 i (re) and k + 1 (im).  (After an expired wait the
    // stage is overwritten all the same: the launch has failed.)
    const uint32_t chunk = (uint32_t)(pol * 4 + (j >> 1)), within = (uint32_t)(j & 1) * 8;
    const int k0 = 2 * s0, steps = Kpad / (4 * kGroup);
    unsigned char *re = sbase + kRingOff + (size_t)s * L.stage_max + (size_t)grp * (Kpad * 128) + k0 * 128 + within;
    unsigned char *im = re + 128 + ((chunk ^ (uint32_t)((k0 + 1) & 7)) << 4);
    re += (chunk ^ (uint32_t)(k0 & 7)) << 4;
    const uint32_t slice = (uint32_t)Kpad * 256;
    // on to the next tile
    ptr += kTileSpec;
    if (++t == t1) {
      item += gridDim.x;
      more = item < L.items;
      if (more) enter();
    }
    const int nS = more ? plan().S : 0, nM = plan().M;
    const float2 mg = make_float2(kMagic, kMagic), mg2 = make_float2(kMagic2, kMagic2), m1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      float2 h[4], m[4], l[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 x = make_float2(r[i][2 * e], r[i][2 * e + 1]), sx = make_float2(sc[e], sc[e]);
        h[e] = __ffma2_rn(__ffma2_rn(x, sx, mg), m1, mg);   // minus the first slice
        l[e] = __ffma2_rn(x, sx, h[e]);
        m[e] = __ffma2_rn(__fadd2_rn(l[e], mg2), m1, mg2);   // minus the second
        l[e] = __fadd2_rn(l[e], m[e]);
      }
      if (i < steps) {
        *reinterpret_cast<uint2 *>(re + i * (kGroup * 512)) = make_uint2(pack_half2(-h[0].x, -h[1].x), pack_half2(-h[2].x, -h[3].x));
        *reinterpret_cast<uint2 *>(im + i * (kGroup * 512)) = make_uint2(pack_half2(-h[0].y, -h[1].y), pack_half2(-h[2].y, -h[3].y));
        *reinterpret_cast<uint2 *>(re + slice + i * (kGroup * 512)) = make_uint2(pack_half2(-m[0].x, -m[1].x), pack_half2(-m[2].x, -m[3].x));
        *reinterpret_cast<uint2 *>(im + slice + i * (kGroup * 512)) = make_uint2(pack_half2(-m[0].y, -m[1].y), pack_half2(-m[2].y, -m[3].y));
        *reinterpret_cast<uint2 *>(re + 2 * slice + i * (kGroup * 512)) = make_uint2(pack_half2(l[0].x, l[1].x), pack_half2(l[2].x, l[3].x));
        *reinterpret_cast<uint2 *>(im + 2 * slice + i * (kGroup * 512)) = make_uint2(pack_half2(l[0].y, l[1].y), pack_half2(l[2].y, l[3].y));
      }
      if (kMulti) clear(i);                   // the next plan may have fewer stations
      load_tile(i, nS, nM);
    }
    if (!failed) {
      if (wg == 0 && lane < 16) *reinterpret_cast<float4 *>(scales + slot * kCols + grp * 64 + cc) = inv;
      if (wg == 0 && lane == 0) nonfinite[slot * 2 + grp] = fix ? 1 : 0;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the slices visible to the MMA
      __syncwarp();
      if (lane == 0) mbar_arrive(full_bar(s));
    }
    slot = (slot + 1) & (kSlots - 1);
    ++n;
    if (++s == L.nstages) { s = 0; ph ^= 1u; }
  }
}

template <int NS, int Q, bool kMulti>
__global__ void __launch_bounds__(kThreads, 1)
bf_split_kernel(const __grid_constant__ SpLaunch L) {
  using St = Stage<NS, Q>;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *sbase = smem_raw + (base - raw);
  const uint32_t bar0 = base;
  const int nst = L.nstages;
  const uint32_t sB = base + kRingOff;
  unsigned char *after = sbase + kRingOff + (size_t)nst * L.stage_max;
  const float *const scales = reinterpret_cast<const float *>(sbase + kScaleOff);   // [kSlots][kCols]
  float *const stage_out = reinterpret_cast<float *>(after);
  float2 *const wstage = reinterpret_cast<float2 *>(after + St::kBytes);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 64u + 8u * s; };
  const uint32_t d1full = bar0 + 128u, d1empty = bar0 + 136u, d2full = bar0 + 144u, d2empty = bar0 + 152u;
  const uint32_t wfull = bar0 + 160u, drain_bar = bar0 + 168u;
  auto pair_bar = [&](int q) { return bar0 + 176u + 8u * q; };
  const uint32_t fix_bar = bar0 + 208u, wready = bar0 + 216u, wfree = bar0 + 320u;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sbase + 224);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(sbase + kAbortOff);
  volatile int *gfail = reinterpret_cast<volatile int *>(sbase + kGfailOff);          // [group][parity]
  volatile int *nonfinite = reinterpret_cast<volatile int *>(sbase + kNonfOff);      // [kSlots][group]

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(full_bar(s), kConvWarps);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(d1full, 1);
    mbar_init(d2full, 1);
    mbar_init(d1empty, kEpiWarps);
    mbar_init(d2empty, kEpiWarps);
    mbar_init(wfull, kEpiWarps);
    mbar_init(drain_bar, 1);
    mbar_init(fix_bar, kEpiWarps);
    mbar_init(wready, kEvalWarps);
    mbar_init(wfree, kEpiWarps);
    for (int q = 0; q < 4; ++q) mbar_init(pair_bar(q), 2);
    *abort_flag = 0;
    for (int i = 0; i < 4; ++i) gfail[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 1 && lane == 0) {
      // -------------------------------------------------------------- MMA issuer
      bool issued = false, ok = true;
      int s = 0, it = 0;
      uint32_t ph = 0, gpar = 0;
      int *err = L.plan[0].err;
      // the tile kPrefetch tiles on goes to L2 (one box of all its rows) while the MMAs run
      const bool pf = !kMulti && L.plan[0].align >= 16;
      int pitem = blockIdx.x, pt = 0, pt1 = 0, pfc = 0;
      auto prefetch = [&](bool fetch) {
        if (pitem >= L.items) return;
        if (pt == pt1) {
          const Item w = item_of(L.plan[0], pitem);
          pt = w.t0;
          pt1 = w.t1;
          pfc = w.fc;
        }
        if (fetch)
          asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];"
                       ::"l"(reinterpret_cast<uint64_t>(&L.map[0])), "r"(pt * 2 * kTileSpec), "r"(0), "r"(pfc)
                       : "memory");
        if (++pt == pt1) pitem += gridDim.x;
      };
      for (int i = 0; pf && i < kPrefetch; ++i) prefetch(i > 0);
      for (int item = blockIdx.x; item < L.items && ok; item += gridDim.x, ++it) {
        const SpParams &p = L.plan[kMulti ? plan_of(L, item) : 0];
        err = p.err;
        const Item w = item_of(p, item);
        const int ksteps = p.Kpad >> 4;
        const uint64_t slice = (uint64_t)((uint32_t)(p.Kpad * 256) >> 4);   // to the next slice of the block, / 16
        const uint64_t desc0 = smem_desc(sB, (uint32_t)(p.Kpad * 128));
        const uint32_t a0 = tmem + kW0;
        if (!mbar_wait_suspended(wfull, (uint32_t)it & 1u, abort_flag)) { fail(abort_flag, err, ERR_MMA); break; }
        for (int t = w.t0; t < w.t1; ++t, gpar ^= 1u) {
          if (!mbar_wait_suspended(full_bar(s), ph, abort_flag) || !mbar_wait_suspended(d2empty, gpar ^ 1u, abort_flag)) {
            fail(abort_flag, err, ERR_MMA); ok = false; break;
          }
          tc_fence_after();
          const uint64_t b0 = desc0 + (uint64_t)((uint32_t)(s * L.stage_max) >> 4);
          for (int ks = 0; ks < ksteps; ++ks) {      // D2 = W2 Y1 + W3 Y1 + W1 Y2 + W2 Y2 + W1 Y3
            const uint64_t b = b0 + (uint64_t)(ks * ((16 * 128) >> 4));
            const uint32_t a = a0 + 8u * ks;
            umma(tmem + kD2, a + kWPlane, b, ks != 0);
            umma(tmem + kD2, a + 2 * kWPlane, b, 1);
            umma(tmem + kD2, a, b + slice, 1);
            umma(tmem + kD2, a + kWPlane, b + slice, 1);
            umma(tmem + kD2, a, b + 2 * slice, 1);
          }
          umma_commit(d2full);
          issued = true;
          if (!mbar_wait_suspended(d1empty, gpar ^ 1u, abort_flag)) { fail(abort_flag, err, ERR_MMA); ok = false; break; }
          tc_fence_after();
          for (int ks = 0; ks < ksteps; ++ks)        // D1 = W1 Y1
            umma(tmem + kD1, a0 + 8u * ks, b0 + (uint64_t)(ks * ((16 * 128) >> 4)), ks != 0);
          umma_commit(empty_bar(s));
          umma_commit(d1full);
          if (pf) prefetch(true);
          if (++s == nst) { s = 0; ph ^= 1u; }
        }
      }
      if (issued) {   // every MMA (and its barrier arrivals) retired before TMEM is released
        umma_commit(drain_bar);
        volatile int never = 0;
        if (!mbar_wait(drain_bar, 0, &never)) fail(abort_flag, err, ERR_MMA);
      }
    } else if (warp != 1) {
      // -------------------------------------------------------------- weight evaluators
      const int ew = warp == 0 ? 0 : warp - 1;
      uint32_t k = 0;
      for (int item = blockIdx.x; item < L.items; item += gridDim.x, k ^= 1u) {
        const SpParams &p = L.plan[kMulti ? plan_of(L, item) : 0];
        if (!warp_wait_suspended(wfree, k ^ 1u, abort_flag)) { fail(abort_flag, p.err, ERR_EPILOGUE); break; }
        eval_weights(p, wstage, item_of(p, item), ew, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(wready);
      }
    }
    __syncwarp();
  } else if (warp < 4 + kEpiWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    // ---------------------------------------------------------------- epilogue
    const int ew = warp - 4, quad = warp & 3, half = ew >> 2;
    const int ro = lane & 1, jq = lane >> 1;
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t acol = (uint32_t)(half * 2 * kSpec);        // this half's columns of an accumulator
    float *const qbuf = stage_out + quad * 2 * St::kBuf;
    uint32_t gpar = 0, fpar = 0;
    int fl = 0, eit = 0, slot = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < L.items && ok; item += gridDim.x, ++eit) {
      const SpParams &p = L.plan[kMulti ? plan_of(L, item) : 0];
      const Item w = item_of(p, item);
      const int f = w.fc / kN, c = w.fc - f * kN;
      int bad = 0;
      const int Mq = NS == 0 ? 0 : p.M / Q;
      const long long pstride = (long long)p.F * kN * Mq;        // between Stokes parameters
      const int b0 = w.bb * kItemBeams + quad * 16;               // the warp's 16 beams, of which nb exist
      const int nb = min(16, p.B - b0);
      float *const row0 = p.out + (NS == 0 ? 0 : (((long long)b0 * NS * p.F + f) * kN + c) * Mq);
      const int ni = item + (int)gridDim.x;
      const bool more = ni < L.items;
      const SpParams &pn = L.plan[kMulti ? plan_of(L, more ? ni : item) : 0];
      // the weights of item number k (of this CTA) to TMEM
      auto put = [&](const SpParams &q, int k) -> bool {
        if (!warp_wait(wready, (uint32_t)k & 1u, abort_flag)) { fail(abort_flag, q.err, ERR_EPILOGUE); return false; }
        put_weights(q, wstage, tl + kW0, quad * 16 + jq, ro, half);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(wfull);
          mbar_arrive(wfree);
        }
        return true;
      };
      if (eit == 0 && !put(p, 0)) break;
      for (int t = w.t0; t < w.t1; ++t, gpar ^= 1u) {
        float2 vx[16], vy[16];
        if (nb <= 0) {   // no beams in this lane quadrant: keep the barriers and the weights going
          if (!warp_wait(d2full, gpar, abort_flag)) { fail(abort_flag, p.err, ERR_EPILOGUE); ok = false; break; }
          if (lane == 0) mbar_arrive(d2empty);
          if (!warp_wait(d1full, gpar, abort_flag)) { fail(abort_flag, p.err, ERR_EPILOGUE); ok = false; break; }
          tc_fence_after();   // put() overwrites the weights that the MMAs of D1 have read
          if (t == w.t1 - 1 && more && !put(pn, eit + 1)) { ok = false; break; }
          if (lane == 0) mbar_arrive(d1empty);
          bad |= nonfinite[slot * 2] | nonfinite[slot * 2 + 1];
          slot = (slot + 1) & (kSlots - 1);
          continue;
        }
        if (!warp_wait(d2full, gpar, abort_flag)) { fail(abort_flag, p.err, ERR_EPILOGUE); ok = false; break; }
        tc_fence_after();
        {
          float a[2][16], d[2][16];
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            tmem_ld16(tl + kD2 + acol + (uint32_t)(ch * 16), a[ch]);
            tmem_ld16(tl + kD2 + acol + (uint32_t)(kSpec + ch * 16), d[ch]);
          }
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            vx[i] = make_float2(a[i >> 3][(2 * i) & 15], a[i >> 3][(2 * i + 1) & 15]);
            vy[i] = make_float2(d[i >> 3][(2 * i) & 15], d[i >> 3][(2 * i + 1) & 15]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(d2empty);
        if (!warp_wait(d1full, gpar, abort_flag)) { fail(abort_flag, p.err, ERR_EPILOGUE); ok = false; break; }
        tc_fence_after();
        // every MMA that reads this item's weights is complete
        if (t == w.t1 - 1 && more && !put(pn, eit + 1)) { ok = false; break; }
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          float a[16], d[16];
          tmem_ld16(tl + kD1 + acol + (uint32_t)(ch * 16), a);
          tmem_ld16(tl + kD1 + acol + (uint32_t)(kSpec + ch * 16), d);
          tmem_wait_ld();
          if (ch == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(d1empty);
          }
          const float4 *sx = reinterpret_cast<const float4 *>(scales + slot * kCols + acol + ch * 16);
          const float4 *sy = sx + kSpec / 4;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 a4 = sx[i], d4 = sy[i];
            const int k = ch * 8 + 2 * i;
            vx[k] = __fmul2_rn(__fadd2_rn(make_float2(a[4 * i], a[4 * i + 1]), vx[k]), make_float2(a4.x, a4.y));
            vx[k + 1] = __fmul2_rn(__fadd2_rn(make_float2(a[4 * i + 2], a[4 * i + 3]), vx[k + 1]), make_float2(a4.z, a4.w));
            vy[k] = __fmul2_rn(__fadd2_rn(make_float2(d[4 * i], d[4 * i + 1]), vy[k]), make_float2(d4.x, d4.y));
            vy[k + 1] = __fmul2_rn(__fadd2_rn(make_float2(d[4 * i + 2], d[4 * i + 3]), vy[k + 1]), make_float2(d4.z, d4.w));
          }
        }
        bad |= nonfinite[slot * 2] | nonfinite[slot * 2 + 1];
        slot = (slot + 1) & (kSlots - 1);
        const int m0 = t * kTileSpec + half * kSpec;
        const int wbase = (t / St::kPeriod) * 8;
        float *const buf = qbuf + (fl & 1) * St::kBuf;
        if constexpr (NS == 0) {
          float2 *const v0 = reinterpret_cast<float2 *>(p.out) + (((long long)b0 * p.F + f) * kN + c) * kP * p.M;
          voltage_half(vx, vy, m0, lane, nb, p.M, v0, (long long)p.F * kN * kP * p.M,
                       stage_out + ew * (kVStageBytes / 4));
        } else {
          stokes_half<NS, Q>(vx, vy, m0, lane, nb, p.M, row0, NS * pstride, pstride, buf + jq * St::kRow,
                             stage_out + ew * (kVStageBytes / 4), wbase);
          if constexpr (St::kOn) {
            if ((t + 1) % St::kPeriod == 0 || t == w.t1 - 1) {
              __syncwarp();
              if (lane == 0) mbar_arrive(pair_bar(quad));
              if (!warp_wait(pair_bar(quad), (uint32_t)fl & 1u, abort_flag)) {
                fail(abort_flag, p.err, ERR_EPILOGUE); ok = false; break;
              }
              flush_stage<NS, Q>(p, buf, half * 32 + lane, quad, w.bb, f, c, wbase);
              ++fl;
            }
          }
        }
      }
      if (ok && bad) {   // the same value in every epilogue warp; all of them have stored the item first
        __syncwarp();
        if (lane == 0) mbar_arrive(fix_bar);
        if (!warp_wait(fix_bar, fpar, abort_flag)) { fail(abort_flag, p.err, ERR_EPILOGUE); break; }
        fpar ^= 1u;
        fix_item<NS, Q>(p, w, tid - 128);
      }
    }
  } else {
    // ---------------------------------------------------------------- converters
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int cw = warp - 4 - kEpiWarps;
    const int nld = L.plan[0].Kpad / 16, al = L.plan[0].align;
    if (kMulti || al == 8) convert<8, 8, kMulti>(L, sbase, cw, lane);
    else if (al == 16) convert<8, 16, kMulti>(L, sbase, cw, lane);
    else if (nld <= 2) convert<2, 32, kMulti>(L, sbase, cw, lane);
    else if (nld <= 4) convert<4, 32, kMulti>(L, sbase, cw, lane);
    else if (nld <= 6) convert<6, 32, kMulti>(L, sbase, cw, lane);
    else convert<8, 32, kMulti>(L, sbase, cw, lane);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

template <int NS, int Q, bool kMulti>
cudaError_t launch_q(SpLaunch &L, int grid, cudaStream_t st) {
  auto kern = bf_split_kernel<NS, Q, kMulti>;
  const int wstage = weight_stage_bytes(L.stage_max / (6 * 128));   // of the largest Kpad
  L.nstages = (kSmemLimit - kFixed - Stage<NS, Q>::kBytes - wstage) / L.stage_max;
  if (L.nstages > kMaxStages) L.nstages = kMaxStages;
  if (L.nstages < 1) return cudaErrorInvalidValue;
  int smem = kFixed + L.nstages * L.stage_max + Stage<NS, Q>::kBytes + wstage;
  if (smem < kMinSmem) smem = kMinSmem;
  // the register split of the kernel's warpgroups draws on what the CTA was launched with
  static std::atomic<int> regs{0};   // of this kernel, once known
  cudaError_t e = cudaSuccess;
  if (regs.load(std::memory_order_relaxed) == 0) {
    cudaFuncAttributes a;
    e = cudaFuncGetAttributes(&a, kern);
    if (e != cudaSuccess) return e;
    regs.store(a.numRegs, std::memory_order_relaxed);
  }
  if (regs.load(std::memory_order_relaxed) < kLaunchRegs) return cudaErrorInvalidConfiguration;
  e = allow_shared(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, kThreads, smem, st>>>(L);
  return cudaGetLastError();
}

template <int NS, bool kMulti>
cudaError_t launch_ns(int Q, SpLaunch &L, int grid, cudaStream_t st) {
  switch (Q) {
    case 1: return launch_q<NS, 1, kMulti>(L, grid, st);
    case 2: return launch_q<NS, 2, kMulti>(L, grid, st);
    case 4: return launch_q<NS, 4, kMulti>(L, grid, st);
    case 8: return launch_q<NS, 8, kMulti>(L, grid, st);
    case 16: return launch_q<NS, 16, kMulti>(L, grid, st);
    case 32: return launch_q<NS, 32, kMulti>(L, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

template <bool kMulti>
cudaError_t launch_kind(SpLaunch &L, int out_kind, int Q, int grid, cudaStream_t st) {
  if (out_kind == OUT_VOLTAGES) return launch_q<0, 1, kMulti>(L, grid, st);
  if (out_kind == OUT_STOKES_IQUV) return launch_ns<4, kMulti>(Q, L, grid, st);
  if (out_kind == OUT_STOKES_I) return launch_ns<1, kMulti>(Q, L, grid, st);
  return cudaErrorInvalidValue;
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? n : 0;
}

bool fill_plan(SpLaunch &L, int i, const Geometry &g, int out_kind, const float2 *ct, void *out, int sms) {
  SpParams &p = L.plan[i];
  p.S = g.S; p.F = g.F; p.B = g.B; p.M = g.M;
  p.Kpad = ((2 * g.S + 15) / 16) * 16;
  p.stage_bytes = 6 * p.Kpad * 128;
  p.ntiles = (g.M + kTileSpec - 1) / kTileSpec;
  p.ipf = (g.B + kItemBeams - 1) / kItemBeams;
  const long long rows = (long long)g.F * kN * p.ipf;
  p.tpc = split_tiles_per_item(rows, p.ntiles, sms);
  p.chunks = (p.ntiles + p.tpc - 1) / p.tpc;
  const long long items = rows * p.chunks;
  const long long first = i == 0 ? 0 : (long long)L.plan[i - 1].first_item + L.plan[i - 1].items;
  if (items + first >= (1ll << 31) - 65536) return false;
  p.items = (int)items;
  p.first_item = (int)first;
  p.phase0 = g.phase0; p.step = g.step;
  p.ct = ct;
  p.out = static_cast<float *>(out);
  p.err = g.err;
  const bool aligned = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  p.vec = aligned && (out_kind == OUT_VOLTAGES ? g.M % 2 == 0 : (g.M / g.Q) % 4 == 0);
  const uintptr_t ca = reinterpret_cast<uintptr_t>(ct);
  p.align = g.M % 4 == 0 && (ca & 31) == 0 ? 32 : g.M % 2 == 0 && (ca & 15) == 0 ? 16 : 8;
  if (p.align >= 16 && encode_ct32_tile_map(&L.map[i], ct, 2 * g.S, g.M, (long long)g.F * kN, kTileSpec) != cudaSuccess)
    return false;
  L.items = p.first_item + p.items;
  L.stage_max = p.stage_bytes > L.stage_max ? p.stage_bytes : L.stage_max;
  L.nplans = i + 1;
  return true;
}

}  // namespace

int split_max_stations() { return kMaxKpad / 2; }

// Whole (f, c) rows per item; an observation of few rows is cut along the spectra, in spans of whole output
// flushes (at most 4 tiles), so that every SM has a few items.
int split_tiles_per_item(long long rows, int ntiles, int sms) {
  int tpc = ntiles;
  while (tpc > 4 && rows * ((ntiles + tpc - 1) / tpc) < 4ll * sms) tpc = ((tpc / 2 + 3) / 4) * 4;
  return tpc;
}

int split_max_plans_per_launch() { return kMaxPlans; }

cudaError_t launch_bf_split(const SplitPlanRef *plans, int n, int out_kind, int Q, cudaStream_t st) {
  if (n < 1 || n > kMaxPlans) return cudaErrorInvalidValue;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  SpLaunch L;
  L.nplans = 0; L.items = 0; L.nstages = 0; L.stage_max = 0;
  int k = 0;
  for (int i = 0; i < n; ++i) {
    const SplitPlanRef &r = plans[i];
    if (r.g.S > split_max_stations() || !r.g.err || (r.g.Q != Q && out_kind != OUT_VOLTAGES))
      return cudaErrorInvalidValue;
    if (r.g.M == 0 || r.g.B == 0) continue;
    if (!fill_plan(L, k, r.g, out_kind, r.ct, r.out, sms)) return cudaErrorInvalidValue;
    ++k;
  }
  if (L.items == 0) return cudaSuccess;
  const int grid = L.items < sms ? L.items : sms;
  return L.nplans > 1 ? launch_kind<true>(L, out_kind, Q, grid, st) : launch_kind<false>(L, out_kind, Q, grid, st);
}

}  // namespace lbf
