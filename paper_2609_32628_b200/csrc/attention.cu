// Kernel 4: phased mixed-precision block-sparse attention (Sec. 3.3 "Phased execution" and "Cross-precision
// accumulation", App. C.3 / C.4).
//
// Every query block (64 tokens) walks its own list: NVFP4 segment, then INT8/E4M3 segment, then BF16 segment.  All
// segments share the fp32 running row maximum h, the fp32 denominator l (which always sums the exponential weights
// BEFORE they are converted to a matrix operand) and ONE output accumulator in tensor memory; at a segment boundary
// the accumulator only changes units (Eq. "precision-state-conversion"), and the output is normalised once.
//
// Mapping onto sm_100a
//   A CTA owns two neighbouring query blocks ("streams" 0 and 1; in the last wave of CTAs, if its blocks are no more than the
//   SMs, each block has its own) and 1024 threads in six roles, with four softmax sets:
//     warps 0..15     softmax, set k = warp/4 takes the steps i = k (mod 4); inside a set stream = (warp%4)/2 and one
//                     thread owns one full 64-key row.  A thread reads its S row from TMEM, takes the running maximum
//                     of step i-1 from the thread of the previous set through a shared-memory word tagged with the
//                     step, keeps a partial denominator, and writes P~ (and its NVFP4 scale factors) into its set's
//                     operand image.  These warps hold most of the register file (setmaxnreg).
//     next 8 warps    correction + epilogue, four per stream.  Every step passes through them between the softmax
//                     and the product: they read the step's "maximum moved" ballots and, only if one is set or the
//                     segment changes, wait for the previous product and rescale those accumulator columns (and apply
//                     the per-channel unit change); then they release the product.  Most steps move no maximum, and
//                     the check is off the issuing warp's instruction stream (and it does not pay to move it back:
//                     all-4-bit call of 16x48x48, 13.75 ms; with the ballots read by the issuing warp 13.94).  Finally
//                     they combine the sets' partial denominators, normalise, exchange channel pairs between lanes and
//                     store straight from TMEM
//     next 2 warps    S = Q K^T issue, one warp per stream (tcgen05.mma, accumulators in TMEM), two steps ahead
//     next 2 warps    O^T += V^T P~^T issue, one warp per stream.  The issuing warps' instruction
//                     counts are on the critical path of every step: their loops are warp-uniform (one elected lane
//                     issues), operand descriptors are built once and only offset inside the loop
//     last 4 warps    loaders: per stream one warp for K (and the Q records) and one for V^T, 1-D bulk copies into
//                     rings of their own (a K block is needed as soon as a score buffer is free, a V block only after
//                     the step's weights are written); a ring entry takes two blocks of the list under one barrier (one of
//                     the 16-bit tier); lane l holds list entry 32*batch + l (address, mask, key scale)
//   S   = Q K^T   : M = 128, N = 64 keys, K = d.  The block-scaled instruction only exists at M = 128, so stream 0's
//                   queries sit in rows 0..63 and stream 1's in rows 64..127 (its operand descriptor starts 1 KB
//                   early); the other 64 rows of each product are don't-care.  S is double buffered.
//   O^T = V^T P^T : M = 128 channels, N = 64 queries, K = 64 keys.  Keeping O transposed makes the online-softmax
//                   correction a per-COLUMN scale, so only queries whose maximum moved are touched, and makes the
//                   per-channel unit changes (eta*delta_c^V, g_V/2688) per-lane scalars.
//   kinds         : kind::f16 (BF16); kind::i8 for QK^T + kind::f8f6f4 E4M3 x E4M3 for PV (App. C.1); and
//                   kind::mxf4nvf4 with E4M3 scales per 16 elements (NVFP4), scale factors moved by tcgen05.cp.
// What bounds it: the fetch of instructions, together with the latency of the hand-offs.  Eight warps of a scheduler are at
// eight places of the code, so that nearly every line comes from the SM's instruction cache (32 KB, shared by all roles).  Taken
// block by block, its request rate was 94 % of the peak (all-4-bit call of 16x48x48, 24 heads; special-function pipe 70 %, issue
// slots 69 %, tensor pipe 22 %).  So the instructions of a step are what is saved, in the roles around the softmax above all: the
// loaders, the Q K^T warps and the PV warps take the blocks of a list in pairs, with one ring entry, one wait and one round of
// the loop for two.  Requests fell by 18 % (1.59 -> 1.30 G), instructions by 8 % (9.34 -> 8.61 G) and the time by 5 %
// (12.59 -> 11.99 ms): at 81 % of the peak rate the fetch is no longer alone.  Taking PV and correction in pairs as well makes
// the products late (13.3 ms), and softmax steps of two blocks have 7.33 G instructions and 67 % of the request rate, but leave
// two warps a scheduler, which do not cover the latencies (13.7 ms).
// The softmax keeps the work inside the chain of hand-offs short: the row maximum is taken on raw accumulator values, the
// scale and the maximum are folded into one packed FMA feeding ex2, the NVFP4 group scale is folded into the exponent so the
// scaled weight needs no extra multiply, narrow weights are packed by the conversions themselves, and the exponentiate phase
// runs over the whole row in batches (all arguments, all exponentials, then sums and packing), which gives the single warp the
// instruction-level parallelism it lacks when the three are interleaved per pair.  And the code is kept small: beyond about 47
// KB in all the hits fall (99.9 % 11.9 ms, 99.0 % 12.0 to 12.1 with the same instructions; 97.6 % 14.4 and 93.8 % 15.1 in
// earlier states).
// Measured (kernel alone, ms, before -> with pairs):  12 heads of 32,760 tokens 2.92 -> 2.77, one ranking per head 2.91 ->
// 2.77, with a 226-token prefix, whose blocks are bf16, 3.90 -> 3.57;  24 heads of 36,864 tokens all in 8 bit at d = 64 11.79
// -> 10.75; 40 heads of 75,600 tokens, 20 % bf16 + 40 % 8-bit, 86.1 -> 82.7. And the first list entries' masks and key scales
// are fetched while a block is set up (three tiers at d = 64, whole call, 395.0 -> 390.8 us).
// Every wait on an mbarrier is bounded; a wait that gives up records device status "timeout", all roles leave their
// loops and the CTA exits normally after releasing TMEM.
#include <type_traits>
#include <cuda_fp8.h>

#include "da2_internal.cuh"
#include "tc05.cuh"

namespace da2 {

namespace {

// Softmax warp sets: set k takes the steps i = k (mod 4), one thread per 64-key row, four warps (one per TMEM lane
// quarter) per set.
constexpr int kSets = 4, kShift = 2, kMask = kSets - 1;
constexpr int kSoftmaxWarps = 4 * kSets, kCorrWarps = 8;  // four correction warps per stream
constexpr int kMmaWarp0 = kSoftmaxWarps + kCorrWarps;     // Q K^T issue for stream 0, 1
constexpr int kPvWarp0 = kMmaWarp0 + 2;                   // V^T P^T issue for stream 0, 1
constexpr int kLoadWarp0 = kPvWarp0 + 2;                  // K loaders for stream 0, 1, then V loaders
constexpr int NT = (kLoadWarp0 + 4) * 32;                 // 1024
constexpr uint32_t kTmemCols = 512;
// TMEM column map
__host__ __device__ constexpr uint32_t col_s(int s, int buf) { return (uint32_t)(s * 2 + buf) * 64u; }
__host__ __device__ constexpr uint32_t col_o(int s) { return 256u + (uint32_t)s * 64u; }
// scale factors: every region starts on a multiple of 4 columns (one 4-column group holds 128 rows x 4 scales)
__host__ __device__ constexpr uint32_t col_sfq(int s) { return 384u + (uint32_t)s * 8u; }  // 4 columns per K step
__host__ __device__ constexpr uint32_t col_sfk(int s) { return 400u + (uint32_t)s * 8u; }
__host__ __device__ constexpr uint32_t col_sfv(int s) { return 416u + (uint32_t)s * 4u; }
__host__ __device__ constexpr uint32_t col_sfp(int s) { return 424u + (uint32_t)s * 4u; }

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kEtaP8 = 0.0022326917f;  // probability dequantisation scale of the 8-bit path
constexpr float kOffsetP8 = 8.807f;      // base-2 exponent offset (about log2 448)

// barrier indices inside one stream's group
// (a parity wait can only tell the latest completion from the one before, so every barrier is laid out such that no
// waiter can fall two completions behind: buffers indexed by step parity get one barrier per buffer)
constexpr int kMaxK = 3, kMaxV = 4, kInfoRing = 16;  // (steps between a K request and its scores: at most 2 nk + 3)
// barriers, factors, ballots and scale atoms of the steps between softmax and product (kSets of them unless SEGMENTED, where a
// softmax warp may wait for the last product of the segment before: twice as many keep that use the barrier's latest)
constexpr int kStepBars = 8;
enum {
  B_FULLK = 0, B_KFREE = B_FULLK + kMaxK, B_FULLV = B_KFREE + kMaxK, B_VFREE = B_FULLV + kMaxV, B_SREADY = B_VFREE + kMaxV,
  B_SFREE = B_SREADY + kSets, B_PREADY = B_SFREE + 2, B_CORROK = B_PREADY + kStepBars, B_PVDONE = B_CORROK + kStepBars,
  B_ELL = B_PVDONE + kStepBars, B_Q = B_ELL + 1, B_COUNT = B_Q + 1
};

// Shared memory.  An entry of the operand rings holds two consecutive blocks of a list, or one of the 16-bit tier (which is
// about as large as two of the others): one wait, one barrier and one round of a loader's loop for both.  The Q records of the
// 4- and the 8-bit tier are resident; that of the 16-bit tier takes their place when its segment starts.
// With a 16-bit tier at head_dim 128 (8 KB P images) the layout is SEGMENTED: every segment cuts the bytes of the P slots into
// slots of its own tier, four, four and two.
struct SmemMap {
  uint32_t q[2][3];               // Q record per stream and tier
  uint32_t kring[2], vring[2];    // per stream: K blocks (K image + scale atoms), V blocks (V^T image + scale atom)
  uint32_t kbytes[3], vbytes[3];  // bytes to copy per block
  uint32_t kstage, vstage;        // from the first block of a ring entry to the second
  uint32_t kentry, ventry;        // bytes of a ring entry
  int nk, nv;                     // ring entries
  uint32_t p[2];                  // P operand images per stream
  uint32_t pbytes[3];             // bytes of a P slot (there are four, or SEGMENTED 4, 4, 2)
  uint32_t sfp[2];    // P scale atoms (512 B), one per step barrier
  uint32_t factor;    // float [2 streams][kStepBars][64]
  uint32_t hx;        // {float h, int step} [2][sets][64]: running maximum after a step, handed from thread to thread
  uint32_t href;      // float [2][sets][64]: reference of each set's partial denominator
  uint32_t ell;       // float [2][sets][64]
  uint32_t info;      // per stream, ring of kInfoRing steps: {float key scale, uint32 "has padding keys"}
  uint32_t lim;       // beside it, float [64] per step: +inf, -inf at padding keys (written where there are any)
  uint32_t bars;      // uint64 [2][B_COUNT]
  uint32_t tok;       // int [2 streams][64]: token of each query slot, -1 at padding
  uint32_t chg;       // uint32 [2 streams][kStepBars][2]: ballots of the queries whose maximum moved this step
  uint32_t total;
  int pair_ctas;      // CTAs with two query blocks; the CTAs after them have one each,
  int first_single;   // from this one on (head * Rt + block): stream 1 has none
  bool fits;          // the layout fits the 227 KB a block may use
};

__host__ SmemMap make_smem_map(const Params &p, bool segmented) {
  SmemMap m;
  // Two query blocks per CTA, but one in the last wave of CTAs if its blocks are no more than the SMs: the wave lasts as long
  // as one list, and a stream that has the SM to itself walks its list faster (calls of one such wave: 144 blocks of 144
  // 4- and 8-bit entries 59.9 -> 52.6 us, the smallest call's 32 blocks 13.3 -> 12.5 us).
  const int pairs = (p.Rt + 1) / 2, total = p.BH * pairs;
  auto block_of = [&](int cta) { return cta / pairs * p.Rt + cta % pairs * 2; };
  m.pair_ctas = total - total % kSms;
  if (p.BH * p.Rt - block_of(m.pair_ctas) > kSms) m.pair_ctas = total;
  m.first_single = block_of(m.pair_ctas);
  uint32_t cur = 0;
  auto r128 = [](uint32_t b) { return (b + 127u) / 128u * 128u; };
  auto take = [&](uint32_t bytes) { uint32_t o = cur; cur = r128(cur + bytes); return o; };
  uint32_t qlow = 0, pmax = 0;
  m.kstage = m.vstage = m.kentry = m.ventry = 0;
  for (int t = 0; t < 3; ++t) {
    m.kbytes[t] = p.qrec_bytes[t];                     // the K part of a record is laid out like a Q record
    m.vbytes[t] = p.kvrec_bytes[t] - p.qrec_bytes[t];
    if (!p.tier_active[t]) continue;
    pmax = 2048u << t;
    if (t < 2) {
      m.kstage = max(m.kstage, r128(m.kbytes[t]));
      m.vstage = max(m.vstage, r128(m.vbytes[t]));
      qlow += r128(p.qrec_bytes[t]);
    }
    m.kentry = max(2 * m.kstage, t < 2 ? 0u : r128(m.kbytes[t]));
    m.ventry = max(2 * m.vstage, t < 2 ? 0u : r128(m.vbytes[t]));
  }
  // stream 1's Q descriptors start 1 KB before its images: stream 0's records precede them, so that is valid memory
  for (int s = 0; s < 2; ++s) {
    m.q[s][0] = m.q[s][2] = take(p.tier_active[2] ? max(qlow, p.qrec_bytes[2]) : qlow);
    m.q[s][1] = m.q[s][0] + (p.tier_active[0] ? r128(p.qrec_bytes[0]) : 0u);
  }
  const uint32_t pregion = segmented ? 16384u : kSets * pmax;  // per stream
  const uint32_t fixed = 2 * (pregion + kStepBars * 512) + r128(2 * kStepBars * 64 * 4) + 2 * r128(2 * kSets * 64 * 4) +
                         r128(2 * kStepBars * 2 * 4) + r128(2 * kSets * 64 * 8) + r128(2 * kInfoRing * 8) + 2 * kInfoRing * 256 + r128(2 * 64 * 4) +
                         r128(2 * B_COUNT * 8);
  constexpr uint32_t kLimit = 232448u - 128u;  // less the static shared variables
  const uint32_t left = cur + fixed < kLimit ? (kLimit - cur - fixed) / 256u * 128u : 0u;  // ring bytes per stream
  // Three K and four V entries where they fit (a K block is consumed as soon as a score buffer is free, a V block only after the
  // weights of its step are written): d = 64, and d = 128 with a 4-bit tier alone.  Two of each at d = 128 otherwise.
  m.nk = kMaxK;
  m.nv = kMaxV;
  if (m.nk * m.kentry + m.nv * m.ventry > left) m.nk = m.nv = 2;
  m.fits = m.nk * m.kentry + m.nv * m.ventry <= left;
  for (int t = 0; t < 3; ++t) m.pbytes[t] = segmented ? 2048u << t : pmax;
  for (int s = 0; s < 2; ++s) m.kring[s] = take(m.nk * m.kentry);
  for (int s = 0; s < 2; ++s) m.vring[s] = take(m.nv * m.ventry);
  for (int s = 0; s < 2; ++s) m.p[s] = take(pregion);
  for (int s = 0; s < 2; ++s) m.sfp[s] = take(kStepBars * 512);
  m.factor = take(2 * kStepBars * 64 * 4);
  m.chg = take(2 * kStepBars * 2 * 4);
  m.hx = take(2 * kSets * 64 * 8);
  m.href = take(2 * kSets * 64 * 4);
  m.ell = take(2 * kSets * 64 * 4);
  m.info = take(2 * kInfoRing * 8);
  m.lim = take(2 * kInfoRing * 256);
  m.tok = take(2 * 64 * 4);
  m.bars = take(2 * B_COUNT * 8);
  m.total = cur;
  if (cur > kLimit) m.fits = false;
  return m;
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// the packed pairs of da2_internal.cuh taken apart and added; a three-input maximum, a minimum that keeps a NaN
__device__ __forceinline__ void unf2(uint64_t x, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
// eight accumulator columns of one channel times the columns' factors (and the channel's change of unit)
__device__ __forceinline__ void scale8(uint32_t (&o)[8], const float *fac, float lane_factor) {
  const float4 f0 = *reinterpret_cast<const float4 *>(fac), f1 = *reinterpret_cast<const float4 *>(fac + 4);
  const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
  const uint64_t l2 = f2(lane_factor, lane_factor);
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    float a, b;
    unf2(mul2(f2(__uint_as_float(o[j]), __uint_as_float(o[j + 1])), mul2(f2(f[j], f[j + 1]), l2)), a, b);
    o[j] = __float_as_uint(a);
    o[j + 1] = __float_as_uint(b);
  }
}
// maximum of 16 values in 8 instructions
__device__ __forceinline__ float max16(const float *x) {
  const float m0 = max3(x[0], x[1], x[2]), m1 = max3(x[3], x[4], x[5]), m2 = max3(x[6], x[7], x[8]);
  const float m3 = max3(x[9], x[10], x[11]), m4 = max3(x[12], x[13], x[14]);
  return fmaxf(max3(m0, m1, m2), max3(m3, m4, x[15]));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ uint32_t pack_e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return (uint32_t)r;
}
// two E4M3 codes -> two floats
__device__ __forceinline__ void decode_e4m3x2(uint32_t codes, float &lo, float &hi) {
  asm("{ .reg .b32 t; .reg .b16 a, b; cvt.rn.f16x2.e4m3x2 t, %2; mov.b32 {a, b}, t; cvt.f32.f16 %0, a; cvt.f32.f16 %1, b; }"
      : "=f"(lo), "=f"(hi)
      : "h"((uint16_t)codes));
}

// bounded wait that also gives up as soon as another thread of the CTA has flagged a failure
// (the flag then holds 1 + the shared-memory offset of the barrier that was never completed, for diagnosis)
//
// A plain mbarrier.try_wait blocks in hardware for a while (7,760 cycles, about 4 us) before it reports failure, so the retry loop
// issues next to nothing.  The bound is on elapsed clock cycles.  Barriers are named by their shared-memory address, and
// the loop is kept short: every wait is a copy of it, and the hot code of all roles shares a 32 KB instruction cache.
constexpr uint32_t kWaitLimitCycles = 400000000u;  // about 0.2 s
__device__ __forceinline__ uint32_t clock32() {
  uint32_t t;
  asm volatile("mov.u32 %0, %%clock;" : "=r"(t));
  return t;
}
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, int *abort_flag,
                                              uint32_t limit = kWaitLimitCycles) {
  if (tc::mbar_try_wait(bar, parity)) return true;
  const uint32_t t0 = clock32();
#pragma unroll 1
  do {
    if (tc::mbar_try_wait(bar, parity)) return true;
  } while (!*(volatile int *)abort_flag && clock32() - t0 <= limit);
  if (!*(volatile int *)abort_flag) *(volatile int *)abort_flag = 1 + (int)(bar & 0xffffu);
  return false;
}

// One arrival per warp: every lane's earlier writes are ordered before the elected lane's arrive by the warp barrier.
// (A per-thread arrive is a shared-memory atomic per thread; hundreds of them per step dominate the step time.)
__device__ __forceinline__ void warp_arrive(uint32_t bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) tc::mbar_arrive(bar);
}

// register rebalancing between warpgroups: the softmax warps hold a whole score row, the others a few scalars
template <int N> __device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

__device__ __forceinline__ uint2 ld_shared_volatile_v2(uint32_t saddr) {
  uint2 r;
  asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "r"(saddr) : "memory");
  return r;
}

// Valid-slot mask and token index of a block, from the frame's region table (prefix blocks are runs of 64 tokens)
__device__ __forceinline__ unsigned long long table_mask(const Params &p, int a) {
  if (a >= p.R) {
    const int rem = p.P - (a - p.R) * kSlots;
    return rem >= kSlots ? ~0ull : ((1ull << rem) - 1ull);
  }
  return p.region_mask[a % p.R_f];
}
__device__ __forceinline__ long long table_token(const Params &p, int a, int j) {
  if (a >= p.R) return (long long)(a - p.R) * kSlots + j;
  const int t = a / p.R_f, r = a - t * p.R_f;
  return p.P + (long long)t * (p.Hg * p.Wg) + p.region_cell[r * kSlots + j];
}

struct StreamInfo {
  int a;         // query block, or -1
  int n4, n48;   // end of the NVFP4 segment, end of the INT8 segment (list positions)
  int L;
  const uint16_t *ids;
  __device__ __forceinline__ int tier(int i) const { return i < n4 ? 0 : (i < n48 ? 1 : 2); }
};

// Per-row budgets (ROW scope) give every video row the same bounds and a fixed place in the id array, so that nothing has to
// be read before the ids; in HEAD scope (ORDERED) the bounds are the counts that came with the list.
template <bool ORDERED> __device__ __forceinline__ StreamInfo load_stream(const Params &p, int bh, int a) {
  StreamInfo st;
  st.a = a < p.Rt ? a : -1;
  st.n4 = st.n48 = st.L = 0;
  st.ids = nullptr;
  if (a < p.Rt) {
    int4 c;
    if (ORDERED) c = *reinterpret_cast<const int4 *>(p.counts + ((size_t)bh * p.Rt + a) * 4);
    else if (a < p.R) c = make_int4((int)p.quota[0], (int)p.quota[1], (int)p.quota[2] + p.Rp, a * p.row_stride);
    else c = make_int4(0, 0, p.Rt, p.R * p.row_stride + (a - p.R) * ((p.Rt + 7) / 8 * 8));  // a prefix row keeps every block
    st.n4 = c.x; st.n48 = c.x + c.y; st.L = c.x + c.y + c.z;
    st.ids = p.ids + (size_t)bh * p.ids_per_head + c.w;
  }
  return st;
}

// ORDERED: the CTA's two query blocks come from the scheduling order of the head (rows of unequal length, HEAD scope);
// otherwise they are blocks 2p and 2p+1 (per-row budgets: every row has the same length, the order is the identity).
// FP4: the plan has an NVFP4 tier.  Without one the exponentiate phase keeps the per-pair interleaved form, which is
// the faster one for the 8-bit and bf16 bodies alone (the compiler's schedule of the unrolled softmax body decides).
template <int D, bool ORDERED, bool FP4, bool B16>
__global__ void __launch_bounds__(NT, 1) attention_kernel(Params p, SmemMap sm, __nv_bfloat16 *__restrict__ out) {
  constexpr bool SEGMENTED = B16 && D == 128;
  constexpr int kStepShift = SEGMENTED ? 3 : kShift, kStepMask = (1 << kStepShift) - 1;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint32_t s_tmem_base;
  __shared__ int s_abort;

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction
  const int R = p.R, Rt = p.Rt;
  const bool single = (int)blockIdx.x >= sm.pair_ctas;
  int bh, pr;
  if (single) {
    const int idx = (int)blockIdx.x + (sm.first_single - sm.pair_ctas);
    bh = idx / Rt; pr = idx % Rt;
  } else {
    const int pairs = (Rt + 1) / 2;
    bh = blockIdx.x / pairs; pr = blockIdx.x % pairs;
  }
  __nv_bfloat16 *out_head = out + (size_t)bh * p.Ntot * D;
  grid_wait();
  // this warp's stream and its query block: block 2 pr or 2 pr + 1, or that entry of the scheduling order (equally long rows
  // of the head)
  const int stream = warp < kSoftmaxWarps ? (warp & 3) >> 1 : (warp < kMmaWarp0 ? (warp - kSoftmaxWarps) >> 2 : warp & 1);
  int a = single ? (stream ? Rt : pr) : 2 * pr + stream;
  if (ORDERED) {
    if (a < Rt) a = p.order[(size_t)bh * ((Rt + 1) / 2) * 2 + a];
  }
  StreamInfo S = load_stream<ORDERED>(p, bh, a);
  // the loaders' first ids (for K with their blocks' masks and key scales) and the correction warps' table of query tokens are
  // on their way while the block is set up
  int pre0 = 0, pre1 = 0;
  unsigned long long pre_mask = 0;
  float pre_dk = 0.f;
  if (warp >= kLoadWarp0) {
    if (lane < S.L) pre0 = S.ids[lane];
    if (32 + lane < S.L) pre1 = S.ids[32 + lane];
    if (warp < kLoadWarp0 + 2) {
      const int b = pre0 < Rt ? pre0 : 0;  // (an id beyond the head's blocks is reported by the loader)
      pre_mask = table_mask(p, b);
      if (lane < S.n48 && lane >= S.n4) pre_dk = p.dk8[(size_t)bh * R + b];
    }
  } else if (warp >= kSoftmaxWarps && warp < kMmaWarp0 && (warp & 3) < 2 && S.a >= 0) {
    const int j = (warp & 1) * 32 + lane;
    reinterpret_cast<int *>(smem + sm.tok)[stream * 64 + j] =
        (table_mask(p, S.a) >> j) & 1ull ? (int)table_token(p, S.a, j) : -1;
  }

  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + sm.bars);
  const uint32_t bars0 = tc::smem_u32(bars);
  auto bar = [&](int s, int which) -> uint32_t { return bars0 + (uint32_t)(s * B_COUNT + which) * 8u; };
  float *s_factor = reinterpret_cast<float *>(smem + sm.factor);      // [s][kStepBars][64]
  uint32_t *s_chg = reinterpret_cast<uint32_t *>(smem + sm.chg);      // [s][kStepBars][2]
  uint2 *s_hx = reinterpret_cast<uint2 *>(smem + sm.hx);              // [s][set][64]
  float *s_href = reinterpret_cast<float *>(smem + sm.href);          // [s][set][64]
  float *s_ell = reinterpret_cast<float *>(smem + sm.ell);            // [s][set][64]
  uint2 *s_info = reinterpret_cast<uint2 *>(smem + sm.info);          // [s][kInfoRing]

  for (int k_ = tid; k_ < 2 * kSets * 64; k_ += NT) s_hx[k_] = make_uint2(0u, 0xffffffffu);  // no step has this tag
  if (warp == 0) {
    tc::tmem_alloc(&s_tmem_base, kTmemCols);
    tc::tmem_relinquish();
  }
  if (warp == 1) {
    // arrivals per barrier: 1 (a commit or a copy), but two softmax warps per step (scores in registers, weights written),
    // four correction warps (accumulator rescaled), and two warps of each set for the denominators
#pragma unroll 1
    for (int k = lane; k < 2 * B_COUNT; k += 32) {
      const int b = k % B_COUNT;
      tc::mbar_init(bars0 + (uint32_t)k * 8u, (b >= B_SFREE && b < B_CORROK) ? 2 : ((b >= B_CORROK && b < B_PVDONE) ? 4 : (b == B_ELL ? 2 * kSets : 1)));
    }
    tc::fence_barrier_init();
    if (lane == 0) s_abort = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem_base;
  int *abortp = &s_abort;

  // =========================================================================================== softmax warps
  if (warp < kSoftmaxWarps) {
    reg_inc<88>();
    // The warps w, w+4, w+8, ... share a scheduler and own the same 32 query rows; they take the steps of their sets
    // in turn, one thread per full 64-key row: while one exponentiates and packs its step (special-function bound),
    // the others fetch, mask and reduce later ones.  The only hand-off between them is the running maximum.
    const int s = stream, set = warp >> 2;
    const int r = (warp & 1) * 32 + lane;  // query row inside the stream's block
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const float gqk = p.gscale[bh * 4 + 0] * p.gscale[bh * 4 + 1] * p.scale * kLog2e;
    const float dq8s = (S.a >= 0 && S.a < R && p.tier_active[1]) ? p.dq8[(size_t)bh * R + S.a] * p.scale * kLog2e : 0.f;
    const float c16 = p.scale * kLog2e;
    // What does not change from step to step is computed here and not in the step, whose every instruction is on the chain
    // (with one row per warp loaded at the start: all-4-bit call of 16x48x48 13.75 -> 12.5 ms, 12 heads of 32,760 tokens
    // 3.17 -> 2.92 ms).
    const uint32_t sb = bars0 + (uint32_t)s * (B_COUNT * 8u);
    auto my_bar = [&](int which) -> uint32_t { return sb + (uint32_t)which * 8u; };
    float h_own = -INFINITY, ell = 0.f;  // log2-domain maximum after this warp's last step; its partial denominator
    uint2 *my_hx = s_hx + (s * kSets + set) * 64 + r;                // running maximum after my steps, tagged with the step
    const uint32_t prev_hx = tc::smem_u32(s_hx + (s * kSets + ((set + kSets - 1) % kSets)) * 64 + r);
    uint8_t *const p_row0 = smem + sm.p[s] + r * 16;
    uint8_t *const sf_row0 = smem + sm.sfp[s] + (r & 31) * 16 + (r >> 5) * 4;

    const uint32_t s_col = tmem + lane_addr + col_s(s, set & 1);  // (i and set have the same parity)
    for (int i = set; i < S.L; i += kSets) {
      const int tier = B16 ? S.tier(i) : (FP4 && i < S.n4 ? 0 : 1);
      const int g = SEGMENTED ? i & kStepMask : set;  // barriers, factors, ballots, scale atom
      // the step's P slot, and the product that last used it: step i - 4, or i - 2 in the 16-bit segment of a SEGMENTED plan,
      // where the first steps of every segment also wait for the last product of the segment before, whose slots were cut
      // differently.  (A parity wait for product b must find the barrier's previous use, b - kStepBars, complete: the set's
      // step before, i - 4, has waited for product i - 8 at least, and b - 8 <= i - 9.)
      const int seg0 = tier == 0 ? 0 : (tier == 1 ? S.n4 : S.n48), pm = SEGMENTED && tier == 2 ? 1 : kMask;
      uint8_t *prow = p_row0 + (SEGMENTED ? (set & pm) << (11 + tier) : set * sm.pbytes[0]);
      const int busy = SEGMENTED && i - seg0 <= pm ? seg0 - 1 : i - 1 - pm;
      if (!wait_or_abort(my_bar(B_SREADY + set), (i >> kShift) & 1, abortp)) break;
      tc::fence_after_sync();
      // the step's mask and key scale (written before its K block was requested) are read while the scores load
      const uint2 info = s_info[s * kInfoRing + (i & (kInfoRing - 1))];
      const bool padded = info.y != 0u;
      float coef;
      if (B16 && tier == 2) coef = c16;
      else if (tier == 1) coef = dq8s * __uint_as_float(info.x);
      else coef = gqk;
      float v[64];
      {
        uint32_t a0[16], a1[16], a2[16], a3[16];
        tc::tmem_ld16(s_col, a0);
        tc::tmem_ld16(s_col + 16, a1);
        tc::tmem_ld16(s_col + 32, a2);
        tc::tmem_ld16(s_col + 48, a3);
        tc::wait_ld();
        // int32 accumulators (exact as floats: |S| < 2^22)
        if (tier == 1) {
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            v[c] = (float)(int)a0[c]; v[16 + c] = (float)(int)a1[c];
            v[32 + c] = (float)(int)a2[c]; v[48 + c] = (float)(int)a3[c];
          }
        } else {
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            v[c] = __uint_as_float(a0[c]); v[16 + c] = __uint_as_float(a1[c]);
            v[32 + c] = __uint_as_float(a2[c]); v[48 + c] = __uint_as_float(a3[c]);
          }
        }
      }
      tc::fence_before_sync();
      warp_arrive(my_bar(B_SFREE + (set & 1)));
      // Padding keys take no part: the loader left -inf for them and +inf for the others.  A score that is no number stays one
      // (at a padding key only a query that is not finite makes it one, and then every score of the row is not finite).
      if (padded) {
        const float4 *lim = reinterpret_cast<const float4 *>(smem + sm.lim + (s * kInfoRing + (i & (kInfoRing - 1))) * 256);
#pragma unroll
        for (int c = 0; c < 64; c += 4) {
          const float4 x = lim[c >> 2];
          v[c] = min_nan(v[c], x.x); v[c + 1] = min_nan(v[c + 1], x.y); v[c + 2] = min_nan(v[c + 2], x.z); v[c + 3] = min_nan(v[c + 3], x.w);
        }
      }
      // maxima of the four 16-key groups (pairwise trees), then of the row
      float gm[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) gm[q] = max16(v + q * 16);
      const float pmax = fmaxf(max3(gm[0], gm[1], gm[2]), gm[3]) * coef;  // log2 domain
      // the step's P slot, factors and ballots are free
      if (busy >= 0 && !wait_or_abort(my_bar(B_PVDONE + (SEGMENTED ? busy & kStepMask : set)), (busy >> kStepShift) & 1, abortp)) break;
      // running maximum after step i-1: the thread that owns this row in the previous set leaves it, tagged with its
      // step, in shared memory (one 8-byte store, one 8-byte load: no barrier on this chain)
      float h_prev = -INFINITY;
      if (i > 0) {
        uint2 hv = ld_shared_volatile_v2(prev_hx);
        for (uint32_t spin = 0; hv.y != (uint32_t)(i - 1); ++spin) {
          if ((spin & 1023u) == 1023u && (*(volatile int *)abortp || spin > (1u << 24))) break;
          hv = ld_shared_volatile_v2(prev_hx);
        }
        const bool got = hv.y == (uint32_t)(i - 1);
        if (!__all_sync(0xffffffffu, got)) {
          atomicCAS(abortp, 0, 1 + (int)(my_bar(B_CORROK) & 0xffffu));
          break;
        }
        h_prev = __uint_as_float(hv.x);
      }
      const float m_new = fmaxf(h_prev, pmax);
      *my_hx = make_uint2(__float_as_uint(m_new), (uint32_t)i);
      s_factor[(s * kStepBars + g) * 64 + r] = ex2(h_prev - m_new);  // 0 on the first block (h_prev = -inf)
      const uint32_t moved = __ballot_sync(0xffffffffu, m_new != h_prev);
      if (lane == 0) s_chg[(s * kStepBars + g) * 2 + (warp & 1)] = moved;
      ell *= ex2(h_own - m_new);
      h_own = m_new;

      const uint64_t coef2 = f2(coef, coef);
      if (!FP4 && B16 && tier == 2) {
        const uint64_t bias2 = f2(-m_new, -m_new);
        uint64_t sum2 = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          uint32_t w4[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float t0, t1;
            unf2(fma2(f2(v[c * 8 + 2 * j], v[c * 8 + 2 * j + 1]), coef2, bias2), t0, t1);
            const float w0 = ex2(t0), w1 = ex2(t1);
            sum2 = add2(sum2, f2(w0, w1));
            w4[j] = pack_bf16x2(w0, w1);
          }
          *reinterpret_cast<uint4 *>(prow + c * 1024) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
        }
        float s0, s1;
        unf2(sum2, s0, s1);
        ell += s0 + s1;
      } else if (!FP4) {
        const uint64_t bias2 = f2(kOffsetP8 - m_new, kOffsetP8 - m_new);
        uint64_t sum2 = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t w4[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float t0, t1, t2, t3;
            unf2(fma2(f2(v[c * 16 + 4 * j + 0], v[c * 16 + 4 * j + 1]), coef2, bias2), t0, t1);
            unf2(fma2(f2(v[c * 16 + 4 * j + 2], v[c * 16 + 4 * j + 3]), coef2, bias2), t2, t3);
            const float w0 = ex2(t0), w1 = ex2(t1), w2 = ex2(t2), w3 = ex2(t3);
            sum2 = add2(add2(sum2, f2(w0, w1)), f2(w2, w3));
            const float w[4] = {w0, w1, w2, w3};
            w4[j] = pack_e4m3x4(w);
          }
          *reinterpret_cast<uint4 *>(prow + c * 1024) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
        }
        float s0, s1;
        unf2(sum2, s0, s1);
        ell += kEtaP8 * (s0 + s1);  // the denominator sums the amplified fp32 weights; eta restores the unit
      } else if (tier != 0) {
        // the scores of the row become the exponent arguments, then the weights, in place: all 64 exponentials are
        // issued before any is consumed (the 8-bit path carries the 2^8.807 offset in the exponent)
        const float b = !B16 || tier == 1 ? kOffsetP8 - m_new : -m_new;
        const uint64_t bias2 = f2(b, b);
#pragma unroll
        for (int j = 0; j < 32; ++j) unf2(fma2(f2(v[2 * j], v[2 * j + 1]), coef2, bias2), v[2 * j], v[2 * j + 1]);
#pragma unroll
        for (int j = 0; j < 64; ++j) v[j] = ex2(v[j]);
        uint64_t sum2 = 0;
#pragma unroll
        for (int j = 0; j < 32; j += 2) sum2 = add2(sum2, add2(f2(v[2 * j], v[2 * j + 1]), f2(v[2 * j + 2], v[2 * j + 3])));
        float s0, s1;
        unf2(sum2, s0, s1);
        if (B16 && tier == 2) {
#pragma unroll
          for (int c = 0; c < 8; ++c)
            *reinterpret_cast<uint4 *>(prow + c * 1024) =
                make_uint4(pack_bf16x2(v[c * 8 + 0], v[c * 8 + 1]), pack_bf16x2(v[c * 8 + 2], v[c * 8 + 3]),
                           pack_bf16x2(v[c * 8 + 4], v[c * 8 + 5]), pack_bf16x2(v[c * 8 + 6], v[c * 8 + 7]));
          ell += s0 + s1;
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t w4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              w4[j] = pack_e4m3x4(v + c * 16 + 4 * j);
            *reinterpret_cast<uint4 *>(prow + c * 1024) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
          }
          ell += kEtaP8 * (s0 + s1);  // the denominator sums the amplified fp32 weights; eta restores the unit
        }
      } else {
        // Group scales from each group's largest weight (Eq. "v2-nvfp4-probability"), folded into the exponent:
        // sigma = E4M3(448 * max w); scaled weight u = w * 2688 / sigma = 2^(x - m + log2(2688) - log2(sigma)).
        // The four scale chains run first (interleaved), then the exponentials in batches of 32 that are all issued
        // before any is consumed.
        // A group whose scale code is 0 takes the smallest scale for u: its codes do not matter, the product multiplies
        // them by the stored scale 0, and the denominator gets w = u * sigma / 2688 either way.
        float bb[4], sl[4];
        const uint64_t nm2 = f2(-m_new, -m_new);
        uint32_t sfw[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float x0, x1, s0, s1;
          unf2(fma2(f2(gm[2 * h], gm[2 * h + 1]), coef2, nm2), x0, x1);
          unf2(mul2(f2(ex2(x0), ex2(x1)), f2(448.0f, 448.0f)), x0, x1);
          sfw[h] = pack_e4m3x2(x0, x1);
          decode_e4m3x2(sfw[h], s0, s1);
          s0 = fmaxf(s0, 0.001953125f);
          s1 = fmaxf(s1, 0.001953125f);
          unf2(mul2(f2(s0, s1), f2(1.0f / 2688.0f, 1.0f / 2688.0f)), sl[2 * h], sl[2 * h + 1]);
          // log2(2688) - log2(sigma) - m (log2(2688) = 11.3923...)
          unf2(add2(fma2(f2(lg2(s0), lg2(s1)), f2(-1.0f, -1.0f), f2(11.392317422778762f, 11.392317422778762f)), nm2), bb[2 * h], bb[2 * h + 1]);
        }
        const uint32_t sfword = __byte_perm(sfw[0], sfw[1], 0x5410);
        *reinterpret_cast<uint32_t *>(sf_row0 + g * 512) = sfword;
        {
          // the scores of the row become the exponent arguments, then the scaled weights, in place
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float b = bb[j >> 3];
            unf2(fma2(f2(v[2 * j], v[2 * j + 1]), coef2, f2(b, b)), v[2 * j], v[2 * j + 1]);
          }
#pragma unroll
          for (int j = 0; j < 64; ++j) v[j] = ex2(v[j]);
#pragma unroll
          for (int gp = 0; gp < 2; ++gp) {  // 32 keys = two groups = one 16-byte chunk of the row
            uint32_t cw[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float *x = v + gp * 32 + h * 16;
              const uint64_t sa = add2(f2(x[0], x[1]), f2(x[2], x[3])), sb = add2(f2(x[4], x[5]), f2(x[6], x[7]));
              const uint64_t sc2 = add2(f2(x[8], x[9]), f2(x[10], x[11])), sd = add2(f2(x[12], x[13]), f2(x[14], x[15]));
              float s0, s1;
              unf2(add2(add2(sa, sb), add2(sc2, sd)), s0, s1);
              ell = fmaf(s0 + s1, sl[gp * 2 + h], ell);
              cw[h * 2 + 0] = pack_e2m1x8(x);
              cw[h * 2 + 1] = pack_e2m1x8(x + 8);
            }
            *reinterpret_cast<uint4 *>(prow + gp * 1024) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
          }
        }
      }
      tc::fence_async_smem();
      warp_arrive(my_bar(B_PREADY + g));
    }
    if (S.L > 0) {
      s_ell[(s * kSets + set) * 64 + r] = ell;
      s_href[(s * kSets + set) * 64 + r] = h_own;  // reference of this partial denominator
      warp_arrive(my_bar(B_ELL));
    }
  }
  // =========================================================================================== loader warps
  else {
  reg_dec<40>();
  if (warp >= kLoadWarp0) {
    // Warps kLoadWarp0 + s request the K blocks of stream s (and its Q records), warps kLoadWarp0 + 2 + s its V
    // blocks: a K block is consumed as soon as a score buffer is free, a V block only once the weights of its step
    // are written, several steps later, so the two rings advance independently.
    // Warp-uniform loop.  Lane l holds list entry 32 * batch + l ready for use: the record's address, the valid-key
    // mask and the INT8 key scale; the ids of the next two batches and the scales of the next one are already on
    // their way while a batch is used, so that a step costs a few shuffles and the copy request of one elected lane.
    const int s = stream;
    const bool is_v = warp >= kLoadWarp0 + 2;
    S.n4 = __shfl_sync(0xffffffffu, S.n4, 0);
    S.n48 = __shfl_sync(0xffffffffu, S.n48, 0);
    S.L = __shfl_sync(0xffffffffu, S.L, 0);
    if (S.L > 0) {
      // Q records: of the 4- and the 8-bit segment at once, that of the 16-bit segment when it starts
      auto load_q = [&](int first, int last) {
        if (is_v || !tc::elect_one()) return;
        const int nn[3] = {S.n4, S.n48 - S.n4, S.L - S.n48};
        uint32_t bytes = 0;
        for (int t = first; t <= last; ++t) if (nn[t] > 0) bytes += p.qrec_bytes[t];
        if (bytes == 0) return;
        tc::mbar_arrive_expect_tx(bar(s, B_Q), bytes);
        for (int t = first; t <= last; ++t)
          if (nn[t] > 0)
            tc::bulk_g2s(tc::smem_u32(smem + sm.q[s][t]), p.qrec[t] + ((size_t)bh * rec_blocks(p, t) + S.a) * p.qrec_bytes[t], p.qrec_bytes[t],
                         bar(s, B_Q));
      };
      load_q(0, 1);
      __syncwarp();
      const size_t head_blocks = (size_t)bh * R;
      auto checked = [&](int b) -> int {
        if (b >= Rt) { atomicExch(p.status, kDevBadList); b = 0; }
        return b;
      };
      auto list_id = [&](int idx) -> int { return checked(idx < S.L ? (int)S.ids[idx] : 0); };
      auto key_scale = [&](int idx, int b) -> float {
        return (!is_v && idx < S.L && S.tier(idx) == 1) ? p.dk8[head_blocks + b] : 0.f;
      };
      int nxt_b = checked(pre0), nn_b = checked(pre1);
      float cur_dk = 0.f, nxt_dk = pre_dk;
      unsigned long long cur_mask = 0;
      uint32_t padded_lanes = 0;
      const uint32_t dst = tc::smem_u32(smem) + (is_v ? sm.vring[s] : sm.kring[s]);
      const int b_full = is_v ? B_FULLV : B_FULLK, b_free = is_v ? B_VFREE : B_KFREE;
      const uint32_t stage = is_v ? sm.vstage : sm.kstage, entry = is_v ? sm.ventry : sm.kentry;
      const int depth = is_v ? sm.nv : sm.nk;  // ring entries
      int kk = 0;                              // ring entry
      uint32_t kpar = 1;                       // parity of the consumption that frees the entry
      bool kwrapped = false;                   // ring gone round
      uint32_t q_par = 0;                      // parity of the last request for Q records (one comes before the first wait)
      // lane l holds the record's address, the mask and the key scale of list entry 32 * batch + l
      auto record = [&](int idx, int b) -> unsigned long long {
        const int t = S.tier(idx);
        return reinterpret_cast<unsigned long long>(p.kvrec[t] + ((size_t)bh * rec_blocks(p, t) + b) * p.kvrec_bytes[t] + (is_v ? sm.kbytes[t] : 0u));
      };
      const uint32_t nb0 = is_v ? sm.vbytes[0] : sm.kbytes[0], nb1 = is_v ? sm.vbytes[1] : sm.kbytes[1], nb2 = is_v ? sm.vbytes[2] : sm.kbytes[2];
      uint2 *const infos = s_info + s * kInfoRing;
      unsigned long long cur_rec = 0;
      // The 16-bit segment has a loop of its own where the plan has no 4-bit tier: its blocks come one by one, and in the loop
      // for pairs the second one's instructions cost plans of the 16-bit tier alone 2 % (24 heads of 8,192 tokens at d = 64, 30 %
      // kept: 343 and 336 us).  Beside a 4-bit tier the one loop for both is the faster one, as the code is smaller.
      constexpr bool kOwnLoop = B16 && !FP4;
      bool ok = true;
      int i = 0;
#pragma unroll 1
      while (i < (kOwnLoop ? S.n48 : S.L)) {
        const int src = i & 31;
        const bool two = i + 1 < (B16 ? S.n48 : S.L);
        if (src == 0) {  // next batch: its ids and scales were requested one batch ago
          const int b = nxt_b;
          cur_dk = nxt_dk;
          cur_rec = record(i + lane, b);
          cur_mask = is_v ? ~0ull : (i == 0 ? pre_mask : table_mask(p, b));
          padded_lanes = __ballot_sync(0xffffffffu, cur_mask != ~0ull);
          nxt_b = nn_b;
          nxt_dk = key_scale(i + 32 + lane, nxt_b);
          nn_b = list_id(i + 64 + lane);
        }
        const uint32_t lo0 = __shfl_sync(0xffffffffu, (uint32_t)cur_rec, src), hi0 = __shfl_sync(0xffffffffu, (uint32_t)(cur_rec >> 32), src);
        const uint32_t lo1 = __shfl_sync(0xffffffffu, (uint32_t)cur_rec, src + 1), hi1 = __shfl_sync(0xffffffffu, (uint32_t)(cur_rec >> 32), src + 1);
        const uint32_t n0 = B16 && i >= S.n48 ? nb2 : (FP4 && i < S.n4 ? nb0 : nb1), n1 = !two ? 0u : (FP4 && i + 1 < S.n4 ? nb0 : nb1);
        if (B16 && !kOwnLoop && i == S.n48 && !is_v) {
          // the Q buffer is free once every product of the segments before is done: their last K blocks are consumed
          if (i > 0 && !wait_or_abort(bar(s, B_KFREE) + (uint32_t)(kk == 0 ? depth - 1 : kk - 1) * 8u, kk == 0 ? kpar : kpar ^ 1u, abortp)) break;
          load_q(2, 2);
          __syncwarp();
          q_par = S.n48 > 0;
        }
        if (kwrapped && !(ok = wait_or_abort(bar(s, b_free + kk), kpar, abortp))) break;
        if (!is_v) {
          // the steps' masks and key scales are written before the data the softmax waits for is requested
          const int e = i & (kInfoRing - 1);
          if ((padded_lanes >> src) & (!B16 || two ? 3u : 1u)) {
            float *lim = reinterpret_cast<float *>(smem + sm.lim) + (s * kInfoRing + e) * 64;
#pragma unroll 1
            for (int x = 0; x <= (!B16 || two); ++x) {
              const uint32_t mlo = __shfl_sync(0xffffffffu, (uint32_t)cur_mask, src + x);
              const uint32_t mhi = __shfl_sync(0xffffffffu, (uint32_t)(cur_mask >> 32), src + x);
              lim[x * 64 + lane] = (mlo >> lane) & 1u ? INFINITY : -INFINITY;
              lim[x * 64 + 32 + lane] = (mhi >> lane) & 1u ? INFINITY : -INFINITY;
            }
          }
          if (B16 ? lane == src || (two && lane == src + 1) : (lane & ~1) == src) infos[lane & (kInfoRing - 1)] = make_uint2(__float_as_uint(cur_dk), cur_mask != ~0ull);
          __syncwarp();
        }
        if (tc::elect_one()) {
          const uint32_t full = bar(s, b_full + kk), to = dst + (uint32_t)kk * entry;
          tc::mbar_arrive_expect_tx(full, n0 + n1);
          tc::bulk_g2s(to, reinterpret_cast<const uint8_t *>(((unsigned long long)hi0 << 32) | lo0), n0, full);
          if (n1) tc::bulk_g2s(to + stage, reinterpret_cast<const uint8_t *>(((unsigned long long)hi1 << 32) | lo1), n1, full);
        }
        __syncwarp();
        i += !B16 || two ? 2 : 1;
        if (++kk == depth) { kk = 0; kpar ^= 1u; kwrapped = true; }
      }
      if (kOwnLoop && ok && i < S.L) {  // (the steps are those of the loop above, which compiles to slower code with any of them shared)
        if (!is_v) {
          ok = i == 0 || wait_or_abort(bar(s, B_KFREE) + (uint32_t)(kk == 0 ? depth - 1 : kk - 1) * 8u, kk == 0 ? kpar : kpar ^ 1u, abortp);
          if (ok) {
            load_q(2, 2);
            q_par = S.n48 > 0;
          }
          __syncwarp();
        }
#pragma unroll 1
        for (; ok && i < S.L; ++i) {
          const int src = i & 31;
          if (src == 0) {
            const int b = nxt_b;
            cur_rec = record(i + lane, b);
            cur_mask = is_v ? ~0ull : (i == 0 ? pre_mask : table_mask(p, b));
            padded_lanes = __ballot_sync(0xffffffffu, cur_mask != ~0ull);
            nxt_b = nn_b;
            nn_b = list_id(i + 64 + lane);
          }
          const uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)cur_rec, src), hi = __shfl_sync(0xffffffffu, (uint32_t)(cur_rec >> 32), src);
          if (kwrapped && !wait_or_abort(bar(s, b_free + kk), kpar, abortp)) break;
          if (!is_v) {
            const int e = i & (kInfoRing - 1);
            const bool padded = (padded_lanes >> src) & 1u;
            if (padded) {
              float *lim = reinterpret_cast<float *>(smem + sm.lim) + (s * kInfoRing + e) * 64;
              const uint32_t mlo = __shfl_sync(0xffffffffu, (uint32_t)cur_mask, src), mhi = __shfl_sync(0xffffffffu, (uint32_t)(cur_mask >> 32), src);
              lim[lane] = (mlo >> lane) & 1u ? INFINITY : -INFINITY;
              lim[32 + lane] = (mhi >> lane) & 1u ? INFINITY : -INFINITY;
            }
            if (lane == 0) infos[e] = make_uint2(0u, padded);  // (no key scale in the 16-bit tier)
            __syncwarp();
          }
          if (tc::elect_one()) {
            const uint32_t full = bar(s, b_full + kk);
            tc::mbar_arrive_expect_tx(full, nb2);
            tc::bulk_g2s(dst + (uint32_t)kk * entry, reinterpret_cast<const uint8_t *>(((unsigned long long)hi << 32) | lo), nb2, full);
          }
          __syncwarp();
          if (++kk == depth) { kk = 0; kpar ^= 1u; kwrapped = true; }
        }
      }
      // A block exits only when its copies have landed, also those that nobody waits for any more after a give-up (bounded).
      // Entries before kk were used in this round of the ring, the others in the round before.
      const uint32_t used = kwrapped ? (1u << depth) - 1u : (1u << kk) - 1u;
      const uint32_t par = kpar ? (kwrapped ? ((1u << depth) - 1u) & ~((1u << kk) - 1u) : 0u) : (1u << kk) - 1u;
#pragma unroll 1
      for (int k = 0; k < (is_v ? kMaxV : kMaxK); ++k)
        if ((used >> k) & 1u) tc::mbar_wait(bar(s, b_full + k), (par >> k) & 1u, 1u << 14);
      if (!is_v) tc::mbar_wait(bar(s, B_Q), q_par, 1u << 14);
    }
  }
  // =========================================================================================== MMA warps
  else if (warp >= kMmaWarp0 && warp < kPvWarp0) {
    // The whole warp runs this loop with warp-uniform control flow and values; only the tcgen05 instructions
    // themselves are issued by one elected lane.  (Under a lane-0 branch every descriptor would have to be moved from
    // vector to uniform registers before each issue, which costs more than the MMA itself.)
    const int s = warp - kMmaWarp0;
    S.n4 = __shfl_sync(0xffffffffu, S.n4, 0);
    S.n48 = __shfl_sync(0xffffffffu, S.n48, 0);
    S.L = __shfl_sync(0xffffffffu, S.L, 0);
    if (S.L > 0 && wait_or_abort(bar(s, B_Q), 0, abortp)) {
      // operand descriptors, built once; inside the loop only the 16-byte-unit start address (low bits) moves
      const uint64_t qd0 = tc::smem_desc(tc::smem_u32(smem + sm.q[s][0]) - (s ? 1024u : 0u), 1024, 128);
      const uint64_t qd1 = tc::smem_desc(tc::smem_u32(smem + sm.q[s][1]) - (s ? 1024u : 0u), 1024, 128);
      const uint64_t qd2 = tc::smem_desc(tc::smem_u32(smem + sm.q[s][2]) - (s ? 1024u : 0u), 1024, 128);
      const uint64_t kd0 = tc::smem_desc(tc::smem_u32(smem + sm.kring[s]), 1024, 128);
      const uint64_t ksf0 = tc::smem_desc(tc::smem_u32(smem + sm.kring[s]) + kSlots * D / 2, 128, 128);
      const uint32_t t_sfq = tmem + col_sfq(s), t_sfk = tmem + col_sfk(s);
      if (S.n4 > 0) {  // Q scale factors go to TMEM once; the record carries them for rows 0..63 and again for rows
        if (tc::elect_one()) {  // 64..127, so the same atom serves either stream
#pragma unroll
          for (int k = 0; k < D / 64; ++k)
            tc::tmem_cp_sf(t_sfq + 4 * k, tc::smem_desc(tc::smem_u32(smem + sm.q[s][0]) + kSlots * D / 2 + k * kSfAtomBytes,
                                                         128, 128));
        }
        __syncwarp();
      }
      // the score tiles are double buffered, so Q K^T runs up to two steps ahead of the softmax
      const uint32_t full0 = bar(s, B_FULLK), last = full0 + (uint32_t)sm.nk * 8u, kstep = sm.kstage >> 4, kentry = sm.kentry >> 4;
      uint32_t full = full0, kpar = 0;  // ring entry, parity of its next use
      uint32_t ko = 0, spar = 1;             // its place in the ring; parity of the consumption that frees a score buffer
      auto next_entry = [&]() {
        full += 8u;
        ko += kentry;
        if (full == last) { full = full0; ko = 0; kpar ^= 1u; }
      };
      bool ok = true;
#pragma unroll 1
      for (int j = 0; ok && j < S.n48; j += 2) {
        if (!(ok = wait_or_abort(full, kpar, abortp))) break;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (e == 1 && j + 1 >= S.n48) break;
          if (!(ok = wait_or_abort(bar(s, B_SFREE + e), spar, abortp))) break;
          tc::fence_after_sync();
          const uint32_t d_s = tmem + col_s(s, e);
          const uint32_t kde = ko + (e ? kstep : 0u);
          if (tc::elect_one()) {
            if (!FP4 || j + e >= S.n4) {
#pragma unroll
              for (int ks = 0; ks < D / 32; ++ks) tc::mma_i8(d_s, qd1 + ks * 128, kd0 + kde + ks * 128, tc::idesc_i8(64), ks > 0);
            } else {
              const uint64_t ksf = ksf0 + kde;
#pragma unroll
              for (int k = 0; k < D / 64; ++k) tc::tmem_cp_sf(t_sfk + 4 * k, ksf + k * (kSfAtomBytes >> 4));
#pragma unroll
              for (int ks = 0; ks < D / 64; ++ks)
                tc::mma_nvfp4(d_s, qd0 + ks * 128, kd0 + kde + ks * 128, tc::idesc_nvfp4(64), ks > 0, t_sfq + 4 * ks, t_sfk + 4 * ks);
            }
            tc::mma_commit(bar(s, B_SREADY + e) + (uint32_t)(j & 2) * 8u);
            if (e == 1 || (B16 && j + 1 == S.n48)) tc::mma_commit(full + (B_KFREE - B_FULLK) * 8u);
          }
          __syncwarp();
        }
        spar ^= 1u;
        next_entry();
      }
      if (B16 && ok && S.n48 < S.L && wait_or_abort(bar(s, B_Q), S.n48 > 0 ? 1u : 0u, abortp)) {
#pragma unroll 1
        for (int j = S.n48; j < S.L; ++j) {
          const int g = j & 1;
          if (!wait_or_abort(full, kpar, abortp)) break;
          if (!wait_or_abort(bar(s, B_SFREE + g), ((j >> 1) & 1) ^ 1, abortp)) break;
          tc::fence_after_sync();
          if (tc::elect_one()) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) tc::mma_f16(tmem + col_s(s, g), qd2 + ks * 128, kd0 + ko + ks * 128, tc::idesc_bf16(64), ks > 0);
            tc::mma_commit(bar(s, B_SREADY + (j & kMask)));
            tc::mma_commit(full + (B_KFREE - B_FULLK) * 8u);
          }
          __syncwarp();
          next_entry();
        }
      }
    }
  }
  // =========================================================================================== PV warps
  else if (warp >= kPvWarp0) {
    const int s = stream;
    S.n4 = __shfl_sync(0xffffffffu, S.n4, 0);
    S.n48 = __shfl_sync(0xffffffffu, S.n48, 0);
    S.L = __shfl_sync(0xffffffffu, S.L, 0);
    if (S.L > 0) {
      const uint64_t vd0 = tc::smem_desc(tc::smem_u32(smem + sm.vring[s]), D * 16, 128);
      const uint64_t vsf0 = tc::smem_desc(tc::smem_u32(smem + sm.vring[s]) + D * kSlots / 2, 128, 128);
      const uint64_t pd0 = tc::smem_desc(tc::smem_u32(smem + sm.p[s]), 1024, 128);
      const uint64_t sfpd0 = tc::smem_desc(tc::smem_u32(smem + sm.sfp[s]), 128, 128);
      const uint32_t t_sfv = tmem + col_sfv(s), t_sfp = tmem + col_sfp(s), t_o = tmem + col_o(s);
      const uint32_t full0 = bar(s, B_FULLV), last = full0 + (uint32_t)sm.nv * 8u, vstep = sm.vstage >> 4, ventry = sm.ventry >> 4;
      uint32_t full = full0, vpar = 0, vo = 0;  // ring entry, parity of its next use, its place in the ring
      auto next_entry = [&]() {
        full += 8u;
        vo += ventry;
        if (full == last) { full = full0; vo = 0; vpar ^= 1u; }
      };
      // O^T += V(j)^T P(j)^T, once P(j) is written and the stream's correction warps have rescaled the accumulator where step j
      // asked for it
      bool ok = true;
      uint32_t par = 0;
#pragma unroll 1
      for (int j = 0; ok && j < S.n48; j += 2) {
        if (!(ok = wait_or_abort(full, vpar, abortp))) break;
        const uint32_t g0 = (uint32_t)j & kStepMask;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (e == 1 && j + 1 >= S.n48) break;
          if (!(ok = wait_or_abort(bar(s, B_CORROK + e) + g0 * 8u, par, abortp))) break;
          tc::fence_after_sync();
          const uint32_t ve = vo + (e ? vstep : 0u), acc = (e == 0) ? j > 0 : 1u;
          const bool four = FP4 && j + e < S.n4;
          const uint64_t vd = vd0 + ve;
          const uint64_t pdg = pd0 + (uint64_t)(((g0 & 2u) + e) * (SEGMENTED ? (four ? 128u : 256u) : sm.pbytes[0] >> 4));
          if (tc::elect_one()) {
            if (!four) {
#pragma unroll
              for (int ks = 0; ks < 2; ++ks)
                tc::mma_f8f6f4(t_o, vd + ks * (2 * D), pdg + ks * 128, tc::idesc_e4m3(64), acc | (ks > 0));
            } else {
              tc::tmem_cp_sf(t_sfv, vsf0 + ve);
              tc::tmem_cp_sf(t_sfp, sfpd0 + (uint64_t)((g0 + e) * 32));
              tc::mma_nvfp4(t_o, vd, pdg, tc::idesc_nvfp4(64), acc, t_sfv, t_sfp);
            }
            tc::mma_commit(bar(s, B_PVDONE + e) + g0 * 8u);
            if (e == 1 || (B16 && j + 1 == S.n48)) tc::mma_commit(full + (B_VFREE - B_FULLV) * 8u);
          }
          __syncwarp();
        }
        if (g0 + 2u > (uint32_t)kStepMask) par ^= 1u;
        next_entry();
      }
      if (B16 && ok) {
#pragma unroll 1
        for (int j = S.n48; j < S.L; ++j) {
          const uint32_t g = (uint32_t)j & kStepMask;
          if (!wait_or_abort(full, vpar, abortp)) break;
          if (!wait_or_abort(bar(s, B_CORROK) + g * 8u, (j >> kStepShift) & 1, abortp)) break;
          tc::fence_after_sync();
          const uint64_t vd = vd0 + vo, pdg = pd0 + (uint64_t)((g & (SEGMENTED ? 1u : 3u)) * (sm.pbytes[2] >> 4));
          const uint32_t acc = j > 0;
          if (tc::elect_one()) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              tc::mma_f16(t_o, vd + ks * (2 * D), pdg + ks * 128, tc::idesc_bf16(64), acc | (ks > 0));
            tc::mma_commit(bar(s, B_PVDONE) + g * 8u);
            tc::mma_commit(full + (B_VFREE - B_FULLV) * 8u);
          }
          __syncwarp();
          next_entry();
        }
      }
    }
  }
  // =========================================================================================== correction warps
  else {
    const int s = stream;
    const int cw = (warp - kSoftmaxWarps) & 3;  // lane quarter
    const int ch = cw * 32 + lane;              // channel (TMEM lane)
    const uint32_t lane_addr = (uint32_t)(cw * 32) << 16;
    const float gv = p.gscale[bh * 4 + 2];
    const float dv8 = (p.tier_active[1] && ch < D) ? p.dv8[(size_t)bh * D + ch] : 0.f;
    auto unit_of = [&](int t) -> float {  // common units per accumulator unit, for this thread's channel
      return t == 0 ? __fdiv_rn(gv, 2688.0f) : (t == 1 ? kEtaP8 * dv8 : 1.0f);
    };
    // Every step passes through these warps between the softmax and the product: once P(i) is written they read the
    // step's "maximum moved" ballots and, only if one is set or the segment changes, wait for product i-1 and rescale
    // their lane quarter of the accumulator; then they let product i go.  Most steps move no maximum.
    for (int i = 0; i < S.L; ++i) {
      const int g = i & kStepMask;
      if (!wait_or_abort(bar(s, B_PREADY + g), (i >> kStepShift) & 1, abortp)) break;
      const bool tier_switch = (i == S.n4) || (i == S.n48);
      const uint2 moved = ld_shared_volatile_v2(tc::smem_u32(s_chg + (s * kStepBars + g) * 2));
      if (i == 0 || ((moved.x | moved.y) == 0u && !tier_switch)) {
        if (lane == 0) tc::mbar_arrive(bar(s, B_CORROK + g));
        continue;
      }
      const int tier = S.tier(i);
      // everything that does not need the accumulator comes before the wait for product i-1
      float lane_factor = 1.0f;
      if (tier_switch && ch < D) {
        const float un = unit_of(tier), up = unit_of(S.tier(i - 1));
        lane_factor = un > 0.f ? __fdiv_rn(up, un) : 0.f;
      }
      const float *fac = s_factor + (s * kStepBars + g) * 64;
      // column groups (eight queries each) with a moved maximum; all of them when the segment changes.  Two groups
      // are in flight at a time: their loads are issued together, so a rescale costs one TMEM round trip per pair.
      uint32_t todo = 0xffu;
      if (!tier_switch) {  // a bit per byte that is not zero: into the byte's top bit, then four of them gathered by a product
        const uint32_t nx = (((moved.x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | moved.x) & 0x80808080u;
        const uint32_t ny = (((moved.y & 0x7f7f7f7fu) + 0x7f7f7f7fu) | moved.y) & 0x80808080u;
        todo = ((nx >> 7) * 0x10204080u >> 28) | (((ny >> 7) * 0x10204080u >> 28) << 4);
      }
      if (!wait_or_abort(bar(s, B_PVDONE + ((i - 1) & kStepMask)), ((i - 1) >> kStepShift) & 1, abortp)) break;
      tc::fence_after_sync();
#pragma unroll 1
      while (todo) {
        const int c0 = __ffs(todo) - 1;
        todo &= todo - 1;
        const int c1 = todo ? __ffs(todo) - 1 : -1;
        if (c1 >= 0) todo &= todo - 1;
        uint32_t o0[8], o1[8];
        tc::tmem_ld8(tmem + lane_addr + col_o(s) + c0 * 8, o0);
        if (c1 >= 0) tc::tmem_ld8(tmem + lane_addr + col_o(s) + c1 * 8, o1);
        tc::wait_ld();
        scale8(o0, fac + c0 * 8, lane_factor);
        tc::tmem_st8(tmem + lane_addr + col_o(s) + c0 * 8, o0);
        if (c1 >= 0) {
          scale8(o1, fac + c1 * 8, lane_factor);
          tc::tmem_st8(tmem + lane_addr + col_o(s) + c1 * 8, o1);
        }
      }
      tc::wait_st();
      tc::fence_before_sync();
      warp_arrive(bar(s, B_CORROK + g));
    }
    // ---------------------------------------------------------- epilogue: O = U / l, back to raster order
    if (S.a >= 0) {
      bool ok = S.L > 0 && !*(volatile int *)abortp;
      if (ok) ok = wait_or_abort(bar(s, B_ELL), 0, abortp);
      if (ok) ok = wait_or_abort(bar(s, B_PVDONE + ((S.L - 1) & kStepMask)), ((S.L - 1) >> kStepShift) & 1, abortp);
      const int ltid = tid - (kSoftmaxWarps + 4 * s) * 32;  // thread index inside the stream's correction group
      float *s_inv = s_factor + (s * kStepBars) * 64;        // 1 / l per query (the factors are no longer needed)
      const int *s_tok = reinterpret_cast<const int *>(smem + sm.tok) + s * 64;
      if (ltid < 64) {
        // the sets of a row kept partial denominators relative to their own last maximum (a set without a step has ell = 0
        // and reference -inf); rows without a retained key return zero (App. C.1)
        float l = 0.f;
        if (ok) {
          float hf = -INFINITY;
#pragma unroll
          for (int k = 0; k < kSets; ++k) hf = fmaxf(hf, s_href[(s * kSets + k) * 64 + ltid]);
#pragma unroll
          for (int k = 0; k < kSets; ++k) {
            const float lk = s_ell[(s * kSets + k) * 64 + ltid];
            if (lk > 0.f) l += lk * ex2(s_href[(s * kSets + k) * 64 + ltid] - hf);
          }
        }
        s_inv[ltid] = l > 0.f ? __fdiv_rn(1.0f, l) : 0.f;
      }
      if (s == 0) asm volatile("bar.sync 1, 128;" ::: "memory"); else asm volatile("bar.sync 2, 128;" ::: "memory");
      if ((ok || S.L == 0) && cw * 32 < D) {
        tc::fence_after_sync();
        const float unit = ok ? unit_of(S.tier(S.L - 1)) : 0.f;
        uint32_t *out_ch = reinterpret_cast<uint32_t *>(out_head + (ch & ~1));
#pragma unroll 1
        for (int c = 0; c < 8; ++c) {
          uint32_t o[8];
          tc::tmem_ld8(tmem + lane_addr + col_o(s) + c * 8, o);
          tc::wait_ld();
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            // lanes 2x and 2x+1 hold neighbouring channels: after one exchange the even lane writes both of query j, the odd
            // lane both of query j + 1 (64 contiguous bytes per query and warp, no staging tile, no barrier)
            const float2 inv = *reinterpret_cast<const float2 *>(s_inv + c * 8 + j);
            const float x = inv.x > 0.f ? __uint_as_float(o[j]) * unit * inv.x : 0.f;
            const float y = inv.y > 0.f ? __uint_as_float(o[j + 1]) * unit * inv.y : 0.f;
            const float got = __shfl_xor_sync(0xffffffffu, (lane & 1) ? x : y, 1);
            const uint32_t word = (lane & 1) ? pack_bf16x2(got, y) : pack_bf16x2(x, got);
            const int tok = s_tok[c * 8 + j + (lane & 1)];
            if (tok >= 0) out_ch[(size_t)tok * (D / 2)] = word;
          }
        }
      }
    }
  }

  }  // warps without a score row

  tc::fence_before_sync();
  __syncthreads();
  if (s_abort && tid == 0) {
    atomicExch(p.status, kDevTimeout);
    atomicCAS(p.status + 1, 0, s_abort - 1 - (int)(tc::smem_u32(bars) & 0xffff));  // byte offset of the stuck barrier
  }
  if (warp == 0) tc::tmem_dealloc(tmem, kTmemCols);
}

// Failure-path probe: one warp waits, through the very wait the attention kernel uses, on an mbarrier that nothing
// ever completes.  The wait gives up after `limit` cycles, the kernel records the same status the attention kernel
// would (timeout + the barrier's offset) and returns normally: no trap, no endless loop, the context stays usable.
__global__ void bounded_wait_probe_kernel(int *status, uint32_t limit) {
  __shared__ uint64_t never;
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&never), 1);
    tc::fence_barrier_init();
    s_abort = 0;
  }
  __syncthreads();
  const bool ok = wait_or_abort(tc::smem_u32(&never), 0, &s_abort, limit);
  __syncthreads();
  if (threadIdx.x == 0 && (!ok || s_abort)) {
    atomicExch(status, kDevTimeout);
    atomicCAS(status + 1, 0, s_abort - 1);
  }
}

}  // namespace

cudaError_t launch_bounded_wait_probe(int *status, long long limit_cycles, cudaStream_t st) {
  bounded_wait_probe_kernel<<<1, 32, 0, st>>>(status, (uint32_t)limit_cycles);  // 1 .. 2e9: well inside the 32-bit clock's range
  return cudaGetLastError();
}

cudaError_t launch_attention(const Params &p, __nv_bfloat16 *out, cudaStream_t st, int *launches) {
  const bool b16 = p.tier_active[2] != 0;
  const SmemMap sm = make_smem_map(p, b16 && p.d == 128);
  if (!sm.fits) return cudaErrorInvalidConfiguration;
  cudaError_t e;
  const int grid = sm.pair_ctas + p.BH * p.Rt - sm.first_single;
  auto launch = [&](auto kernel) -> cudaError_t {
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm.total);
    if (err != cudaSuccess) return err;
    return launch_chained(kernel, grid, NT, sm.total, st, p, sm, out);
  };
  const bool ordered = p.rank_scope != 0, fp4 = p.tier_active[0] != 0;
  auto pick = [&](auto dtag, auto stag) -> cudaError_t {
    constexpr int D = decltype(dtag)::value;
    constexpr bool S = decltype(stag)::value;
    return ordered ? (fp4 ? launch(attention_kernel<D, true, true, S>) : launch(attention_kernel<D, true, false, S>))
                   : (fp4 ? launch(attention_kernel<D, false, true, S>) : launch(attention_kernel<D, false, false, S>));
  };
  using I64 = std::integral_constant<int, 64>;
  using I128 = std::integral_constant<int, 128>;
  if (p.d == 128) e = b16 ? pick(I128{}, std::true_type{}) : pick(I128{}, std::false_type{});
  else e = b16 ? pick(I64{}, std::true_type{}) : pick(I64{}, std::false_type{});
  *launches += 1;
  return e;
}

}  // namespace da2

