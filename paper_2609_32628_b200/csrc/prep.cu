// Kernel 3: fused operand preparation.  One pass over Q, K, V reorders every 8 x 8 spatial tile into a contiguous
// block and quantises it to each active format (App. C.3), writing the result directly as the shared-memory image
// the attention kernel streams in (K-major 8 x 16-byte core matrices, V already transposed to [channel][key slot],
// scale factors in the layout the block-scaled tensor-core instruction reads) -- see da2.h for the record layout.
//   INT8  Q/K : one fp32 scale per block, delta = amax/127 + 1e-7, round half away from zero
//   E4M3  V   : per-(head, channel) scale delta_c = max|V_c| / 2.25
//   NVFP4 Q/K : E2M1 with one E4M3 scale per 16 channels; V: per 16 key slots of a channel; per-head scale g_X
//   BF16      : the stored values, reordered only
// Every fp32 operation below is a single correctly rounded operation in the order the format definition gives, so
// codes and scales are reproducible bit for bit.  Reads 3*64*d*2 bytes per block, writes the records.
// HBM would allow it in half the time it takes: what bounds it is the integer and conversion work per element.  So every
// thread takes its 32 channels of a row (Q, K) or 16 slots of two channels (V) out of shared memory once and makes the
// codes of all formats from those registers, in packed pairs where an instruction for pairs exists, and the block needs
// two barriers in all.
// Measured: 40 heads x 75,600 tokens (4.31 GB read and written) 1.41 -> 1.08 ms, 4.0 TB/s; 24 heads x 8,192 tokens 95 -> 73 us
// (before: a thread per 16 channels and format, quotients and casts one by one, a barrier per format); 12 heads x 32,760 tokens
// 166 us (176 with the maxima taken on masked magnitudes as integers, which also let a NaN win).
#include <cuda_fp8.h>

#include "da2_internal.cuh"

namespace da2 {

namespace {

constexpr int NT = 256;

// round half away from zero for |x| < 2^23: adding the largest float below one half (with the sign of x) and truncating
// gives the same integer as roundf for every x in that range (the sum can only round up to the next integer when x
// is at least one half above the integer below it)
__device__ __forceinline__ int round_half_away(float x) { return __float2int_rz(__fadd_rn(x, copysignf(0x1.fffffep-2f, x))); }

__device__ __forceinline__ uint32_t cast_e4m3(float x) {
  return (uint32_t)__nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
}
__device__ __forceinline__ float decode_e4m3(uint32_t c) {
  const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)c, __NV_E4M3);
  return __half2float(*reinterpret_cast<const __half *>(&h));
}
// four ints -> four int8 codes (saturating; the first in the low bits)
__device__ __forceinline__ uint32_t pack_s8x4(int c0, int c1, int c2, int c3) {
  uint32_t r;
  asm("{ .reg .b32 t; cvt.pack.sat.s8.s32.b32 t, %4, %3, 0; cvt.pack.sat.s8.s32.b32 %0, %2, %1, t; }"
      : "=r"(r)
      : "r"(c0), "r"(c1), "r"(c2), "r"(c3));
  return r;
}

// Correctly rounded x / d for many x and one positive divisor d, without a division per element: with r = RN(1/d),
// q0 = RN(x r), e = q0 d - x (exact in one fused multiply-add) and q = RN(q0 - e r) is the correctly rounded quotient
// (Markstein's division theorem).  Checked exhaustively on the device against the IEEE division for every bf16 x
// with |x| >= 2^-100 and millions of divisors in [2^-60, 2^60], significands of all ones included.  The callers hand in
// y = -x, so that all three steps are plain multiply-adds on pairs and a zero quotient keeps the sign of x: q0 = y (-r) is
// a zero of the sign of x, e = +0, and q = (+0)(-r) + q0 = q0.  For |x| < 2^-100 the residual can
// underflow; the quotient is then below 2^-40 in magnitude either way and every format here encodes it as a signed
// zero.  Divisors outside [2^-60, 2^60] (or not finite) keep the plain division.  da2_selfcheck_quantiser_arithmetic
// repeats the check with these very functions.
struct Divider {
  float d, r;
  bool fast;
  __device__ __forceinline__ void quick2(float y0, float y1, float &q0, float &q1) const {  // -y0 / d, -y1 / d
    const uint64_t y = f2(y0, y1), nr = f2(-r, -r);
    const uint64_t q = mul2(y, nr);
    const uint64_t e = fma2(q, f2(d, d), y);
    const uint64_t z = fma2(e, nr, q);
    asm("mov.b64 {%0, %1}, %2;" : "=f"(q0), "=f"(q1) : "l"(z));
  }
  __device__ __forceinline__ float exact(float x) const { return __fdiv_rn(x, d); }
  // the quotients of N bf16 pairs given as words with both signs flipped
  template <int N> __device__ __forceinline__ void quotients(const uint32_t (&nw)[N], float (&x)[2 * N]) const {
    if (fast) {
#pragma unroll
      for (int i = 0; i < N; ++i) quick2(bf16lo(nw[i]), bf16hi(nw[i]), x[2 * i], x[2 * i + 1]);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) { x[2 * i] = exact(-bf16lo(nw[i])); x[2 * i + 1] = exact(-bf16hi(nw[i])); }
    }
  }
};
__device__ __forceinline__ Divider make_divider(float d) {
  Divider v;
  v.d = d;
  v.r = __frcp_rn(d);
  v.fast = d >= 8.6736174e-19f && d <= 1.1529215e18f;
  return v;
}

// NVFP4 group of 16 values (Eq. "v2-nvfp4-quantization") given as sign-flipped bf16 words and their largest magnitude:
// returns the E4M3 scale code, writes 8 bytes of codes
__device__ __forceinline__ uint32_t nvfp4_group(const uint32_t (&nw)[8], float gmax, float g6, float g, uint32_t &lo, uint32_t &hi) {
  const uint32_t sc = cast_e4m3(__fdiv_rn(gmax, g6));
  const float sigma = decode_e4m3(sc);
  lo = 0; hi = 0;
  if (sigma == 0.f) return sc;  // a group whose encoded scale is zero is encoded as zero
  float x[16];
  make_divider(__fmul_rn(g, sigma)).quotients(nw, x);
  lo = pack_e2m1x8(x);
  hi = pack_e2m1x8(x + 8);
  return sc;
}

// POOL: the pass also writes the block's average and max descriptors of Q and K (Eq. "v2-descriptors"), so that a
// call whose quantiser statistics are already known reads Q, K, V from HBM exactly once (Sec. 3.3, "Fused
// quantization and reordering").
template <int D, bool POOL>
__global__ void __launch_bounds__(NT, 4) prep_kernel(Params p, const __nv_bfloat16 *__restrict__ q,
                                                  const __nv_bfloat16 *__restrict__ k,
                                                  const __nv_bfloat16 *__restrict__ v, bool beside_draft) {
  extern __shared__ __align__(16) uint8_t smem[];
  // beside_draft: the kernel before is the draft-logits kernel, which this one does not depend on; its blocks have waited
  // for the pooling kernel before they let this kernel start.  So the two overlap, and the wait comes at the end.  What the
  // kernels before it wrote (scales; caller-fixed ones too) is read only after the block has taken the word that the
  // draft-logits kernel publishes.
  grid_trigger();
  if (!beside_draft) grid_wait();
  // Q, K: rows padded by 16 bytes, so that threads that read the same channels of consecutive slots fall on different
  // banks.  V: the 64-byte halves of a 128-byte line are swapped in every other group of 16 rows, so that the two groups a
  // warp reads at a time fall on different banks.
  constexpr int LD = D + 8, ROW = LD * 2;
  uint8_t *tq = smem, *tk = tq + kSlots * ROW, *tv = tk + kSlots * ROW;
  uint8_t *sf_img = tv + kSlots * D * 2;  // scale atoms: Q and K D/64 each, V one
  constexpr int NATOM = D / 64;
  uint8_t *sf_v = sf_img + 2 * NATOM * kSfAtomBytes;
  __shared__ uint32_t s_red[2][NT / 32];
  __shared__ bool s_pooled;

  const int a = blockIdx.x, bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned long long mask = block_valid_mask(p, a);
  const size_t head_off = (size_t)bh * p.Ntot * D;
  const size_t blk = (size_t)bh * p.R + a;        // record index in the quantised tiers (video blocks only)
  const size_t blk16 = (size_t)bh * p.Rt + a;     // record index in the 16-bit tier (video and prefix blocks)
  const bool video = a < p.R;                      // prefix blocks only ever run in the 16-bit tier (App. C.1)
  const bool t4 = p.tier_active[0] && video, t8 = p.tier_active[1] && video, t16 = p.tier_active[2];
  // the regions of the first frame also leave the frame's region table for the attention kernel
  if (bh == 0 && a < p.R_f) {
    if (tid < kSlots) p.region_cell[a * kSlots + tid] = (int)(slot_token(p, a, tid) - p.P);
    if (tid == 0) p.region_mask[a] = mask;
  }

  // stage the three tiles, padding slots as zeros; track max|Q|, max|K| of the block
  {
    constexpr int CPR = D / 8, PASSES = kSlots * CPR / NT;
    const int c8 = tid % CPR;
    uint4 xq[PASSES], xk[PASSES], xv[PASSES];
#pragma unroll
    for (int i = 0; i < PASSES; ++i) {
      const int j = (tid + i * NT) / CPR;
      xq[i] = xk[i] = xv[i] = make_uint4(0, 0, 0, 0);
      if ((mask >> j) & 1ull) {
        const size_t off = head_off + (size_t)slot_token(p, a, j) * D + c8 * 8;
        xq[i] = __ldg(reinterpret_cast<const uint4 *>(q + off));
        xk[i] = __ldg(reinterpret_cast<const uint4 *>(k + off));
        xv[i] = __ldg(reinterpret_cast<const uint4 *>(v + off));
      }
    }
    if (beside_draft && tid == 0) s_pooled = published(p.status + kPooledWord);
    uint32_t aq = 0, ak = 0;
#pragma unroll
    for (int i = 0; i < PASSES; ++i) {
      const int j = (tid + i * NT) / CPR;
      *reinterpret_cast<uint4 *>(tq + j * ROW + c8 * 16) = xq[i];
      *reinterpret_cast<uint4 *>(tk + j * ROW + c8 * 16) = xk[i];
      *reinterpret_cast<uint4 *>(tv + j * (D * 2) + (c8 ^ (((j >> 4) & 1) << 2)) * 16) = xv[i];
      aq = max_abs2(max_abs2(aq, xq[i].x, xq[i].y), xq[i].z, xq[i].w);
      ak = max_abs2(max_abs2(ak, xk[i].x, xk[i].y), xk[i].z, xk[i].w);
    }
    if (t8) {
      aq = magnitudes2(aq);
      ak = magnitudes2(ak);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        aq = __vmaxu2(aq, __shfl_xor_sync(0xffffffffu, aq, o));
        ak = __vmaxu2(ak, __shfl_xor_sync(0xffffffffu, ak, o));
      }
      if (lane == 0) { s_red[0][warp] = aq; s_red[1][warp] = ak; }
    }
    // head_dim 64 leaves the atom of V half empty (channels 64..127)
    if (D == 64 && tid < kSfAtomBytes / 16) *reinterpret_cast<uint4 *>(sf_v + tid * 16) = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  if (beside_draft && !s_pooled) grid_wait();

  if (POOL && video) {
    // one thread per (tensor, channel): sum and maximum over the valid slots of the staged tile.  A sum of at most
    // 64 bf16 values is exact in fp64, so the mean is correctly rounded whatever the order.
    const int n_valid = __popcll(mask);
    for (int idx = tid; idx < 2 * D; idx += NT) {
      const uint8_t *src = (idx < D ? tq : tk) + (idx % D) * 2;
      double sum = 0.0;
      float mx = -INFINITY;
#pragma unroll 8
      for (int j = 0; j < kSlots; ++j) {
        if ((mask >> j) & 1ull) {
          const float x = bf16lo(*reinterpret_cast<const uint16_t *>(src + j * ROW));
          sum += (double)x;
          mx = fmaxf(mx, x);
        }
      }
      const size_t o = blk * D + (idx % D);
      p.desc[idx < D ? 0 : 2][o] = (float)(sum / (double)n_valid);
      p.desc[idx < D ? 1 : 3][o] = mx;
    }
  }

  // ------------------------------------------------------------------ Q and K: 32 channels of one slot per thread
#pragma unroll 1
  for (int u = tid; u < 2 * kSlots * (D / 32); u += NT) {
    const int which = u / (kSlots * (D / 32)), r = u % kSlots, kc = (u / kSlots) % (D / 32);  // 0: Q, 1: K (warp-uniform)
    uint32_t w[16];
    const uint8_t *src = (which ? tk : tq) + r * ROW + kc * 64;
#pragma unroll
    for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4 *>(w + 4 * i) = *reinterpret_cast<const uint4 *>(src + 16 * i);
    if (t16) {  // chunk (c, r): channels c*8.. of slot r
      uint8_t *dst = (which ? p.kvrec[2] + blk16 * p.kvrec_bytes[2] : p.qrec[2] + blk16 * p.qrec_bytes[2]) + (kc * 4 * kSlots + r) * 16;
#pragma unroll
      for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4 *>(dst + i * kSlots * 16) = *reinterpret_cast<const uint4 *>(w + 4 * i);
    }
    if (!t8 && !t4) continue;
    uint32_t nw[2][8];  // signs flipped (see Divider)
#pragma unroll
    for (int i = 0; i < 16; ++i) nw[i >> 3][i & 7] = w[i] ^ 0x80008000u;
    if (t8) {  // chunk (c, r): channels c*16.. of slot r
      uint32_t m = 0;
#pragma unroll
      for (int i = 0; i < NT / 32; ++i) m = __vmaxu2(m, s_red[which][i]);
      const float delta = __fadd_rn(__fdiv_rn(fmaxf(bf16lo(m), bf16hi(m)), 127.0f), 1e-7f);
      if (r == 0 && kc == 0) (which ? p.dk8 : p.dq8)[blk] = delta;
      const Divider dv = make_divider(delta);  // delta >= 1e-7: always in the quick range (unless it is not finite)
      uint8_t *dst = (which ? p.kvrec[1] + blk * p.kvrec_bytes[1] : p.qrec[1] + blk * p.qrec_bytes[1]) + (kc * 2 * kSlots + r) * 16;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float x[16];
        dv.quotients(nw[h], x);
        uint32_t c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          c[i] = pack_s8x4(round_half_away(x[4 * i]), round_half_away(x[4 * i + 1]), round_half_away(x[4 * i + 2]), round_half_away(x[4 * i + 3]));
        *reinterpret_cast<uint4 *>(dst + h * kSlots * 16) = make_uint4(c[0], c[1], c[2], c[3]);
      }
    }
    if (t4) {  // chunk (kc, r): channels kc*32.. of slot r
      const float g = __ldcg(&p.gscale[bh * 4 + which]), g6 = __fmul_rn(6.0f, g);
      uint32_t c[4], sc[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t m = max_abs2(max_abs2(0u, nw[h][0], nw[h][1]), nw[h][2], nw[h][3]);
        m = magnitudes2(max_abs2(max_abs2(m, nw[h][4], nw[h][5]), nw[h][6], nw[h][7]));
        sc[h] = nvfp4_group(nw[h], fmaxf(bf16lo(m), bf16hi(m)), g6, g, c[2 * h], c[2 * h + 1]);
      }
      uint8_t *dst = which ? p.kvrec[0] + blk * p.kvrec_bytes[0] : p.qrec[0] + blk * p.qrec_bytes[0];
      *reinterpret_cast<uint4 *>(dst + (kc * kSlots + r) * 16) = make_uint4(c[0], c[1], c[2], c[3]);
      // rows 0..63 and, duplicated, rows 64..127: the attention kernel places a block's queries in either half
      uint8_t *sfp = sf_img + (which * NATOM + (kc >> 1)) * kSfAtomBytes + (r & 31) * 16 + (r >> 5) * 4 + (kc & 1) * 2;
      const uint16_t two = (uint16_t)(sc[0] | (sc[1] << 8));
      *reinterpret_cast<uint16_t *>(sfp) = two;
      *reinterpret_cast<uint16_t *>(sfp + 8) = two;
    }
  }

  // ------------------------------------------------------------------ V: 16 slots of two channels per thread
  // Lanes 2x and 2x + 1 hold neighbouring groups of 16 slots of the same channels; before a store they exchange halves, so
  // that lane parity stands for the channel and a warp writes 512 contiguous bytes.
  if (tid < 2 * D) {
    const int h = lane & 1, pair = (warp % (D / 32)) * 16 + (lane >> 1), gh = warp / (D / 32), g = gh * 2 + h;
    uint32_t w[16];  // slot g*16 + i: channels 2 * pair (low half) and 2 * pair + 1
    const uint8_t *src = tv + g * 16 * (D * 2) + ((pair >> 2) ^ (h << 2)) * 16 + (pair & 3) * 4;
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = *reinterpret_cast<const uint32_t *>(src + i * (D * 2));
    uint32_t nw[2][8], m = 0;  // per channel, slots in pairs, signs flipped
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      m = max_abs2(m, w[2 * i], w[2 * i + 1]);
      nw[0][i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410) ^ 0x80008000u;
      nw[1][i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632) ^ 0x80008000u;
    }
    m = magnitudes2(m);
    // Hands over the channel the other lane stores; mine[e]: this lane's 16 bytes of channel e.  Afterwards out[0] / out[1]
    // are the 16 bytes of slot groups gh*2 / gh*2 + 1 of channel 2 * pair + h.
    auto exchange = [&](const uint4 (&mine)[2], uint4 (&both)[2]) {
      const uint4 give = h ? mine[0] : mine[1], own = h ? mine[1] : mine[0];
      uint4 got;
      got.x = __shfl_xor_sync(0xffffffffu, give.x, 1); got.y = __shfl_xor_sync(0xffffffffu, give.y, 1);
      got.z = __shfl_xor_sync(0xffffffffu, give.z, 1); got.w = __shfl_xor_sync(0xffffffffu, give.w, 1);
      both[0] = h ? got : own;
      both[1] = h ? own : got;
    };
    const int ch = 2 * pair + h;
    if (t16) {  // chunk (c, ch): slots c*8.. of channel ch
      uint8_t *dst = p.kvrec[2] + blk16 * p.kvrec_bytes[2] + kSlots * D * 2;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint4 mine[2], both[2];
#pragma unroll
        for (int e = 0; e < 2; ++e)
          mine[e] = make_uint4(nw[e][half * 4] ^ 0x80008000u, nw[e][half * 4 + 1] ^ 0x80008000u, nw[e][half * 4 + 2] ^ 0x80008000u,
                               nw[e][half * 4 + 3] ^ 0x80008000u);
        exchange(mine, both);
#pragma unroll
        for (int e = 0; e < 2; ++e) *reinterpret_cast<uint4 *>(dst + (((gh * 2 + e) * 2 + half) * D + ch) * 16) = both[e];
      }
    }
    if (t8) {  // chunk (c, ch): slots c*16.. of channel ch (padding slots hold +0: code 0)
      const float2 dv = __ldcg(reinterpret_cast<const float2 *>(p.dv8 + (size_t)bh * D + 2 * pair));
      uint4 mine[2], both[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float d = e ? dv.y : dv.x;
        mine[e] = make_uint4(0, 0, 0, 0);
        if (d > 0.f) {  // an all-zero channel is encoded as zero
          float x[16];
          make_divider(d).quotients(nw[e], x);
          mine[e] = make_uint4(pack_e4m3x4(x), pack_e4m3x4(x + 4), pack_e4m3x4(x + 8), pack_e4m3x4(x + 12));
        }
      }
      exchange(mine, both);
      uint8_t *dst = p.kvrec[1] + blk * p.kvrec_bytes[1] + kSlots * D + (gh * 2 * D + ch) * 16;
      *reinterpret_cast<uint4 *>(dst) = both[0];
      *reinterpret_cast<uint4 *>(dst + D * 16) = both[1];
    }
    if (t4) {  // chunk (gh, ch): slots gh*32.. of channel ch
      const float gv = __ldcg(&p.gscale[bh * 4 + 2]), g6 = __fmul_rn(6.0f, gv);
      uint2 mine[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int c = 2 * pair + e;
        sf_v[(c & 31) * 16 + (c >> 5) * 4 + g] = (uint8_t)nvfp4_group(nw[e], e ? bf16hi(m) : bf16lo(m), g6, gv, mine[e].x, mine[e].y);
      }
      const uint2 give = h ? mine[0] : mine[1], own = h ? mine[1] : mine[0];
      uint2 got;
      got.x = __shfl_xor_sync(0xffffffffu, give.x, 1); got.y = __shfl_xor_sync(0xffffffffu, give.y, 1);
      *reinterpret_cast<uint4 *>(p.kvrec[0] + blk * p.kvrec_bytes[0] + kSlots * D / 2 + NATOM * kSfAtomBytes + (gh * D + ch) * 16) =
          h ? make_uint4(got.x, got.y, own.x, own.y) : make_uint4(own.x, own.y, got.x, got.y);
    }
  }
  if (t4) {  // the scale atoms: Q, K (behind their images), V (behind its image)
    __syncthreads();
    constexpr int QK_IMG = kSlots * D / 2, ATOM16 = kSfAtomBytes / 16;
    for (int i = tid; i < (2 * NATOM + 1) * ATOM16; i += NT) {
      uint8_t *dst;
      if (i < NATOM * ATOM16) dst = p.qrec[0] + blk * p.qrec_bytes[0] + QK_IMG + i * 16;
      else if (i < 2 * NATOM * ATOM16) dst = p.kvrec[0] + blk * p.kvrec_bytes[0] + QK_IMG + (i - NATOM * ATOM16) * 16;
      else dst = p.kvrec[0] + blk * p.kvrec_bytes[0] + QK_IMG + NATOM * kSfAtomBytes + D * kSlots / 2 + (i - 2 * NATOM * ATOM16) * 16;
      *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(sf_img + i * 16);
    }
  }
  if (beside_draft) grid_wait();
}

// Self-check of Divider::quick2 and round_half_away against the IEEE division and roundf (see da2.h).
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16; x *= 0x7feb352dU; x ^= x >> 15; x *= 0x846ca68bU; x ^= x >> 16;
  return x;
}
__global__ void selfcheck_quotient_kernel(int n_divisors, int all_ones, uint32_t seed, unsigned long long *bad_out) {
  const int di = blockIdx.x * blockDim.x + threadIdx.x;
  if (di >= n_divisors) return;
  const uint32_t h = mix32((uint32_t)di * 2654435761u + seed);
  const uint32_t man = all_ones ? 0x7fffffu : (h & 0x7fffffu);
  const uint32_t ex = 127u - 60u + mix32(h) % 120u;  // binades 2^-60 .. 2^59: inside the quick range
  const Divider div = make_divider(__uint_as_float((ex << 23) | man));
  unsigned long long bad = div.fast ? 0ull : 1ull;
  for (uint32_t b = 0; b < 65536u; ++b) {
    const float x = __uint_as_float(b << 16);
    if (!(fabsf(x) <= 3.0e38f) || (x != 0.f && fabsf(x) < 7.9e-31f)) continue;  // finite, zero or at least 2^-100
    const float ref = div.exact(x);
    if (!(fabsf(ref) < 3.0e38f) || (ref != 0.f && fabsf(ref) < 1e-30f)) continue;  // quotient in the normal range
    float q0, q1;
    div.quick2(-x, x, q0, q1);
    if (__float_as_uint(q0) != __float_as_uint(ref) || __float_as_uint(q1) != (__float_as_uint(ref) ^ 0x80000000u)) ++bad;
  }
  if (bad) atomicAdd(bad_out, bad);
}
__global__ void selfcheck_round_kernel(unsigned long long *bad_out) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long bad = 0;
  for (unsigned long long b = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; b < (1ull << 32); b += stride) {
    const float x = __uint_as_float((uint32_t)b);
    if (!(fabsf(x) < 8388608.0f)) continue;
    if ((int)roundf(x) != round_half_away(x)) ++bad;
  }
  if (bad) atomicAdd(bad_out, bad);
}

}  // namespace

cudaError_t launch_quantiser_selfcheck(int mode, int n_divisors, uint32_t seed, unsigned long long *out, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  if (mode == 2) selfcheck_round_kernel<<<kSms * 8, 256, 0, st>>>(out);
  else selfcheck_quotient_kernel<<<(n_divisors + 127) / 128, 128, 0, st>>>(n_divisors, mode == 1, seed, out);
  return cudaGetLastError();
}

cudaError_t launch_prep(const Params &p, const __nv_bfloat16 *q, const __nv_bfloat16 *k, const __nv_bfloat16 *v,
                        cudaStream_t st, int *launches, bool pool, bool beside_draft) {
  dim3 grid(p.Rt, p.BH);
  const size_t smem = (size_t)kSlots * (2 * (p.d + 8) + p.d) * 2 + (2 * (p.d / 64) + 1) * kSfAtomBytes;
  auto launch = [&](auto kernel) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, grid, NT, smem, st, p, q, k, v, beside_draft);
  };
  cudaError_t e;
  if (p.d == 128) e = pool ? launch(prep_kernel<128, true>) : launch(prep_kernel<128, false>);
  else e = pool ? launch(prep_kernel<64, true>) : launch(prep_kernel<64, false>);
  if (e != cudaSuccess) return e;
  *launches += 1;
  return cudaSuccess;
}

}  // namespace da2
