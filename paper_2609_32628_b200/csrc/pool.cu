// Kernel 1: spatial-tile reorder + 2D average / max pooling of Q and K into per-block draft tokens
// (Eq. "v2-descriptors"; padding of ragged edge tiles excluded, App. C.1), plus the statistics the quantisers
// need before they can run: per-head max|Q|, max|K|, max|V| and per-(head, channel) max|V| (App. C.3), and the scales
// derived from them.
//
// A block is an 8 x 8 tile of one frame (or a run of 64 tokens).  A warp walks tokens of one block and every lane owns
// D / 32 channels of it, so a token row is one coalesced load and sums and maxima stay in registers from the first token
// to the last: no shuffles and no shared memory per block.  SPLIT warps share a block (1, 2, 4 or 8 by the waves that the
// blocks make, see launch_pool); only their results are combined.
// HBM-bound: reads Q, K, V once (3*N*d*2 bytes per head), writes 4*R*d*4 bytes.
// Measured: 40 heads x 75,600 tokens (2.42 GB) 0.94 -> 0.41 ms, 5.9 TB/s (before: a CTA per block, sums across threads through
// shared memory, scales in a launch of their own); 24 heads x 8,192 tokens 72 -> 38 us.
//
// Sums are carried in fp64: a sum of at most 64 bf16 values is exact there, so the fp32 descriptor equals the
// correctly rounded mean regardless of summation order.
#include <type_traits>

#include "da2_internal.cuh"

namespace da2 {

namespace {

constexpr int kPoolWarps = 8;
constexpr int kBatch = 8;  // tokens whose loads are in flight together

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ float abs_max_of(uint32_t m) { return fmaxf(bf16lo(m), bf16hi(m)); }

template <int W> struct Row { uint32_t w[W]; };  // one token's channels of a lane
template <int W> __device__ __forceinline__ Row<W> load_row(const uint16_t *p) {
  Row<W> r;
  if (W == 2) {
    const uint2 x = __ldg(reinterpret_cast<const uint2 *>(p));
    r.w[0] = x.x; r.w[W - 1] = x.y;
  } else {
    r.w[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
  }
  return r;
}

template <int D, int SPLIT>
__global__ void __launch_bounds__(kPoolWarps * 32) pool_kernel(Params p, const uint16_t *__restrict__ q, const uint16_t *__restrict__ k,
                                                               const uint16_t *__restrict__ v) {
  constexpr int W = D / 64;                  // words (channel pairs) per lane
  constexpr int BLOCKS = kPoolWarps / SPLIT;  // blocks per CTA
  constexpr int TOK = kSlots / SPLIT;        // tokens per warp
  constexpr int BATCH = kBatch;
  const int bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int a = blockIdx.x * BLOCKS + warp / SPLIT, part = warp % SPLIT;
  const bool live = a < p.R;
  grid_trigger();
  grid_wait();

  double sq[2 * W], sk[2 * W];
  uint32_t mq[W], mk[W], av[W], aq = 0, ak = 0;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    sq[2 * i] = sq[2 * i + 1] = sk[2 * i] = sk[2 * i + 1] = 0.0;
    mq[i] = mk[i] = 0xff80ff80u;  // -inf
    av[i] = 0;
  }
  int n_valid = 0;
  if (live) {
    const unsigned long long mask = block_valid_mask(p, a);
    n_valid = __popcll(mask);
    const size_t base = (size_t)bh * p.Ntot * D + lane * (2 * W);
    // the tokens of a warp: lane l keeps the index of slot part * TOK + l (+ 32), -1 at padding
    int tok[(TOK + 31) / 32];
#pragma unroll
    for (int i = 0; i < (TOK + 31) / 32; ++i) {
      const int j = part * TOK + i * 32 + lane;
      tok[i] = i * 32 + lane < TOK && ((mask >> (j & 63)) & 1ull) ? (int)slot_token(p, a, j) : -1;
    }
#pragma unroll 1
    for (int j0 = 0; j0 < TOK; j0 += BATCH) {
      Row<W> xq[BATCH], xk[BATCH], xv[BATCH];
      int t[BATCH];
#pragma unroll
      for (int i = 0; i < BATCH; ++i) {
        const int src = TOK > 32 && j0 >= 32 ? tok[(TOK + 31) / 32 - 1] : tok[0];
        t[i] = __shfl_sync(0xffffffffu, src, (j0 + i) & 31);
        const size_t off = base + (size_t)max(t[i], 0) * D;
        xq[i] = load_row<W>(q + off);
        xk[i] = load_row<W>(k + off);
        xv[i] = load_row<W>(v + off);
      }
#pragma unroll
      for (int i = 0; i < BATCH; ++i) {
        if (t[i] < 0) continue;  // (uniform) padding takes no part
#pragma unroll
        for (int c = 0; c < W; ++c) {
          sq[2 * c] += (double)bf16lo(xq[i].w[c]); sq[2 * c + 1] += (double)bf16hi(xq[i].w[c]);
          sk[2 * c] += (double)bf16lo(xk[i].w[c]); sk[2 * c + 1] += (double)bf16hi(xk[i].w[c]);
          mq[c] = max_bf16x2(mq[c], xq[i].w[c]);
          mk[c] = max_bf16x2(mk[c], xk[i].w[c]);
          av[c] = max_abs2(av[c], xv[i].w[c]);
        }
        aq = W == 2 ? max_abs2(aq, xq[i].w[0], xq[i].w[W - 1]) : max_abs2(aq, xq[i].w[0]);
        ak = W == 2 ? max_abs2(ak, xk[i].w[0], xk[i].w[W - 1]) : max_abs2(ak, xk[i].w[0]);
      }
    }
  }

  __shared__ uint32_t s_av[kPoolWarps][D / 2];
  __shared__ uint32_t s_a[2][kPoolWarps];
  __shared__ int s_last;
  if (SPLIT > 1) {  // the warps of a block hand their sums and maxima to its first warp
    __shared__ double s_sum[2][kPoolWarps][D];
    __shared__ uint32_t s_max[2][kPoolWarps][D / 2];
#pragma unroll
    for (int c = 0; c < W; ++c) {
      s_sum[0][warp][lane * 2 * W + 2 * c] = sq[2 * c]; s_sum[0][warp][lane * 2 * W + 2 * c + 1] = sq[2 * c + 1];
      s_sum[1][warp][lane * 2 * W + 2 * c] = sk[2 * c]; s_sum[1][warp][lane * 2 * W + 2 * c + 1] = sk[2 * c + 1];
      s_max[0][warp][lane * W + c] = mq[c];
      s_max[1][warp][lane * W + c] = mk[c];
    }
    __syncthreads();
    if (part == 0) {
#pragma unroll
      for (int w = 1; w < SPLIT; ++w)
#pragma unroll
        for (int c = 0; c < W; ++c) {
          sq[2 * c] += s_sum[0][warp + w][lane * 2 * W + 2 * c]; sq[2 * c + 1] += s_sum[0][warp + w][lane * 2 * W + 2 * c + 1];
          sk[2 * c] += s_sum[1][warp + w][lane * 2 * W + 2 * c]; sk[2 * c + 1] += s_sum[1][warp + w][lane * 2 * W + 2 * c + 1];
          mq[c] = max_bf16x2(mq[c], s_max[0][warp + w][lane * W + c]);
          mk[c] = max_bf16x2(mk[c], s_max[1][warp + w][lane * W + c]);
        }
    }
  }
  if (live && part == 0) {
    const size_t o = ((size_t)bh * p.R + a) * D + lane * 2 * W;
    const double n = (double)n_valid;
#pragma unroll
    for (int c = 0; c < W; ++c) {
      *reinterpret_cast<float2 *>(p.desc[0] + o + 2 * c) = make_float2((float)(sq[2 * c] / n), (float)(sq[2 * c + 1] / n));
      *reinterpret_cast<float2 *>(p.desc[1] + o + 2 * c) = make_float2(bf16lo(mq[c]), bf16hi(mq[c]));
      *reinterpret_cast<float2 *>(p.desc[2] + o + 2 * c) = make_float2((float)(sk[2 * c] / n), (float)(sk[2 * c + 1] / n));
      *reinterpret_cast<float2 *>(p.desc[3] + o + 2 * c) = make_float2(bf16lo(mk[c]), bf16hi(mk[c]));
    }
  }
  // statistics of the head: combined over the CTA first, then one atomic per channel (non-negative floats order like
  // their bit patterns)
#pragma unroll
  for (int c = 0; c < W; ++c) s_av[warp][lane * W + c] = magnitudes2(av[c]);
  aq = magnitudes2(aq);
  ak = magnitudes2(ak);
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    aq = __vmaxu2(aq, __shfl_xor_sync(0xffffffffu, aq, off));
    ak = __vmaxu2(ak, __shfl_xor_sync(0xffffffffu, ak, off));
  }
  if (lane == 0) { s_a[0][warp] = aq; s_a[1][warp] = ak; }
  __syncthreads();
  if (tid < D / 2) {
    uint32_t m = 0;
#pragma unroll
    for (int w = 0; w < kPoolWarps; ++w) m = __vmaxu2(m, s_av[w][tid]);
    atomicMax(&p.vmax[(size_t)bh * D + 2 * tid], m << 16);
    atomicMax(&p.vmax[(size_t)bh * D + 2 * tid + 1], m & 0xffff0000u);
    // head maximum of |V| from the channel maxima: reduce within the warp first
    float hv = abs_max_of(m);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) hv = fmaxf(hv, __shfl_xor_sync(0xffffffffu, hv, off));
    if (lane == 0) atomicMax(&p.amax[bh * 4 + 2], __float_as_uint(hv));
  } else if (tid >= 128 && tid < 130) {
    uint32_t m = 0;
#pragma unroll
    for (int w = 0; w < kPoolWarps; ++w) m = __vmaxu2(m, s_a[tid - 128][w]);
    atomicMax(&p.amax[bh * 4 + tid - 128], __float_as_uint(abs_max_of(m)));
  }
  // the last CTA of the head derives the scales (App. C.3): NVFP4 per-tensor scale g_X = amax_X / 2688 (1 for an all-zero
  // head), and the E4M3 per-channel value scale delta_c = max_v |V_vc| / 2.25 (0 marks an all-zero channel)
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&p.amax[bh * 4 + 3], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (tid < D)
    p.dv8[(size_t)bh * D + tid] = __fdiv_rn(__uint_as_float(__ldcg(&p.vmax[(size_t)bh * D + tid])), 2.25f);
  if (tid < 3) {
    const float am = __uint_as_float(__ldcg(&p.amax[bh * 4 + tid]));
    p.gscale[bh * 4 + tid] = am > 0.f ? __fdiv_rn(am, 2688.0f) : 1.0f;
  }
}

}  // namespace

cudaError_t launch_pool(const Params &p, const __nv_bfloat16 *q, const __nv_bfloat16 *k, const __nv_bfloat16 *v,
                        cudaStream_t st, int *launches) {
  // Warps per block: the number with the shortest waves.  An SM holds two CTAs at d = 128 and three at d = 64 (registers); a wave
  // lasts the batches of loads that a warp walks one after the other, and start, combination and atomics cost about three more.
  // So a call whose blocks fit one wave with eight warps each takes eight (it is the latency of one block), and a last wave that
  // would be nearly empty is made shorter.  (With the split by the number of blocks alone, 8 below 592, 4 below 2,368, else 1
  // -> now, us; da2_prepare at d = 128, 128 blocks a head: 8 heads 63.6 -> 59.7, 12 heads 86.4 -> 80.0, 17 heads 113.5 -> 102.5,
  // 24 heads 143.3 -> 138.3; d = 64, 8 heads of 168 blocks 53.2 -> 51.0; whole calls, 4 heads of 128 blocks 97.8 -> 92.0, 5 heads
  // 118.4 -> 115.7, one head of 588 blocks 220.8 -> 215.0.  Eight and four warps at d = 64, da2_refresh_operands: 20 heads of 16
  // blocks 18.8 and 20.6, 24 heads 19.4 and 20.7, 5 heads of 64 blocks 19.1 and 20.6, of 80 blocks 20.5 and 20.7.)
  const long long wave = (long long)kSms * (p.d == 128 ? 2 : 3);
  int split = 1;
  long long best = 0;
  for (int s = 1; s <= kPoolWarps; s *= 2) {
    const long long ctas = (long long)p.BH * ((p.R * s + kPoolWarps - 1) / kPoolWarps);
    const long long cost = (ctas + wave - 1) / wave * (kSlots / kBatch / s + 3);
    if (s == 1 || cost < best) { best = cost; split = s; }
  }
  const dim3 grid((p.R * split + kPoolWarps - 1) / kPoolWarps, p.BH);
  const uint16_t *q16 = reinterpret_cast<const uint16_t *>(q), *k16 = reinterpret_cast<const uint16_t *>(k),
                 *v16 = reinterpret_cast<const uint16_t *>(v);
  auto launch = [&](auto kernel) { return launch_chained(kernel, grid, kPoolWarps * 32, 0, st, p, q16, k16, v16); };
  auto pick = [&](auto dtag) -> cudaError_t {
    constexpr int D = decltype(dtag)::value;
    return split == 1 ? launch(pool_kernel<D, 1>) : (split == 2 ? launch(pool_kernel<D, 2>) : (split == 4 ? launch(pool_kernel<D, 4>) : launch(pool_kernel<D, 8>)));
  };
  const cudaError_t e = p.d == 128 ? pick(std::integral_constant<int, 128>{}) : pick(std::integral_constant<int, 64>{});
  *launches += 1;
  return e;
}

}  // namespace da2
