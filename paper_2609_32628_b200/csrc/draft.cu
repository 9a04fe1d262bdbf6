// Kernel 2, first half: low-resolution draft logits (Def. 3.1, Eq. "v2-draft").
//   logits[0][bh][a][b] = scale * Qavg_a . Kavg_b      logits[1][bh][a][b] = scale * Qmax_a . Kmax_b
// The row softmaxes, their mixture and the ranking follow in rank.cu.
//
// The ranking compares scores to about 1e-5 relative and a softmax turns an ABSOLUTE logit error into a RELATIVE
// score error, so the contraction accumulates in fp64 (products of fp32 descriptors are exact there) and only the
// final logit is rounded to fp32; with large logits (outlier channels) fp32 accumulation alone would already move
// scores by 1e-4.  It is a small GEMM: 4*R*R*d flops per head, against 4*64*64*d flops per retained block pair in
// the attention kernel.
// The plain fp64 pipe sustains about half of what the fp64 tensor-core path does on this part, so the products run as
// mma.sync m8n8k4 (fp64 in, fp64 accumulate): 64 x 64 output tile per CTA of four warps, 32 x 32 per warp (4 x 4
// fragments).  Both operand tiles are requested at once, as fp32 and for all channels (64 KB at d = 128), by asynchronous
// copies in groups of 32 channels: the first products start when the first group is there, and with three CTAs an SM the
// loads of one hide behind the products of the others.  Fragments are widened to fp64 as they are read (8 conversions for
// 16 products of 15 cycles each).  64 x 64 tiles instead of 128 x 64 give small maps (a few hundred blocks, a few heads)
// enough CTAs to fill the GPU evenly.
// Measured: 40 heads, R = 1260 (32.5 GFLOP) 1.29 -> 1.04 ms, 31 TFLOP/s; 12 heads, R = 588 107 -> 87 us.
#include "da2_internal.cuh"

namespace da2 {

namespace {

constexpr int TILE = 64, TK = 32, kChunk = 128;  // channels per copy group, channels staged at a time

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}
__device__ __forceinline__ void copy16(uint32_t dst, const float *src, bool valid) {  // zeros where not valid
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
template <int N> __device__ __forceinline__ void copies_left() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__global__ void __launch_bounds__(128) draft_logits_kernel(Params p) {
  extern __shared__ __align__(16) float dsm[];
  const int d = p.d, ld = min(d, kChunk) + 4;  // row stride = 4 mod 32 words: the 8 rows x 4 channels of a fragment hit 32 banks
  float *As = dsm, *Bs = dsm + TILE * ld;  // [block][channel]
  const int which = blockIdx.z & 1, bh = blockIdx.z >> 1;
  const float *__restrict__ Qd = p.desc[which] + (size_t)bh * p.R * d;       // Qavg or Qmax
  const float *__restrict__ Kd = p.desc[2 + which] + (size_t)bh * p.R * d;   // Kavg or Kmax
  float *__restrict__ out = p.logits[which] + (size_t)bh * p.R * p.R;
  const int a0 = blockIdx.y * TILE, b0 = blockIdx.x * TILE;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t as = (uint32_t)__cvta_generic_to_shared(As), bs = (uint32_t)__cvta_generic_to_shared(Bs);

  const int wm = (warp & 1) * 32, wn = (warp >> 1) * 32;  // warp tile origin inside the CTA tile
  const int fr = lane >> 2, fc = lane & 3;                // fragment row (or column of B) and channel inside a k4 step
  const bool live = a0 + wm < p.R && b0 + wn < p.R;
  double acc[4][4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc[i][j][0] = 0.0; acc[i][j][1] = 0.0; }
  grid_wait();
  if (p.status != nullptr && tid == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) publish(p.status + kPooledWord);
  grid_trigger();  // only now: what runs beside this kernel finds the kernels before it complete (and the word, as a rule, set)
  // 64 rows x 8 quarters of four channels per operand and group: 4 + 4 copies per thread
  const int lc = (tid & 7) * 4, lr = tid >> 3;
  for (int base = 0; base < d; base += kChunk) {
    const int n = min(kChunk, d - base), groups = (n + TK - 1) / TK;
    if (base > 0) __syncthreads();
    for (int g = 0; g < groups; ++g) {
      const int c = g * TK + lc;
      if (c < n) {
#pragma unroll
        for (int i = 0; i < TILE; i += 16) {
          const int a = a0 + lr + i, b = b0 + lr + i;
          copy16(as + ((lr + i) * ld + c) * 4, Qd + (size_t)min(a, p.R - 1) * d + base + c, a < p.R);
          copy16(bs + ((lr + i) * ld + c) * 4, Kd + (size_t)min(b, p.R - 1) * d + base + c, b < p.R);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int g = 0; g < groups; ++g) {
      const int left = groups - 1 - g;
      if (left >= 3) copies_left<3>(); else if (left == 2) copies_left<2>(); else if (left == 1) copies_left<1>(); else copies_left<0>();
      __syncthreads();
      if (!live) continue;
      const int c1 = min(n, (g + 1) * TK);
#pragma unroll 2
      for (int c = g * TK; c < c1; c += 4) {
        double af[4], bf[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) af[i] = (double)As[(wm + i * 8 + fr) * ld + c + fc];
#pragma unroll
        for (int j = 0; j < 4; ++j) bf[j] = (double)Bs[(wn + j * 8 + fr) * ld + c + fc];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) dmma(acc[i][j], af[i], bf[j]);
      }
    }
  }
  if (!live) return;
  // accumulator fragment: row = lane / 4, columns 2 * (lane % 4) and + 1
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = a0 + wm + i * 8 + fr;
    if (a >= p.R) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = b0 + wn + j * 8 + fc * 2;
      if (b < p.R) out[(size_t)a * p.R + b] = (float)((double)p.scale * acc[i][j][0]);
      if (b + 1 < p.R) out[(size_t)a * p.R + b + 1] = (float)((double)p.scale * acc[i][j][1]);
    }
  }
}

}  // namespace

cudaError_t launch_draft(const Params &p, cudaStream_t st, int *launches) {
  const dim3 grid((p.R + TILE - 1) / TILE, (p.R + TILE - 1) / TILE, p.BH * 2);
  // Three CTAs fit an SM, but the kernel starts while the pooling kernel still fills the SMs, and the few CTAs of a small map
  // would be packed three to an SM wherever there is room, to share its fp64 pipe while others stay idle.  So a grid of up to
  // one, or two, CTAs per SM asks for so much shared memory that no more than that fit.  Rows of up to half a tile give a CTA
  // one working warp and the pipe nothing to share.  (da2_prepare, us: 2 heads of 128 blocks 36.8 -> 28.2, 8 heads 59.3 -> 52.5,
  // 12 heads 80.0 -> 76.7, 24 heads 138.1 -> 134.6; d = 64, 8 heads of 168 blocks 50.7 -> 47.5; larger grids as before.)
  // The operand kernel's blocks run beside these CTAs.  Where they are one wave (four an SM), the SMs keep all of their shared
  // memory: set to what a CTA of this kernel needs they take no such block until it has ended, and the last blocks then start
  // late (whole calls, d = 128: 4 heads of 128 blocks 117.8 -> 110.5, 6 heads of 80 95.8 -> 89.9; d = 64: 4 heads of 128 blocks
  // 103.4 -> 98.7).  With more blocks there is a second wave anyway, and the logits are the sooner ready if they have the SM to
  // themselves (6 heads of 128 blocks 154.4, with blocks beside them 156.8).
  const int tiles = 2 * TILE * ((p.d < kChunk ? p.d : kChunk) + 4) * (int)sizeof(float);
  const long long ctas = (long long)grid.x * grid.y * grid.z;
  constexpr int kOne = 116 * 1024, kTwo = 78 * 1024;  // one CTA to an SM's 228 KB, two
  const bool spread = p.R > TILE / 2 && ctas <= 2 * kSms;
  const int smem = !spread ? tiles : (ctas <= kSms ? kOne : kTwo);
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(draft_logits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOne);
    if (e != cudaSuccess) return e;
  }
  *launches += 1;
  return launch(true, spread && (long long)p.BH * p.Rt <= 4 * kSms, draft_logits_kernel, grid, 128, smem, st, p);
}

}  // namespace da2
