// Kernel 2, second half: draft attention map, block-importance ranking and per-row block lists.
//   A = (1-lambda) softmax_row(logits_avg) + lambda softmax_row(logits_max)        (Def. 3.1, Eq. "v2-draft")
//   stable descending order of the scores, first quota -> 16-bit, next -> 8-bit, next -> 4-bit, rest skipped;
//   ties go to the lower index (Alg. 1, App. C.1).
// Output per query-block row: key-block ids grouped in execution order NVFP4 | INT8 | BF16 (Sec. 3.3 "Phased
// execution"), ascending inside a group, plus the three counts and the row's offset in its head's id array.
//
// Exact top-k without sorting: for each tier boundary a search on the fp32 bit patterns (scores are non-negative, so bit
// patterns order like values) finds the boundary score and how many entries equal to it are still admitted; equal
// entries are admitted in index order through a prefix count.
//
// ROW scope: one warp per (row, head) does everything while the row fits its registers (rank_warp_kernel), else one CTA.
// HEAD scope (Alg. 1 as printed, one ranking over all R*R pairs of a head): small kernels with per-head histograms in the
// workspace.
#include "da2_internal.cuh"

namespace da2 {

namespace {

constexpr int NT = 256;
constexpr int kRowWarps = 4;  // rows per CTA where a warp takes a row

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ float block_max(float v, float *red) {
  v = warp_max(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = red[0];
#pragma unroll
  for (int w = 1; w < NT / 32; ++w) r = fmaxf(r, red[w]);
  return r;
}
__device__ float block_sum(float v, float *red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = 0.f;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) r += red[w];
  return r;
}

// Draft map row a of head bh into keys[] (fp32 bit patterns, shared memory) and into the global map.
__device__ void draft_map_row(const Params &p, int bh, int a, uint32_t *keys, float *red) {
  const float *l0 = p.logits[0] + ((size_t)bh * p.R + a) * p.R;
  const float *l1 = p.logits[1] + ((size_t)bh * p.R + a) * p.R;
  float *mp = p.map + ((size_t)bh * p.R + a) * p.R;
  float m0 = -INFINITY, m1 = -INFINITY;
  for (int i = threadIdx.x; i < p.R; i += NT) { m0 = fmaxf(m0, l0[i]); m1 = fmaxf(m1, l1[i]); }
  m0 = block_max(m0, red);
  m1 = block_max(m1, red);
  float z0 = 0.f, z1 = 0.f;
  for (int i = threadIdx.x; i < p.R; i += NT) { z0 += expf(l0[i] - m0); z1 += expf(l1[i] - m1); }
  z0 = block_sum(z0, red);
  z1 = block_sum(z1, red);
  const float w0 = 1.0f - p.lambda, w1 = p.lambda;
  for (int i = threadIdx.x; i < p.R; i += NT) {
    const float s = __fmaf_rn(w0, __fdiv_rn(expf(l0[i] - m0), z0), __fmul_rn(w1, __fdiv_rn(expf(l1[i] - m1), z1)));
    keys[i] = __float_as_uint(s);
    mp[i] = s;
  }
  __syncthreads();
}

// One radix-select digit step on a 256-bin histogram (counts of the candidates' current digit), done by warp 0:
// finds the bin holding the need-th largest candidate.  out[0] = bin, out[1] = need minus the count above the bin.
__device__ void pick_bin(const uint32_t *hist, uint32_t need, uint32_t *out) {
  const int lane = threadIdx.x & 31;
  uint32_t c[8], local = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) { c[i] = hist[255 - (lane * 8 + i)]; local += c[i]; }
  uint32_t incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  uint32_t above = incl - local;  // candidates in higher bins than this lane's
  if (above < need && need <= incl) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (need <= above + c[i]) { out[0] = 255 - (lane * 8 + i); out[1] = need - above; break; }
      above += c[i];
    }
  }
}

// c-th largest of keys[0..n) (1 <= c <= n): value bits and how many entries equal to it are admitted.
__device__ void radix_select(const uint32_t *keys, int n, uint32_t c, uint32_t *hist, uint32_t *out,
                             uint32_t *value, uint32_t *take) {
  uint32_t prefix = 0, mask = 0, need = c;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = threadIdx.x; i < 256; i += NT) hist[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += NT) {
      const uint32_t key = keys[i];
      if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) pick_bin(hist, need, out);
    __syncthreads();
    prefix |= out[0] << shift;
    mask |= 255u << shift;
    need = out[1];
    __syncthreads();
  }
  *value = prefix;
  *take = need;
}

// exclusive prefix over the block of NS counters per thread (thread order); totals returned to every thread
template <int NS>
__device__ void block_scan(int (&v)[NS], int (&total)[NS], int *scratch /* NS*NT */) {
  __syncthreads();
#pragma unroll
  for (int s = 0; s < NS; ++s) scratch[s * NT + threadIdx.x] = v[s];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < NS) {
    int *arr = scratch + warp * NT;
    int x[8], local = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) { x[i] = arr[lane * 8 + i]; local += x[i]; }
    int incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    int run = incl - local;
#pragma unroll
    for (int i = 0; i < 8; ++i) { arr[lane * 8 + i] = run; run += x[i]; }
    if (lane == 31) scratch[NS * NT + warp] = incl;
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < NS; ++s) { v[s] = scratch[s * NT + threadIdx.x]; total[s] = scratch[NS * NT + s]; }
  __syncthreads();
}

struct Boundary { uint32_t value, take; };

__device__ __forceinline__ int tier_of(uint32_t key, const Boundary *bd, const int *eqrank) {
  // bd[0]: 16-bit boundary, bd[1]: 8-bit, bd[2]: 4-bit (cumulative).  Returns 2 (16-bit), 1, 0 or -1 (skip).
  if (key > bd[0].value || (key == bd[0].value && (uint32_t)eqrank[0] < bd[0].take)) return 2;
  if (key > bd[1].value || (key == bd[1].value && (uint32_t)eqrank[1] < bd[1].take)) return 1;
  if (key > bd[2].value || (key == bd[2].value && (uint32_t)eqrank[2] < bd[2].take)) return 0;
  return -1;
}

// ------------------------------------------------------------------------------ one warp per row, row in registers
// Lane l holds entries 32 e + l, e < E.  The boundary scores are found by bisection on the bit patterns between the row's
// smallest and largest score; a step costs two instructions per register and one warp reduction, and a step whose count
// hits the quota exactly ends the search (about log2(R) + 2 steps; only ties need all of them).  No barrier and no shared
// memory: the CTA version spends 32 barriers a row, and its 12 histogram passes three times the instructions
// (R = 1260, two boundaries).  Bound by instruction issue: the exponentials of both branches, the bisection, the prefix counts.
// Measured (kernel alone, cold cache): 40 heads, R = 1260 1.05 -> 0.84 ms; 12 heads, R = 588 115 -> 42 us; 24 heads, R = 128
// 38 -> 7 us.
struct Cut { int value, take; };  // admitted: keys above value, and the first `take` keys equal to it

template <int E> __device__ __forceinline__ int count_at_least(const int (&key)[E], int t) {
  int n = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) n += key[e] >= t;
  return (int)__reduce_add_sync(0xffffffffu, (unsigned)n);
}

// Sum of a row, in the order of the CTA version (256 threads, entry i with thread i mod 256), so that the scores, and with
// them the ties among scores that round to the same bits, do not depend on which version ranks a row.
template <int E> __device__ __forceinline__ float row_sum(const float (&x)[E]) {
  float r = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w >= E) break;
    float v = 0.f;
#pragma unroll
    for (int e = w; e < E; e += 8) v += x[e];
    r += warp_sum(v);
  }
  return r;
}

// x / z, correctly rounded, for 0 <= x <= 1 <= z: reciprocal and two corrections by the exact residual (Markstein's theorem:
// the first brings the quotient within one unit in the last place, the second rounds it) where nothing can underflow, else
// the division itself
struct Quotient {
  float z, r;
  __device__ __forceinline__ float of(float x) const {
    if (x < 7.8886091e-31f) return __fdiv_rn(x, z);  // 2^-100
    float q = __fmul_rn(x, r);
    q = __fmaf_rn(__fmaf_rn(-q, z, x), r, q);
    return __fmaf_rn(__fmaf_rn(-q, z, x), r, q);
  }
};

// RANK: ranking and lists (ROW scope); otherwise the draft map rows only
// (20 entries fit the 80 registers of six CTAs an SM; the compiler's own choice is 96, five CTAs: logits and ranking of 12 heads
// at 588 entries 84.6 us instead of 82.5)
template <int E, bool RANK>
__global__ void __launch_bounds__(kRowWarps * 32, E == 20 ? 6 : 0) rank_warp_kernel(Params p) {
  const int lane = threadIdx.x & 31, a = blockIdx.x * kRowWarps + (threadIdx.x >> 5), bh = blockIdx.y, R = p.R;
  grid_trigger();
  grid_wait();
  if (a >= R) return;
  const size_t row = ((size_t)bh * R + a) * R;
  const float *l0 = p.logits[0] + row, *l1 = p.logits[1] + row;
  float x0[E], x1[E];
  float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * 32 + lane;
    x0[e] = i < R ? l0[i] : -INFINITY;
    x1[e] = i < R ? l1[i] : -INFINITY;
  }
#pragma unroll
  for (int e = 0; e < E; ++e) { m0 = fmaxf(m0, x0[e]); m1 = fmaxf(m1, x1[e]); }
  m0 = warp_max(m0);
  m1 = warp_max(m1);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    x0[e] = expf(x0[e] - m0);
    x1[e] = expf(x1[e] - m1);
  }
  const float z0 = row_sum(x0), z1 = row_sum(x1);
  const Quotient d0 = {z0, __frcp_rn(z0)}, d1 = {z1, __frcp_rn(z1)};
  const float w0 = 1.0f - p.lambda, w1 = p.lambda;
  float *mp = p.map + row;
  int key[E];  // scores are non-negative: their bit patterns order like integers; -1 beyond the row
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * 32 + lane;
    const float s = __fmaf_rn(w0, d0.of(x0[e]), __fmul_rn(w1, d1.of(x1[e])));
    key[e] = i < R ? __float_as_int(s) : -1;
    if (i < R) mp[i] = s;
  }
  if (!RANK) return;

  int kmin = 0x7fffffff, kmax = -1;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    kmax = max(kmax, key[e]);
    kmin = min(kmin, key[e] < 0 ? 0x7fffffff : key[e]);
  }
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  Cut cut[3];  // cumulative: 16-bit, 16 + 8, 16 + 8 + 4
  // Keys >= top: `above` of them, fewer than any boundary still to come.  A row of NaN scores (one in a row makes all of them
  // NaN, 0x7fffffff) has no key above: its search is over at once, and the boundary's ties go to the lower indices.
  int cum = 0, top = kmax < 0x7fffffff ? kmax + 1 : kmax, above = 0;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const int c = cum + (int)p.quota[2 - t];
    if (c <= 0) { cut[t].value = 0x7fffffff; cut[t].take = 0; }
    else if (c >= R) { cut[t].value = -1; cut[t].take = 0; }
    else if (t > 0 && c == cum) cut[t] = cut[t - 1];
    else {
      int lo = kmin, hi = top, n_hi = above;  // count(>= lo) >= c > count(>= hi)
      cut[t].take = -1;
#pragma unroll 1
      while (hi - lo > 1) {
        const int mid = lo + ((hi - lo) >> 1);
        const int n = count_at_least(key, mid);
        if (n == c) { cut[t].value = mid - 1; cut[t].take = 0; top = mid; above = n; break; }
        if (n > c) lo = mid; else { hi = mid; n_hi = n; }
      }
      if (cut[t].take < 0) {  // entries tie at the boundary: the lower indices among them
        cut[t].value = lo;
        cut[t].take = c - n_hi;
        top = hi;
        above = n_hi;
      }
    }
    cum = c;
  }

  uint16_t *ids = p.ids + (size_t)bh * p.ids_per_head + (size_t)a * p.row_stride;
  const unsigned below = (1u << lane) - 1u;
  const int k4 = (int)p.quota[0], k8 = (int)p.quota[1], k16 = (int)p.quota[2];
  int pos4 = 0, pos8 = k4, pos16 = k4 + k8;
  int eq0 = 0, eq1 = 0, eq2 = 0;  // keys equal to each boundary so far
  const bool ties = cut[0].take > 0 || cut[1].take > 0 || cut[2].take > 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    bool in16 = key[e] > cut[0].value, in8 = key[e] > cut[1].value, in4 = key[e] > cut[2].value;
    if (ties) {
      const unsigned q0 = __ballot_sync(0xffffffffu, key[e] == cut[0].value), q1 = __ballot_sync(0xffffffffu, key[e] == cut[1].value),
                     q2 = __ballot_sync(0xffffffffu, key[e] == cut[2].value);
      in16 |= ((q0 >> lane) & 1u) && eq0 + __popc(q0 & below) < cut[0].take;
      in8 |= ((q1 >> lane) & 1u) && eq1 + __popc(q1 & below) < cut[1].take;
      in4 |= ((q2 >> lane) & 1u) && eq2 + __popc(q2 & below) < cut[2].take;
      eq0 += __popc(q0); eq1 += __popc(q1); eq2 += __popc(q2);
    }
    const unsigned b16 = __ballot_sync(0xffffffffu, in16), b8 = __ballot_sync(0xffffffffu, in8) & ~b16,
                   b4 = __ballot_sync(0xffffffffu, in4) & ~(b16 | b8);
    const unsigned mine = ((b16 >> lane) & 1u) ? b16 : (((b8 >> lane) & 1u) ? b8 : b4);
    const int base = ((b16 >> lane) & 1u) ? pos16 : (((b8 >> lane) & 1u) ? pos8 : pos4);
    if ((mine >> lane) & 1u) ids[base + __popc(mine & below)] = (uint16_t)(e * 32 + lane);
    pos16 += __popc(b16); pos8 += __popc(b8); pos4 += __popc(b4);
  }
  // prefix interactions lie outside the budget: every video row keeps all prefix blocks, in the 16-bit segment
  for (int j = lane; j < p.Rp; j += 32) ids[k4 + k8 + k16 + j] = (uint16_t)(R + j);
  if (lane == 0)
    *reinterpret_cast<int4 *>(p.counts + ((size_t)bh * p.Rt + a) * 4) = make_int4(k4, k8, k16 + p.Rp, a * p.row_stride);
}

// Launches the kernel whose registers hold a row: entries per lane in steps of 2 up to 16, of 4 up to 32 and of 8 up to 64, so
// that the entries a row pays for beyond its own stay few; false for rows above 2,048 entries.  (With seven sizes, 2 to 64,
// da2_prepare of 12 heads took 261 us at 609 entries and 978 us at 1,400 instead of 236 and 765.)
template <bool RANK, int E = 2> bool launch_rank_warp(const Params &p, cudaStream_t st, cudaError_t *err) {
  if ((p.R + 31) / 32 > E) {
    constexpr int next = E < 16 ? E + 2 : (E < 32 ? E + 4 : E + 8);
    if constexpr (next <= 64) return launch_rank_warp<RANK, next>(p, st, err);
    else return false;
  }
  const dim3 grid((p.R + kRowWarps - 1) / kRowWarps, p.BH);
  // Chained to the kernel before only where the rows are few: there it hides the launch, while waiting blocks of a larger grid
  // hold registers that the kernel before still wants.  da2_prepare chained / not, us: 32 rows of 16 19.2 / 22.0, 512 rows of
  // 128 30.1 / 31.0; 960 rows of 480 55.8 / 51.5, 1,176 rows of 588 61.9 / 58.9 (and 1,280 rows of 160, 49.7 / 50.6, lose it
  // again in the call: 264 / 262).
  const bool chained = (long long)p.R * p.BH <= 512;
  *err = launch(chained, rank_warp_kernel<E, RANK>, grid, kRowWarps * 32, 0, st, p);
  return true;
}

// ---------------------------------------------------------------------------------------------- ROW scope, long rows
__global__ void __launch_bounds__(NT) rank_row_kernel(Params p) {
  extern __shared__ uint32_t dyn[];
  uint32_t *keys = dyn;  // [R]
  __shared__ float red[NT / 32];
  __shared__ uint32_t hist[256];
  __shared__ uint32_t pick[2];
  __shared__ int scratch[3 * NT + 8];
  __shared__ Boundary bd[3];
  const int a = blockIdx.x, bh = blockIdx.y, R = p.R;

  grid_trigger();
  grid_wait();
  draft_map_row(p, bh, a, keys, red);

  // cumulative boundaries: 16-bit, 16+8, 16+8+4
  long long cum = 0;
  for (int t = 0; t < 3; ++t) {
    const long long prev = cum;
    cum += p.quota[2 - t];
    uint32_t value, take;
    if (cum <= 0) { value = 0xffffffffu; take = 0; }
    else if (cum >= R) { value = 0u; take = (uint32_t)R; }
    else if (t > 0 && cum == prev) { value = bd[t - 1].value; take = bd[t - 1].take; }
    else radix_select(keys, R, (uint32_t)cum, hist, pick, &value, &take);
    __syncthreads();
    if (threadIdx.x == 0) { bd[t].value = value; bd[t].take = take; }
    __syncthreads();
  }

  // contiguous chunk per thread so that prefix counts follow index order
  const int per = (R + NT - 1) / NT;
  const int lo = min(R, (int)threadIdx.x * per), hi = min(R, lo + per);
  int eq[3] = {0, 0, 0}, tot[3];
  for (int i = lo; i < hi; ++i) {
    const uint32_t key = keys[i];
#pragma unroll
    for (int t = 0; t < 3; ++t) eq[t] += key == bd[t].value;
  }
  block_scan<3>(eq, tot, scratch);
  int cnt[3] = {0, 0, 0};
  {
    int er[3] = {eq[0], eq[1], eq[2]};
    for (int i = lo; i < hi; ++i) {
      const uint32_t key = keys[i];
      const int tr = tier_of(key, bd, er);
      if (tr >= 0) ++cnt[tr];
#pragma unroll
      for (int t = 0; t < 3; ++t) er[t] += key == bd[t].value;
    }
  }
  int pos[3] = {cnt[0], cnt[1], cnt[2]};
  block_scan<3>(pos, tot, scratch);
  const int stride = p.row_stride;
  uint16_t *ids = p.ids + (size_t)bh * p.ids_per_head + (size_t)a * stride;
  const int base[3] = {0, tot[0], tot[0] + tot[1]};
  {
    int er[3] = {eq[0], eq[1], eq[2]};
    for (int i = lo; i < hi; ++i) {
      const uint32_t key = keys[i];
      const int tr = tier_of(key, bd, er);
      if (tr >= 0) { ids[base[tr] + pos[tr]] = (uint16_t)i; ++pos[tr]; }
#pragma unroll
      for (int t = 0; t < 3; ++t) er[t] += key == bd[t].value;
    }
  }
  // prefix interactions lie outside the budget: every video row keeps all prefix blocks, in the 16-bit segment
  for (int j = threadIdx.x; j < p.Rp; j += NT) ids[tot[0] + tot[1] + tot[2] + j] = (uint16_t)(R + j);
  if (threadIdx.x == 0) {
    int *c = p.counts + ((size_t)bh * p.Rt + a) * 4;
    c[0] = tot[0]; c[1] = tot[1]; c[2] = tot[2] + p.Rp; c[3] = a * stride;
  }
}

// Prefix query rows are not sparse (App. C.1): their list is every block of the head, video and prefix, 16-bit.
__global__ void __launch_bounds__(NT) prefix_rows_kernel(Params p) {
  const int j = blockIdx.x, bh = blockIdx.y, a = p.R + j;
  grid_trigger();
  grid_wait();
  const int pstride = (p.Rt + 7) / 8 * 8;
  const int off = p.R * p.row_stride + j * pstride;
  uint16_t *ids = p.ids + (size_t)bh * p.ids_per_head + off;
  for (int b = threadIdx.x; b < p.Rt; b += NT) ids[b] = (uint16_t)b;
  if (threadIdx.x == 0) {
    int *c = p.counts + ((size_t)bh * p.Rt + a) * 4;
    c[0] = 0; c[1] = 0; c[2] = p.Rt; c[3] = off;
  }
}

__global__ void __launch_bounds__(NT) head_map_kernel(Params p) {
  extern __shared__ uint32_t dyn[];
  __shared__ float red[NT / 32];
  grid_trigger();
  grid_wait();
  draft_map_row(p, blockIdx.y, blockIdx.x, dyn, red);
}

// --------------------------------------------------------------------------------------------- HEAD scope
// Three radix passes (11, 10 and 10 bits of the 31 that a non-negative score has) narrow the three boundary scores of a
// head; the first digit spreads the scores over 8 bins an octave, after it only the entries in a boundary's bin count at
// all.  A CTA counts a share of the head's R*R scores in shared memory, and the last CTA of the head picks the bins.  Then
// a warp per row counts, one CTA per head turns counts into offsets, and a warp per row writes its list.
// Measured with the call around it (12 heads, R = 588, step time): 4.29 -> 3.68 ms, against 4.11 -> 3.47 ms in ROW scope (four
// passes of 8 bits for each boundary in turn and a CTA per row before).
//
// select scratch per head (uint32): [0..11]  (value or prefix, take or need, mode, pad) x 3 boundaries   [12] ticket
//                                   [16..16+2048) histogram of pass 0; [16..16+3072) 3 x 1024 of passes 1 and 2
//                                   [4096..4096+3R) per row and boundary: equal scores -> equal scores in earlier rows
//                                   [4096+3R..4096+6R) higher scores
constexpr int kBins0 = 2048, kBins = 1024;
__device__ __forceinline__ uint32_t *sel_base(const Params &p, int bh) {
  return p.select + (size_t)bh * (4096 + 8 * (size_t)p.R);
}

__global__ void __launch_bounds__(NT) head_init_kernel(Params p) {
  grid_trigger();
  grid_wait();
  uint32_t *s = sel_base(p, blockIdx.x);
  const long long M = (long long)p.R * p.R;
  if (threadIdx.x < 3) {
    long long cum = 0;
    for (int t = 0; t <= (int)threadIdx.x; ++t) cum += p.quota[2 - t];
    uint32_t *b = s + threadIdx.x * 4;
    // mode: 0 = select normally, 1 = nothing admitted, 2 = everything admitted
    const uint32_t mode = cum <= 0 ? 1u : (cum >= M ? 2u : 0u);
    b[0] = mode == 1 ? 0xffffffffu : 0u;
    b[1] = mode == 1 ? 0u : (mode == 2 ? 0xffffffffu : (uint32_t)cum);
    b[2] = mode;
  }
  if (threadIdx.x == 12) s[12] = 0;
  for (int i = threadIdx.x; i < 3 * kBins; i += NT) s[16 + i] = 0;
}

// The bin that holds the need-th largest of a histogram's candidates (N bins, one warp): out[0] = bin, out[1] = need minus
// the count above the bin.
template <int N> __device__ void pick_bin_of(const uint32_t *hist, uint32_t need, uint32_t *out) {
  const int lane = threadIdx.x & 31;
  constexpr int PER = N / 32;
  uint32_t local = 0;
#pragma unroll 8
  for (int i = 0; i < PER; ++i) local += __ldcg(&hist[N - 1 - (lane * PER + i)]);
  uint32_t incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  uint32_t above = incl - local;  // candidates in higher bins than this lane's
  if (above < need && need <= incl) {
    for (int i = 0; i < PER; ++i) {
      const uint32_t c = __ldcg(&hist[N - 1 - (lane * PER + i)]);
      if (need <= above + c) { out[0] = N - 1 - (lane * PER + i); out[1] = need - above; break; }
      above += c;
    }
  }
}

template <int PASS>
__global__ void __launch_bounds__(NT) head_hist_kernel(Params p) {
  constexpr int BINS = PASS == 0 ? kBins0 : 3 * kBins, SHIFT = PASS == 0 ? 20 : (PASS == 1 ? 10 : 0);
  __shared__ uint32_t h[BINS];
  __shared__ uint32_t out[3][2];
  __shared__ bool s_last;
  const int bh = blockIdx.y, tid = threadIdx.x;
  uint32_t *s = sel_base(p, bh);
  for (int i = tid; i < BINS; i += NT) h[i] = 0;
  grid_trigger();
  grid_wait();
  __syncthreads();
  const size_t M = (size_t)p.R * p.R, share = (M + gridDim.x - 1) / gridDim.x;
  const size_t lo = min(M, share * blockIdx.x), hi = min(M, lo + share);
  const uint32_t *keys = reinterpret_cast<const uint32_t *>(p.map) + (size_t)bh * M;
  const uint32_t pf[3] = {s[0] >> (SHIFT + 10), s[4] >> (SHIFT + 10), s[8] >> (SHIFT + 10)};
  const bool on[3] = {s[2] == 0u, s[6] == 0u, s[10] == 0u};
#pragma unroll 4
  for (size_t i = lo + tid; i < hi; i += NT) {
    const uint32_t key = __ldg(&keys[i]);
    if (PASS == 0) {
      atomicAdd(&h[(key >> 20) & (kBins0 - 1)], 1u);  // (a score has no sign)
    } else {
#pragma unroll
      for (int t = 0; t < 3; ++t)
        if (on[t] && (key >> (SHIFT + 10)) == pf[t]) atomicAdd(&h[t * kBins + ((key >> SHIFT) & (kBins - 1))], 1u);
    }
  }
  __syncthreads();
  for (int i = tid; i < BINS; i += NT)
    if (h[i]) atomicAdd(&s[16 + i], h[i]);
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&s[12], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int t = tid >> 5;  // 3 warps, one per boundary
  if (t < 3 && s[t * 4 + 2] == 0u) {
    if (PASS == 0) pick_bin_of<kBins0>(s + 16, s[t * 4 + 1], out[t]);
    else pick_bin_of<kBins>(s + 16 + t * kBins, s[t * 4 + 1], out[t]);
  }
  __syncthreads();
  if (tid < 3 && s[tid * 4 + 2] == 0u) {
    s[tid * 4] |= out[tid][0] << SHIFT;
    s[tid * 4 + 1] = out[tid][1];
  }
  if (tid == 12) s[12] = 0;
  if (PASS < 2)
    for (int i = tid; i < 3 * kBins; i += NT) s[16 + i] = 0;
}

// one warp per row: entries equal to, and above, each boundary score
__global__ void __launch_bounds__(kRowWarps * 32) head_count_kernel(Params p) {
  const int lane = threadIdx.x & 31, a = blockIdx.x * kRowWarps + (threadIdx.x >> 5), bh = blockIdx.y, R = p.R;
  grid_trigger();
  grid_wait();
  if (a >= R) return;
  uint32_t *s = sel_base(p, bh);
  const uint32_t v[3] = {s[0], s[4], s[8]};
  const uint32_t *keys = reinterpret_cast<const uint32_t *>(p.map + ((size_t)bh * R + a) * R);
  int eq[3] = {0, 0, 0}, gt[3] = {0, 0, 0};
#pragma unroll 4
  for (int i = lane; i < R; i += 32) {
    const uint32_t key = keys[i];
#pragma unroll
    for (int t = 0; t < 3; ++t) { eq[t] += key == v[t]; gt[t] += key > v[t]; }
  }
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const unsigned e = __reduce_add_sync(0xffffffffu, (unsigned)eq[t]), g = __reduce_add_sync(0xffffffffu, (unsigned)gt[t]);
    if (lane == 0) { s[4096 + t * R + a] = e; s[4096 + (3 + t) * R + a] = g; }
  }
}

// of `eq` entries equal to a boundary score, after `before` of them in earlier rows, those among the first `take`
__device__ __forceinline__ int admitted(uint32_t take, int before, int eq) {
  return take > (uint32_t)before ? (int)min(take - (uint32_t)before, (uint32_t)eq) : 0;
}

// one CTA per head: counts of a row per tier, its offset, and the equal scores in earlier rows
__global__ void __launch_bounds__(NT) head_offsets_kernel(Params p) {
  __shared__ int scratch[3 * NT + 8];
  const int bh = blockIdx.x, R = p.R;
  grid_trigger();
  grid_wait();
  uint32_t *s = sel_base(p, bh), *eqs = s + 4096, *gts = s + 4096 + 3 * R;
  const uint32_t take[3] = {s[1], s[5], s[9]};
  const int per = (R + NT - 1) / NT, lo = min(R, (int)threadIdx.x * per), hi = min(R, lo + per);
  int eq[3] = {0, 0, 0}, tot[3];
  for (int a = lo; a < hi; ++a)
#pragma unroll
    for (int t = 0; t < 3; ++t) eq[t] += (int)eqs[t * R + a];
  block_scan<3>(eq, tot, scratch);
  int run[3] = {eq[0], eq[1], eq[2]}, len[1] = {0}, total[1];
  for (int a = lo; a < hi; ++a) {
    int c[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int e = (int)eqs[t * R + a];
      c[t] = (int)gts[t * R + a] + admitted(take[t], run[t], e);
      eqs[t * R + a] = (uint32_t)run[t];
      run[t] += e;
    }
    len[0] += c[2];
    *reinterpret_cast<int4 *>(p.counts + ((size_t)bh * R + a) * 4) = make_int4(c[2] - c[1], c[1] - c[0], c[0], 0);
  }
  block_scan<1>(len, total, scratch);
  int off = len[0];
  for (int a = lo; a < hi; ++a) {
    int *c = p.counts + ((size_t)bh * R + a) * 4;
    c[3] = off;
    off += c[0] + c[1] + c[2];
  }
}

// one warp per row: the row's list
__global__ void __launch_bounds__(kRowWarps * 32) head_emit_kernel(Params p) {
  const int lane = threadIdx.x & 31, a = blockIdx.x * kRowWarps + (threadIdx.x >> 5), bh = blockIdx.y, R = p.R;
  grid_trigger();
  grid_wait();
  if (a >= R) return;
  const uint32_t *s = sel_base(p, bh);
  const uint32_t v[3] = {s[0], s[4], s[8]}, take[3] = {s[1], s[5], s[9]};
  int before[3];
#pragma unroll
  for (int t = 0; t < 3; ++t) before[t] = (int)s[4096 + t * R + a];
  const int4 c = *reinterpret_cast<const int4 *>(p.counts + ((size_t)bh * R + a) * 4);
  uint16_t *ids = p.ids + (size_t)bh * p.ids_per_head + c.w;
  int pos4 = 0, pos8 = c.x, pos16 = c.x + c.y;
  const uint32_t *keys = reinterpret_cast<const uint32_t *>(p.map + ((size_t)bh * R + a) * R);
  const unsigned below = (1u << lane) - 1u;
#pragma unroll 4
  for (int i0 = 0; i0 < R; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < R ? keys[i] : 0u;
    bool in[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const unsigned q = __ballot_sync(0xffffffffu, i < R && key == v[t]);
      in[t] = i < R && (key > v[t] || (((q >> lane) & 1u) && (uint32_t)(before[t] + __popc(q & below)) < take[t]));
      before[t] += __popc(q);
    }
    const unsigned b16 = __ballot_sync(0xffffffffu, in[0]), b8 = __ballot_sync(0xffffffffu, in[1]) & ~b16,
                   b4 = __ballot_sync(0xffffffffu, in[2]) & ~(b16 | b8);
    const unsigned mine = ((b16 >> lane) & 1u) ? b16 : (((b8 >> lane) & 1u) ? b8 : b4);
    const int base = ((b16 >> lane) & 1u) ? pos16 : (((b8 >> lane) & 1u) ? pos8 : pos4);
    if ((mine >> lane) & 1u) ids[base + __popc(mine & below)] = (uint16_t)i;
    pos16 += __popc(b16); pos8 += __popc(b8); pos4 += __popc(b4);
  }
}

}  // namespace

// Draft map rows only (softmax of both logit branches and their mixture into p.map); used by callers that want
// the map without the ranking.
cudaError_t launch_map_rows(const Params &p, cudaStream_t st, int *launches) {
  cudaError_t e;
  if (launch_rank_warp<false>(p, st, &e)) {
    *launches += 1;
    return e;
  }
  dim3 grid(p.R, p.BH);
  const size_t smem = (size_t)p.R * sizeof(uint32_t);
  if (smem > 48 * 1024) {
    e = cudaFuncSetAttribute(head_map_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  *launches += 1;
  return launch_chained(head_map_kernel, grid, NT, smem, st, p);
}

cudaError_t launch_rank(const Params &p, cudaStream_t st, int *launches) {
  dim3 grid(p.R, p.BH);
  const size_t smem = (size_t)p.R * sizeof(uint32_t);
  cudaError_t e;
  if (p.rank_scope == DA2_RANK_ROW) {
    if (launch_rank_warp<true>(p, st, &e)) {
      *launches += 1;
      return e;
    }
    if (smem > 48 * 1024) {
      e = cudaFuncSetAttribute(rank_row_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    *launches += 1;
    return launch_chained(rank_row_kernel, grid, NT, smem, st, p);
  }
  e = launch_map_rows(p, st, launches);
  if (e != cudaSuccess) return e;
  // about eight CTAs an SM share the scores of all heads; a share is at least one pass of the CTA's threads
  const long long M = (long long)p.R * p.R, most = (M + 4 * NT - 1) / (4 * NT), fair = (kSms * 8 + p.BH - 1) / p.BH;
  const dim3 shares((unsigned)(most < fair ? most : fair), p.BH), rows((p.R + kRowWarps - 1) / kRowWarps, p.BH);
  auto next = [&](auto kernel, dim3 grid, int threads) {  // enqueued only if the one before was
    if (e == cudaSuccess) e = launch_chained(kernel, grid, threads, 0, st, p);
  };
  next(head_init_kernel, p.BH, NT);
  next(head_hist_kernel<0>, shares, NT);
  next(head_hist_kernel<1>, shares, NT);
  next(head_hist_kernel<2>, shares, NT);
  next(head_count_kernel, rows, kRowWarps * 32);
  next(head_offsets_kernel, p.BH, NT);
  next(head_emit_kernel, rows, kRowWarps * 32);
  *launches += 7;
  return e;
}

// Scheduling order of the query blocks of a head for the attention kernel: by decreasing list length, ties by index.
// O(R^2) comparisons per head on lengths staged in shared memory (R is a few thousand at most).
namespace {
__global__ void __launch_bounds__(256) order_rows_kernel(Params p) {
  extern __shared__ int s_len[];
  const int bh = blockIdx.y, R = p.R, Rp = 2 * ((R + 1) / 2);
  grid_trigger();
  grid_wait();
  const int4 *cnt = reinterpret_cast<const int4 *>(p.counts + (size_t)bh * R * 4);
  for (int a = threadIdx.x; a < R; a += 256) {
    const int4 c = cnt[a];
    s_len[a] = c.x + c.y + c.z;
  }
  __syncthreads();
  uint16_t *ord = p.order + (size_t)bh * Rp;
  if (blockIdx.x == 0 && threadIdx.x == 0 && Rp > R) ord[R] = 0xFFFFu;
  // eight threads per row, each against an eighth of the others
  const int a = blockIdx.x * 32 + (threadIdx.x >> 3), part = threadIdx.x & 7;
  int pos = 0;
  if (a < R) {
    const int la = s_len[a];
#pragma unroll 4
    for (int b = part; b < R; b += 8) {
      const int lb = s_len[b];
      pos += (lb > la) || (lb == la && b < a);
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) pos += __shfl_xor_sync(0xffffffffu, pos, o);
  if (a < R && part == 0) ord[pos] = (uint16_t)a;
}
}  // namespace

cudaError_t launch_prefix_rows(const Params &p, cudaStream_t st, int *launches) {
  if (p.Rp == 0) return cudaSuccess;
  *launches += 1;
  return launch_chained(prefix_rows_kernel, dim3(p.Rp, p.BH), NT, 0, st, p);
}

cudaError_t launch_order(const Params &p, cudaStream_t st, int *launches) {
  const size_t smem = (size_t)p.R * sizeof(int);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(order_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  *launches += 1;
  return launch_chained(order_rows_kernel, dim3((p.R + 31) / 32, p.BH), 256, smem, st, p);
}

}  // namespace da2
