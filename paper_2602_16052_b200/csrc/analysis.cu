// Analysis mode: oracle (greedy reconstruction-error) ranking of Eq. 6 and the reconstruction error
// of Section 4.5.  Both work on what an unbudgeted pass of the layer leaves in the workspace: the rows
// y[row(t, a)] = E_i(h_t) of every (token, natural top-k expert) pair, their mixing weights and the
// gather order.
//
// With c_{t,i} = g_i(h_t) E_i(h_t) the objective of Eq. 6 for a set S is
//     sum_t || sum_{j in T_k(h_t) \ S} c_{t,j} ||^2,
// so adding expert i lowers it by
//     gain_i(S) = sum_{t : i in T_k(h_t)} ( 2 * sum_{j in T_k(h_t) \ S} c_{t,j}.c_{t,i}  -  c_{t,i}.c_{t,i} ).
// Everything the greedy loop needs is therefore the k x k Gram matrix of each token's weighted rows.
// Kernel 1 forms the Gram matrices (fp32 inputs, fp64 products and sums, fixed order); kernel 2 runs
// the whole greedy loop in one CTA (fp64, ties -> lower expert index, a fixed summation order).
#include "internal.h"

namespace moespec {

namespace {

constexpr unsigned kFullMask = 0xffffffffu;

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_float(__half v) { return __half2float(v); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    int lo = __double2loint(v), hi = __double2hiint(v);
    lo = __shfl_xor_sync(kFullMask, lo, o);
    hi = __shfl_xor_sync(kFullMask, hi, o);
    v += __hiloint2double(hi, lo);
  }
  return v;
}

// G[t][a][b] = (w_a y_a) . (w_b y_b) for the k slots of token t; slots without a row give zeros.
// One CTA per token.  What bounds it is the conversion of fp32 to fp64 (a product needs two, and they run at a
// fraction of the FMA rate), so a warp takes row a against up to four rows b at a time: five conversions for four
// products instead of eight, and the rows come from L1 after the first read.  Twelve warps are one round of k = 8.
constexpr int kGramThreads = 384, kGramB = 4;

__global__ void __launch_bounds__(kGramThreads) gram_kernel(const float *y, const float *gate_w, const int *tokslot2row,
                                                            double *__restrict__ gram, int *__restrict__ row2slot,
                                                            int d, int k) {
  const int t = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x < k) {
    const int row = tokslot2row[(size_t)t * k + threadIdx.x];
    if (row >= 0) row2slot[row] = threadIdx.x;
  }
  int item = warp;                       // items: (a, group of b), a ascending, k - a rows b = a .. k - 1 in groups
  for (int a = 0; a < k; ++a) {
    const int groups = (k - a + kGramB - 1) / kGramB;
    for (; item < groups; item += kGramThreads / 32) {
      const int b0 = a + item * kGramB;
      const int ra = tokslot2row[(size_t)t * k + a];
      int rb[kGramB];
      double acc[kGramB];
      const float4 *pb[kGramB];
      const float4 *pa = reinterpret_cast<const float4 *>(y + (size_t)max(ra, 0) * d);
#pragma unroll
      for (int q = 0; q < kGramB; ++q) {
        acc[q] = 0.0;
        rb[q] = b0 + q < k ? tokslot2row[(size_t)t * k + b0 + q] : -1;
        pb[q] = rb[q] >= 0 ? reinterpret_cast<const float4 *>(y + (size_t)rb[q] * d) : pa;
      }
      if (ra >= 0)
#pragma unroll 4
        for (int c = lane; c < d / 4; c += 32) {
          const float4 u = pa[c];
          const double ux = (double)u.x, uy = (double)u.y, uz = (double)u.z, uw = (double)u.w;
#pragma unroll
          for (int q = 0; q < kGramB; ++q) {
            const float4 v = pb[q][c];
            acc[q] += ux * (double)v.x;
            acc[q] += uy * (double)v.y;
            acc[q] += uz * (double)v.z;
            acc[q] += uw * (double)v.w;
          }
        }
#pragma unroll
      for (int q = 0; q < kGramB; ++q) {
        const int b = b0 + q;
        if (b >= k) break;                               // the same for the whole warp
        double g = 0.0;
        if (ra >= 0 && rb[q] >= 0)
          g = warp_sum(acc[q]) * ((double)gate_w[(size_t)t * k + a] * (double)gate_w[(size_t)t * k + b]);
        if (lane == 0) {
          gram[((size_t)t * k + a) * k + b] = g;
          gram[((size_t)t * k + b) * k + a] = g;
        }
      }
    }
    item -= groups;
  }
}

// Greedy loop of Eq. 6 in one CTA, for trees that greedy_rows_kernel below does not take.  gain(row) = 2 * sum of the row's Gram entries over the token's experts outside S,
// minus its own: kept per routed row, so that a step recomputes only the rows of tokens that hold the expert just
// picked (the same sum in the same order as from scratch) and otherwise adds up kept numbers.  Eight lanes take one
// expert: they stride its rows in gather order and their partial sums meet in a shuffle tree, the same shape for every
// expert, so identical experts tie exactly.  Every warp then finds the largest gain for itself (ties -> lower index; an
// expert without rows has gain 0) by integer warp reductions of the order-preserving bit pattern.  What bounds a step is
// its chain of dependent loads, additions and barriers, so everything it reads lies in shared memory where it fits (a
// tree of 63 tokens with k = 8 needs 42 KB).  Ranking the first 32 of 64 experts at that size, layer pass included:
// recomputing every row in every step 481 us; keeping row gains 266; eight-lane sums and integer maxima 235; the working
// set in shared memory 227.
constexpr int kGreedyThreads = 512;      // 1024: 9 us a ranking more (barriers), 256: 9 us more (longer sums)

__device__ __forceinline__ double row_gain(const double *gram, const int *assign_idx, int t, int a, int k,
                                           const unsigned char *s_in, int also) {
  const double *G = gram + ((size_t)t * k + a) * k;
  const int *as = assign_idx + (size_t)t * k;
  double cross = 0.0;
  for (int b0 = 0; b0 < k; b0 += 8) {            // the loads of eight terms are in flight together
    int j[8];
    double g[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      j[b] = b0 + b < k ? as[b0 + b] : -1;
      g[b] = b0 + b < k ? G[b0 + b] : 0.0;
    }
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if (j[b] >= 0 && j[b] != also && !s_in[j[b]]) cross += g[b];
  }
  return 2.0 * cross - G[a];
}

// larger double, larger key; a NaN (an expert that overflowed, or one that shares a token with it) is below every number
__device__ __forceinline__ unsigned long long order_bits(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v), size = u & 0x7fffffffffffffffull;
  if (size > 0x7ff0000000000000ull) return 0ull;
  return (u >> 63) && size != 0ull ? ~u : (size | 0x8000000000000000ull);      // -0 and +0 share a key
}

// Bytes of the working set: row gains, Gram matrices, kept experts, rows of the slots, tokens of the rows.
size_t greedy_bytes(int M, int k) { return (size_t)M * k * (8 + 8 * (size_t)k + 4 + 4 + 4); }
constexpr size_t kGreedySmem = 200 * 1024;

// gain_mem: scratch, one double per routed row; used when the working set stays in global memory (in_smem = 0).
__global__ void __launch_bounds__(kGreedyThreads) greedy_kernel(
    const double *gram, const int *assign_idx, const int *offset, const int *perm_row2tok,
    const int *tokslot2row, const int *row2slot, const int *status, double *gain_mem, int M,
    int N, int k, int n_pick, int in_smem, RankingResult res) {
  extern __shared__ double s_work[];
  __shared__ unsigned char s_in[kMaxExperts];
  __shared__ double s_gain[kMaxExperts];
  __shared__ unsigned long long s_key[kMaxExperts];
  __shared__ int s_offset[kMaxExperts + 1];
  __shared__ double s_part[kGreedyThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  for (int i = tid; i < N; i += kGreedyThreads) s_in[i] = 0;
  for (int i = tid; i <= N; i += kGreedyThreads) s_offset[i] = offset[i];
  double *gain = gain_mem;
  const int pairs = M * k;
  if (in_smem) {
    gain = s_work;
    double *sg = s_work + pairs;
    int *sa = reinterpret_cast<int *>(sg + (size_t)pairs * k), *sr = sa + pairs, *sp = sr + pairs;
    for (int i = tid; i < pairs * k; i += kGreedyThreads) sg[i] = gram[i];
    const int R = offset[N];
    for (int i = tid; i < pairs; i += kGreedyThreads) {
      sa[i] = assign_idx[i];
      sr[i] = tokslot2row[i];
      sp[i] = i < R ? perm_row2tok[i] : 0;
    }
    gram = sg;
    assign_idx = sa;
    tokslot2row = sr;
    perm_row2tok = sp;
  }
  __syncthreads();
  // objective of the empty set: sum_t || O*_t ||^2 = sum_t sum_{a,b} G_t[a][b], in a fixed order
  double err = 0.0;
  {
    double acc = 0.0;
    const size_t n = (size_t)pairs * k;
    for (size_t i = tid; i < n; i += kGreedyThreads) acc += gram[i];
    acc = warp_sum(acc);
    if (lane == 0) s_part[warp] = acc;
    __syncthreads();
    for (int w = 0; w < kGreedyThreads / 32; ++w) err += s_part[w];
    if (tid == 0) {
      *res.gold = err;
      *res.status = *status;
    }
  }
  const int R = s_offset[N];
  for (int r = tid; r < R; r += kGreedyThreads)
    gain[r] = row_gain(gram, assign_idx, perm_row2tok[r], row2slot[r], k, s_in, -1);
  __syncthreads();
  for (int step = 0; step < n_pick; ++step) {
    for (int i0 = 0; i0 < N; i0 += kGreedyThreads / 8) {
      const int i = i0 + (tid >> 3), sub = tid & 7;
      double g = 0.0;
      if (i < N && !s_in[i])
        for (int r = s_offset[i] + sub; r < s_offset[i + 1]; r += 8) g += gain[r];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        int lo = __double2loint(g), hi = __double2hiint(g);
        lo = __shfl_xor_sync(kFullMask, lo, o);
        hi = __shfl_xor_sync(kFullMask, hi, o);
        g += __hiloint2double(hi, lo);
      }
      if (sub == 0 && i < N) {
        s_gain[i] = g;
        s_key[i] = order_bits(g);
      }
    }
    __syncthreads();
    unsigned long long best = 0;
    int best_i = 0x7fffffff;
    for (int i = lane; i < N; i += 32) {
      const unsigned long long key = s_key[i];
      if (!s_in[i] && (best_i == 0x7fffffff || key > best)) {      // ascending i: an equal gain keeps the lower index
        best = key;
        best_i = i;
      }
    }
    const unsigned hi = __reduce_max_sync(kFullMask, (unsigned)(best >> 32));
    const unsigned lo = __reduce_max_sync(kFullMask, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
    const bool mine = (unsigned)(best >> 32) == hi && (unsigned)best == lo;
    best_i = (int)__reduce_min_sync(kFullMask, mine ? (unsigned)best_i : 0x7fffffffu);
    err -= s_gain[best_i];
    if (tid == 0) {
      res.order[step] = best_i;
      res.objective[step] = err;
    }
    // rows of the tokens that hold the expert just picked
    const int first = s_offset[best_i], items = (s_offset[best_i + 1] - first) * k;
    for (int q = tid; q < items; q += kGreedyThreads) {
      const int t = perm_row2tok[first + q / k], a = q % k;
      const int r = tokslot2row[(size_t)t * k + a];
      if (r >= 0) gain[r] = row_gain(gram, assign_idx, t, a, k, s_in, best_i);
    }
    __syncthreads();
    if (tid == 0) s_in[best_i] = 1;
    __syncthreads();
  }
}

// The same loop for trees whose routed rows fit the registers of one CTA: up to 512 * ROWS (token, slot) pairs of k <= 8.
// A thread keeps its pairs' Gram rows, the experts of their tokens and which of those are still outside S, so a pick is
// answered by a compare and at most eight additions without a load, and a step is two barriers with an expert sum and an
// argmax between them.  The sums are those of greedy_kernel in its order (the energy of the empty set apart, which is
// added up pair by pair).  What bounds that one was a step's chain of dependent shared-memory loads (picked expert ->
// its rows -> their tokens -> slots -> membership), integer divisions and a third barrier.  us a ranking of the first 32 of
// 64 experts, layer pass included: 63 tokens 228 -> 188, 127 265 -> 213, 15 tokens (16 picks) 151 -> 134 (with the Gram
// kernel and this one launched behind the layer's CTAs instead of behind its end).  A step is 0.9 us: sums 0.35, argmax
// 0.1, the pick's rows 0.25, barriers.
template <int ROWS, int W>
__global__ void __launch_bounds__(kGreedyThreads) greedy_rows_kernel(
    const double *gram, const int *assign_idx, const int *offset, const int *tokslot2row, const int *status, int M, int N,
    int k, int n_pick, RankingResult res) {
  __shared__ double s_row[kGreedyThreads * ROWS];         // gains of the routed rows, in gather order
  __shared__ double s_gain[kMaxExperts];
  __shared__ unsigned long long s_key[kMaxExperts];
  __shared__ int s_offset[kMaxExperts + 1];
  __shared__ double s_part[kGreedyThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  for (int i = tid; i <= N; i += kGreedyThreads) s_offset[i] = offset[i];
  double G[ROWS][8], own[ROWS];
  unsigned id[ROWS][2], out[ROWS][2];      // experts of the token's slots, a byte each; 0xff where outside S, else 0
  int row[ROWS];
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < ROWS; ++q) {
    // (no load behind a branch: they would be waited for one by one)
    const int pair = tid + q * kGreedyThreads, p = min(pair, M * k - 1), t = p / k, a = p - t * k;
    int e[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      e[b] = assign_idx[t * k + min(b, k - 1)];
      G[q][b] = gram[(size_t)p * k + min(b, k - 1)];
    }
    row[q] = tokslot2row[p];
    own[q] = gram[(size_t)p * k + a];
    if (pair >= M * k) row[q] = -1;
    id[q][0] = id[q][1] = out[q][0] = out[q][1] = 0u;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      if (pair >= M * k || b >= k) G[q][b] = 0.0;
      if (b < k && e[b] >= 0) {
        id[q][b >> 2] |= (unsigned)e[b] << (8 * (b & 3));
        out[q][b >> 2] |= 0xffu << (8 * (b & 3));
      }
      acc += G[q][b];
    }
  }
  // objective of the empty set: sum_t || O*_t ||^2 = sum_t sum_{a,b} G_t[a][b], in a fixed order
  double err = 0.0;
  acc = warp_sum(acc);
  if (lane == 0) s_part[warp] = acc;
  __syncthreads();
  for (int w = 0; w < kGreedyThreads / 32; ++w) err += s_part[w];
  if (tid == 0) {
    *res.gold = err;
    *res.status = *status;
  }
  auto store_gain = [&](int q) {
    double cross = 0.0;
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if ((out[q][b >> 2] >> (8 * (b & 3))) & 1u) cross += G[q][b];
    if (row[q] >= 0) s_row[row[q]] = 2.0 * cross - own[q];
  };
#pragma unroll
  for (int q = 0; q < ROWS; ++q) store_gain(q);
  __syncthreads();
  unsigned taken = 0;        // this lane's experts lane, lane + 32, ... that are in S, or beyond the last: bit i / 32
#pragma unroll
  for (int slot = 0; slot < W; ++slot)
    if (lane + 32 * slot >= N) taken |= 1u << slot;
  for (int step = 0; step < n_pick; ++step) {
    // eight lanes an expert
    for (int i0 = 0; i0 < N; i0 += kGreedyThreads / 8) {
      const int i = i0 + (tid >> 3), sub = tid & 7;
      double g = 0.0;
      if (i < N) {
        const int end = s_offset[i + 1];
#pragma unroll 4
        for (int r = s_offset[i] + sub; r < end; r += 8) g += s_row[r];
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        int lo = __double2loint(g), hi = __double2hiint(g);
        lo = __shfl_xor_sync(kFullMask, lo, o);
        hi = __shfl_xor_sync(kFullMask, hi, o);
        g += __hiloint2double(hi, lo);
      }
      if (sub == 0 && i < N) {
        s_gain[i] = g;
        s_key[i] = order_bits(g);
      }
    }
    __syncthreads();
    // every warp finds the largest gain for itself (ties: lower index)
    unsigned long long best = 0;
    unsigned best_slot = 32;        // none
#pragma unroll
    for (int slot = W - 1; slot >= 0; --slot) {      // descending: an equal gain goes to the lower index
      const unsigned long long key = s_key[lane + 32 * slot];
      if (!((taken >> slot) & 1u) && key >= best) {
        best = key;
        best_slot = slot;
      }
    }
    const unsigned hi = __reduce_max_sync(kFullMask, (unsigned)(best >> 32));
    const unsigned lo = __reduce_max_sync(kFullMask, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
    const bool mine = best_slot < 32 && (unsigned)(best >> 32) == hi && (unsigned)best == lo;
    const int best_i = (int)__reduce_min_sync(kFullMask, mine ? best_slot * 32 + lane : 0x7fffffffu);
    if (lane == (best_i & 31)) taken |= 1u << (best_i >> 5);
    err -= s_gain[best_i];
    if (tid == 0) {
      res.order[step] = best_i;
      res.objective[step] = err;
    }
    // rows of the tokens that hold it
    const unsigned pattern = (unsigned)best_i * 0x01010101u;
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      const unsigned hit0 = __vcmpeq4(id[q][0], pattern) & out[q][0], hit1 = __vcmpeq4(id[q][1], pattern) & out[q][1];
      if (hit0 | hit1) {
        out[q][0] &= ~hit0;
        out[q][1] &= ~hit1;
        store_gain(q);
      }
    }
    __syncthreads();
  }
}

// sum (a - b)^2 and sum b^2 over n elements: every CTA reduces one contiguous slice in a fixed order,
// the partial sums are added by a one-CTA launch.
template <typename T>
__global__ void __launch_bounds__(256) sqdiff_partial_kernel(const T *__restrict__ a, const T *__restrict__ b, size_t n,
                                                             double *__restrict__ partial) {
  const size_t per = (n + gridDim.x - 1) / gridDim.x;
  const size_t lo = (size_t)blockIdx.x * per, hi = lo + per < n ? lo + per : n;
  double num = 0.0, den = 0.0;
  for (size_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const double x = (double)to_float(a[i]), r = (double)to_float(b[i]);
    num += (x - r) * (x - r);
    den += r * r;
  }
  __shared__ double s_n[8], s_d[8];
  num = warp_sum(num);
  den = warp_sum(den);
  if ((threadIdx.x & 31) == 0) {
    s_n[threadIdx.x >> 5] = num;
    s_d[threadIdx.x >> 5] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tn = 0.0, td = 0.0;
    for (int w = 0; w < 8; ++w) {
      tn += s_n[w];
      td += s_d[w];
    }
    partial[2 * blockIdx.x] = tn;
    partial[2 * blockIdx.x + 1] = td;
  }
}

__global__ void sqdiff_final_kernel(const double *__restrict__ partial, int n_parts, double *__restrict__ out) {
  if (threadIdx.x == 0) {
    double tn = 0.0, td = 0.0;
    for (int i = 0; i < n_parts; ++i) {
      tn += partial[2 * i];
      td += partial[2 * i + 1];
    }
    out[0] = tn;
    out[1] = td;
  }
}

}  // namespace

cudaError_t launch_gram(const LaunchCtx &c, double *gram, int *row2slot) {
  return launch_kernel(gram_kernel, dim3(c.M), dim3(kGramThreads), 0, c.stream, (const float *)c.ws->y,
                       (const float *)c.ws->gate_w, (const int *)c.ws->tokslot2row, gram, row2slot, c.desc->d, c.k);
}

cudaError_t launch_greedy(const LaunchCtx &c, const double *gram, const int *row2slot, int n_pick, double *row_gain,
                          const RankingResult &res) {
  const int pairs = c.M * c.k;
  if (c.k <= 8 && pairs <= 4 * kGreedyThreads) {
    auto go = [&](auto kernel) {
      return launch_kernel(kernel, dim3(1), dim3(kGreedyThreads), 0, c.stream, gram, (const int *)c.ws->assign_idx,
                           (const int *)c.ws->offset, (const int *)c.ws->tokslot2row, (const int *)c.ws->status, c.M,
                           c.desc->n_experts, c.k, n_pick, res);
    };
    const bool narrow = c.desc->n_experts <= 64;
    if (pairs <= kGreedyThreads) return narrow ? go(greedy_rows_kernel<1, 2>) : go(greedy_rows_kernel<1, 8>);
    if (pairs <= 2 * kGreedyThreads) return narrow ? go(greedy_rows_kernel<2, 2>) : go(greedy_rows_kernel<2, 8>);
    return narrow ? go(greedy_rows_kernel<4, 2>) : go(greedy_rows_kernel<4, 8>);
  }
  const size_t bytes = greedy_bytes(c.M, c.k);
  const bool in_smem = bytes <= kGreedySmem;
  cudaError_t e = cudaFuncSetAttribute(greedy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGreedySmem);
  if (e != cudaSuccess) return e;
  return launch_kernel(greedy_kernel, dim3(1), dim3(kGreedyThreads), in_smem ? bytes : 0, c.stream, gram,
                       (const int *)c.ws->assign_idx, (const int *)c.ws->offset, (const int *)c.ws->perm_row2tok,
                       (const int *)c.ws->tokslot2row, row2slot, (const int *)c.ws->status, row_gain, c.M,
                       c.desc->n_experts, c.k, n_pick, (int)in_smem, res);
}

cudaError_t launch_sqdiff(const void *a, const void *b, size_t n, int dtype, double *partial, double *out,
                          cudaStream_t stream) {
  if (dtype == MOESPEC_FP32)
    sqdiff_partial_kernel<float><<<kSqdiffParts, 256, 0, stream>>>((const float *)a, (const float *)b, n, partial);
  else if (dtype == MOESPEC_FP16)
    sqdiff_partial_kernel<__half><<<kSqdiffParts, 256, 0, stream>>>((const __half *)a, (const __half *)b, n, partial);
  else
    sqdiff_partial_kernel<__nv_bfloat16><<<kSqdiffParts, 256, 0, stream>>>((const __nv_bfloat16 *)a,
                                                                           (const __nv_bfloat16 *)b, n, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  sqdiff_final_kernel<<<1, 32, 0, stream>>>(partial, kSqdiffParts, out);
  return cudaGetLastError();
}

}  // namespace moespec
