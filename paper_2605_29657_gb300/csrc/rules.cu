// rules.cu -- the selection rules of the paper's component ablation, beside
// the register-anchored threshold of the method (Eqs. 5 and 8):
//   mean_ref_kernel     the "mean threshold" reference: per segment or per
//                       sample, the mean score of the unit's candidate rows
//                       (visual rows, restricted to a previous keep mask);
//                       the threshold is then s(v) >= lambda * mean;
//   budget_keep_kernel  the "fixed budget" rule, i.e. the top-K rule of
//                       Sec. 2, S = top-K(V, s): per sample the budget[b]
//                       candidate rows with the largest score, equal scores
//                       taken lower row first.
//   pool_scores_kernel  scores of merged tokens from their patches' scores
//                       (a 2x2 patch merger puts a merged token's patches on
//                       consecutive rows): the sum, mean or max of each
//                       group of consecutive rows.
// All are deterministic: fixed-order sums, and a selection whose result
// does not depend on thread timing.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.cuh"

namespace occam {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A cluster of C CTAs of 256 threads per unit (segment or sample). Thread t of
// CTA c sums the candidate rows 256 c + t, 256 (c + C) + t, ... in fp64; warps
// then combine in a fixed tree, a CTA's lane 0 adds its eight warp sums in
// order and the first CTA's the C sums. What bounds it is the rounds of loads
// and the slow fp64 adds of one SM, so units of more than kMeanSplitRows rows
// take eight CTAs: 5 samples of 3,500 to 14,900 rows 31.3 us with one CTA each
// and a row a round, 6.2 so; 64 samples of 2,900 rows 17.0 and 8.2. Below, the
// rounds of four rows alone: 21 samples of 420 to 890 rows 5.9 and 4.0.
template <int C>
__device__ __forceinline__ void mean_ref(const MeanRefParams& p) {
  constexpr int PER = 4;
  __shared__ double wsum[8], csum[C];
  __shared__ int wcnt[8], ccnt[C];
  __shared__ uint32_t bits[kRegBitWords];
  const int u = blockIdx.x / C, rank = blockIdx.x % C, tid = threadIdx.x;
  const int64_t lo = p.scope == OCCAM_REF_SEGMENT ? p.bt.seg_off[u] : p.bt.row_off[u];
  const int64_t hi = p.scope == OCCAM_REF_SEGMENT ? p.bt.seg_off[u + 1] : p.bt.row_off[u + 1];
  if (!p.role) {
    const int sa = p.scope == OCCAM_REF_SEGMENT ? u : p.bt.seg_first[u];
    const int sz = p.scope == OCCAM_REF_SEGMENT ? u + 1 : p.bt.seg_first[u + 1];
    mark_register_bits(bits, lo, (int)min(hi - lo, (int64_t)kRegBitRows), p.bt.reg_idx, p.bt.reg_off[sa],
                       p.bt.reg_off[sz]);
  }
  double acc = 0.0;
  int cnt = 0;
  // PER rows' loads are in flight together
  for (int64_t r0 = lo + rank * 256 + tid; r0 < hi; r0 += PER * C * 256) {
    float s[PER];
    bool cand[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int64_t r = r0 + k * C * 256;
      const bool in = r < hi;
      s[k] = in ? p.s[r] : 0.f;
      const bool kept = in && (!p.prev_keep || p.prev_keep[r] != 0);
      const bool reg = in && p.role && p.role[r] != 0;
      cand[k] = kept && !reg;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      if (cand[k] && (p.role || !test_bit(bits, (int)(r0 - lo) + k * C * 256))) {
        acc += (double)s[k];
        ++cnt;
      }
    }
  }
  acc = warp_sum_d(acc);
  cnt = warp_sum_i(cnt);
  if ((tid & 31) == 0) {
    wsum[tid >> 5] = acc;
    wcnt[tid >> 5] = cnt;
  }
  __syncthreads();
  double a = 0.0;
  int c = 0;
  if (tid == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += wsum[w];
      c += wcnt[w];
    }
  if constexpr (C > 1) {
    // every CTA runs, then every sum is in the first one's shared memory
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (tid == 0) {
      cl.map_shared_rank(csum, 0)[rank] = a;
      cl.map_shared_rank(ccnt, 0)[rank] = c;
    }
    cl.sync();
    if (rank != 0) return;
    if (tid == 0) {
      a = 0.0;
      c = 0;
      for (int i = 0; i < C; ++i) {
        a += csum[i];
        c += ccnt[i];
      }
    }
  }
  if (tid == 0) {
    const float ref = c > 0 ? (float)(a / (double)c) : 0.f;
    p.ref[u] = ref;
    if (p.tau) p.tau[u] = p.lambda * ref;
  }
}
__global__ void __launch_bounds__(256) mean_ref_kernel(MeanRefParams p) { mean_ref<1>(p); }
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(256) mean_ref_split_kernel(MeanRefParams p) { mean_ref<8>(p); }

// Order-preserving 32-bit key of a float: larger values give larger keys
// (-0 is taken as +0, so equal values have equal keys; NaN is undefined).
__device__ __forceinline__ uint32_t order_key(float v) {
  const uint32_t u = __float_as_uint(v == 0.f ? 0.f : v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// One CTA of 1,024 threads per sample.
//   1. Candidate keys (STAGED: once from global memory into shared memory,
//      with the candidates and registers as bits; else read again by every
//      pass) and the histogram of their top 11 bits; n = the candidate count,
//      K = clamp(budget[b], 0, n).
//   2. If 0 < K < n: the K-th largest candidate key t, eleven bits at a time
//      (bits 31-21, 20-10, 9-0): a block scan over the 2,048 buckets finds
//      the one where the running count from the top reaches K. need = how
//      many keys equal to t are kept = K - #(keys > t).
//   3. Keys above t are kept, and those equal to t if all of them are
//      needed; else they are ranked in row order (each thread a contiguous
//      run of rows, a block scan) and the first `need` kept. Register rows
//      get keep_registers.
// The chain of passes bounds it. With four 8-bit passes over global memory
// and a serial search of each histogram a sample of 2,900 rows took 30 us.
template <bool STAGED>
__global__ void __launch_bounds__(1024) budget_keep_kernel(BudgetParams p) {
  extern __shared__ uint32_t keys[];  // STAGED: the sample's keys
  __shared__ uint32_t hist[2048];
  __shared__ uint32_t regs[kRegBitWords], cands[STAGED ? kRegBitWords : 1];
  __shared__ uint32_t s_prefix, s_k;
  __shared__ int tmp[40];
  const int b = blockIdx.x, tid = threadIdx.x;
  const int64_t lo = p.bt.row_off[b];
  const int nrows = (int)(p.bt.row_off[b + 1] - lo);
  const int budget = p.budget[b];
  if (!p.role) {
    const int ra = p.bt.reg_off[p.bt.seg_first[b]], rb = p.bt.reg_off[p.bt.seg_first[b + 1]];
    mark_register_bits(regs, lo, min(nrows, kRegBitRows), p.bt.reg_idx, ra, rb);
  }
  auto is_reg = [&](int i) { return p.role ? p.role[lo + i] != 0 : test_bit(regs, i); };
  auto global_cand = [&](int i) { return !is_reg(i) && (!p.prev_keep || p.prev_keep[lo + i] != 0); };
  if (STAGED) {
    // rows i, i + 1024, ...: a warp's 32 rows are one word of bits. Four
    // rows' loads in flight per thread.
    for (int i0 = 0; i0 < nrows; i0 += 4096) {
      float s[4];
      bool c[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * 1024 + tid;
        s[k] = i < nrows ? p.s[lo + i] : 0.f;
        c[k] = i < nrows && global_cand(i);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * 1024 + tid;
        const uint32_t w = __ballot_sync(0xffffffffu, c[k]);
        if (i < nrows) {
          keys[i] = order_key(s[k]);
          if ((tid & 31) == 0) cands[i >> 5] = w;
        }
      }
    }
  }
  auto cand = [&](int i) { return STAGED ? test_bit(cands, i) : global_cand(i); };
  auto key_of = [&](int i) { return STAGED ? keys[i] : order_key(p.s[lo + i]); };
  // t = 0 with need = n keeps every candidate (every key is >= 0)
  uint32_t t = 0, prefix = 0, mask = 0;
  int need = 0, K = 0;
  bool select = true;
  for (int level = 0; level < 3 && select; ++level) {
    const int shift = level == 0 ? 21 : level == 1 ? 10 : 0;
    const uint32_t digit = level == 2 ? 1023u : 2047u;
    hist[tid] = hist[tid + 1024] = 0;
    __syncthreads();
    for (int i = tid; i < nrows; i += 1024) {
      if (!cand(i)) continue;
      const uint32_t key = key_of(i);
      if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & digit], 1u);
    }
    __syncthreads();
    // thread t holds buckets 2047 - 2t and 2046 - 2t
    const int hi = 2047 - 2 * tid;
    const int chi = (int)hist[hi], clo = (int)hist[hi - 1];
    int total;
    const int above = block_exclusive_scan(chi + clo, tmp, &total);
    int k;
    if (level == 0) {
      const int n = total;  // every candidate
      K = min(max(budget, 0), n);
      need = n;
      if (K == 0) {
        t = 0xffffffffu;
        need = 0;
      }
      select = K > 0 && K < n;
      if (!select) break;
      k = K;
    } else {
      k = need;
    }
    if (above < k && k <= above + chi + clo) {
      const int bucket = above + chi >= k ? hi : hi - 1;
      s_k = (uint32_t)(bucket == hi ? k - above : k - above - chi);
      s_prefix = prefix | ((uint32_t)bucket << shift);
    }
    __syncthreads();
    prefix = s_prefix;
    need = (int)s_k;
    mask |= digit << shift;
    t = prefix;
  }
  // whether the keys equal to t are all needed (hist holds the last level's
  // counts: the bucket of t counts exactly the keys equal to it)
  __syncthreads();
  const bool all_ties = !select || (int)hist[t & 1023u] == need;
  if (all_ties) {
    for (int i = tid; i < nrows; i += 1024) {
      bool k = false;
      if (is_reg(i)) {
        k = p.keep_registers != 0;
      } else if (cand(i)) {
        const uint32_t key = key_of(i);
        k = key > t || (key == t && need > 0);
      }
      p.keep[lo + i] = k ? 1 : 0;
    }
  } else {
    // contiguous runs of rows per thread keep the tie ranking in row order
    const int per = (nrows + 1023) / 1024;
    const int a = min(nrows, tid * per), z = min(nrows, a + per);
    int ties = 0;
    for (int i = a; i < z; ++i)
      if (cand(i) && key_of(i) == t) ++ties;
    int ties_total;
    int rank = block_exclusive_scan(ties, tmp, &ties_total);
    for (int i = a; i < z; ++i) {
      bool k = false;
      if (is_reg(i)) {
        k = p.keep_registers != 0;
      } else if (cand(i)) {
        const uint32_t key = key_of(i);
        if (key == t) {
          k = rank < need;
          ++rank;
        } else {
          k = key > t;
        }
      }
      p.keep[lo + i] = k ? 1 : 0;
    }
  }
  if (tid == 0 && p.count_vis) p.count_vis[b] = K;
}

// Samples of up to kBudgetStagedRows rows are staged in shared memory (their
// keys, 160 KB at most); the bits of larger ones would not fit beside it.
constexpr int kBudgetStagedRows = 40960;
static_assert(kBudgetStagedRows <= kRegBitRows, "candidate and register bits");

int launch_budget_keep(const BudgetParams& p, int64_t max_sample_rows, cudaStream_t st) {
  if (max_sample_rows <= kBudgetStagedRows) {
    const size_t smem = (size_t)max_sample_rows * 4;
    if (smem > 16 * 1024 &&
        cudaFuncSetAttribute(budget_keep_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kBudgetStagedRows * 4) != cudaSuccess)
      return 1;
    budget_keep_kernel<true><<<p.bt.B, 1024, smem, st>>>(p);
  } else {
    budget_keep_kernel<false><<<p.bt.B, 1024, 0, st>>>(p);
  }
  count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// One thread per merged row; the group's values are added in row order.
__global__ void __launch_bounds__(256) pool_scores_kernel(const float* __restrict__ s_in, int64_t rows_out, int group,
                                                          int mode, float* __restrict__ s_out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows_out; i += (int64_t)gridDim.x * blockDim.x) {
    const float* g = s_in + i * group;
    float acc = g[0];
    for (int k = 1; k < group; ++k) acc = mode == OCCAM_POOL_MAX ? fmaxf(acc, g[k]) : acc + g[k];
    s_out[i] = mode == OCCAM_POOL_MEAN ? acc / (float)group : acc;
  }
}

}  // namespace occam
