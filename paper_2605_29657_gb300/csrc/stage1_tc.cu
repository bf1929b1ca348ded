// stage1_tc.cu -- mutual Stage-I scoring on the 5th-generation tensor cores
// (tcgen05 + TMEM + TMA).
//
// What it computes (Sec. 3.4, Eq. 6; App. A, Eq. 13): in segment s with n
// rows, every row u attends to every row v per head h with
// A_h(u -> v) = softmax_v(q_{u,h} k_{v,h} / sqrt(d1)), and
// s1[v] = 1/n sum_u 1/H sum_h A_h(u -> v).
// Two launches of one kernel template:
//   pass 1: per (segment, tile of 256 query rows, head) the query rows'
//           softmax log-sums L[h][u] = log2 sum_v exp2(c q_u k_v), with
//           c = log2(e) / sqrt(d1), over all the segment's keys (stored
//           negated, as the second pass adds them);
//   pass 2: per (segment, tile of 256 key rows, group of heads) the
//           attention each key receives, sum_h sum_u exp2(c q_u k_v - L[h][u]),
//           over the group's heads and all query rows; a small third kernel
//           sums the groups' shares in order into s1.
// An item is worked by a pair of CTAs (a 2-CTA cluster, tcgen05 cta_group::2):
// each CTA's half of the tile, 128 rows, are its TMEM lanes (the MMA's A
// operand), and the other side streams in blocks of 256 rows (the B operand),
// half of every block in either CTA's shared memory. S = A B^T is 128 x 256
// fp32 in each CTA's TMEM, from 4-5 tcgen05.mma of K = 16 over both SMs.
// The pair lets the operand feed keep up with the softmax: one CTA alone
// loads 40 KB (512 box rows) a block, and at the TMA unit's rate that takes
// 0.44 ms a pass on 32 images of 256-4,096 tokens (0.31 ms for a pair's half).
// What bounds it: the exponential unit, 32 a clock and SM (measured), 523 ns
// for a block of 128 x 256, and the 256 columns a TMEM lane quadrant is read
// in, which add to it (130 ns); the MMAs take 335 ns of a block. On those 32
// images (657 blocks an SM) pass 1 takes 560 us and pass 2 493 us, against 642
// and 550 us with one CTA an item, every softmax warp on the same block and a
// maximum taken for each block.
// Q1 and K1 are read as 3-D TMA boxes {64 dims, 1 head, 128 rows} with the
// 128-byte swizzle, plus {16 dims, 1 head, 128 rows} with the 32-byte swizzle
// for dims 64-79; dims past d1 (72 -> 80) come zero-filled by the box, so the
// padded K-step adds nothing.
// Roles (640 threads a CTA): warp 0 issues the TMA loads, warp 1 of the
// leader CTA (rank 0) the MMAs, warps 2-3 tell the leader's MMA warp that
// this CTA's tiles have landed (and fold the log-sums in, below), warps 4-19
// (two groups of eight, one per accumulator; in a group two warps per TMEM
// lane quadrant, each taking 128 of the 256 columns) do the softmax
// arithmetic, their TMEM loads in flight while they compute. A tiles and the
// accumulator are double buffered, B blocks come through a ring. Every wait
// is bounded; on a timeout the CTA records OCCAM_ERR_TIMEOUT, lets its copies
// land, frees TMEM and returns (its peer's waits then run out too).
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc5.cuh"

namespace occam {

namespace m1 {
constexpr int AR = 128;                   // tile rows of one CTA (TMEM lanes)
constexpr int TR = kMutTileRows;          // tile rows of the pair (MMA M)
constexpr int BR = 256;                   // block rows (MMA N)
constexpr int BH = BR / 2;                // ... of which each CTA holds half
constexpr int ABYTES = AR * 128;          // K-block 0 (dims 0-63) of a CTA's A tile
constexpr int BBYTES = BH * 128;          // K-block 0 of a CTA's half of a B block
constexpr int ABYTES1 = AR * 32;          // K-block 1 (dims 64-79, 32-byte rows)
constexpr int BBYTES1 = BH * 32;
static_assert(TR == 2 * AR && BH == AR, "one 128-row box per A tile and per half block");
constexpr int NGRP = 2;                   // softmax groups, one per accumulator
constexpr int GW = 8;                     // warps of a group: two per TMEM lane quadrant
constexpr int COLS = BR / 2;              // accumulator columns per softmax warp (128)
constexpr int EPI0 = 4;                   // first softmax warp
constexpr int THREADS = (EPI0 + NGRP * GW) * 32;
constexpr int NPP = 4;                    // partial-exchange slots, by item & 3 (see the softmax warps)
constexpr int NIT = 16;                   // item hand-out slots
constexpr uint64_t kLimitNs = 2000000000ull;

// A decoded work item: first row of its tile in the segment, first head, the
// segment's rows (-1: no more items), its first row in the batch.
struct alignas(16) MutItem {
  int a0, h, n, sb;
  int it;  // its number
  __device__ int first_group(int hgsize) const { return (h / hgsize + a0 / TR) & 1; }
};

// Pass 2 of 72-dim heads carries the log-sums in the free dims 72-74 of the
// last K-step (the fold warps). 64- and 80-dim heads have none; there a K-step
// of its own for the log-sums was faster (32 against 41 us on 6 images of
// 353-1,709 rows, 12 heads) but up to twice as far from 64 bits as adding
// them in the softmax warps, which is what is done.
template <int PASS, int D>
struct Cfg {
  static constexpr int T1 = D > 64 ? 1 : 0;        // a 16-dim K-step for dims 64-79
  static constexpr bool FOLD = PASS == 2 && D == 72;
  static constexpr bool LSM = PASS == 2 && !FOLD;  // the softmax warps take the log-sums from shared memory
  static constexpr int NBB = LSM && T1 ? 6 : 8;     // half blocks of B in flight (a ring; A tiles and accumulators: 2 each)
};

template <int PASS, int D>
struct Smem {
  using C = Cfg<PASS, D>;
  uint8_t a[2][ABYTES];     // K-block 0 per buffer
  uint8_t b[C::NBB][BBYTES];
  uint8_t a1[2][C::T1 ? ABYTES1 : 16];  // the 16-dim K-step per buffer
  uint8_t b1[C::NBB][C::T1 ? BBYTES1 : 16];
  float lsm[C::LSM ? 2 : 1][C::LSM ? NGRP * GW : 1][COLS];  // minus the log-sums of each softmax warp's columns (a ring of two steps)
  float2 part[NPP][3][4][32];  // partials of the quadrant's other warps per (item & 3, warp, quadrant, lane)
  MutItem itm[NIT];         // the ii-th work item, by ii % NIT, written by the leader's TMA producer
  uint64_t afull[2], aempty[2], bfull[C::NBB], bempty[C::NBB], dfull[2], dfree[2], hb[NPP][4], hfree[NPP][4], inext[NIT], mdone;
  uint64_t aready[2], bready[C::NBB];  // leader: the tile lies complete in both CTAs
  uint32_t tmem_base;
  int abort;
};
}  // namespace m1

static_assert(sizeof(m1::Smem<2, 80>) + 1024 <= 227 * 1024 && sizeof(m1::Smem<1, 80>) + 1024 <= 227 * 1024 &&
                  sizeof(m1::Smem<2, 64>) + 1024 <= 227 * 1024 && sizeof(m1::Smem<2, 72>) + 1024 <= 227 * 1024,
              "shared memory per CTA");

namespace {

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(tc::su32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(tc::su32(bar))
      : "memory");
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::su32(dst)), "l"(src) : "memory");
}

// Waits for the warp's TMEM load and ties the registers it wrote to the wait.
template <int N>
__device__ __forceinline__ void wait_ld(uint32_t (&v)[N]) {
  tc::tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < N; i += 8)
    asm volatile(""
                 : "+r"(v[i]), "+r"(v[i + 1]), "+r"(v[i + 2]), "+r"(v[i + 3]), "+r"(v[i + 4]), "+r"(v[i + 5]),
                   "+r"(v[i + 6]), "+r"(v[i + 7]));
}

// sum of exp2(c v + o) over N columns, added into the four pair sums ap
template <int N>
__device__ __forceinline__ void exp_sum(const uint32_t (&v)[N], float c, float o, float2 (&ap)[4]) {
  const float2 cc = make_float2(c, c), oo = make_float2(o, o);
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    float2 x = __ffma2_rn(make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), cc, oo);
    x.x = tc::ex2(x.x);
    x.y = tc::ex2(x.y);
    ap[i & 3] = __fadd2_rn(ap[i & 3], x);
  }
}
// the same with an offset per column (16-byte aligned, shared memory)
__device__ __forceinline__ void exp_sum_cols(const uint32_t (&v)[32], float c, const float* o, float2 (&ap)[4]) {
  const float2 cc = make_float2(c, c);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 o4 = reinterpret_cast<const float4*>(o)[i];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float2 x = __ffma2_rn(make_float2(__uint_as_float(v[4 * i + 2 * k]), __uint_as_float(v[4 * i + 2 * k + 1])), cc,
                            k == 0 ? make_float2(o4.x, o4.y) : make_float2(o4.z, o4.w));
      x.x = tc::ex2(x.x);
      x.y = tc::ex2(x.y);
      ap[(2 * i + k) & 3] = __fadd2_rn(ap[(2 * i + k) & 3], x);
    }
  }
}
__device__ __forceinline__ float pair_total(const float2 (&ap)[4]) {
  const float2 a2 = __fadd2_rn(__fadd2_rn(ap[0], ap[1]), __fadd2_rn(ap[2], ap[3]));
  return a2.x + a2.y;
}
__device__ __forceinline__ void pair_zero(float2 (&ap)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) ap[i] = make_float2(0.f, 0.f);
}

// the largest of 32 values, as a tree of three-input maxima
__device__ __forceinline__ float max32(const uint32_t (&v)[32]) {
  float t[11];
#pragma unroll
  for (int i = 0; i < 10; ++i)
    t[i] = tc::fmax3(__uint_as_float(v[3 * i]), __uint_as_float(v[3 * i + 1]), __uint_as_float(v[3 * i + 2]));
  t[10] = fmaxf(__uint_as_float(v[30]), __uint_as_float(v[31]));
  return fmaxf(tc::fmax3(tc::fmax3(t[0], t[1], t[2]), tc::fmax3(t[3], t[4], t[5]), tc::fmax3(t[6], t[7], t[8])),
               fmaxf(t[9], t[10]));
}

// masks the columns of a 32-column piece past the segment out of the softmax
__device__ __forceinline__ void mask32(uint32_t (&v)[32], int lim) {
  if (lim < 32) {
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = i < lim ? v[i] : 0xff800000u;  // -inf
  }
}

// Pass 1's running softmax of one row, log2 units: the sum (z plus the pair
// sums ap) is relative to a reference m that need not be the exact maximum:
// fp32 sums have the same relative precision whatever the reference, and a
// term small enough to underflow is below 2^-100 of the sum. A warp's first
// piece of an item sets m for the whole item; the maxima of the pieces after
// it (a tree of operations each, 0.10 of 0.65 ms a pass on 32 images of
// 256-4,096 tokens) are not taken. Only logits more than 127 above the first
// piece's overflow that sum: such an item is put on a list, and a launch
// behind this one works the list through with move_ref at every piece, which
// moves m when a piece's maximum mx lies more than 64 above it.
__device__ __forceinline__ void move_ref(float mx, float& m, float& z, float2 (&ap)[4]) {
  if (__any_sync(0xffffffffu, mx > m + 64.f)) {
    const float mn = fmaxf(m, mx);
    const float e = mn == -INFINITY ? 0.f : tc::ex2(m - mn);
    z = (z + pair_total(ap)) * e;
    pair_zero(ap);
    m = mn;
  }
}

}  // namespace

// Work items, taken from a queue by a persistent grid (one CTA pair per two SMs):
// PASS 1: (segment, tile of 256 query rows, head), A = query tile, B = key
//         blocks of that head;
// PASS 2: (segment, tile of 256 key rows, group of hgsize heads), A = key tile,
//         B = query blocks, for the group's heads in turn.
// The leader's producer thread draws items (skipping tiles past a segment's
// rows) and hands each, decoded, to every role of both CTAs through an
// ring in shared memory. It is at most 3 items ahead of the MMAs (two A
// tiles), they at most 2 steps ahead of the softmax group they feed, and no
// softmax warp more than NPP items behind another, so each slot of the NIT is
// read before it comes round again; buffer and phase counters run on across
// items, so the next item's loads overlap the current item's tail.

template <int PASS>
__device__ __forceinline__ bool mut_item(const MutualTcParams& p, int it, m1::MutItem& w) {
  w.it = it;
  const int sub_n = PASS == 1 ? p.H : p.hgroups;  // heads (pass 1) or head groups (pass 2) per tile
  const int per_seg = p.tiles * sub_n;
  const int seg = it / per_seg;
  const int rem = it - seg * per_seg;
  const int tile = rem / sub_n;
  w.h = (rem - tile * sub_n) * (PASS == 1 ? 1 : p.hgsize);  // first head of the item
  w.a0 = tile * m1::TR;
  const int64_t sb = p.bt.seg_off[seg];
  w.sb = (int)sb;
  w.n = (int)(p.bt.seg_off[seg + 1] - sb);
  return w.a0 < w.n;
}

// The ii-th item, once the leader has handed it out; false if it did not
// arrive in time.
template <class SM>
__device__ __forceinline__ bool mut_take(SM& sm, int ii, volatile int* abort, m1::MutItem& w) {
  using m1::NIT;
  if (!tc::bar_wait(&sm.inext[ii % NIT], (ii / NIT) & 1, abort, m1::kLimitNs, true)) return false;
  const int4 v = *reinterpret_cast<const int4*>(&sm.itm[ii % NIT]);
  w.a0 = v.x;
  w.h = v.y;
  w.n = v.z;
  w.sb = v.w;
  w.it = sm.itm[ii % NIT].it;
  return true;
}

// Hands item w (w.n = -1: no more) to both CTAs as their ii-th.
template <class SM>
__device__ __forceinline__ void mut_hand_out(SM& sm, int ii, const m1::MutItem& w) {
  using m1::NIT;
#pragma unroll
  for (uint32_t r = 0; r < 2; ++r) {
    tc::st_cluster_u32(&sm.itm[ii % NIT].a0, r, (uint32_t)w.a0);
    tc::st_cluster_u32(&sm.itm[ii % NIT].h, r, (uint32_t)w.h);
    tc::st_cluster_u32(&sm.itm[ii % NIT].n, r, (uint32_t)w.n);
    tc::st_cluster_u32(&sm.itm[ii % NIT].sb, r, (uint32_t)w.sb);
    tc::st_cluster_u32(&sm.itm[ii % NIT].it, r, (uint32_t)w.it);
  }
#pragma unroll
  for (uint32_t r = 0; r < 2; ++r) tc::bar_arrive_remote(&sm.inext[ii % NIT], r);
}

template <int PASS, int D, bool REDO = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(m1::THREADS, 1)
    mutual_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                     const __grid_constant__ CUtensorMap mapA1, const __grid_constant__ CUtensorMap mapB1,
                     MutualTcParams p) {
  using namespace m1;
  using CF = Cfg<PASS, D>;
  constexpr int NBB = CF::NBB;
  constexpr bool FOLD = CF::FOLD;
  extern __shared__ unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<Smem<PASS, D>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)tc::cluster_rank();  // 0: the pair's leader
  const int H = p.H;
  // (the redo launch draws from the list of the launch before it, and leaves
  // at once when, as nearly always, that is empty)
  if (REDO && *p.n_redo == 0) return;
  const int total = REDO ? *p.n_redo : p.bt.S_tot * p.tiles * (PASS == 1 ? H : p.hgroups);
  constexpr int NRW = FOLD ? 2 : 1;          // warps that report this CTA's tiles to the leader
  int* queue = p.queue + (REDO ? 2 : PASS - 1);
  volatile int* abort = &sm.abort;

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::bar_init(&sm.afull[i], 1);
      tc::bar_init(&sm.aempty[i], 1);
      tc::bar_init(&sm.aready[i], 2 * NRW);
      tc::bar_init(&sm.dfull[i], 1);
      tc::bar_init(&sm.dfree[i], 2 * GW);
    }
    for (int i = 0; i < NBB; ++i) {
      tc::bar_init(&sm.bfull[i], 1);
      tc::bar_init(&sm.bempty[i], 1);
      tc::bar_init(&sm.bready[i], 2 * NRW);
    }
    for (int i = 0; i < 4 * NPP; ++i) {
      tc::bar_init(&sm.hb[i >> 2][i & 3], 3);
      tc::bar_init(&sm.hfree[i >> 2][i & 3], 1);
    }
    for (int i = 0; i < NIT; ++i) tc::bar_init(&sm.inext[i], 1);
    tc::bar_init(&sm.mdone, 1);
    sm.abort = 0;
    tc::bar_fence_init();
    tc::prefetch_map(&mapA);
    tc::prefetch_map(&mapB);
    tc::prefetch_map(&mapA1);
    tc::prefetch_map(&mapB1);
  }
  if (warp == 1) tc::tmem_alloc_pair(&sm.tmem_base, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  // the peer's barriers must be initialised before anything arrives on them
  tc::cluster_sync_all();
  const uint32_t tmem = sm.tmem_base;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t na = 0, nbk = 0;
      int next = rank == 0 ? atomicAdd(queue, 1) : 0;
      for (int ii = 0;; ++ii) {
        MutItem w;
        if (rank == 0) {
          while (next < total && !mut_item<PASS>(p, REDO ? p.redo[next] : next, w)) next = atomicAdd(queue, 1);
          if (next >= total || *abort) w.n = -1;
          mut_hand_out(sm, ii, w);
          if (w.n < 0) break;
          next = atomicAdd(queue, 1);  // the next item's index travels while this one's tiles load
        } else {
          if (!mut_take(sm, ii, abort, w)) {
            sm.abort = 1;
            set_status(p.status, OCCAM_ERR_TIMEOUT);
            break;
          }
          if (w.n < 0) break;
        }
        const int nb = (w.n + BR - 1) / BR;
        const int nheads = PASS == 1 ? 1 : min(p.hgsize, H - w.h);
        const int ya = w.sb + w.a0 + rank * AR, yb = w.sb + rank * BH;
        bool ok = true;
        // step s is block jb of head h (counters instead of a division per step)
        for (int s = 0, h = w.h, jb = 0; s < nheads * nb && ok; ++s, jb = jb + 1 == nb ? 0 : jb + 1, h += jb == 0) {
          if (jb == 0) {
            const int ab = na & 1;
            if (!tc::bar_wait(&sm.aempty[ab], ((na >> 1) & 1) ^ 1, abort, kLimitNs)) {
              ok = false;
              break;
            }
            tc::bar_expect_tx(&sm.afull[ab], (uint32_t)(ABYTES + CF::T1 * ABYTES1));
            tma_load_3d(sm.a[ab], &mapA, 0, h, ya, &sm.afull[ab]);
            if (CF::T1) tma_load_3d(sm.a1[ab], &mapA1, 64, h, ya, &sm.afull[ab]);
            ++na;
          }
          const int bb = nbk % NBB;
          if (!tc::bar_wait(&sm.bempty[bb], ((nbk / NBB) & 1) ^ 1, abort, kLimitNs)) {
            ok = false;
            break;
          }
          tc::bar_expect_tx(&sm.bfull[bb], (uint32_t)(BBYTES + CF::T1 * BBYTES1));
          tma_load_3d(sm.b[bb], &mapB, 0, h, yb + jb * BR, &sm.bfull[bb]);
          if (CF::T1) tma_load_3d(sm.b1[bb], &mapB1, 64, h, yb + jb * BR, &sm.bfull[bb]);
          ++nbk;
        }
        if (!ok) {
          sm.abort = 1;
          set_status(p.status, OCCAM_ERR_TIMEOUT);
          if (rank == 0) {
            // tell the other roles to stop at the next hand-out
            w.n = -1;
            mut_hand_out(sm, ii + 1, w);
          }
          break;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = tc::idesc_bf16(TR, BR);
      uint32_t na = 0, sg = 0, use[2] = {0, 0};
      for (int ii = 0;; ++ii) {
        MutItem w;
        if (!mut_take(sm, ii, abort, w)) {
          sm.abort = 1;
          set_status(p.status, OCCAM_ERR_TIMEOUT);
          break;
        }
        if (w.n < 0) break;
        const int nb = (w.n + BR - 1) / BR;
        const int nheads = PASS == 1 ? 1 : min(p.hgsize, H - w.h);
        const int g0 = w.first_group(PASS == 1 ? 1 : p.hgsize);
        bool ok = true;
        for (int s = 0, jb = 0; s < nheads * nb; ++s, ++sg, jb = jb + 1 == nb ? 0 : jb + 1) {
          const int ab = na & 1, bb = sg % NBB;
          const int db = (s + g0) & 1;  // the accumulator, and softmax group, of this step
          if (jb == 0) ok = tc::bar_wait(&sm.aready[ab], (na >> 1) & 1, abort, kLimitNs);
          if (ok) ok = tc::bar_wait(&sm.bready[bb], (sg / NBB) & 1, abort, kLimitNs);
          const uint32_t u = db ? use[1]++ : use[0]++;
          if (ok && u > 0) ok = tc::bar_wait(&sm.dfree[db], (u - 1) & 1, abort, kLimitNs);
          if (!ok) break;
          tc::fence_after();
          const uint32_t abase = tc::su32(sm.a[ab]), bbase = tc::su32(sm.b[bb]);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            tc::mma_bf16_pair(tmem + db * BR, tc::sdesc_sw128(abase + ks * 32), tc::sdesc_sw128(bbase + ks * 32), idesc,
                              ks > 0 ? 1u : 0u);
          // dims 64-79 (for 72-dim heads in pass 2: and the log-sums)
          if (CF::T1)
            tc::mma_bf16_pair(tmem + db * BR, tc::sdesc_sw32(tc::su32(sm.a1[ab])),
                              tc::sdesc_sw32(tc::su32(sm.b1[bb])), idesc, 1u);
          tc::mma_commit_pair(&sm.dfull[db]);
          tc::mma_commit_pair(&sm.bempty[bb]);
          if (jb == nb - 1) {
            tc::mma_commit_pair(&sm.aempty[ab]);
            ++na;
          }
        }
        if (!ok) {
          sm.abort = 1;
          set_status(p.status, OCCAM_ERR_TIMEOUT);
          break;
        }
      }
      tc::mma_commit_pair(&sm.mdone);
      if (!tc::bar_wait(&sm.mdone, 0, nullptr, kLimitNs)) set_status(p.status, OCCAM_ERR_TIMEOUT);
    }
    __syncwarp();
  } else if (!FOLD && warp == 2) {
    // ------------------------------------------------------------ relay warp
    // tells the leader's MMA warp of every tile that has landed in this CTA
    if (lane == 0) {
      uint32_t na = 0, nbk = 0;
      for (int ii = 0;; ++ii) {
        MutItem w;
        bool ok = mut_take(sm, ii, abort, w);
        if (ok && w.n < 0) break;
        const int nb = (w.n + BR - 1) / BR;
        const int steps = ok ? (PASS == 1 ? 1 : min(p.hgsize, H - w.h)) * nb : 0;
        for (int s = 0, jb = 0; s < steps && ok; ++s, ++nbk, jb = jb + 1 == nb ? 0 : jb + 1) {
          if (jb == 0) {
            ok = tc::bar_wait(&sm.afull[na & 1], (na >> 1) & 1, abort, kLimitNs);
            if (ok) tc::bar_signal_remote(&sm.aready[na & 1], 0);
            ++na;
          }
          if (ok) ok = tc::bar_wait(&sm.bfull[nbk % NBB], (nbk / NBB) & 1, abort, kLimitNs);
          if (ok) tc::bar_signal_remote(&sm.bready[nbk % NBB], 0);
        }
        if (!ok) {
          sm.abort = 1;
          set_status(p.status, OCCAM_ERR_TIMEOUT);
          break;
        }
      }
    }
    __syncwarp();
  } else if (FOLD && (warp == 2 || warp == 3)) {
    // ------------------------------------------------------------ fold warps
    // Dims 72-79 of the last K-step arrive zero-filled by the TMA box. Into
    // dims 72-74 go 1.0 on the key side (A) and, on the query side (B), a
    // three-term bf16 split of -L_u / c (each term the rounding of what the
    // previous ones leave, so the three hold 24 significant bits), so the MMA
    // yields S - L_u / c and the softmax warps need only c times it. A
    // query row past the segment gets -1e30, whose exponential is 0. In the
    // 32-byte-swizzled rows, 16-byte chunk k of row r sits in chunk
    // k ^ ((r >> 2) & 1). Warp 2 takes the first half of the rows of this
    // CTA's tiles, warp 3 the second; each then tells the leader's MMA warp.
    const float inv_c = 1.0f / p.scale_log2;
    const int half = warp - 2;
    const int64_t R = p.bt.total_rows;
    uint32_t na = 0, nbk = 0;
    for (int ii = 0;; ++ii) {
      MutItem w;
      if (!__all_sync(0xffffffffu, mut_take(sm, ii, nullptr, w))) {
        sm.abort = 1;
        set_status(p.status, OCCAM_ERR_TIMEOUT);
        break;
      }
      if (w.n < 0) break;
      const int n = w.n;
      const int64_t sb = w.sb;
      const int nb = (n + BR - 1) / BR;
      const int steps = min(p.hgsize, H - w.h) * nb;
      // -L of the block's query rows lane + 32 k, loaded a step ahead
      // (clamped to the segment; rows past it are replaced below)
      constexpr int KR = BH / 64;  // B rows per lane and step
      float lpre[KR];
      auto load_l = [&](int ht, int tb) {  // block tb of head ht
        const int base = tb * BR + rank * BH + half * (BH / 2);
#pragma unroll
        for (int k = 0; k < KR; ++k)
          lpre[k] = __ldcg(&p.lsum[(int64_t)ht * R + sb + min(base + lane + 32 * k, n - 1)]);
      };
      load_l(w.h, 0);
      bool ok = true;
      for (int s = 0, h = w.h, jb = 0; s < steps; ++s, jb = jb + 1 == nb ? 0 : jb + 1, h += jb == 0) {
        if (jb == 0) {
          const int ab = na & 1;
          if (!__all_sync(0xffffffffu, tc::bar_wait(&sm.afull[ab], (na >> 1) & 1, nullptr, kLimitNs))) {
            ok = false;
            break;
          }
          for (int r = half * (AR / 2) + lane; r < (half + 1) * (AR / 2); r += 32)
            *reinterpret_cast<uint4*>(sm.a1[ab] + r * 32 + 16 * (1 ^ ((r >> 2) & 1))) =
                make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);  // bf16 1.0 in dims 72, 73, 74
          tc::fence_proxy_async();
          __syncwarp();
          if (lane == 0) tc::bar_signal_remote(&sm.aready[ab], 0);
          ++na;
        }
        const int bb = nbk % NBB;
        if (!__all_sync(0xffffffffu, tc::bar_wait(&sm.bfull[bb], (nbk / NBB) & 1, nullptr, kLimitNs))) {
          ok = false;
          break;
        }
        float cur[KR];
#pragma unroll
        for (int k = 0; k < KR; ++k) cur[k] = lpre[k];
        if (s + 1 < steps) {
          if (jb + 1 == nb) load_l(h + 1, 0);
          else load_l(h, jb + 1);
        }
#pragma unroll
        for (int k = 0; k < KR; ++k) {
          const int r = half * (BH / 2) + lane + 32 * k;
          uint4 t4 = make_uint4(__bfloat16_as_ushort(__float2bfloat16_rn(-1e30f)), 0u, 0u, 0u);
          if (jb * BR + rank * BH + r < n) {
            const float y = cur[k] * inv_c;  // -L / c
            const __nv_bfloat16 h1 = __float2bfloat16_rn(y);
            const float r1 = y - __bfloat162float(h1);
            const __nv_bfloat16 h2 = __float2bfloat16_rn(r1);
            const float r2 = r1 - __bfloat162float(h2);
            const __nv_bfloat16 h3 = __float2bfloat16_rn(fmaf(y, kMutFoldBias, r2));
            t4.x = (uint32_t)__bfloat16_as_ushort(h1) | ((uint32_t)__bfloat16_as_ushort(h2) << 16);
            t4.y = (uint32_t)__bfloat16_as_ushort(h3);
          }
          *reinterpret_cast<uint4*>(sm.b1[bb] + r * 32 + 16 * (1 ^ ((r >> 2) & 1))) = t4;
        }
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) tc::bar_signal_remote(&sm.bready[bb], 0);
        ++nbk;
      }
      if (!ok) {
        sm.abort = 1;
        set_status(p.status, OCCAM_ERR_TIMEOUT);
        break;
      }
    }
  } else if (warp >= EPI0) {
    // ------------------------------------------------------------ softmax warps
    const int ew = warp - EPI0;
    const int quad = warp & 3, grp = ew / GW, half = (ew >> 2) & 1;  // TMEM lane quadrant; accumulator; column half
    const int row = quad * 32 + lane;                   // tile row = TMEM lane
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    const float c = p.scale_log2;
    const int64_t R = p.bt.total_rows;
    uint32_t use = 0;  // uses of this group's accumulator
    for (int ii = 0;; ++ii) {
      MutItem w;
      if (!__all_sync(0xffffffffu, mut_take(sm, ii, nullptr, w))) {
        sm.abort = 1;
        set_status(p.status, OCCAM_ERR_TIMEOUT);
        break;
      }
      if (w.n < 0) break;
      const int n = w.n;
      const int64_t sb = w.sb;
      const int nb = (n + BR - 1) / BR;
      const int steps = (PASS == 1 ? 1 : min(p.hgsize, H - w.h)) * nb;
      const int arow = w.a0 + rank * AR + row;            // this thread's row of the segment
      const bool vrow = arow < n;
      const int pp = ii & (NPP - 1);
      float m = -INFINITY, z = 0.f;  // pass 1: running reference / sum (log2 domain)
      float acc = 0.f;               // pass 2: attention received by this key row
      // The two groups of eight warps take the item's blocks in turn, each
      // from its own accumulator, so that one group's exponentials fill the
      // exponential unit while the other waits, loads or adds up: with every
      // warp on the same block they did that together, and a block took
      // 1,460 cycles against the unit's 1,024 (8 exponentials a cycle and SM
      // sub-partition, measured). A warp's 128 columns of a block come in
      // four loads, each in flight while the piece before it is computed; the
      // accumulator is released as soon as it lies in registers.
      const uint32_t d = tmem + lane_base + grp * BR + half * COLS;
      float2 ap[4];
      pair_zero(ap);
      bool ok = true;
      // step s is block s % nb of a head; this group's are s0, s0 + 2, ...
      const int s0 = (grp + w.first_group(PASS == 1 ? 1 : p.hgsize)) & 1;
      int lim = n - s0 * BR - half * COLS;  // pass 1: this warp's columns left in the segment
      uint32_t v0[32], v1[32];
      const float* lcol = nullptr;
      auto piece = [&](uint32_t (&v)[32], int left, bool first = false) {
        if (PASS == 1) {
          mask32(v, left);
          // c > 0: the max of c l is c times the max of l
          if (REDO || first) move_ref(max32(v) * c, m, z, ap);
          exp_sum<32>(v, c, m == -INFINITY ? 0.f : -m, ap);
        } else {
          if (CF::FOLD)
            exp_sum<32>(v, c, 0.f, ap);  // the accumulator holds S - L / c
          else
            exp_sum_cols(v, c, lcol, ap);
        }
      };
      // Without the fold, minus the log-sums of this warp's columns of a step
      // (past the segment: -inf, which contributes 0) come by cp.async into a
      // ring of two slots, one of the group's steps ahead. The slot refilled
      // was last read in the step before, which every lane has finished.
      int fh = w.h, fj = s0;  // head and block of the step fetched next
      auto fetch = [&](int slot) {
        while (fj >= nb) {
          fj -= nb;
          ++fh;
        }
        if (fh < min(w.h + p.hgsize, H)) {
#pragma unroll
          for (int i = 0; i < COLS / 32; ++i) {
            const int qq = fj * BR + half * COLS + lane * (COLS / 32) + i;
            float* dst = &sm.lsm[slot][ew][lane * (COLS / 32) + i];
            if (qq < n)
              cp_async4(dst, &p.lsum[(int64_t)fh * R + sb + qq]);
            else
              *dst = -INFINITY;
          }
        }
        cp_async_commit();
        fj += 2;
      };
      int slot = 0;
      if (CF::LSM) fetch(slot);
      for (int s = s0; s < steps; s += 2, ++use, lim -= 2 * BR) {
        ok = __all_sync(0xffffffffu, tc::bar_wait(&sm.dfull[grp], use & 1, nullptr, kLimitNs));
        if (!ok) break;
        tc::fence_after();
        tc::tmem_ld32(d, v0);
        if (CF::LSM) {
          cp_async_wait<0>();
          __syncwarp();
          lcol = sm.lsm[slot][ew];
          slot ^= 1;
          fetch(slot);
        }
        wait_ld(v0);
        tc::tmem_ld32(d + 32, v1);
        piece(v0, lim, s == s0);
        wait_ld(v1);
        tc::tmem_ld32(d + 64, v0);
        if (CF::LSM) lcol += 32;
        piece(v1, lim - 32);
        wait_ld(v0);
        tc::tmem_ld32(d + 96, v1);
        if (CF::LSM) lcol += 32;
        piece(v0, lim - 64);
        wait_ld(v1);
        tc::fence_before();
        __syncwarp();
        if (lane == 0) {
          if (rank == 0)
            tc::bar_arrive(&sm.dfree[grp]);
          else
            tc::bar_signal_remote(&sm.dfree[grp], 0);
        }
        if (CF::LSM) lcol += 32;
        piece(v1, lim - 96);
        const float t = pair_total(ap);
        pair_zero(ap);
        if (PASS == 1)
          z += t;
        else
          acc += t;
      }
      if (ok) {
        // the quadrant's four partials meet in the first group's first warp,
        // in fixed order; the others wait until it has read their slot's
        // last use, so no softmax warp is more than NPP items ahead of it
        const int src = grp * 2 + half - 1;
        if (src >= 0) {
          if (ii >= NPP)
            ok = __all_sync(0xffffffffu, tc::bar_wait(&sm.hfree[pp][quad], (ii / NPP - 1) & 1, nullptr, kLimitNs));
          if (ok) {
            sm.part[pp][src][quad][lane] = make_float2(PASS == 1 ? m : acc, z);
            __syncwarp();
            if (lane == 0) tc::bar_arrive(&sm.hb[pp][quad]);
          }
        } else if (!__all_sync(0xffffffffu, tc::bar_wait(&sm.hb[pp][quad], (ii / NPP) & 1, nullptr, kLimitNs))) {
          ok = false;
        } else {
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float2 o = sm.part[pp][q][quad][lane];
            if (PASS == 2) {
              acc += o.x;
            } else if (o.x != -INFINITY) {
              const bool up = o.x > m;
              const float e = tc::ex2(up ? m - o.x : o.x - m);
              z = up ? fmaf(z, e, o.y) : fmaf(o.y, e, z);
              m = fmaxf(m, o.x);
            }
          }
          __syncwarp();
          if (lane == 0) tc::bar_arrive(&sm.hfree[pp][quad]);
          // an infinite sum (or one that is no number) is not < inf
          if (PASS == 1 && !REDO && !__all_sync(0xffffffffu, !vrow || z < INFINITY)) {
            if (lane == 0) p.redo[atomicAdd(p.n_redo, 1)] = w.it;
          }
          if (vrow && in_bounds(sb + arow < R, p.status, kSiteMutualRow)) {
            if (PASS == 1)
              // -L, L = log2 of the row's sum of exp2(c q k) over the segment's keys
              p.lsum[(int64_t)w.h * R + sb + arow] = -(m + log2f(z));
            else
              // this head group's share of s1 (summed over the groups in order afterwards)
              p.part[(int64_t)(w.h / p.hgsize) * R + sb + arow] = acc * p.inv_h / (float)n;
          }
        }
      }
      if (!ok) {
        sm.abort = 1;
        set_status(p.status, OCCAM_ERR_TIMEOUT);
        break;
      }
    }
  }

  // ------------------------------------------------------------ teardown
  tc::fence_before();
  __syncthreads();
  if (sm.abort && tid == 0) {
    // let the TMA copies still in flight land before the CTA's shared memory goes away
    const uint64_t t0 = tc::globaltimer();
    while (tc::globaltimer() - t0 < 100000ull) {
    }
  }
  __syncthreads();
  // neither CTA leaves (or frees its TMEM) while the pair's MMAs or the
  // peer's arrivals may still reach it
  tc::cluster_sync_all();
  tc::fence_after();
  if (warp == 1) tc::tmem_dealloc_pair(tmem, 512);
  tc::cluster_sync_all();
}

// s1 = the sum of the head groups' shares, in group order (deterministic)
__global__ void __launch_bounds__(256) mutual_reduce_kernel(MutualTcParams p) {
  const int64_t R = p.bt.total_rows;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < R; r += (int64_t)gridDim.x * blockDim.x) {
    float v = 0.f;
    for (int g = 0; g < p.hgroups; ++g) v += __ldcg(&p.part[(int64_t)g * R + r]);
    p.s1[r] = v;
    if (p.s2_zero) p.s2_zero[r] = 0.f;
  }
  pdl_trigger();  // the finalize kernel may start its input-only prologue
}

namespace {
template <int D>
void launch_passes(const MutualTcParams& p, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mq1,
                   const CUtensorMap& mk1, int grid, cudaStream_t st) {
  constexpr int smem1 = (int)sizeof(m1::Smem<1, D>) + 1024, smem2 = (int)sizeof(m1::Smem<2, D>) + 1024;
  cudaFuncSetAttribute(mutual_tc_kernel<1, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem1);
  cudaFuncSetAttribute(mutual_tc_kernel<2, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
  cudaFuncSetAttribute(mutual_tc_kernel<1, D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem1);
  mutual_tc_kernel<1, D><<<grid, m1::THREADS, smem1, st>>>(mq, mk, mq1, mk1, p);
  mutual_tc_kernel<1, D, true><<<grid, m1::THREADS, smem1, st>>>(mq, mk, mq1, mk1, p);
  mutual_tc_kernel<2, D><<<grid, m1::THREADS, smem2, st>>>(mk, mq, mk1, mq1, p);
  count_launch(3);
}
}  // namespace

void launch_mutual_tc(const MutualTcParams& p, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mq1,
                      const CUtensorMap& mk1, int sms, cudaStream_t st) {
  const int grid = std::max(2, sms & ~1);  // CTA pairs
  if (p.tile_rows != kMutTileRows)
    launch_mutual_short(p, mq, mk, mq1, mk1, sms, st);
  else if (p.d1 == 64)
    launch_passes<64>(p, mq, mk, mq1, mk1, grid, st);
  else if (p.d1 == 72)
    launch_passes<72>(p, mq, mk, mq1, mk1, grid, st);
  else
    launch_passes<80>(p, mq, mk, mq1, mk1, grid, st);
  mutual_reduce_kernel<<<sms * 2, 256, 0, st>>>(p);
  count_launch();
}

}  // namespace occam
