// plan.cuh -- the Stage-II work plan (internal header): which Stage-II path
// each sample takes and the item lists of those paths. Run by one CTA (the
// last Stage-I finalize CTA to finish) once every sample's S1 size n1[b] is
// known.
#pragma once

#include "common.cuh"
#include "kernels.cuh"

namespace occam {

// Routes every sample (the fused tensor-core kernel with 4-, 8- or 16-CTA
// clusters where its S1 keys and text keys fit, else the two-pass kernels)
// and writes the item lists, the per-sample item and partial-slot offsets,
// and the item counts. blockDim.x threads, tmp: >= 40 ints of shared memory.
// The two-pass kernels get per-sample item offsets, not item lists.
__device__ __forceinline__ void plan_stage2(const Stage2Params& p, int* tmp) {
  const int tid = threadIdx.x;
  const int nhg = (p.H + kHeadGroup - 1) / kHeadGroup;
  int runA = 0, runB = 0, runF = 0, runF8 = 0, runF16 = 0, runS = 0, runHS = 0, runP = 0;
  // A small batch leaves most SMs idle with 4-CTA clusters: when every text
  // tile of the batch can run at once as a resident 16- (or 8-) CTA cluster,
  // samples take the wider cluster, whose CTAs hold fewer keys and finish
  // each head sooner.
  int wide = 0, hsg = 1, hs16 = 1;  // hsg: head groups of a split tile (1: no split), on 16-CTA clusters or on 4 and 8
  // the first blockDim.x samples' text lengths and S1 sizes, loaded together
  // up front (one memory round trip instead of two in a row)
  int M0 = 0, n10 = 0;
  if (tid < p.bt.B) {
    M0 = (int)(p.bt.text_off[tid + 1] - p.bt.text_off[tid]);
    n10 = *((volatile int32_t*)&p.n1[tid]);
  }
  if (p.use_fused) {
    // the batch's text tiles and, for one that may split its heads, the CTAs
    // that one group of every tile takes (in the high bits; a sample's tiles
    // count as 100 at most, far above any rule)
    int tiles = 0;
    bool fit = true;
    if (p.has_ppart) {  // (at most kHsMaxTiles samples)
      if (tid < p.bt.B) {
        const bool fit4 = fused_fits(kFusedCluster, n10, M0, p.H);
        fit = fit4 || (p.split8 && fused_fits(8, n10, M0, p.H)) || M0 == 0;
        tiles = min((M0 + 127) / 128, 100);
        tiles |= tiles * (fit4 ? kFusedCluster : 8) << 12;
      }
    } else {
      for (int b = tid; b < p.bt.B; b += blockDim.x)
        tiles += b == tid ? (M0 + 127) / 128 : (int)((p.bt.text_off[b + 1] - p.bt.text_off[b] + 127) / 128);
    }
    int total_tiles, ctas = 0;
    block_exclusive_scan(tiles, tmp, &total_tiles);
    if (p.has_ppart) {
      ctas = total_tiles >> 12;
      total_tiles &= 4095;
    }
    wide = total_tiles <= p.res16 ? 16 : total_tiles <= p.res8 ? 8 : 0;
    // Head split: each tile's heads go to hsg items (whole key groups, at
    // least 4 heads each), all resident at once. An item's time is its heads
    // times about 2 us (the chain of one head: MMA, statistics, exchange,
    // probabilities), on clusters of any size, so the smallest clusters, 4
    // CTAs (36 resident) or 8 for the samples that do not fit those, take the
    // most groups: 8 tiles of 64 text rows and 540 S1 keys took 77 us on
    // 8-CTA clusters, a head after the other, and take 33 us and about 8 of
    // merge in 4 groups; one tile of 32 text rows and 270 S1 keys 17 and 7 in
    // 8 groups, where 16-CTA clusters in 4 groups take 21 and 7. (One tile
    // does so only where the host can tell, p.sure4: else the launches for
    // either would cost more than that.) More than kHsMaxTiles fill the device
    // unsplit.
    if (p.has_ppart && total_tiles <= kHsMaxTiles) {
      const bool small = __syncthreads_and(fit) && total_tiles > (p.sure4 ? 0 : 1) && p.res4 > 0;
      // the most groups that divide the heads (hs_valid) and fit at once
      int most = 0;
      if (small)
        most = p.res4 * kFusedCluster / ctas;
      else if (wide == 16 && total_tiles > 0)
        most = p.res16 / total_tiles;
      const uint32_t fits = p.hs_valid & ((2u << min(most, kHsGroups)) - 1u);
      if (fits) hsg = 31 - __clz(fits);
      if (small && hsg > 1) {
        hs16 = 0;
        wide = 0;
      }
    }
  }
  const int hsg4 = hs16 ? 1 : hsg, hsg16 = hs16 ? hsg : 1;  // of tiles on 4- and 8-, and on 16-CTA clusters (1: no split)
  for (int b0 = 0; b0 < p.bt.B; b0 += blockDim.x) {
    const int bb = b0 + tid;
    int nA = 0, nB = 0, tF = 0, tF8 = 0, tF16 = 0;  // (tF..: text tiles, each of hsg4 / hsg16 items)
    if (bb < p.bt.B) {
      const int M = b0 == 0 ? M0 : (int)(p.bt.text_off[bb + 1] - p.bt.text_off[bb]);
      const int n1 = b0 == 0 ? n10 : *((volatile int32_t*)&p.n1[bb]);
      // the fused tensor-core kernel takes a sample when its S1 keys and its
      // causal text keys fit the cluster's TMEM / shared memory
      const bool w16 = wide == 16 && fused_fits(16, n1, M, p.H);
      const bool w8 = !w16 && wide >= 8 && fused_fits(8, n1, M, p.H);
      const bool fused4 = !w16 && !w8 && p.use_fused && fused_fits(kFusedCluster, n1, M, p.H);
      const bool fused8 = w8 || (!w16 && !fused4 && p.use_fused && fused_fits(8, n1, M, p.H));
      const bool fused16 = w16 || (!fused4 && !fused8 && p.use_fused && fused_fits(16, n1, M, p.H));
      if (fused4) {
        tF = (M + 127) / 128;
      } else if (fused8) {
        tF8 = (M + 127) / 128;
      } else if (fused16) {
        tF16 = (M + 127) / 128;
      } else {
        const int nch = (n1 + kKeyChunk - 1) / kKeyChunk;
        nA = (M + kStatsTile - 1) / kStatsTile * nhg * s2_stat_splits(n1, M);
        nB = (M + kTextTile - 1) / kTextTile * nch;
      }
      if (M == 0) {
        set_status(p.status, OCCAM_ERR_INVALID_ARG);
        p.ref2[bb] = 0.f;
        p.tau2[bb] = 0.f;
      }
    }
    const int nS = tF * kFusedSlotsPerItem + tF8 * kFusedSlotsPerItem8 + tF16 * kFusedSlotsPerItem16 +
                   nB;  // s2(r) partial slots of this sample (a split tile's items share its slots)
    // this sample's head-split tiles, and the scratch slots of their items' CTAs
    const int nHS = hsg > 1 ? (hs16 ? tF16 : tF + tF8) : 0;
    const int hsC = hs16 ? 16 : tF ? kFusedCluster : 8;
    // the eight item and slot counts, scanned together
    __shared__ int mtmp[8 * 33];
    const int cnt[8] = {nA, nB, tF * hsg4, tF8 * hsg4, tF16 * hsg16, nS, nHS, nHS * hsg * hsC};
    int ex[8], tot[8];
    block_exclusive_scan_n<8>(cnt, ex, tot, mtmp);
    const int totA = tot[0], totB = tot[1], totF = tot[2], totF8 = tot[3], totF16 = tot[4], totS = tot[5],
              totHS = tot[6];
    const int offA = runA + ex[0], offB = runB + ex[1], offF = runF + ex[2], offF8 = runF8 + ex[3],
              offF16 = runF16 + ex[4], offS = runS + ex[5], offHS = runHS + ex[6], offP = runP + ex[7];
    if (bb < p.bt.B) {
      // the sample's tiles, all on clusters of one size; a tile's items: one, or
      // its head groups in turn (one rolled loop: this code runs once a call, on
      // one CTA, and waits for its instructions)
      int4* const items = tF ? p.itemsF : tF8 ? p.itemsF8 : p.itemsF16;
      const int C = tF ? kFusedCluster : tF8 ? 8 : 16, g_n = tF16 ? hsg16 : hsg4;
      const int tiles = tF + tF8 + tF16, slots = C * kFusedPartialWarps;
      int off = tF ? offF : tF8 ? offF8 : offF16;
#pragma unroll 1
      for (int t = 0; t < tiles; ++t)
#pragma unroll 1
        for (int g = 0; g < g_n; ++g, ++off)
          if (off < p.maxF)
            items[off] = make_int4(bb, t * 128, offS + t * slots,
                                   g_n > 1 ? ((offP + (t * g_n + g) * C) << 8) | (g << 4) | g_n : 0);
#pragma unroll 1
      for (int t = 0; t < nHS; ++t)
        if (offHS + t < kHsMaxTiles)
          p.itemsHS[offHS + t] = make_int4(bb, t * 128, offS + t * hsC * kFusedPartialWarps,
                                           hsg | (hsC << 8) | ((offP + t * hsg * hsC) << 16));
      p.itemA_off[bb] = offA;
      p.itemB_off[bb] = offB;
      p.slot_off[bb] = offS;
    }
    runA += totA;
    runB += totB;
    runF += totF;
    runF8 += totF8;
    runF16 += totF16;
    runS += totS;
    runHS += totHS;
    runP += tot[7];
  }
  if (tid == 0) {
    p.itemA_off[p.bt.B] = runA;
    p.itemB_off[p.bt.B] = runB;
    p.slot_off[p.bt.B] = runS;
    if (runA > p.maxA || runB > p.maxB || runF > p.maxF || runF8 > p.maxF || runF16 > p.maxF)
      set_status(p.status, OCCAM_ERR_CAPACITY);
    p.counters[CNT_NA] = (int)(runA < p.maxA ? runA : p.maxA);
    p.counters[CNT_NB] = (int)(runB < p.maxB ? runB : p.maxB);
    p.counters[CNT_NF] = (int)(runF < p.maxF ? runF : p.maxF);
    p.counters[CNT_NF8] = (int)(runF8 < p.maxF ? runF8 : p.maxF);
    p.counters[CNT_NF16] = (int)(runF16 < p.maxF ? runF16 : p.maxF);
    p.counters[CNT_NHS] = runHS < kHsMaxTiles ? runHS : kHsMaxTiles;
  }
}

}  // namespace occam
