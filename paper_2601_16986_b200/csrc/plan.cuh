// Launch plan of a layer's attention kernel: which warp streams which groups of which head.
//
// Every head is cut into k = ceil(g / T) pieces of nearly equal length, at most T groups (pages of
// 16 keys) each, one piece per warp, and all pieces of a head are placed in consecutive warps of
// ONE CTA, where the head is merged in shared memory (a head of more than eight pieces takes whole
// CTAs and one shorter run).  T is the smallest bound for which such a placement fits the grid,
// whatever the heads' lengths are (after the budgets have been reallocated heads hold a few hundred
// to a few thousand entries); longer pieces are taken where they keep heads inside one CTA at less
// cost than the merge through global memory they avoid.  With more heads than warps every head is
// one piece and a warp takes several in turn.  The plan only depends on the heads' lengths, so it
// is written by whichever kernel changed them (the LRFU kernel of the layer's previous step once a
// head has drifted from the planned length, the shrink pass of a reallocation, the prompt
// insertion) and the attention kernel starts streaming without deriving anything but its pieces'
// bounds from the heads' current lengths.
#pragma once
#include "common.cuh"

namespace ckv {

// CTAs a set of heads needs when the pieces of a head have to sit in consecutive warps of one CTA:
// `full` CTAs are taken whole (eight pieces of a head with eight or more), cnt[s] runs of s < 8
// pieces are packed best fit, longest first.  A run goes to the open CTA with the fewest free
// warps that still holds it, so a CTA with c free warps takes c / s runs of length s one after the
// other: the loop below moves whole classes of CTAs at once and counts exactly what the
// run-by-run placement does.
__host__ __device__ __forceinline__ int ctas_needed(int full, const int (&cnt)[8]) {
  int open[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};   // open[c]: CTAs with c free warps
  int ctas = full;
#pragma unroll
  for (int s = 7; s >= 1; --s) {
    int n = cnt[s];
#pragma unroll
    for (int c = s; c <= 8; ++c) {
      const int q = c / s;                              // runs one such CTA takes
      const int have = (c == 8) ? (n + q - 1) / q : open[c];   // fresh CTAs are not counted in open[]
      const int nb = have < n / q ? have : n / q;       // CTAs filled with q runs
      int left = c - q * s;
      if (c == 8) ctas += nb; else open[c] -= nb;
      open[left] += nb;
      n -= nb * q;
      if (n > 0 && n < q && have > nb) {                // one more takes the rest
        if (c == 8) ++ctas; else --open[c];
#pragma unroll
        for (int nn = 1; nn < 8; ++nn)
          if (nn < q && n == nn) open[c - nn * s] += 1;
        n = 0;
      }
    }
  }
  return ctas;
}

// Where the runs go.  Heads of one length are spread where spread_pays(): a run goes to a fresh CTA while there is
// one and then to an open CTA with the most free warps, longest runs first, so that no SM idles while another one's CTA streams eight
// pieces.  Heads of unequal lengths gain in some launches (96 of 512 .. 1536 entries 15.9 us a layer and 16.2) and lose in others (720 of 150 .. 450
// 25.9 and 25.4: Algorithm 1's kernels then run on SMs without an attention CTA).  All these, and runs that do not fit the other
// way, are placed by the walk of ctas_needed(), which fits them whenever that counts no more CTAs than there are.  Both walk over
// ranges of consecutive CTAs instead of CTAs, class by class of free warps.
// An entry says: the runs [r0, r0 + n) of length s (in head order) fill CTAs base, base + 1, ... with q
// runs each, from warp `off` on.  A range of CTAs visited for a length is cut into at most a consumed, a
// partly consumed and an untouched part, so no more than 13 ranges and 35 entries arise in the walk of ctas_needed(); a spread
// that runs out of either is one that does not fit.
constexpr int PL_SCRATCH = 320;   // ints of shared scratch that write_plan() wants
constexpr int PL_ENTRIES = 40, PL_RANGES = 16;
struct Placement {
  int first[9];                  // entries of length s: [first[s], first[s - 1]), s = 7 .. 1
  int r0[PL_ENTRIES], n[PL_ENTRIES], base[PL_ENTRIES], qoff[PL_ENTRIES];   // qoff = q | off << 8
  int rb[PL_RANGES], rn[PL_RANGES], rc[PL_RANGES];   // ranges of open CTAs: first, count, free warps
};
static_assert(sizeof(Placement) <= (PL_SCRATCH - 64) * sizeof(int), "the placement lives in the planner's scratch");
// cnt[s]: runs of length s; full: CTAs taken whole (the first ones).  One thread.  False if they do not fit.
template <bool SPREAD>
__host__ __device__ inline bool place_runs_by(int full, const int* cnt, int grid, Placement& p) {
  int ne = 0, nr = 0, fresh = full;
  p.first[8] = p.first[7] = 0;
  for (int s = 7; s >= 1; --s) {
    p.first[s] = ne;
    int todo = cnt[s], done = 0;
    for (int k = s; k <= 8 && todo > 0; ++k) {
      const int c = SPREAD ? 8 + s - k : k;             // free warps of the CTAs visited: most first, or fewest
      const int q = SPREAD ? 1 : c / s, live = nr;      // runs one such CTA takes now
      for (int x = 0; x < (c == 8 ? 1 : live) && todo > 0; ++x) {
        int base, have;
        if (c == 8) {
          base = fresh; have = (todo + q - 1) / q;
          if (SPREAD) have = have < grid - fresh ? have : grid - fresh;
          if (fresh + have > grid) return false;
          if (have <= 0) continue;
          fresh += have;
        } else {
          if (p.rc[x] != c || p.rn[x] == 0) continue;
          base = p.rb[x]; have = p.rn[x];
        }
        const int wholes = todo / q < have ? todo / q : have;
        const int rest = wholes < have ? (todo - wholes * q < q ? todo - wholes * q : 0) : 0;
        const int used = wholes + (rest > 0 ? 1 : 0), runs = wholes * q + rest;
        if (ne >= PL_ENTRIES || nr + 2 > PL_RANGES) return false;
        p.r0[ne] = done; p.n[ne] = runs; p.base[ne] = base; p.qoff[ne] = q | ((8 - c) << 8);
        ++ne;
        done += runs;
        todo -= runs;
        if (c < 8) { p.rb[x] += used; p.rn[x] -= used; }
        if (wholes > 0 && c - q * s > 0) { p.rb[nr] = base; p.rn[nr] = wholes; p.rc[nr] = c - q * s; ++nr; }
        if (rest > 0) { p.rb[nr] = base + wholes; p.rn[nr] = 1; p.rc[nr] = c - rest * s; ++nr; }
      }
    }
    if (todo > 0) return false;
    int keep = 0;   // drop emptied ranges
    for (int x = 0; x < nr; ++x)
      if (p.rn[x] > 0) { p.rb[keep] = p.rb[x]; p.rn[keep] = p.rn[x]; p.rc[keep] = p.rc[x]; ++keep; }
    nr = keep;
  }
  p.first[0] = ne;
  return true;
}
__host__ __device__ inline bool place_runs(int full, const int* cnt, int grid, bool spread, Placement& p) {
  return (spread && place_runs_by<true>(full, cnt, grid, p)) || place_runs_by<false>(full, cnt, grid, p);
}

// Whether U heads of g groups each, in k pieces, are spread: from 33 groups a CTA on, unless Algorithm 1's kernel
// then misses the SMs without an attention CTA: its CTAs of eight warps (heads of more than 20 groups), of which two fit beside an attention CTA, come in
// several waves with more than two heads an SM, and they show while the streams are short.  us a layer, spread and with CTAs filled up one after the other:
// 150 heads of 76 groups 19.8 and 22.1, 160 of 44 14.4 and 16.1, 160 of 32 11.9 and 13.1, 256 of 65 25.0 and 25.6, 1024 of 17 26.3 and 26.8, 96 of 51 (33 a CTA) 11.65
// and 11.7; but 480 of 10 (32) 11.4 and 10.8, 192 of 19 (25) 9.9 and 9.55.  More than 296 heads that would fill 128 CTAs: 512 of 20 17.3 and 17.7, of 25 23.8 and 21.3,
// of 37 31.2 and 29.2, of 44 33.5 and 33.7, 1024 of 21 38.4 and 34.5, of 34 51.1 and 50.4; 104 CTAs: 832 of 26 36.0 and 33.0, of 34 41.0 and 42.5; 92 CTAs: 736 of 22 28.8 and 27.1, of
// 26 30.6 and 31.8; 90 CTAs: 360 of 22 15.0 and 16.7; 80 CTAs: 640 of 25 25.2 and 29.0.
// (So many heads are in one or two pieces.  The planner is part of Algorithm 1's kernels, whose launches got slower by 0.3 per cent with a second
// count of the CTAs, or branches, here.)
__host__ __device__ __forceinline__ bool spread_pays(int U, int g, int k, int grid) {
  const int filled = (U * k + NW - 1) / NW;   // CTAs, filled up one after the other
  const int line = U > 2 * grid && (unsigned)(g - 21) < 20u ? (g <= 22 ? 61 : g <= 32 ? 70 : 80) : 100;   // hundredths of the grid
  return U * g >= 33 * grid && 100 * filled <= line * grid;
}

// The first warp (CTA x NW + its place in the CTA) of run r of length s.
__host__ __device__ __forceinline__ int run_warp(const Placement& p, int s, int r) {
  int e = p.first[s];
  while (e + 1 < p.first[s - 1] && r >= p.r0[e] + p.n[e]) ++e;
  const int q = p.qoff[e] & 255, off = p.qoff[e] >> 8, d = r - p.r0[e];
  return (p.base[e] + d / q) * NW + off + (d % q) * s;
}

// Called by all NTH threads of one CTA.  `gs` is memory for U + 1 ints, `red` shared memory for 320.
// The plan is for a decode step: every head one entry longer than now, or, with shrink > 0, than once the heads that are
// `shrink` or more entries over their budgets have come down to them.
// A function of its own: inlined at the end of the LRFU kernel (48 registers) its counts and placement cost the
// kernel's common path registers.  14B shape with unequal budgets 27.95 us a layer instead of 28.1, 8B shape 29.0
// instead of 30.1, 64 heads of 4097 entries 31.5 instead of 32.9.  The kernels that call it take the state as a
// __grid_constant__, so that its address is passed without a copy on the stack.
template <int NTH = NT>
__device__ __noinline__ void write_plan(const State& st, const Plan& pl, int layer, int nWarps, int grid, int cl,
                                        int* gs, int* red, int shrink = 0) {
  const int U = st.batch * st.H, tid = threadIdx.x, lane = tid & 31;
  // ---- groups per head
  int mine = 0, gmax = 0;
  for (int u = tid; u < U; u += NTH) {
    const int uid = ((u / st.H) * st.L + layer) * st.H + (u % st.H);
    int n = __ldcg(st.n_cur + uid);   // (other CTAs of the calling kernel may just have written it: not from L1)
    if (shrink > 0 && n > 1 && n - __ldcg(st.budget + uid) >= shrink) n = max(1, __ldcg(st.budget + uid));
    // A head without entries (an insertion that found no pages, a head that is yet to be imported) has no page
    // to read: it gets no pieces.  The LRFU kernel flags it when a step meets it.
    const int g = n > 0 ? (n + 1 + GRP - 1) / GRP : 0;
    gs[u] = g;
    mine += g;
    gmax = max(gmax, g);
  }
  int Gtot;
  block_excl_scan<NTH>(mine, red, Gtot);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) gmax = max(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
  __syncthreads();
  if (lane == 0) red[tid >> 5] = gmax;
  __syncthreads();
  for (int x = 0; x < NTH / 32; ++x) gmax = max(gmax, red[x]);
  __syncthreads();
  // ---- the piece bound T.  Heads are cut into ceil(g_u / T) pieces; the smallest T is wanted for
  // which all heads can be placed with every head's pieces inside one CTA (such a head is merged in
  // shared memory; one that straddles CTAs goes through global memory and a ticket, which costs the
  // launch several microseconds at its end).  32 candidates are tried at once: warp x counts the
  // runs of every length over the heads u = x mod 8, lane c for T0 + c; warp 0 then packs them.
  int T = 0x7fffffff;
  bool packed = false;
  int* hist = red + 16;   // [32][4]: counts of two run lengths per word, 16 bits each (U < 65536)
  if (cl > 1) {
    // few heads: the cl CTAs of a cluster share each of them, in pieces of nearly equal length (at least
    // two groups) dealt evenly to the CTAs
    T = max(2, (gmax + NW * cl - 1) / (NW * cl));
  } else if (Gtot > 0 && U <= nWarps && grid * NW == nWarps && grid <= 256 && nWarps < 4096) {
    // A launch with few groups per warp is bound by the steps a head's result goes through, not by
    // bytes: pieces are then made long enough (up to GLAT groups) for the longest head to stay inside
    // one CTA, whose merge is one barrier instead of a trip through global memory.
    const int gfloor = min(gmax, max(GMIN, min(GLAT, (gmax + NW - 1) / NW)));
    const int T0 = max(max(1, (Gtot + nWarps - 1) / nWarps), gfloor);   // pieces shorter than GMIN groups
                                                                                // cost more in starts and merges than they gain
    // first feasible bound among Tfirst .. Tfirst + 31, or -1
    auto first_that_packs = [&](int Tfirst) {
      const int Tc = Tfirst + lane;
      for (int x = tid; x < 128; x += NTH) hist[x] = 0;
      __syncthreads();
      unsigned h4[4] = {0u, 0u, 0u, 0u};
      for (int u = tid >> 5; u < U; u += NTH / 32) {
        const int k = (gs[u] + Tc - 1) / Tc;
        const int r = k & 7;   // 0: nothing beyond whole CTAs
#pragma unroll
        for (int x = 0; x < 4; ++x) h4[x] += ((x > 0 && r == 2 * x) ? 1u : 0u) + ((r == 2 * x + 1) ? 0x10000u : 0u);
        h4[0] += (unsigned)(k >> 3);   // the low half of word 0 counts whole CTAs (there is no run of length 0)
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) atomicAdd(reinterpret_cast<unsigned*>(hist) + lane * 4 + x, h4[x]);
      __syncthreads();
      if (tid < 32) {
        int cnt[8];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const unsigned v = (unsigned)hist[lane * 4 + x];
          cnt[2 * x] = (int)(v & 0xffffu);
          cnt[2 * x + 1] = (int)(v >> 16);
        }
        const int full = cnt[0];
        const int ok = ctas_needed(full, cnt) <= grid;
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) red[0] = m ? Tfirst + (__ffs(m) - 1) : -1;
      }
      __syncthreads();
      const int found = red[0];
      __syncthreads();
      return found;
    };
    for (int round = 0; round < 4 && !packed; ++round) {
      const int found = first_that_packs(T0 + round * 32);
      if (found > 0) { T = found; packed = true; }
    }
    // Heads of more than eight pieces go through global memory, which costs the end of the launch
    // about as much as seven groups of streaming.  When pieces long enough for the longest head to fit
    // one CTA (gmax / 8 groups) cost less than that -- streaming is bound by the longer of a warp's own
    // groups and its share of the HBM rate, 7/4 group times per group at full occupancy -- they are taken.
    const int Tb = (gmax + NW - 1) / NW;
    if (packed && Tb > T) {
      const int hbm = (int)(((long long)Gtot * 7 / 4 + nWarps - 1) / nWarps);
      if (Tb <= max(T, hbm) + 7) {
        const int found = first_that_packs(Tb);
        if (found > 0 && found <= Tb + 2) T = found;
      }
    }
  }
  if (!packed && cl == 1 && Gtot > 0 && U <= nWarps) {
    // fallback: the smallest T for which sum ceil(g_u / T) <= nWarps, heads laid over the warps end to end
    int lo = max(1, (Gtot + nWarps - 1) / nWarps), hi = max(lo, gmax);   // feasible at hi: one piece per head
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      int cnt = 0;
      for (int u = tid; u < U; u += NTH) cnt += (gs[u] + mid - 1) / mid;
      int tot;
      block_excl_scan<NTH>(cnt, red, tot);
      __syncthreads();
      if (tot <= nWarps) hi = mid; else lo = mid + 1;
    }
    T = max(lo, min(GMIN, gmax));
  }
  // ---- pieces per head, their prefix sums, the descriptors; when packing, also the CTAs a head takes
  // whole and its place among the runs of its length
  Placement& place = *reinterpret_cast<Placement*>(red + 64);
  int pieces = 0, wholes = 0;
  int runs[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // runs of each length among the heads so far
  if (packed)
    for (int pw = tid; pw < nWarps; pw += NTH) pl.wrange[pw] = make_int4(0, 0, -1, 0);
  for (int b0 = 0; b0 < U; b0 += NTH) {
    const int u = b0 + tid;
    const int g = (u < U && Gtot > 0) ? gs[u] : 0;
    const int k = g == 0 ? 0 : (T == 0x7fffffff ? 1 : (g + T - 1) / T);
    int tot;
    const int start = pieces + block_excl_scan<NTH>(k, red, tot);
    pieces += tot;
    if (u < U) {
      pl.npc[u] = k;
      pl.gplan[u] = g;
      // the last word: 1 when the head's k pieces sit in consecutive warps of one CTA, each warp with
      // nothing else to stream; 2 when they sit that way in runs of eight (whole CTAs) and one shorter run
      const int together = k <= 1 ? 0 : cl > 1 ? 3 : (packed ? (k <= NW ? 1 : 2) : ((start & (NW - 1)) + k <= NW ? 1 : 0));
      for (int j = 0; j < k; ++j) pl.desc[start + j] = make_int4(u, j, k, together);
    }
    if (cl > 1 && u < U) gs[u] = start;
    if (packed) {
      const int f = k >> 3, s = k & 7;
      const int c0 = wholes + block_excl_scan<NTH>(f, red, tot);
      wholes += tot;
      if ((c0 + f) * NW <= nWarps)
        for (int x = 0; x < f * NW; ++x)
          pl.wrange[c0 * NW + x] = make_int4(start + x, start + x + 1, u, x | (k << 12) | ((k <= NW ? 1 : 2) << 24));
      int r = 0;   // this head's place among the runs of its length: two lengths per scan
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int v = (x > 0 && s == 2 * x ? 1 : 0) | (s == 2 * x + 1 ? 0x10000 : 0);
        const int e = block_excl_scan<NTH>(v, red, tot);
        if (x > 0 && s == 2 * x) r = runs[2 * x] + (e & 0xffff);
        if (s == 2 * x + 1) r = runs[2 * x + 1] + (e >> 16);
        runs[2 * x] += tot & 0xffff;
        runs[2 * x + 1] += tot >> 16;
      }
      if (u < U) gs[u] = (start << 12) | r;   // (both below 4096: packing wants fewer pieces than 4096 warps)
    }
  }
  if (packed) {
    // One thread walks the classes of CTAs, then every head looks its run up.  (A
    // plan of 128 heads takes 9 us; one warp placing the runs one by one took it to 26.)
    if (tid == 0) {
      const bool ok = wholes <= grid && place_runs(wholes, runs, grid, Gtot == gmax * U && spread_pays(U, gmax, (gmax + T - 1) / T, grid), place);
      place.first[8] = ok;
      if (!ok) atomicOr(st.errword, ERR_PLAN);   // cannot happen while ctas_needed() counts the same walk
    }
    __syncthreads();   // (also: the empty ranges above are written)
    const bool ok = place.first[8] != 0;
    for (int u = tid; u < U && ok; u += NTH) {
      const int k = pl.npc[u], s = k & 7, start = gs[u] >> 12, r = gs[u] & 4095, j0 = k - s;   // the pieces before took whole CTAs
      if (s == 0) continue;
      int4* w = pl.wrange + run_warp(place, s, r);
      for (int x = 0; x < s; ++x)
        w[x] = make_int4(start + j0 + x, start + j0 + x + 1, u, (j0 + x) | (k << 12) | ((k <= 1 ? 0 : (k <= NW ? 1 : 2)) << 24));
    }
    if (!ok) nWarps = -1;   // no launch accepts the plan
  } else if (cl > 1) {
    __syncthreads();   // (every head's pieces and first piece are known)
    // head u belongs to CTAs u cl .. u cl + cl - 1; CTA x of them takes the pieces from shared_first(k, x, cl) on
    for (int pw = tid; pw < nWarps; pw += NTH) {
      const int cta = pw / NW, u = cta / cl, x = cta % cl, k = u < U ? pl.npc[u] : 0;
      const int j = shared_first(k, x, cl) + (pw & (NW - 1));
      const bool mine = j < shared_first(k, x + 1, cl);
      pl.wrange[pw] = mine ? make_int4(gs[u] + j, gs[u] + j + 1, u, j | (k << 12) | ((k <= 1 ? 0 : 3) << 24)) : make_int4(0, 0, -1, 0);
    }
  } else {
    // heads end to end: consecutive pieces go to consecutive warps; with more pieces than warps
    // every warp takes a run of consecutive pieces
    const int per = (pieces + nWarps - 1) / max(nWarps, 1);
    for (int pw = tid; pw < nWarps; pw += NTH) {
      int4 r = make_int4(0, 0, -1, 0);
      if (pieces <= nWarps) {
        if (pw < pieces) r = make_int4(pw, pw + 1, -1, 0);
      } else {
        const int i0 = min(pieces, pw * per);
        r = make_int4(i0, min(pieces, i0 + per), -1, 0);
      }
      pl.wrange[pw] = r;
    }
  }
  if (tid == 0) {
    pl.hdr[0] = pieces;
    pl.hdr[1] = Gtot;
    pl.hdr[2] = nWarps;   // (-1 after a failed placement: no launch accepts the plan)
    pl.hdr[3] = 1;        // (a decode step's; read by the debug export only)
  }
}

}  // namespace ckv
