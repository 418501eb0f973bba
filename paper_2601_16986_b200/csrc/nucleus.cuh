// The top-p threshold of one head, found exactly: the value theta of pbar such that the entries
// above it (and the earliest of those equal to it) are the smallest descending-pbar prefix whose
// exclusive mass is below p.  One histogram of 1024 bins of 1/64 octave around 1/n (256 of 1/16 for
// CTAs of 64 threads) locates theta's bin, the few entries of that bin are ranked against one
// another; a bin outside the window or with more entries than max_cand() falls back to four 8-bit radix
// passes over all bits.
// The mass walk uses 2^-40 fixed-point integers so it is exact and order independent; the
// threshold is relative to the integer total, so a common factor on pbar changes nothing.
#pragma once
#include "common.cuh"

namespace ckv {

constexpr float MASS_ONE = 1099511627776.0f;   // 2^40
// A bin's mass is summed in two 32-bit words: the low LOW_BITS of every term, and the bits above.  The masses
// of a head add up to 2^40, so the upper word stays below 2^31, and the lower one holds 2^22 terms (with 16
// low bits it wrapped at 2^16 terms of one bin: a prompt of 100 003 equal keys lost 351 hits).
constexpr int LOW_BITS = 10;
constexpr unsigned LOW_MASK = (1u << LOW_BITS) - 1u;

// fine bins of CTAs of NTH threads and the key bits below a bin: 16 octaves in all
__host__ __device__ constexpr int fine_bins(int nth) { return nth < 256 ? 256 : 1024; }
__host__ __device__ constexpr int fine_shift(int nth) { return nth < 256 ? 19 : 17; }
// Entries of the threshold's bin that are ranked against one another; they take the histogram's place (12 bytes each).
// (With room for 64 a head of 5000 entries fell back to the radix passes in some steps and not in others, a prompt of
// 9350 tokens in all: 18 of its selection's 40 us.)
__host__ __device__ constexpr int max_cand(int nth) { return nth < 256 ? 128 : 512; }

template <int NTH>
struct NucleusSmem {
  alignas(8) unsigned hist_lo[fine_bins(NTH)];   // per-bin mass, low bits of every term
  unsigned hist_hi[fine_bins(NTH)];   // per-bin mass, the bits above
  unsigned long long redu[NTH / 32 + 1];
  unsigned long long A_theta;    // fast path result: mass strictly above the threshold key
  unsigned theta;                //                   the threshold key
  int cnt_theta;                 //                   entries that carry it
  int ncand;
  int star;
  int eq[NTH / 32];
};

struct Nucleus {
  uint32_t theta;             // the threshold's key (bits of pbar); 0xffffffff: nothing is a hit
  int cnt_eq;                 // entries that carry it
  unsigned long long A;       // mass of the entries above it
  unsigned long long Pthr;    // the mass below which an entry's predecessors must stay
  bool found;
};

// pbar of one entry: the mean over its G query heads (at most N) of exp(s_g - m_g) / l_g, il_g = 1 / (l_g G).  m_g is the
// head's reference point as a natural logarithm (to_natural()): its rounding is a factor all entries share, which cancels
// in the search, and the difference is exact where the two are near.  (2^(s log2(e) - m) from one multiply-add rounds
// an entry's own exponent instead: with one query head and logits of deviation 8 entries were off against one another by
// 3e-7 instead of less than 1e-7, and after reallocations a head now and then kept another entry.  It saved next to
// nothing: 14B shape with unequal budgets 26.4 us a layer instead of 26.5, 8B shape 28.85 instead of 29.0.)
__device__ __forceinline__ float to_natural(float m_log2) { return m_log2 * 0.693147180559945309f; }
template <int N>
__device__ __forceinline__ float group_mean(const float (&s)[N], const float (&m)[N], const float (&il)[N], int G = N) {
  float pm = 0.f;
#pragma unroll
  for (int g = 0; g < N; ++g)
    if (g < G) pm = fmaf(expf(s[g] - m[g]), il[g], pm);
  return pm;
}

__device__ __forceinline__ unsigned long long mass_of(float pm) { return (unsigned long long)(pm * MASS_ONE); }

// Inclusive suffix sum over the lanes of a warp (higher lane = higher bins).
__device__ __forceinline__ unsigned long long warp_suffix(unsigned long long v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long x = __shfl_down_sync(0xffffffffu, v, o);
    if (lane + o < 32) v += x;
  }
  return v;
}

// The search in three parts, all called by the NTH threads of a CTA: nucleus_clear, a barrier, nucleus_add for every
// entry (a histogram of mass in fine bins around 1/n: bin(key) = clamp((key >> FINE_SHIFT) - base, 0, FINE_BINS - 1),
// monotone in key), a barrier, nucleus_find.
template <int NTH>
__device__ __forceinline__ void nucleus_clear(NucleusSmem<NTH>& sh) {
  for (int b = threadIdx.x; b < fine_bins(NTH); b += NTH) { sh.hist_lo[b] = 0u; sh.hist_hi[b] = 0u; }
  if (threadIdx.x == 0) { sh.star = -1; sh.ncand = 0; sh.theta = 0xffffffffu; sh.cnt_theta = 0; }
}
template <int NTH>
__device__ __forceinline__ int nucleus_base(int n) {
  return (int)(__float_as_uint(1.0f / (256.0f * (float)n)) >> fine_shift(NTH));
}
template <int NTH>
__device__ __forceinline__ void nucleus_add(NucleusSmem<NTH>& sh, int base, float pm) {
  const unsigned long long m = mass_of(pm);
  const int b = min(fine_bins(NTH) - 1, max(0, (int)(__float_as_uint(pm) >> fine_shift(NTH)) - base));
  atomicAdd(&sh.hist_lo[b], (unsigned)m & LOW_MASK);
  atomicAdd(&sh.hist_hi[b], (unsigned)(m >> LOW_BITS));
}

// `each(f)` calls f(pbar) for every entry the calling thread owns; `mid()` is called once on the way, where the search
// waits for other threads (a caller's loads that should be under way by then).
template <int NTH, class Each, class Mid>
__device__ __forceinline__ Nucleus nucleus_find(int base, float top_p, NucleusSmem<NTH>& sh, int* errword, Each each, Mid mid) {
  constexpr int WARPS = NTH / 32, FINE_BINS = fine_bins(NTH);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  Nucleus r;
  unsigned long long W = 0, A = 0;   // A: mass of keys strictly above the threshold's bin / prefix range
  {
    // suffix sums from the top bin: thread k owns bins [PER k, PER (k + 1))
    constexpr int PER = FINE_BINS / NTH;
    unsigned long long hb[PER], loc = 0;
#pragma unroll
    for (int b = 0; b < PER; ++b) hb[b] = ((unsigned long long)sh.hist_hi[tid * PER + b] << LOW_BITS) + sh.hist_lo[tid * PER + b];
#pragma unroll
    for (int b = 0; b < PER; ++b) loc += hb[b];
    const unsigned long long suf = warp_suffix(loc, lane);
    if (lane == 0) sh.redu[w] = suf;
    __syncthreads();
    mid();
    unsigned long long above = 0;
    for (int x = 0; x < WARPS; ++x) {
      const unsigned long long v = sh.redu[x];
      W += v;
      if (x > w) above += v;
    }
    // hit  <=>  mass strictly before the entry  <  p * W
    r.Pthr = (unsigned long long)ceil((double)top_p * (double)W);
    unsigned long long sab = above + (suf - loc);   // mass above this thread's top bin
#pragma unroll
    for (int b = PER - 1; b >= 0; --b) {
      if (sab < r.Pthr && r.Pthr <= sab + hb[b]) {
        sh.star = tid * PER + b;
        sh.redu[WARPS] = sab;
      }
      sab += hb[b];
    }
    __syncthreads();
  }
  const unsigned long long Pthr = r.Pthr;
  uint32_t theta = 0xffffffffu;
  int cnt_eq = 0;
  bool found = false;
  const int bstar = sh.star;
  if (bstar > 0 && bstar < FINE_BINS - 1) {   // inside the window: rank the bin's entries exactly
    A = sh.redu[WARPS];
    constexpr int MAX_CAND = max_cand(NTH);
    static_assert(MAX_CAND * 12 <= FINE_BINS * 8, "the candidates take the histogram's place");
    unsigned long long* cmass = reinterpret_cast<unsigned long long*>(sh.hist_lo);   // (every thread has read its bins)
    unsigned* cand = reinterpret_cast<unsigned*>(cmass + MAX_CAND);
    each([&](float pm) {
      const uint32_t key = __float_as_uint(pm);
      if ((int)(key >> fine_shift(NTH)) == bstar + base) {   // (no bin at the window's ends)
        const int x = atomicAdd(&sh.ncand, 1);
        if (x < MAX_CAND) { cand[x] = key; cmass[x] = mass_of(pm); }
      }
    });
    __syncthreads();
    const int c = sh.ncand;
    if (c <= MAX_CAND) {
      // candidate x carries the threshold iff  A + mass(keys above it) < Pthr <= that + mass(keys equal)
      for (int y = tid; y < c; y += NTH) {
        const uint32_t mine = cand[y];
        const unsigned long long wm = cmass[y];
        unsigned long long gt = 0;
        int eqc = 0;
#pragma unroll 4
        for (int x = 0; x < c; ++x) {
          const uint32_t kx = cand[x];
          if (kx > mine) gt += cmass[x];
          eqc += (kx == mine);
        }
        if (A + gt < Pthr && Pthr <= A + gt + (unsigned long long)eqc * wm) {
          sh.theta = mine;            // every carrier writes the same three values
          sh.A_theta = A + gt;
          sh.cnt_theta = eqc;
        }
      }
      __syncthreads();
      if (sh.cnt_theta > 0) {
        theta = sh.theta;
        A = sh.A_theta;
        cnt_eq = sh.cnt_theta;
        found = true;
      }
    }
  }
  if (!found) {
    // ---- general path: MSB-first radix passes over the fp32 bits of pbar, 8 bits each
    A = 0;
    uint32_t prefix = 0;
    found = true;
    for (int pass = 0; pass < 4; ++pass) {
      const int sft = 24 - 8 * pass;
      constexpr int NB = 256, PER = NB > NTH ? NB / NTH : 1;
      __syncthreads();
      for (int b = tid; b < NB; b += NTH) { sh.hist_lo[b] = 0u; sh.hist_hi[b] = 0u; }
      if (tid == 0) sh.star = -1;
      __syncthreads();
      each([&](float pm) {
        const uint32_t key = __float_as_uint(pm);
        const bool match = (pass == 0) || ((key >> (sft + 8)) == (prefix >> (sft + 8)));
        if (match) {
          const unsigned long long m = mass_of(pm);
          const int b = (key >> sft) & (NB - 1);
          atomicAdd(&sh.hist_lo[b], (unsigned)m & LOW_MASK);
          atomicAdd(&sh.hist_hi[b], (unsigned)(m >> LOW_BITS));
        }
      });
      __syncthreads();
      // suffix sums from the top bin: thread k owns bins [PER k, PER (k + 1))
      unsigned long long hb[PER], loc = 0;
#pragma unroll
      for (int b = 0; b < PER; ++b) {
        const int bin = tid * PER + b;
        hb[b] = bin < NB ? ((unsigned long long)sh.hist_hi[bin] << LOW_BITS) + sh.hist_lo[bin] : 0ull;
        loc += hb[b];
      }
      const unsigned long long suf = warp_suffix(loc, lane);
      if (lane == 0) sh.redu[w] = suf;
      __syncthreads();
      unsigned long long above = 0;
      for (int x = w + 1; x < WARPS; ++x) above += sh.redu[x];
      unsigned long long sab = A + above + (suf - loc);   // mass above this thread's top bin
#pragma unroll
      for (int b = PER - 1; b >= 0; --b) {
        if (sab < Pthr && Pthr <= sab + hb[b]) {
          sh.star = tid * PER + b;
          sh.redu[WARPS] = sab;
        }
        sab += hb[b];
      }
      __syncthreads();
      const int dstar = sh.star;
      if (dstar < 0) { found = false; break; }
      prefix |= (uint32_t)dstar << sft;
      A = sh.redu[WARPS];
    }
    __syncthreads();
    if (!found) {
      if (tid == 0) atomicOr(errword, ERR_NUCLEUS);
      prefix = 0xffffffffu;  // nothing is a hit
    }
    // entries whose pbar equals the threshold key share one mass; the earliest positions win
    theta = prefix;
    int eq = 0;
    each([&](float pm) { eq += (__float_as_uint(pm) == theta); });
    eq = warp_sum_i(eq);
    if (lane == 0) sh.eq[w] = eq;
    __syncthreads();
    for (int x = 0; x < WARPS; ++x) cnt_eq += sh.eq[x];
  }
  r.theta = theta;
  r.cnt_eq = cnt_eq;
  r.A = A;
  r.found = found;
  return r;
}

}  // namespace ckv
