// Observation-window prompts: Algorithm 1 replayed over the last W queries of a prompt whose rows are
// already stored.  Which entries a query hits depends on its scores alone, not on what earlier
// queries of the window marked, so the window is one attention kernel over all (query, head) rows,
// one threshold search per (head, query), and one kernel that walks an entry through its queries.
// 128 heads x 1024 tokens, 32 queries of 5 heads: 59 + 20 + 16 us a layer, the pages and the launch plan included; a decode-step launch pair
// per query, each reading the prompt's rows again, took 720 us.
#pragma once
#include "evict.cuh"
#include "nucleus.cuh"
#include "plan.cuh"
#include "window_attn.cuh"
#include "window_mma.cuh"

namespace ckv {

constexpr int WIN_SMEM = 32 * 1024;           // pbar of up to this many bytes stays in shared memory
constexpr int APPLY_WIDE = 1024;              // threads of window_apply_kernel for few heads' prompts of more than APPLY_LINE tokens
constexpr int APPLY_LINE = 2048;
constexpr int WH_SMALL = 1280;                // entries up to which window_hits_kernel may take CTAs of two warps

// The hit bits of one (query, head): Algorithm 1 step 1 with the query of time t over its t + 1 entries.
// grid: (W, U).  G: the query heads whose logits the attention kernel left, 0 if it left their group means.
// Bound: issue slots (some hundred instructions per warp beside those per entry):
// many searches of short prompts take CTAs of two warps.  Few searches are bound by
// the latency of one: the line is as many searches as entries and SMs, and WH_SMALL entries.  us with two warps and with
// eight, while the searches still took the means themselves: 64 heads, 300 entries, 512 searches 6.4 and 6.7, 1024 7.7 and 10.7; 16 heads, 128
// searches 6.0 and 4.5; 1024 entries, 128 searches 10.7 and 5.0, 512 12.0 and 7.7, 1024 13.3 and 12.8, 1536 15.6 and 17.3; 1280 entries, 2048 23.6
// and 28.5; 1600 entries, 4096 searches 61.2 and 60.2.
// 128 heads x 32 queries over 1000 entries: 20 us (36 with the logits of five heads to read and weigh).
// pbar lives in shared memory or, for long prompts, where it is.
template <int NTH, int G>
__global__ void __launch_bounds__(NTH) window_hits_kernel(const __grid_constant__ State st, const WindowParams p, float top_p, int literal,
                                                          int in_smem) {
  constexpr int WARPS = NTH / 32;
  pdl_wait();
  pdl_launch();
  extern __shared__ float s_pbar[];
  __shared__ NucleusSmem<NTH> s_nu;
  __shared__ int s_cnt[WARPS];
  const int u = blockIdx.y, q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int n = p.t0 + q + 1;
  unsigned* bits = p.hits + ((size_t)u * p.W + q) * p.words;
  if (literal) {   // Algorithm 1's first line as printed: nothing runs below the budget
    const int uid = ((u / st.H) * st.L + p.layer) * st.H + u % st.H;
    if (n < st.budget[uid]) {
      for (int x = tid; x < p.words; x += NTH) bits[x] = 0u;
      return;
    }
  }
  float* S = G ? p.logits + ((size_t)u * p.W + q) * G * p.Ps : p.pbar + ((size_t)u * p.W + q) * p.Ps;
  float* pb = in_smem ? s_pbar : S;
  float m[G ? G : 1], il[G ? G : 1];   // reference point, 1 / (normaliser x query heads)
  if constexpr (G > 0) {
    const float* ml = p.ml + ((size_t)u * p.W + q) * 16;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      m[g] = to_natural(ml[g]);
      il[g] = 1.0f / (ml[8 + g] * (float)G);
    }
  }
  const int base = nucleus_base<NTH>(n);
  nucleus_clear<NTH>(s_nu);
  __syncthreads();
  constexpr int BR = 4;   // entries requested together
  for (int i0 = tid; i0 < n; i0 += BR * NTH) {
    float v[BR][G ? G : 1];
#pragma unroll
    for (int x = 0; x < BR; ++x) {
      const float* r = S + min(i0 + x * NTH, n - 1);
#pragma unroll
      for (int g = 0; g < (G ? G : 1); ++g) v[x][g] = r[(size_t)g * p.Ps];
    }
#pragma unroll
    for (int x = 0; x < BR; ++x) {
      float pm = v[x][0];
      if constexpr (G > 0) pm = group_mean(v[x], m, il);
      if (i0 + x * NTH < n) {
        if (G > 0 || in_smem) pb[i0 + x * NTH] = pm;   // (mma.sync, long prompt: in the place of its own logit, which has been read)
        nucleus_add<NTH>(s_nu, base, pm);
      }
    }
  }
  __syncthreads();
  const Nucleus nu = nucleus_find<NTH>(base, top_p, s_nu, st.errword, [&](auto f) {
#pragma unroll 4
    for (int i = tid; i < n; i += NTH) f(pb[i]);
  }, [] {});
  const unsigned long long w_theta = mass_of(__uint_as_float(nu.theta));
  int eq_before = 0;   // entries of earlier rounds that carry the threshold's value
  for (int i0 = 0; i0 < n; i0 += NTH) {   // (uniform: a round may hold a barrier)
    const int i = i0 + tid;
    const uint32_t key = i < n ? __float_as_uint(pb[i]) : 0u;
    bool hit = i < n && nu.found && key > nu.theta;
    const bool eq = i < n && nu.found && key == nu.theta;
    if (nu.cnt_eq > 1) {   // the earliest carriers win: count them in order
      const unsigned m = __ballot_sync(0xffffffffu, eq);
      if (lane == 0) s_cnt[w] = __popc(m);
      __syncthreads();
      int r = eq_before + __popc(m & ((1u << lane) - 1u));
      for (int x = 0; x < WARPS; ++x) {
        if (x < w) r += s_cnt[x];
        eq_before += s_cnt[x];
      }
      if (eq) hit = nu.A + (unsigned long long)r * w_theta < nu.Pthr;
      __syncthreads();
    } else if (eq) {
      hit = nu.A < nu.Pthr;
    }
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    if (lane == 0 && (i >> 5) < p.words) bits[i >> 5] = m;
  }
}

using WindowHits = void (*)(State, WindowParams, float, int, int);
template <int NTH>
WindowHits window_hits_of(int G) {   // 0: the group means are there
  switch (G) {
    case 0: return window_hits_kernel<NTH, 0>;
    case 1: return window_hits_kernel<NTH, 1>;
    case 2: return window_hits_kernel<NTH, 2>;
    case 3: return window_hits_kernel<NTH, 3>;
    case 4: return window_hits_kernel<NTH, 4>;
    case 5: return window_hits_kernel<NTH, 5>;
    case 6: return window_hits_kernel<NTH, 6>;
    case 7: return window_hits_kernel<NTH, 7>;
    default: return window_hits_kernel<NTH, 8>;
  }
}

// Steps 2-3 of the launch's W queries for every entry in turn (an entry takes part from its own time
// on; its CRF and tau only depend on its own hits), and after the last query (last != 0) step 4: the
// head comes down to its budget.  One CTA per head behind CTA 0, which writes the layer's launch plan meanwhile (last):
// from a head's length or, where that is evict_every or more over its budget, from the budget it comes down to, so that it
// does not matter whether the head's CTA has been there.  tmp: U x tmp_stride ints.
// Bound: latency (W dependent multiply-adds per entry; with many heads the plan).  The three kernels of a window with the plan
// written here, and by one CTA of the threshold searches, which starts last and has two warps: 128 heads x 1024 tokens, 32
// queries 151 us and 155, 1024 heads x 300 tokens, 2 queries 144 and 193, 1024 heads x 256 tokens, 32 queries 241 and 292.
// Heads that fill half of the SMs at most take CTAs of 1024 threads for long prompts; with more heads the plan is what takes long, and that
// takes longer with more warps.  us a layer of windows with 1024 threads and with 256: 16 heads x 3000 tokens 96 and 102, x 6000 174 and 197, x
// 12000 338 and 377, 64 heads x 4096 129 and 143, 2 heads x 2100 60.5 and 61; but 128 heads x 2100 119 and 113, x 3000 151 and 146.
template <int NTH>
__global__ void __launch_bounds__(NTH) window_apply_kernel(const __grid_constant__ State st, const WindowParams p, int last, int evict_every,
                                                          int* tmp, int tmp_stride, const __grid_constant__ Plan plan, int plan_grid,
                                                          int plan_cl, int* plan_len) {
  __shared__ __align__(16) int sh[PL_SCRATCH];
  pdl_wait();
  if (!last) pdl_launch();
  if (blockIdx.x == 0) {
    if (last) write_plan<NTH>(st, plan, p.layer, plan_grid * NW, plan_grid, plan_cl, plan_len, sh, evict_every);
    return;
  }
  const int u = blockIdx.x - 1, seq = u / st.H, tid = threadIdx.x;
  const int uid = (seq * st.L + p.layer) * st.H + u % st.H;
  if (st.n_cur[uid] != p.P) return;   // the prompt found no pages: the head is empty
  const size_t mb = (size_t)uid * st.cap;
  int nhit = 0;
  const int lane = tid & 31;
  for (int i0 = tid - lane; i0 < p.P; i0 += NTH) {   // a warp takes 32 entries: one word of hit bits per query, a word per lane
    const int i = i0 + lane, e = min(i, p.P - 1);
    float crf = st.meta_crf[mb + e];
    int tau = st.meta_tau[mb + e];
    const unsigned* bits = p.hits + (size_t)u * p.W * p.words + (i0 >> 5);
    for (int q0 = 0; q0 < p.W; q0 += 32) {
      const unsigned mine = q0 + lane < p.W ? bits[(size_t)(q0 + lane) * p.words] : 0u;
      const int qs = min(32, p.W - q0);
      for (int q = 0; q < qs; ++q) {
        const unsigned m = __shfl_sync(0xffffffffu, mine, q);
        const int t = p.t0 + q0 + q;
        if (i <= t && ((m >> lane) & 1u)) {   // (entries past the prompt's end are later than any query)
          crf = __fadd_rn(__fmul_rn(__ldg(st.tab + (t - tau)), crf), 1.0f);
          tau = t;
          ++nhit;
        }
      }
    }
    if (i < p.P) {
      st.meta_crf[mb + i] = crf;
      st.meta_tau[mb + i] = tau;
    }
  }
  nhit = warp_sum_i(nhit);
  if ((tid & 31) == 0 && nhit) atomicAdd(&st.counters[1], (unsigned long long)nhit);
  if (tid == 0)   // entries attended: t0 + 1, t0 + 2, ..
    atomicAdd(&st.counters[0], (unsigned long long)p.W * (p.t0 + 1) + (unsigned long long)p.W * (p.W - 1) / 2);
  if (!last) return;
  const int B = st.budget[uid];
  __syncthreads();
  if (p.P - B >= evict_every && p.P > 1)
    evict_many<NTH>(st, uid, seq, p.P, min(p.P - B, p.P - 1), p.t0 + p.W - 1, true, sh, tmp + (size_t)u * tmp_stride);
}

}  // namespace ckv
