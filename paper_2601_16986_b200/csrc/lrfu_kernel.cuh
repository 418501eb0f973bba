// Algorithm 1 for the heads of one layer, one CTA per head, from the scaled logits the
// attention kernel left in the scratch (the cache itself is not read again):
//   step 1   softmax weights per query head from the logits, the attention kernel's merged
//            reference point and normaliser, group-mean probability pbar,
//            hit mask = smallest descending-pbar prefix whose exclusive mass is below p
//            (equal pbar: ascending position; nucleus.cuh);
//   step 2-3 hits: CRF <- lambda^(t - tau) CRF + 1, tau <- t; misses only get the decayed
//            CRF_temp, which is not stored;
//   step 4   the entries lowest under (CRF_temp, tau, position) leave until the head is
//            within its budget; the place of a single leaver becomes the head's hole, which
//            the next arriving token fills: nothing is moved.
// A launch without Algorithm 1 (answer stage, full-cache mode) only lets every head keep its new
// entry.  Either way the CTA that finishes last writes the layer's next launch plan (plan.cuh) when
// a head's length has drifted from the one the current plan was made for.
//
// Bound: latency, a chain of a dozen block-wide steps and dependent reads beside an attention kernel
// that saturates HBM; the attention warps of the same SM feel its issue slots and loads.  256 heads of 512 .. 1536
// entries: 22 us beside the attention kernel and 26.3 us a layer; with pbar in register arrays, a spilling path for
// heads of more than ten entries per thread, counters shared by all heads and the heads counted last, 28 and 27.4.
// (Sharing long heads among the CTAs of a cluster did not help: two to four
// CTAs for heads of 4097 entries took 48 us beside the attention kernel instead of 56, and the layer
// 36.3 us instead of 34.4; for heads of 1025 entries 17 us instead of 11.  Nor did fewer instructions by predicated loads at
// fixed offsets: 27.0 us a layer instead of 26.4.)
#pragma once
#include <atomic>

#include "evict.cuh"
#include "lrfu_launch.cuh"
#include "nucleus.cuh"
#include "plan.cuh"

namespace ckv {

template <int NTH>
struct LrfuSmem {
  NucleusSmem<NTH> nu;
  alignas(16) uint32_t least[NTH / 32][4];   // per warp: the lowest (CRF_temp, tau, position) and its list position
  int hits[NTH / 32];
  int is_last;
};
static_assert(sizeof(LrfuSmem<NT>) >= (MAX_UNITS_PER_CALL + 1) * sizeof(int), "the planner's list of lengths reuses this memory");
// Dynamic shared memory: pbar of the head's entries, and once they are dead the scratch of evict_many and of the planner.
static_assert(PL_SCRATCH >= 300, "evict_many wants 300 ints");

// Loads the compiler must leave where they are written: the kernel is bound by the latency of
// its dependent global reads (several microseconds each while the attention kernel saturates
// HBM), so every read whose address is known is requested up front, in one batch.
__device__ __forceinline__ int ld_i32(const int* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float ld_f32(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];\n" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_f32x4(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}

// A row's logits of G query heads (only those are loaded).
template <int G>
struct Row {
  float4 a;
  float b[G > 4 ? G - 4 : 1];
  __device__ __forceinline__ void load(const float* r) {
    a = ld_f32x4(r);
    if (G == 5) {
      b[0] = ld_f32(r + 4);
    } else if (G > 5) {
      const float4 t = ld_f32x4(r + 4);
      const float v[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
      for (int g = 4; g < G; ++g) b[g - 4] = v[g - 4];
    }
  }
  __device__ __forceinline__ float pbar(const float (&m)[G], const float (&invl)[G]) const {
    const float v[4] = {a.x, a.y, a.z, a.w};
    float s[G];
#pragma unroll
    for (int g = 0; g < G; ++g) s[g] = g < 4 ? v[g < 4 ? g : 0] : b[g < 4 ? 0 : g - 4];
    return group_mean(s, m, invl);
  }
};

// What the kernel requests before it knows the head's length.
template <int G>
struct Front {
  Row<G> row[FRONT];             // logit rows of this thread's first entries (index clamped to p.front)
  float m[G], l[G];              // merged reference point (log2 domain) and normaliser per query head
  int budget;
};

// The head's length after this launch, the page that backs its next entry, and the count of finished heads.
// The layer's plan names pieces by (head, j of k), so it stays correct while heads grow or
// shrink a little; a head whose group count has drifted from the planned one by an eighth (at
// least two) marks it stale, and the head that is counted last (its CTA then knows every head's new
// length) writes a new one.  In steady state (one entry arrives, one leaves) nothing is written.
// One thread calls it, once it is known how many entries leave and all threads have read n_cur: the count's release
// makes the length visible to whoever acquires the last count.
__device__ __forceinline__ bool settle_length(const DecodeParams& p, int uid, int seq, int n, int leave, int g_plan) {
  const State& st = p.st;
  int n_new = n - leave;
  if (n <= 1) n_new = n;                                     // (a head without entries stays as it is)
  else if (leave == 0) n_new = keep_all(st, uid, seq, n);
  else st.n_cur[uid] = n_new;
  const int g_new = (n_new + 1 + GRP - 1) / GRP;
  if (abs(g_new - g_plan) >= max(2, g_plan >> 3)) atomicOr(p.done_ctr + 1, 1);
  int done;
  asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;\n" : "=r"(done) : "l"(p.done_ctr) : "memory");
  if (done != (int)gridDim.x - 1) return false;
  *p.done_ctr = 0;
  return atomicExch(p.done_ctr + 1, 0) != 0;   // stale?
}

// Algorithm 1 for a head of n entries, n > 1.  pbar lives in shared memory (room for npb entries) or, for longer heads,
// in the global scratch.  Returns the number of entries that leave; a single leaver's place becomes the head's
// hole, more than one are left to the caller.  The head's length is settled on the way (sh.is_last).
template <int G, int NTH>
__device__ __forceinline__ int lrfu_unit(const DecodeParams& p, int u, int uid, int seq, int n, int g_plan, float* s_pb, int npb,
                                         LrfuSmem<NTH>& sh, const Front<G>& fr) {
  constexpr int WARPS = NTH / 32;
  const State& st = p.st;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const size_t mb = (size_t)uid * st.cap;
  const float* S = p.sc.logits + (size_t)u * p.sc.cap_s * QH;
  float* pb = n <= npb ? s_pb : p.sc.pbar + (size_t)u * p.sc.cap_s;

  // ---- step 1: pbar_i = mean_g exp(s_gi - m_g) / l_g, and the histogram of its mass
  const int base = nucleus_base<NTH>(n);
  {
    float m[G], invl[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      m[g] = to_natural(fr.m[g]);
      invl[g] = 1.0f / (fr.l[g] * (float)G);
    }
    auto put = [&](int i, float pm) {
      pb[i] = pm;
      nucleus_add<NTH>(sh.nu, base, pm);
    };
    const int nf = min(n, min(FRONT * NTH, p.front));   // entries whose rows were requested up front
#pragma unroll
    for (int k = 0; k < FRONT; ++k)
      if (tid + k * NTH < nf) put(tid + k * NTH, fr.row[k].pbar(m, invl));
    // the others in batches whose rows are requested together (clamped index, no branch): while the
    // attention kernel saturates HBM every dependent round of loads costs this CTA microseconds
    constexpr int BR = G <= 5 ? 5 : 4;
#pragma unroll 1
    for (int i0 = nf; i0 < n; i0 += BR * NTH) {
      Row<G> row[BR];
#pragma unroll
      for (int j = 0; j < BR; ++j) row[j].load(S + (size_t)min(i0 + j * NTH + tid, n - 1) * QH);
#pragma unroll
      for (int j = 0; j < BR; ++j)
        if (i0 + j * NTH + tid < n) put(i0 + j * NTH + tid, row[j].pbar(m, invl));
    }
  }
  // stored state of this thread's first entries: the reads complete under the threshold search
  int pos_r[FRONT], tau_r[FRONT];
  float crf_r[FRONT], dec_r[FRONT];
#pragma unroll
  for (int k = 0; k < FRONT; ++k) {
    const size_t i = mb + min(tid + k * NTH, n - 1);
    tau_r[k] = ld_i32(st.meta_tau + i);
    crf_r[k] = ld_f32(st.meta_crf + i);
    pos_r[k] = ld_i32(st.meta_pos + i);
  }
  __syncthreads();
  // The logit rows are dead (every thread has used what it loaded): their L2 lines are dropped instead of being written
  // back to DRAM later.  Four 32-byte rows share a 128-byte line; units start on line boundaries (cap_s is a
  // multiple of four).
  for (int x = tid; x * 4 < n; x += NTH) asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(S + (size_t)x * (4 * QH)) : "memory");
  const Nucleus nu = nucleus_find<NTH>(
      base, p.top_p, sh.nu, st.errword,
      [&](auto f) {
#pragma unroll 4
        for (int i = tid; i < n; i += NTH) f(pb[i]);
      },
      [&] {
#pragma unroll
        for (int k = 0; k < FRONT; ++k) dec_r[k] = __ldg(st.tab + (p.t - min(tau_r[k], p.t)));
      });
  const uint32_t theta = nu.theta;
  const unsigned long long w_theta = mass_of(__uint_as_float(theta));
  // The earliest of the entries that carry the threshold's value are hits: their positions are listed in the histogram's
  // place.  (Among 4097 random entries every seven thousandth search meets two.  Each of them going through all entries' values
  // held the CTA, and with it the layers that wait for it, for 290 us: 16 heads of 4097 entries took 13.9 us a layer in
  // ten passes without such a pair, 15.1, 16.3 and 17.5 with one, two and three.)
  constexpr int LISTED = 256;
  int* eq_pos = reinterpret_cast<int*>(sh.nu.hist_lo);
  static_assert(LISTED <= fine_bins(NTH), "the list takes the histogram's place");
  const bool listed = nu.cnt_eq > 1 && nu.cnt_eq <= LISTED;
  if (listed) {
    if (tid == 0) sh.nu.ncand = 0;
    __syncthreads();
    for (int i = tid; i < n; i += NTH)
      if (__float_as_uint(pb[i]) == theta) eq_pos[atomicAdd(&sh.nu.ncand, 1)] = st.meta_pos[mb + i];
    __syncthreads();
  }

  // ---- steps 2-3: CRF/tau update; step 4 candidates
  // step 4 runs once the head is evict_every entries over its budget, and then for all of them
  const int k_evict = (n - fr.budget >= p.evict_every) ? n - fr.budget : 0;
  // (every thread has read the head's length: the count's round trip runs under the update)
  if (tid == NTH - 32) sh.is_last = settle_length(p, uid, seq, n, min(k_evict, n - 1), g_plan);
  uint32_t bk0 = 0xffffffffu, bk1 = 0xffffffffu, bk2 = 0xffffffffu;
  int bidx = -1, nhit = 0;
  auto update = [&](int i, int pos_i, int tau, float crf, float dec) {
    const float pm = pb[i];
    const uint32_t key = __float_as_uint(pm);
    bool hit = key > theta && nu.found;
    if (key == theta && nu.found) {
      unsigned long long before = 0;
      if (listed) {
#pragma unroll 4
        for (int x = 0; x < nu.cnt_eq; ++x) before += eq_pos[x] < pos_i;
      } else if (nu.cnt_eq > 1) {
#pragma unroll 4
        for (int x = 0; x < n; ++x)
          before += (__float_as_uint(pb[x]) == theta) && (st.meta_pos[mb + x] < pos_i);
      }
      hit = (nu.A + before * w_theta) < nu.Pthr;
    }
    float ct = __fmul_rn(dec, crf);
    if (hit) {
      ct = __fadd_rn(ct, 1.0f);
      tau = p.t;
      st.meta_crf[mb + i] = ct;
      st.meta_tau[mb + i] = tau;
      ++nhit;
    }
    const uint32_t c0 = __float_as_uint(ct), c1 = (uint32_t)tau, c2 = (uint32_t)pos_i;
    const bool less = (c0 != bk0) ? (c0 < bk0) : ((c1 != bk1) ? (c1 < bk1) : (c2 < bk2));
    if (less) { bk0 = c0; bk1 = c1; bk2 = c2; bidx = i; }
  };
#pragma unroll
  for (int k = 0; k < FRONT; ++k)
    if (tid + k * NTH < n) update(tid + k * NTH, pos_r[k], tau_r[k], crf_r[k], dec_r[k]);
#pragma unroll 1
  for (int i0 = FRONT * NTH; i0 < n; i0 += FRONT * NTH) {   // a long head: the next FRONT entries of every thread
#pragma unroll
    for (int k = 0; k < FRONT; ++k) {
      const size_t i = mb + min(i0 + tid + k * NTH, n - 1);
      tau_r[k] = ld_i32(st.meta_tau + i);
      crf_r[k] = ld_f32(st.meta_crf + i);
      pos_r[k] = ld_i32(st.meta_pos + i);
    }
#pragma unroll
    for (int k = 0; k < FRONT; ++k) dec_r[k] = __ldg(st.tab + (p.t - min(tau_r[k], p.t)));
#pragma unroll
    for (int k = 0; k < FRONT; ++k)
      if (i0 + tid + k * NTH < n) update(i0 + tid + k * NTH, pos_r[k], tau_r[k], crf_r[k], dec_r[k]);
  }
  // the lowest (CRF_temp, tau, position) of a warp's lanes, word by word (positions are unique)
  auto least = [&]() {
    const uint32_t m0 = __reduce_min_sync(0xffffffffu, bk0);
    const uint32_t m1 = __reduce_min_sync(0xffffffffu, bk0 == m0 ? bk1 : 0xffffffffu);
    const uint32_t m2 = __reduce_min_sync(0xffffffffu, bk0 == m0 && bk1 == m1 ? bk2 : 0xffffffffu);
    bidx = (int)__reduce_min_sync(0xffffffffu, bk0 == m0 && bk1 == m1 && bk2 == m2 ? (uint32_t)bidx : 0xffffffffu);
    bk0 = m0; bk1 = m1; bk2 = m2;
  };
  least();
  nhit = __reduce_add_sync(0xffffffffu, nhit);
  if (lane == 0) {
    *reinterpret_cast<uint4*>(sh.least[w]) = make_uint4(bk0, bk1, bk2, (uint32_t)bidx);
    sh.hits[w] = nhit;
  }
  __syncthreads();
  if (w == 0) {
    const uint4 a = *reinterpret_cast<const uint4*>(sh.least[min(lane, WARPS - 1)]);
    bk0 = a.x; bk1 = a.y; bk2 = a.z; bidx = (int)a.w;
    least();
    nhit = __reduce_add_sync(0xffffffffu, lane < WARPS ? sh.hits[min(lane, WARPS - 1)] : 0);
    if (lane == 0) {
      if (k_evict == 1) st.hole[uid] = bidx;   // the leaving entry's place is where the next arriving token is written
      count_unit(st, uid, n, nhit, k_evict == 1 ? 1 : 0);
    }
  }
  return k_evict;
}

template <int G, int NTH>
__global__ void __maxnreg__(48) lrfu_kernel(const __grid_constant__ DecodeParams p, int npb) {
  extern __shared__ __align__(16) float s_pb[];
  __shared__ __align__(16) LrfuSmem<NTH> sh;
  const State& st = p.st;
  const int u = blockIdx.x, seq = u / st.H, head = u % st.H;
  const int uid = (seq * st.L + p.layer) * st.H + head;
  // one batch of requests: the length, the budget, the softmax reference, and the logit rows the
  // common path needs (requested for a full thread's worth, clamped to the expected length)
  const int n = ld_i32(st.n_cur + uid) + 1;
  const int g_plan = threadIdx.x == NTH - 32 ? ld_i32(p.plan.gplan + u) : 0;
  bool settled = false;
  if (p.track) {
    // the stored state is asked into L2: every round trip to DRAM costs microseconds beside a saturated HBM
    for (int x = threadIdx.x; x * 32 < p.front; x += NTH) {
      const size_t at = (size_t)uid * st.cap + x * 32;
      asm volatile("prefetch.global.L2 [%0];\n" ::"l"(st.meta_tau + at));
      asm volatile("prefetch.global.L2 [%0];\n" ::"l"(st.meta_crf + at));
      asm volatile("prefetch.global.L2 [%0];\n" ::"l"(st.meta_pos + at));
    }
    Front<G> fr;
    fr.budget = ld_i32(st.budget + uid);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      fr.m[g] = ld_f32(p.sc.mfin + u * (2 * QH) + g);
      fr.l[g] = ld_f32(p.sc.mfin + u * (2 * QH) + QH + g);
    }
    {
      const float* S = p.sc.logits + (size_t)u * p.sc.cap_s * QH;
#pragma unroll
      for (int k = 0; k < FRONT; ++k) fr.row[k].load(S + (size_t)min((int)threadIdx.x + k * NTH, p.front - 1) * QH);
    }
    nucleus_clear<NTH>(sh.nu);
    __syncthreads();
    if (n > 1 && !(p.literal && n < fr.budget)) {   // (Algorithm 1's first line as printed: nothing runs below the budget)
      int leave = lrfu_unit<G, NTH>(p, u, uid, seq, n, g_plan, s_pb, npb, sh, fr);
      settled = true;
      if (leave > 1) {
        __syncthreads();   // every thread's CRFs are written, pbar is dead
        if (leave > p.evict_every && threadIdx.x == 0) atomicOr(st.errword, ERR_OVER_EVICT);
        leave = min(leave, n - 1);
        evict_many<NTH>(st, uid, seq, n, leave, p.t, false, reinterpret_cast<int*>(s_pb), reinterpret_cast<int*>(p.sc.pbar + (size_t)u * p.sc.cap_s));
      }
    }
  }
  if (!settled && threadIdx.x == NTH - 32) {   // no Algorithm 1: the head keeps its new entry
    sh.is_last = settle_length(p, uid, seq, n, 0, g_plan);
    if (n > 1) count_unit(st, uid, n, 0, 0);
    else atomicOr(st.errword, ERR_EMPTY);   // the head has no entries and no page: nothing was attended
  }
  __syncthreads();
  if (!sh.is_last) return;
  // The planner's list of lengths takes the place of this CTA's histogram or, where that is too small, a
  // place of its own.  (Not the pbar scratch: other heads' CTAs may still be reading theirs.)
  write_plan<NTH>(st, p.plan, p.layer, p.plan_warps, p.plan_grid, p.cl,
                  NTH >= NT ? reinterpret_cast<int*>(&sh) : p.plan_len, reinterpret_cast<int*>(s_pb));
}

template <int G, int NTH>
cudaError_t launch_lrfu(const DecodeParams& p, int npb, int heads, cudaStream_t s) {
  // the same shared-memory carve-out as the attention kernel, so that CTAs of both can be
  // resident on one SM at the same time
  // (function attributes are kept per device)
  static std::atomic<bool> prepared[MAX_DEVICES] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  if (!prepared[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(lrfu_kernel<G, NTH>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    prepared[dev].store(true, std::memory_order_release);
  }
  lrfu_kernel<G, NTH><<<heads, NTH, std::max(npb, PL_SCRATCH) * sizeof(float), s>>>(p, npb);
  return cudaGetLastError();
}

}  // namespace ckv
