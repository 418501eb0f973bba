// Prompt insertion.  A prompt with a last query goes through three kernels: the scores of all P
// tokens (prefill_score_kernel), Algorithm 1 on them (prefill_select_kernel: hits, survivors, the
// pages that back them) and the survivors' rows (prefill_rows_kernel, whose first CTA writes the
// layer's launch plan beside the copying).  The pool never holds more than the budget.  A prompt
// that is kept as it is (full cache, observation window) only takes its pages and copies its rows.
#pragma once
#include "attn_kernel.cuh"
#include "nucleus.cuh"
#include "plan.cuh"
#include "tma.cuh"

namespace ckv {

// The plan as a kernel of its own: one CTA per layer of `layers` consecutive layers starting at
// layer0 (after a prompt insertion, a reallocation, or any edit of a head's state from the host).
__global__ void __launch_bounds__(NT) plan_kernel(const __grid_constant__ State st, const Plan* plans, int layer0, int nWarps, int grid, int cl) {
  __shared__ int s_gs[MAX_UNITS_PER_CALL + 1];
  __shared__ int s_red[320];
  write_plan(st, plans[layer0 + blockIdx.x], layer0 + blockIdx.x, nWarps, grid, cl, s_gs, s_red);
}

constexpr int SEL_NT = 1024;            // threads of prefill_select_kernel
constexpr int SEL_SMEM = 160 * 1024;    // pbar of up to this many bytes stays in shared memory

constexpr int SCORE_KEYS = 32;          // keys of an item of prefill_score_kernel: two tiles of 64 channels
constexpr int SCORE_HALF = SCORE_KEYS * 128, SCORE_ITEM = 2 * SCORE_HALF;
constexpr int SCORE_STAGES = 3;
constexpr int SCORE_SMEM = 1024 + NW * SCORE_STAGES * (SCORE_ITEM + 8);

// The scaled logits of the last query's G heads against the prompt's keys, and per item the softmax
// reference point (log2 domain) and normaliser of its keys.  Items are (sequence, 32 tokens, head), head fastest, and a warp takes every
// `warps`-th (a multiple of H where that is 1, 2, 4 or 8: its queries then only change with the sequence).
//   mk: k [batch][P][H][128], boxes of 64 channels x 32 tokens of a head   q_last: [batch][Hq][128]   partials: [U][chunks][16] = m, l
// Bound: HBM.  Every warp keeps a ring of three items full by TMA, like the attention kernel's of pages, and eight warps that
// read the heads of the same tokens keep to the same DRAM pages; the products are mma.sync with keys on M and the (padded) query
// heads on N, 16 per item.  64 heads x 9350 tokens (153 MB of keys, 19 MB of
// logits): 35.5 us (a thread per key with fp32 multiply-adds from shared memory, three
// CTAs of 64 KB an SM: 45.5 us, half of its cycles spent on 16-byte broadcasts of the queries), 128 heads x 512 tokens 8.0 (9.3).
// Which entries survive hangs on the last bits of the logits where an entry lies at the threshold.  Errors of a scaled logit against 64 bits, rms and largest
// of 524288, and of one chain of multiply-adds: keys N(0, 1) 6.95e-8, 8.8e-7 (7.25e-8, 1.1e-6), times 3 (outliers) 2.15e-7, 2.3e-6
// (2.2e-7, 3.7e-6), times 8 (sinks) 5.85e-7, 6.6e-6 (6e-7, 9.6e-6).  Of 17408 heads of prompts with sinks and outliers (2000 tokens to 400, 9350 to
// 2400; 1, 4 and 8 query heads) two keep another entry than in 64 bits, with either kernel.
__global__ void __launch_bounds__(NT, 1) prefill_score_kernel(Scratch sc, const __grid_constant__ CUtensorMap mk, const __nv_bfloat16* __restrict__ q_last,
                                                              int batch, int H, int G, int P, int warps, float scale, float scale_log2, int* errword) {
  extern __shared__ unsigned char s_raw[];
  pdl_launch();   // (an ordinary launch: what was queued before it has ended)
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gid = lane >> 2, tig = lane & 3, mi = lane >> 3, r8 = lane & 7;
  const uint32_t s0 = (smem_u32(s_raw) + 1023) & ~1023u, ring = s0 + w * (SCORE_STAGES * SCORE_ITEM);
  const uint32_t bars = s0 + NW * SCORE_STAGES * SCORE_ITEM + w * (SCORE_STAGES * 8);
  if (lane < SCORE_STAGES) mbar_init(bars + lane * 8, 1);
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  __syncwarp();
  const int chunks = (P + SCORE_KEYS - 1) / SCORE_KEYS, items = batch * chunks * H, first = blockIdx.x * NW + w;
  auto fetch = [&](int i, int stage) {   // by lane 0
    const int head = i % H, at = i / H;
    mbar_expect_tx(bars + stage * 8, SCORE_ITEM);
    for (int x = 0; x < 2; ++x)
      tma_tile(ring + stage * SCORE_ITEM + x * SCORE_HALF, &mk, 64 * x, head, at % chunks * SCORE_KEYS, at / chunks, bars + stage * 8);
  };
  if (first >= warps) return;
  if (lane == 0)
    for (int x = 0; x < SCORE_STAGES; ++x)
      if (first + x * warps < items) fetch(first + x * warps, x);
  uint32_t qb[8][2];
  int have = -1;   // the head whose queries qb holds
  const uint32_t krow = (uint32_t)(((mi & 1) * 8 + r8) * 128), khalf = (uint32_t)(mi >> 1);
  int stage = 0;
  uint32_t phase = 0;
#pragma unroll 1
  for (int i = first; i < items; i += warps) {
    const int head = i % H, at = i / H, chunk = at % chunks, u = at / chunks * H + head;
    if (u != have) {   // the G queries as B fragments
      have = u;
      const unsigned short* q = reinterpret_cast<const unsigned short*>(q_last) + ((size_t)u * G + gid) * HD;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int c = ks * 16 + x * 8 + tig * 2;
          qb[ks][x] = gid < G ? (uint32_t)__ldg(q + c) | ((uint32_t)__ldg(q + c + 1) << 16) : 0u;
        }
    }
    if (!mbar_wait_bounded(bars + stage * 8, phase)) {
      if (lane == 0) atomicOr(errword, ERR_COPY_TIMEOUT);
      for (int x = 0; x < SCORE_STAGES; ++x) mbar_wait_bounded(bars + x * 8, x < stage ? phase ^ 1u : phase);   // what else is on its way
      return;
    }
    const uint32_t tile = ring + stage * SCORE_ITEM;
    float* S = sc.logits + ((size_t)u * sc.cap_s + chunk * SCORE_KEYS) * QH;
    float t[SCORE_KEYS / 16][4];   // logits in the log2 domain
    float c0 = -INFINITY, c1 = -INFINITY;
#pragma unroll
    for (int m = 0; m < SCORE_KEYS / 16; ++m) {
      float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ks = 0; ks < 8; ks += 2) {   // two chains of four
        uint32_t a[4], a2[4];
        const uint32_t ka = tile + (ks >> 2) * SCORE_HALF + m * 16 * 128 + krow;
        ldsm_x4(a, ka + ((((ks & 3) * 2 + khalf) ^ r8) << 4));
        ldsm_x4(a2, ka + ((((ks & 3) * 2 + 2 + khalf) ^ r8) << 4));
        mma_bf16(s, a, qb[ks][0], qb[ks][1]);
        mma_bf16(s2, a2, qb[ks + 1][0], qb[ks + 1][1]);
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int key = m * 16 + x * 8 + gid;
        const float a = s[2 * x] + s2[2 * x], b = s[2 * x + 1] + s2[2 * x + 1];
        const bool there = chunk * SCORE_KEYS + key < P;
        if (there) *reinterpret_cast<float2*>(S + (size_t)key * QH + 2 * tig) = make_float2(__fmul_rn(a, scale), __fmul_rn(b, scale));
        t[m][2 * x] = there ? a * scale_log2 : -INFINITY;
        t[m][2 * x + 1] = there ? b * scale_log2 : -INFINITY;
        c0 = fmaxf(c0, t[m][2 * x]);
        c1 = fmaxf(c1, t[m][2 * x + 1]);
      }
    }
    __syncwarp();   // the stage has been read
    if (lane == 0 && i + SCORE_STAGES * warps < items) fetch(i + SCORE_STAGES * warps, stage);
    if (++stage == SCORE_STAGES) { stage = 0; phase ^= 1u; }
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) {
      c0 = fmaxf(c0, __shfl_xor_sync(0xffffffffu, c0, x));
      c1 = fmaxf(c1, __shfl_xor_sync(0xffffffffu, c1, x));
    }
    float l0 = 0.f, l1 = 0.f;   // (an item has a key, so the reference points are finite)
#pragma unroll
    for (int m = 0; m < SCORE_KEYS / 16; ++m) {
      l0 += ex2(t[m][0] - c0) + ex2(t[m][2] - c0);
      l1 += ex2(t[m][1] - c1) + ex2(t[m][3] - c1);
    }
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) {
      l0 += __shfl_xor_sync(0xffffffffu, l0, x);
      l1 += __shfl_xor_sync(0xffffffffu, l1, x);
    }
    if (gid == 0) {
      float* ml = sc.partials + ((size_t)u * chunks + chunk) * (2 * QH) + 2 * tig;
      *reinterpret_cast<float2*>(ml) = make_float2(c0, c1);
      *reinterpret_cast<float2*>(ml + QH) = make_float2(l0, l1);
    }
  }
}

// Exclusive scan of one int per thread over the SEL_NT threads; red: SEL_NT / 32 ints.
__device__ __forceinline__ int sel_scan(int v, int* red, int& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  __syncthreads();
  if (lane == 31) red[w] = inc;
  __syncthreads();
  const int mine = red[lane];   // SEL_NT / 32 = 32 warps
  int acc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, acc, o);
    if (lane >= o) acc += x;
  }
  total = __shfl_sync(0xffffffffu, acc, 31);
  return __shfl_sync(0xffffffffu, acc - mine, w) + inc - v;
}

// Takes `need` pages for a head from its sequence's free list; the head is empty when there are not
// enough.  All threads of the CTA call it (`threads` of them).
__device__ __forceinline__ bool take_pages(const State& st, int uid, int seq, int need, int n, int threads, int* s_top) {
  if (threadIdx.x == 0) {
    int top = atomicSub(&st.free_top[seq], need);
    if (top < need) {
      atomicAdd(&st.free_top[seq], need);
      atomicOr(st.errword, ERR_FREE_UNDERFLOW);
      top = -1;
      st.n_cur[uid] = 0; st.hole[uid] = 0;
    } else {
      st.n_cur[uid] = n; st.hole[uid] = n; st.npages[uid] = need;
    }
    *s_top = top;
  }
  __syncthreads();
  const int top = *s_top;
  if (top < 0) return false;
  const int* stack = st.free_stack + (size_t)seq * st.pages_per_seq;
  int* pt = st.ptab + (size_t)uid * st.capg;
  for (int j = threadIdx.x; j < need; j += threads) pt[j] = stack[top - 1 - j];
  return true;
}

// Algorithm 1 for a prompt of P tokens scored by its last query at t = P - 1, one CTA per head.
// All entries start with CRF 0 and tau = P - 1, so an entry's CRF_temp is 1 if it is a hit, else 0,
// and the order of leaving, (CRF_temp, tau, position), is: misses by position, then hits by
// position.  Survivors therefore follow from two prefix counts; they are listed by position.
// fixed_budget > 0 sets the heads' budget first.
// Bound: latency (a few block-wide steps over 36 bytes per token); 1024 threads keep a prompt of
// 10 000 tokens at ten entries per thread, pbar in shared memory up to SEL_SMEM bytes.
// 64 heads x 9350 tokens cut to 935: 22 us (25.9 with a pass over the logits for the normalisers, which the items bring now);
// the decode step's Algorithm 1 kernel with its radix
// select over 96-bit keys in global memory took 286 us.  128 heads x 512 tokens: 10.9 us.
__global__ void __launch_bounds__(SEL_NT) prefill_select_kernel(State st, Scratch sc, int layer, int P, int G, int chunks,
                                                                float top_p, int evict_every, int literal,
                                                                int fixed_budget, int in_smem) {
  extern __shared__ float s_pbar[];
  __shared__ NucleusSmem<SEL_NT> s_nu;
  __shared__ float s_m[QH], s_il[QH];
  __shared__ int s_red[SEL_NT / 32];
  __shared__ int s_top;
  const int u = blockIdx.x, seq = u / st.H, head = u % st.H;
  const int uid = (seq * st.L + layer) * st.H + head;
  const size_t mb = (size_t)uid * st.cap;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  nucleus_clear<SEL_NT>(s_nu);   // (a barrier follows long before the histogram is filled)
  pdl_wait();
  pdl_launch();
  const int B = fixed_budget > 0 ? fixed_budget : st.budget[uid];
  if (fixed_budget > 0 && tid == 0) st.budget[uid] = fixed_budget;
  const float* S = sc.logits + (size_t)u * sc.cap_s * QH;
  if (w < G) {   // warp g: query head g's reference point and normaliser
    const float* pp = sc.partials + (size_t)u * chunks * (2 * QH) + w;
    float m = -INFINITY, l = 0.f;
    for (int c = lane; c < chunks; c += 32) m = fmaxf(m, pp[c * (2 * QH)]);
    m = warp_max(m);
#pragma unroll 4
    for (int c = lane; c < chunks; c += 32) l = fmaf(pp[c * (2 * QH) + QH], ex2(pp[c * (2 * QH)] - m), l);
    l = warp_sum(l);
    if (lane == 0) {
      s_m[w] = m;
      s_il[w] = 1.0f / (l * (float)G);
    }
  }
  __syncthreads();
  // ---- step 1: pbar_i = mean_g exp(s_gi - m_g) / l_g
  float mx[QH], il[QH];
#pragma unroll
  for (int g = 0; g < QH; ++g) {
    mx[g] = g < G ? to_natural(s_m[g]) : 0.f;
    il[g] = g < G ? s_il[g] : 0.f;
  }
  float* pb = in_smem ? s_pbar : sc.pbar + (size_t)u * sc.cap_s;
  const bool track = !(literal && P < B);   // Algorithm 1's first line as printed: nothing runs below the budget
  const int base = nucleus_base<SEL_NT>(P);
  constexpr int BR = 3;                       // rows requested together
  for (int i0 = tid; i0 < P; i0 += BR * SEL_NT) {
    float4 ra[BR], rb[BR];
#pragma unroll
    for (int x = 0; x < BR; ++x) {
      const float* r = S + (size_t)min(i0 + x * SEL_NT, P - 1) * QH;
      ra[x] = *reinterpret_cast<const float4*>(r);
      rb[x] = G > 4 ? *reinterpret_cast<const float4*>(r + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int x = 0; x < BR; ++x) {
      const int i = i0 + x * SEL_NT;
      const float sv[8] = {ra[x].x, ra[x].y, ra[x].z, ra[x].w, rb[x].x, rb[x].y, rb[x].z, rb[x].w};
      const float pm = group_mean(sv, mx, il, G);
      if (i < P) {
        pb[i] = pm;
        if (track) nucleus_add<SEL_NT>(s_nu, base, pm);
      }
    }
  }
  __syncthreads();
  Nucleus nu{};
  nu.theta = 0xffffffffu;
  if (track)
    nu = nucleus_find<SEL_NT>(base, top_p, s_nu, st.errword, [&](auto f) {
#pragma unroll 4
      for (int i = tid; i < P; i += SEL_NT) f(pb[i]);
    }, [] {});
  // ---- hits and survivors: every thread owns a run of consecutive tokens (of odd length: the
  // threads of a warp then read different banks)
  const int per = ((P + SEL_NT - 1) / SEL_NT) | 1, lo = min(P, tid * per), hi = min(P, lo + per);
  const uint32_t theta = nu.theta;
  const unsigned long long w_theta = mass_of(__uint_as_float(theta));
  int eq = 0, tot;
  if (nu.found && nu.cnt_eq > 1)
    for (int i = lo; i < hi; ++i) eq += __float_as_uint(pb[i]) == theta;
  const int eq0 = sel_scan(eq, s_red, tot);   // tokens before this run that carry the threshold's value
  auto each_hit = [&](auto f) {               // f(token, hit)
    int r = eq0;
    for (int i = lo; i < hi; ++i) {
      const uint32_t key = __float_as_uint(pb[i]);
      bool hit = nu.found && key > theta;
      if (nu.found && key == theta) { hit = nu.A + (unsigned long long)r * w_theta < nu.Pthr; ++r; }
      f(i, hit);
    }
  };
  int hits = 0, nhit;
  each_hit([&](int, bool hit) { hits += hit; });
  const int hit0 = sel_scan(hits, s_red, nhit);
  const int leave = P - B >= evict_every ? min(P - B, P - 1) : 0, nkeep = P - leave;
  auto each_kept = [&](auto f) {   // f(token, hit) for the survivors of this thread's run
    int h = hit0;
    each_hit([&](int i, bool hit) {
      const bool keep = hit ? h >= nhit - nkeep : i - h >= leave;
      h += hit;
      if (keep) f(i, hit);
    });
  };
  int kept = 0;
  each_kept([&](int, bool) { ++kept; });
  int d = sel_scan(kept, s_red, tot);
  each_kept([&](int i, bool hit) {
    st.meta_pos[mb + d] = i;
    st.meta_tau[mb + d] = P - 1;
    st.meta_crf[mb + d] = hit ? 1.0f : 0.0f;
    ++d;
  });
  if (tid == 0) {
    atomicAdd(&st.counters[0], (unsigned long long)P);
    if (nhit) atomicAdd(&st.counters[1], (unsigned long long)nhit);
    if (leave) atomicAdd(&st.counters[2], (unsigned long long)leave);
  }
  take_pages(st, uid, seq, nkeep / GRP + 1, nkeep, SEL_NT, &s_top);
}

// A prompt that is kept as it is: the pages that back list positions 0 .. P (the P entries and the
// place of the next arrival), one CTA per head.  meta: the entries' stored state as well, tau = the token's own arrival
// time (its queries are replayed).
__global__ void __launch_bounds__(NT) prefill_take_kernel(State st, int layer, int P, int meta) {
  __shared__ int s_top;
  pdl_launch();   // (an ordinary launch: what was queued before it has ended)
  const int u = blockIdx.x, seq = u / st.H, uid = (seq * st.L + layer) * st.H + u % st.H;
  if (meta) {
    const size_t mb = (size_t)uid * st.cap;
    for (int i = threadIdx.x; i < P; i += NT) {
      st.meta_pos[mb + i] = i;
      st.meta_tau[mb + i] = i;
      st.meta_crf[mb + i] = 0.0f;
    }
  }
  take_pages(st, uid, seq, P / GRP + 1, P, NT, &s_top);
}

constexpr int ROWS_SURVIVORS = 0;   // entries are listed in the metadata (their token positions)
constexpr int ROWS_ALL_LAST = 1;    // entry i is token i: metadata written here, tau = P - 1
constexpr int ROWS_ALL = 2;         // ... metadata written before

// The rows of a layer's entries into their pages.  k, v: [batch][P][H][128].  CTA 0 writes the
// layer's launch plan meanwhile (plan_warps > 0); the others, `per_head` for every head, copy a
// page per warp and turn, eight rows of 512 bytes in flight.  Bound: HBM, 1 KB moved per entry, or
// the plan when there is little to copy: 64 heads x 935 entries in 10 us (one
// CTA per head: 85 us), 128 heads x 512 entries in 11 us (insertion, plan kernel and a scoring
// pass of the attention kernel: 81 us).
__global__ void __launch_bounds__(NT) prefill_rows_kernel(const __grid_constant__ State st, const __grid_constant__ Plan plan, int layer, const unsigned char* __restrict__ k,
                                                          const unsigned char* __restrict__ v, int P, int mode, int per_head,
                                                          int plan_warps, int plan_grid, int plan_cl) {
  __shared__ int s_gs[MAX_UNITS_PER_CALL + 1];
  __shared__ int s_red[320];
  pdl_wait();
  if (plan_warps == 0) pdl_launch();   // (a window's kernels follow; else this is the prompt's last)
  if (blockIdx.x == 0) {
    if (plan_warps > 0) write_plan(st, plan, layer, plan_warps, plan_grid, plan_cl, s_gs, s_red);
    return;
  }
  const int u = (blockIdx.x - 1) / per_head, b = (blockIdx.x - 1) % per_head, seq = u / st.H, head = u % st.H;
  const int uid = (seq * st.L + layer) * st.H + head;
  const size_t mb = (size_t)uid * st.cap;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = st.n_cur[uid];
  const int* pt = st.ptab + (size_t)uid * st.capg;
  unsigned char* poolseq = st.pool + (size_t)seq * st.pages_per_seq * PAGE_BYTES;
  const unsigned char* src = (lane < 16 ? k : v) + ((size_t)seq * P * st.H + head) * ROW_BYTES + (lane & 15) * 16;
  const size_t row = (size_t)st.H * ROW_BYTES;
  for (int pg = b * NW + w; pg * GRP < n; pg += per_head * NW) {
    const int cnt = min(GRP, n - pg * GRP), i = pg * GRP + min(lane & 15, cnt - 1);
    const int page = pt[pg];
    int tok = i;
    if (mode == ROWS_SURVIVORS) {
      tok = min(max(st.meta_pos[mb + i], 0), P - 1);
    } else if (mode == ROWS_ALL_LAST && lane < cnt) {
      st.meta_pos[mb + i] = i;
      st.meta_tau[mb + i] = P - 1;
      st.meta_crf[mb + i] = 0.0f;
    }
    unsigned char* dst = poolseq + (size_t)page * PAGE_BYTES;
#pragma unroll
    for (int e0 = 0; e0 < GRP; e0 += 8) {
      uint4 r[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)   // (rows past the head's end repeat its last one and are not stored)
        r[e] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)__shfl_sync(0xffffffffu, tok, e0 + e) * row));
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e0 + e < cnt) *reinterpret_cast<uint4*>(dst + chunk_offset(e0 + e, lane)) = r[e];
    }
  }
}

}  // namespace ckv
