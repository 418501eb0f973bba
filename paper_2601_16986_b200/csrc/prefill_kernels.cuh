// Prompt insertion.  A prompt with a last query goes through three kernels: the scores of all P
// tokens (prefill_score_kernel), Algorithm 1 on them (prefill_select_kernel: hits, survivors, the
// pages that back them) and the survivors' rows (prefill_rows_kernel, whose first CTA writes the
// layer's launch plan beside the copying).  The pool never holds more than the budget.  A prompt
// that is kept as it is (full cache, observation window) only takes its pages and copies its rows.
#pragma once
#include "common.cuh"
#include "nucleus.cuh"
#include "plan.cuh"

namespace ckv {

// The plan as a kernel of its own: one CTA per layer of `layers` consecutive layers starting at
// layer0 (after a prompt insertion, a reallocation, or any edit of a head's state from the host).
__global__ void __launch_bounds__(NT) plan_kernel(State st, const Plan* plans, int layer0, int nWarps, int grid) {
  __shared__ int s_gs[MAX_UNITS_PER_CALL + 1];
  __shared__ int s_red[320];
  write_plan(st, plans[layer0 + blockIdx.x], layer0 + blockIdx.x, nWarps, grid, s_gs, s_red);
}

constexpr int SEL_NT = 1024;            // threads of prefill_select_kernel
constexpr int SEL_SMEM = 160 * 1024;    // pbar of up to this many bytes stays in shared memory

// Keys per CTA of prefill_score_kernel: long enough that a CTA's start (its queries) is paid for by
// several groups per warp, short enough for four CTAs per SM (two are resident) to be there at all.
__host__ __device__ __forceinline__ int score_chunk(int P, int U) {
  int chunk = 512;
  while (chunk > 128 && (long long)U * ((P + chunk - 1) / chunk) < 592) chunk >>= 1;
  return chunk;
}

__device__ __forceinline__ void score_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The scaled logits of the last query's G heads against the prompt's keys, and per CTA the softmax
// reference point (log2 domain) and normaliser of its chunk of keys.
//   k: [batch][P][H][128]   q_last: [batch][Hq][128]   part: [U][chunks][16] = m[8], l[8]
// Bound: HBM (the keys are read once, 256 bytes each).  A warp takes 16 keys at a time straight
// from global memory into MMA fragments: which channels form a k-step is free as long as both
// operands agree, so lane tig of a row takes the 16-byte pieces tig, tig + 4, ... (two whole sectors
// per row and load), and the next 16 keys are requested before the current ones are used.
// 64 heads x 9350 tokens (153 MB): 37.6 us, 4.1 TB/s; one CTA per head with a thread per key and
// fp32 multiply-adds took 252 us.  128 heads x 512 tokens: 9.6 us.
__global__ void __launch_bounds__(NT, 2) prefill_score_kernel(Scratch sc, const __nv_bfloat16* __restrict__ k,
                                                              const __nv_bfloat16* __restrict__ q_last, int H, int P, int G,
                                                              int chunk, float scale, float scale_log2) {
  __shared__ float s_m[NW][QH], s_l[NW][QH];
  const int u = blockIdx.y, seq = u / H, head = u % H;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int end = min(P, (int)(blockIdx.x + 1) * chunk);
  // queries as B fragments: k-step 2 j + h of lane tig holds channels 8 (tig + 4 j) + 4 h .. + 3
  uint32_t qb[8][2];
  {
    const unsigned short* q16 = reinterpret_cast<const unsigned short*>(q_last) + ((size_t)u * G + gid) * HD;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int c = 8 * (tig + 4 * (s >> 1)) + 4 * (s & 1);
#pragma unroll
      for (int x = 0; x < 2; ++x)
        qb[s][x] = gid < G ? (uint32_t)q16[c + 2 * x] | ((uint32_t)q16[c + 2 * x + 1] << 16) : 0u;
    }
  }
  const size_t row = (size_t)H * HD * 2;   // bytes from one token's key of this head to the next one's
  const unsigned char* kb = reinterpret_cast<const unsigned char*>(k) + ((size_t)seq * P * H + head) * (HD * 2) + tig * 16;
  auto load = [&](int i0, uint4 (&a)[4], uint4 (&b)[4]) {
    const unsigned char* pa = kb + (size_t)min(i0 + gid, P - 1) * row;
    const unsigned char* pb = kb + (size_t)min(i0 + gid + 8, P - 1) * row;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a[j] = __ldg(reinterpret_cast<const uint4*>(pa + 64 * j));
      b[j] = __ldg(reinterpret_cast<const uint4*>(pb + 64 * j));
    }
  };
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  float* S = sc.logits + (size_t)u * sc.cap_s * QH + 2 * tig;
  uint4 a[4], b[4];
  int i0 = blockIdx.x * chunk + w * GRP;
  if (i0 < end) load(i0, a, b);
#pragma unroll 1
  for (; i0 < end; i0 += NW * GRP) {
    uint4 na[4], nb[4];
    if (i0 + NW * GRP < end) load(i0 + NW * GRP, na, nb);
    float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      score_mma(s, a[j].x, b[j].x, a[j].y, b[j].y, qb[2 * j][0], qb[2 * j][1]);
      score_mma(s2, a[j].z, b[j].z, a[j].w, b[j].w, qb[2 * j + 1][0], qb[2 * j + 1][1]);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) s[x] += s2[x];
    const bool v0 = i0 + gid < end, v1 = i0 + gid + 8 < end;
    float* lr = S + (size_t)(i0 + gid) * QH;
    if (v0) *reinterpret_cast<float2*>(lr) = make_float2(__fmul_rn(s[0], scale), __fmul_rn(s[1], scale));
    if (v1) *reinterpret_cast<float2*>(lr + 8 * QH) = make_float2(__fmul_rn(s[2], scale), __fmul_rn(s[3], scale));
    const float t0 = v0 ? s[0] * scale_log2 : -INFINITY, t1 = v0 ? s[1] * scale_log2 : -INFINITY;
    const float t2 = v1 ? s[2] * scale_log2 : -INFINITY, t3 = v1 ? s[3] * scale_log2 : -INFINITY;
    const float c0 = fmaxf(t0, t2), c1 = fmaxf(t1, t3);
    if (c0 > m0) { l0 *= ex2(m0 - c0); m0 = c0; }
    if (c1 > m1) { l1 *= ex2(m1 - c1); m1 = c1; }
    if (v0) { l0 += ex2(t0 - m0); l1 += ex2(t1 - m1); }
    if (v1) { l0 += ex2(t2 - m0); l1 += ex2(t3 - m1); }
#pragma unroll
    for (int j = 0; j < 4; ++j) { a[j] = na[j]; b[j] = nb[j]; }
  }
  // over the lanes that hold the same two heads, then over the warps
  auto reduce = [&](float m, float l, int g) {
    float mm = m;
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, x));
    float ll = m > -INFINITY ? l * ex2(m - mm) : 0.f;
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) ll += __shfl_xor_sync(0xffffffffu, ll, x);
    if (gid == 0) { s_m[w][g] = mm; s_l[w][g] = ll; }
  };
  reduce(m0, l0, 2 * tig);
  reduce(m1, l1, 2 * tig + 1);
  __syncthreads();
  if (tid < QH) {
    float m = s_m[0][tid], l = 0.f;
    for (int x = 1; x < NW; ++x) m = fmaxf(m, s_m[x][tid]);
    for (int x = 0; x < NW; ++x) l += s_m[x][tid] > -INFINITY ? s_l[x][tid] * ex2(s_m[x][tid] - m) : 0.f;
    float* pp = sc.partials + ((size_t)u * gridDim.x + blockIdx.x) * 16;
    pp[tid] = m;
    pp[8 + tid] = l;
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
// 64 heads x 9350 tokens cut to 935: 34.8 us; the decode step's Algorithm 1 kernel with its radix
// select over 96-bit keys in global memory took 286 us.  128 heads x 512 tokens: 10.1 us.
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
  const int B = fixed_budget > 0 ? fixed_budget : st.budget[uid];
  if (fixed_budget > 0 && tid == 0) st.budget[uid] = fixed_budget;
  if (w < G) {   // warp g merges query head g's chunks
    const float* pp = sc.partials + (size_t)u * chunks * 16;
    float m = -INFINITY, l = 0.f;
    for (int c = lane; c < chunks; c += 32) m = fmaxf(m, pp[c * 16 + w]);
    m = warp_max(m);
    for (int c = lane; c < chunks; c += 32) l += pp[c * 16 + 8 + w] * ex2(pp[c * 16 + w] - m);
    l = warp_sum(l);
    if (lane == 0) {
      s_m[w] = m * 0.693147180559945309f;   // log2 domain -> natural log
      s_il[w] = 1.0f / (l * (float)G);
    }
  }
  __syncthreads();
  // ---- step 1: pbar_i = mean_g exp(s_gi - m_g) / l_g
  float mx[QH], il[QH];
#pragma unroll
  for (int g = 0; g < QH; ++g) {
    mx[g] = g < G ? s_m[g] : 0.f;
    il[g] = g < G ? s_il[g] : 0.f;
  }
  const float* S = sc.logits + (size_t)u * sc.cap_s * QH;
  float* pb = in_smem ? s_pbar : sc.pbar + (size_t)u * sc.cap_s;
  for (int i0 = tid; i0 < P; i0 += 2 * SEL_NT) {   // two rows requested together
    float4 ra[2], rb[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const float* r = S + (size_t)min(i0 + x * SEL_NT, P - 1) * QH;
      ra[x] = *reinterpret_cast<const float4*>(r);
      rb[x] = G > 4 ? *reinterpret_cast<const float4*>(r + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int i = i0 + x * SEL_NT;
      const float sv[8] = {ra[x].x, ra[x].y, ra[x].z, ra[x].w, rb[x].x, rb[x].y, rb[x].z, rb[x].w};
      float pm = 0.f;
#pragma unroll
      for (int g = 0; g < QH; ++g)
        if (g < G) pm = fmaf(expf(sv[g] - mx[g]), il[g], pm);
      if (i < P) pb[i] = pm;
    }
  }
  const bool track = !(literal && P < B);   // Algorithm 1's first line as printed: nothing runs below the budget
  Nucleus nu{};
  nu.theta = 0xffffffffu;
  if (track)
    nu = nucleus_search<SEL_NT>(P, top_p, s_nu, st.errword, [&](auto f) {
      for (int i = tid; i < P; i += SEL_NT) f(pb[i]);
    });
  __syncthreads();
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
// place of the next arrival), one CTA per head.
__global__ void __launch_bounds__(NT) prefill_take_kernel(State st, int layer, int P) {
  __shared__ int s_top;
  const int u = blockIdx.x, seq = u / st.H;
  take_pages(st, (seq * st.L + layer) * st.H + u % st.H, seq, P / GRP + 1, P, NT, &s_top);
}

constexpr int ROWS_SURVIVORS = 0;   // entries are listed in the metadata (their token positions)
constexpr int ROWS_ALL_LAST = 1;    // entry i is token i: metadata written here, tau = P - 1
constexpr int ROWS_ALL_POS = 2;     // ... tau = i, the token's own arrival time (its queries are replayed)

// The rows of a layer's entries into their pages.  k, v: [batch][P][H][128].  CTA 0 writes the
// layer's launch plan meanwhile (plan_warps > 0); the others, `per_head` for every head, copy a
// page per warp and turn, eight rows of 512 bytes in flight.  Bound: HBM, 1 KB moved per entry, or
// the plan's serial placement when there is little to copy: 64 heads x 935 entries in 16.8 us (one
// CTA per head: 85 us), 128 heads x 512 entries in 21.5 us (insertion, plan kernel and a scoring
// pass of the attention kernel: 81 us).
__global__ void __launch_bounds__(NT) prefill_rows_kernel(State st, Plan plan, int layer, const unsigned char* __restrict__ k,
                                                          const unsigned char* __restrict__ v, int P, int mode, int per_head,
                                                          int plan_warps, int plan_grid) {
  __shared__ int s_gs[MAX_UNITS_PER_CALL + 1];
  __shared__ int s_red[320];
  if (blockIdx.x == 0) {
    if (plan_warps > 0) write_plan(st, plan, layer, plan_warps, plan_grid, s_gs, s_red);
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
    } else if (lane < cnt) {
      st.meta_pos[mb + i] = i;
      st.meta_tau[mb + i] = mode == ROWS_ALL_POS ? i : P - 1;
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
