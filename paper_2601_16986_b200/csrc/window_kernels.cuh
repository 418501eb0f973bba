// Observation-window prompts: Algorithm 1 replayed over the last W queries of a prompt whose rows are
// already stored.  Which entries a query hits depends on its scores alone, not on what earlier
// queries of the window marked, so the window is one attention kernel over all (query, head) rows,
// one threshold search per (head, query), and one kernel that walks an entry through its queries.
// 128 heads x 1024 tokens, 32 queries of 5 heads: 95 + 36 + 16 us a layer, the pages and the launch plan included (as kernels
// of their own they took 20 and 9 us, the three others 85 + 50 + 20); a decode-step launch pair
// per query, each reading the prompt's rows again, took 720 us.
#pragma once
#include "attn_kernel.cuh"
#include "evict.cuh"
#include "nucleus.cuh"
#include "plan.cuh"

namespace ckv {

constexpr int WA_WARPS = 4;                   // warps of a window_attn_kernel CTA, 16 (query, head) rows each
constexpr int WA_ROWS = WA_WARPS * 16;
constexpr int WA_KEYS = 64;                   // keys per tile
constexpr int WA_TILE = WA_KEYS * ROW_BYTES;  // bytes of a K (or V) tile
constexpr int WA_SMEM = 4 * WA_TILE;          // K and V, two stages
constexpr int WIN_SMEM = 32 * 1024;           // pbar of up to this many bytes stays in shared memory
constexpr int WH_SMALL = 1280;                // entries up to which window_hits_kernel may take CTAs of two warps

struct WindowParams {
  const unsigned char* k;      // [batch][P][H][128]
  const unsigned char* v;
  const unsigned char* q;      // [W][batch][Hq][128], from the first query of this launch
  __nv_bfloat16* out;          // the same shape
  float* logits;               // [U][W][G][Ps] scaled logits
  float* ml;                   // [U][W][16] reference point (log2 domain) [8], normaliser [8]
  unsigned* hits;              // [U][W][words] hit bits, bit i % 32 of word i / 32
  int H, G, U, P, Ps, words;
  int W, t0;                   // queries of this launch, time of the first
  int layer, store;            // store: the prompt's rows go to the heads' pages (the launch with the last query)
  float scale, scale_log2;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

// Causal attention of the launch's W x G (query, head) rows of every kv head over the prompt, with the
// scaled logits kept for the threshold search.  grid: (row blocks, U).
// Bound: tensor cores (mma.sync; the weights go in as a bf16 head plus a bf16 remainder like in the
// decode kernel) and the logits written.  Keys on the MMA N dimension, rows on M; a row's channels
// are contracted in the order in which 16-byte pieces of it load (lane tig: pieces tig, tig + 4, ..),
// which makes every K fragment one 16-byte shared load.  Q, S and O live in registers, K and V tiles
// of 64 keys in two cp.async stages; three CTAs fit an SM.  (Two CTAs of five warps for 160 rows, without idle rows but with
// ten warps an SM instead of twelve: 92 us instead of 82.)
// The tiles are also what the heads' pages are filled from (store): the CTAs of a head take its tiles in turn, a tile that
// only the last one sees in full falls to that one.  (A copy kernel of its own reads the prompt again: 20 us.)
template <bool OUT>
__global__ void __launch_bounds__(WA_WARPS * 32, 3) window_attn_kernel(const __grid_constant__ State st, const WindowParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int u = blockIdx.y, seq = u / p.H, head = u % p.H;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int R = p.W * p.G, r_lo = blockIdx.x * WA_ROWS;
  const int ra = r_lo + w * 16 + gid, rb = ra + 8;          // this lane's two rows
  const bool va = ra < R, vb = rb < R;
  const int wa = min(ra, R - 1) / p.G, ga = min(ra, R - 1) % p.G, wb = min(rb, R - 1) / p.G, gb = min(rb, R - 1) % p.G;
  const int ta = p.t0 + wa, tb = p.t0 + wb;                 // times: keys 0 .. t take part
  auto keys_of = [&](int b) { return p.t0 + min(R - 1, (b + 1) * WA_ROWS - 1) / p.G + 1; };   // block b's last query sees these
  const int n_keys = keys_of(blockIdx.x);
  const int ntiles = (n_keys + WA_KEYS - 1) / WA_KEYS;
  const size_t qstride = (size_t)p.U * p.G * ROW_BYTES;     // one query of the window to the next
  uint32_t qa[8][4];
  {
    const unsigned char* pa = p.q + wa * qstride + ((size_t)u * p.G + ga) * ROW_BYTES;
    const unsigned char* pb = p.q + wb * qstride + ((size_t)u * p.G + gb) * ROW_BYTES;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int c = 16 * (tig + 4 * (s >> 1)) + 8 * (s & 1);   // bytes
      qa[s][0] = *reinterpret_cast<const uint32_t*>(pa + c);
      qa[s][1] = *reinterpret_cast<const uint32_t*>(pb + c);
      qa[s][2] = *reinterpret_cast<const uint32_t*>(pa + c + 4);
      qa[s][3] = *reinterpret_cast<const uint32_t*>(pb + c + 4);
    }
  }
  const uint32_t s0 = smem_u32(smem);
  const size_t row = (size_t)p.H * ROW_BYTES;
  const unsigned char* kbase = p.k + ((size_t)seq * p.P * p.H + head) * ROW_BYTES + (tid & 15) * 16;
  const unsigned char* vbase = p.v + ((size_t)seq * p.P * p.H + head) * ROW_BYTES + (tid & 15) * 16;
  // a tile's rows: 16 threads per row, 8 rows per round; K pieces are swizzled by the key's parity (a
  // fragment load takes four neighbouring pieces of eight keys), V pieces by key % 8 (ldmatrix)
  auto fetch = [&](int tile, int stage) {
    const uint32_t ks = s0 + stage * 2 * WA_TILE, vs = ks + WA_TILE;
    const int c = tid & 15;
#pragma unroll
    for (int x = 0; x < WA_KEYS / 8; ++x) {
      const int key = (tid >> 4) + 8 * x;
      const size_t off = (size_t)min(tile * WA_KEYS + key, p.P - 1) * row;   // (keys past the prompt are masked)
      cp_async16(ks + key * ROW_BYTES + ((c ^ ((key & 1) << 2)) << 4), kbase + off);
      if (OUT) cp_async16(vs + key * ROW_BYTES + ((c ^ (key & 7)) << 4), vbase + off);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float o[OUT ? 16 : 1][4];
#pragma unroll
  for (int x = 0; x < (OUT ? 16 : 1); ++x) { o[x][0] = 0.f; o[x][1] = 0.f; o[x][2] = 0.f; o[x][3] = 0.f; }
  float ma = -INFINITY, mb = -INFINITY, la = 0.f, lb = 0.f;
  float* lga = p.logits + (((size_t)u * p.W + wa) * p.G + ga) * p.Ps + 2 * tig;
  float* lgb = p.logits + (((size_t)u * p.W + wb) * p.G + gb) * p.Ps + 2 * tig;
  const int uid = (seq * st.L + p.layer) * st.H + head;
  const bool store = OUT && p.store && st.n_cur[uid] == p.P;   // (a head that found no pages stays empty)
  fetch(0, 0);
#pragma unroll 1
  for (int tile = 0; tile < ntiles; ++tile) {
    const int stage = tile & 1;
    if (tile + 1 < ntiles) {
      fetch(tile + 1, stage ^ 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const uint32_t ks = s0 + stage * 2 * WA_TILE, vs = ks + WA_TILE;
    if (store) {
      const int last = gridDim.x - 1, turn = tile % gridDim.x;
      if (blockIdx.x == ((tile + 1) * WA_KEYS <= keys_of(turn) ? turn : last)) {   // an entry per warp and turn, lane c its chunk c
        const int* pt = st.ptab + (size_t)uid * st.capg + tile * (WA_KEYS / GRP);
        unsigned char* pool = st.pool + (size_t)seq * st.pages_per_seq * PAGE_BYTES;
#pragma unroll 4
        for (int key = w; key < min(WA_KEYS, p.P - tile * WA_KEYS); key += WA_WARPS) {
          const uint32_t at = lane < 16 ? ks + key * ROW_BYTES + ((lane ^ ((key & 1) << 2)) << 4)
                                        : vs + key * ROW_BYTES + (((lane - 16) ^ (key & 7)) << 4);
          uint4 x;
          asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];\n" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "r"(at));
          *reinterpret_cast<uint4*>(pool + (size_t)__ldg(pt + key / GRP) * PAGE_BYTES + chunk_offset(key & (GRP - 1), lane)) = x;
        }
      }
    }
    float s[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      s[nt][0] = 0.f; s[nt][1] = 0.f; s[nt][2] = 0.f; s[nt][3] = 0.f;
      const uint32_t kr = ks + (nt * 8 + gid) * ROW_BYTES;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t x0, x1, x2, x3;
        asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(x0), "=r"(x1), "=r"(x2), "=r"(x3) : "r"(kr + (((tig + 4 * j) ^ ((gid & 1) << 2)) << 4)));
        mma_bf16(s[nt], qa[2 * j], x0, x1);
        mma_bf16(s[nt], qa[2 * j + 1], x2, x3);
      }
    }
    // ---- logits out, masked online softmax
    const int k0 = tile * WA_KEYS + 2 * tig;
    float ca = -INFINITY, cb = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int key = k0 + nt * 8;
      if (va && key <= ta) *reinterpret_cast<float2*>(lga + tile * WA_KEYS + nt * 8) = make_float2(__fmul_rn(s[nt][0], p.scale), __fmul_rn(s[nt][1], p.scale));
      if (vb && key <= tb) *reinterpret_cast<float2*>(lgb + tile * WA_KEYS + nt * 8) = make_float2(__fmul_rn(s[nt][2], p.scale), __fmul_rn(s[nt][3], p.scale));
      s[nt][0] = key <= ta ? s[nt][0] * p.scale_log2 : -INFINITY;
      s[nt][1] = key + 1 <= ta ? s[nt][1] * p.scale_log2 : -INFINITY;
      s[nt][2] = key <= tb ? s[nt][2] * p.scale_log2 : -INFINITY;
      s[nt][3] = key + 1 <= tb ? s[nt][3] * p.scale_log2 : -INFINITY;
      ca = fmaxf(ca, fmaxf(s[nt][0], s[nt][1]));
      cb = fmaxf(cb, fmaxf(s[nt][2], s[nt][3]));
    }
#pragma unroll
    for (int x = 1; x < 4; x <<= 1) {
      ca = fmaxf(ca, __shfl_xor_sync(0xffffffffu, ca, x));
      cb = fmaxf(cb, __shfl_xor_sync(0xffffffffu, cb, x));
    }
    // (key 0 takes part in every row, so the reference points are finite from the first tile on)
    if (__any_sync(0xffffffffu, ca > ma + LAZY || cb > mb + LAZY)) {
      const float na = fmaxf(ma, ca), nb = fmaxf(mb, cb);
      const float xa = ex2(ma - na), xb = ex2(mb - nb);
      la *= xa; lb *= xb;
#pragma unroll
      for (int x = 0; x < (OUT ? 16 : 1); ++x) { o[x][0] *= xa; o[x][1] *= xa; o[x][2] *= xb; o[x][3] *= xb; }
      ma = na; mb = nb;
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {   // 16 keys at a time
      float e[8];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        e[4 * x] = ex2(s[2 * kk + x][0] - ma); e[4 * x + 1] = ex2(s[2 * kk + x][1] - ma);
        e[4 * x + 2] = ex2(s[2 * kk + x][2] - mb); e[4 * x + 3] = ex2(s[2 * kk + x][3] - mb);
        la += e[4 * x] + e[4 * x + 1];
        lb += e[4 * x + 2] + e[4 * x + 3];
      }
      if (OUT) {
        uint32_t ph[4], pl[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {   // x = 0: row a, keys 2 tig; 1: row b; 2, 3: the same for keys + 8
          const __nv_bfloat162 h = __floats2bfloat162_rn(e[2 * x], e[2 * x + 1]);
          ph[x] = *reinterpret_cast<const uint32_t*>(&h);
          pl[x] = pack_bf16(e[2 * x] - __low2float(h), e[2 * x + 1] - __high2float(h));
        }
        const int mi = lane >> 3, r8 = lane & 7;
        const uint32_t vr = vs + (kk * 16 + (mi & 1) * 8 + r8) * ROW_BYTES;
#pragma unroll
        for (int ct = 0; ct < 8; ++ct) {   // 16 channels at a time
          uint32_t b[4];
          ldsm_x4_t(b, vr + (((2 * ct + (mi >> 1)) ^ r8) << 4));
          mma_bf16(o[OUT ? 2 * ct : 0], ph, b[0], b[1]);
          mma_bf16(o[OUT ? 2 * ct + 1 : 0], ph, b[2], b[3]);
          mma_bf16(o[OUT ? 2 * ct : 0], pl, b[0], b[1]);
          mma_bf16(o[OUT ? 2 * ct + 1 : 0], pl, b[2], b[3]);
        }
      }
    }
    __syncthreads();   // the stage may be refilled
  }
#pragma unroll
  for (int x = 1; x < 4; x <<= 1) {
    la += __shfl_xor_sync(0xffffffffu, la, x);
    lb += __shfl_xor_sync(0xffffffffu, lb, x);
  }
  if (tig == 0) {
    float* mla = p.ml + ((size_t)u * p.W + wa) * 16 + ga;
    float* mlb = p.ml + ((size_t)u * p.W + wb) * 16 + gb;
    if (va) { mla[0] = ma; mla[8] = la; }
    if (vb) { mlb[0] = mb; mlb[8] = lb; }
  }
  if (OUT) {
    const float ia = 1.0f / la, ib = 1.0f / lb;
    __nv_bfloat16* oa = p.out + wa * (qstride / 2) + ((size_t)u * p.G + ga) * HD + 2 * tig;
    __nv_bfloat16* ob = p.out + wb * (qstride / 2) + ((size_t)u * p.G + gb) * HD + 2 * tig;
#pragma unroll
    for (int x = 0; x < 16; ++x) {
      if (va) *reinterpret_cast<uint32_t*>(oa + 8 * x) = pack_bf16(o[OUT ? x : 0][0] * ia, o[OUT ? x : 0][1] * ia);
      if (vb) *reinterpret_cast<uint32_t*>(ob + 8 * x) = pack_bf16(o[OUT ? x : 0][2] * ib, o[OUT ? x : 0][3] * ib);
    }
  }
}

// The hit bits of one (query, head): Algorithm 1 step 1 with the query of time t over its t + 1 entries.
// grid: (W, U).
// Bound: issue slots (some hundred instructions per warp beside those per entry), three quarters of which are in use:
// many searches of short prompts take CTAs of two warps, and the query heads are a template argument.  Few searches are bound by
// the latency of one: the line is as many searches as entries and SMs, and WH_SMALL entries.  us with two warps and with
// eight: 64 heads, 300 entries, 512 searches 6.4 and 6.7, 1024 7.7 and 10.7; 16 heads, 128 searches 6.0 and 4.5; 1024 entries, 128
// searches 10.7 and 5.0, 512 12.0 and 7.7, 1024 13.3 and 12.8, 1536 15.6 and 17.3; 1280 entries, 512 searches 14.7 and 10.1, 2048 23.6
// and 28.5, 4096 45.4 and 54.3; 1600 entries, 4096 searches 61.2 and 60.2, 2048 entries 74.7 and 65.4.
// 128 heads x 32 queries over 1000 entries: 36 us.
// pbar lives in shared memory or, for long prompts, in the place of the first query head's logits.
template <int NTH, int G>
__global__ void __launch_bounds__(NTH) window_hits_kernel(const __grid_constant__ State st, const WindowParams p, float top_p, int literal,
                                                          int in_smem) {
  constexpr int WARPS = NTH / 32;
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
  float* S = p.logits + ((size_t)u * p.W + q) * G * p.Ps;
  float* pb = in_smem ? s_pbar : S;
  float m[G], il[G];   // reference point, 1 / (normaliser x query heads)
  const float* ml = p.ml + ((size_t)u * p.W + q) * 16;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    m[g] = to_natural(ml[g]);
    il[g] = 1.0f / (ml[8 + g] * (float)G);
  }
  const int base = nucleus_base<NTH>(n);
  nucleus_clear<NTH>(s_nu);
  __syncthreads();
  constexpr int BR = 4;   // entries requested together
  for (int i0 = tid; i0 < n; i0 += BR * NTH) {
    float sv[BR][G];
#pragma unroll
    for (int x = 0; x < BR; ++x) {
      const float* r = S + min(i0 + x * NTH, n - 1);
#pragma unroll
      for (int g = 0; g < G; ++g) sv[x][g] = r[(size_t)g * p.Ps];
    }
#pragma unroll
    for (int x = 0; x < BR; ++x) {
      const float pm = group_mean(sv[x], m, il);
      if (i0 + x * NTH < n) {
        pb[i0 + x * NTH] = pm;   // (in the place of its own logit, which has been read)
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
WindowHits window_hits_of(int G) {
  switch (G) {
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
__global__ void __launch_bounds__(NT) window_apply_kernel(const __grid_constant__ State st, const WindowParams p, int last, int evict_every,
                                                          int* tmp, int tmp_stride, const __grid_constant__ Plan plan, int plan_grid,
                                                          int plan_cl, int* plan_len) {
  __shared__ __align__(16) int sh[PL_SCRATCH];
  if (blockIdx.x == 0) {
    if (last) write_plan<NT>(st, plan, p.layer, plan_grid * NW, plan_grid, plan_cl, plan_len, sh, evict_every);
    return;
  }
  const int u = blockIdx.x - 1, seq = u / st.H, tid = threadIdx.x;
  const int uid = (seq * st.L + p.layer) * st.H + u % st.H;
  if (st.n_cur[uid] != p.P) return;   // the prompt found no pages: the head is empty
  const size_t mb = (size_t)uid * st.cap;
  int nhit = 0;
  const int lane = tid & 31;
  for (int i0 = tid - lane; i0 < p.P; i0 += NT) {   // a warp takes 32 entries: one word of hit bits per query, a word per lane
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
    evict_many(st, uid, seq, p.P, min(p.P - B, p.P - 1), p.t0 + p.W - 1, true, sh, tmp + (size_t)u * tmp_stride);
}

}  // namespace ckv
