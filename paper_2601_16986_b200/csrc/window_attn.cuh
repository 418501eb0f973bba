// Attention of an observation window's queries over a prompt, on the fifth-generation tensor cores (window_kernels.cuh says
// what comes before and after).  One CTA takes up to 160 (query, head) rows of a kv head over all of the prompt's keys, 128 at a
// time, which makes the rows the N of both products whatever their number:
//   S^T [128 keys x N rows] = K Q^T      A: a tile of keys, B: the rows, both as they lie (K-major)
//   O^T [128 channels x N rows] += V^T P^T   A: a tile of values, B: the weights, both M/N-major
// with S (two buffers) and O in tensor memory.  Three passes over the keys, each of which computes S anew (a tenth of the
// kernel's time): the first finds every row's largest logit, the second the weights against that reference point, the normaliser and O,
// the third the group means of the probabilities, all that Algorithm 1 needs of the queries (a fifth of the bytes of the
// logits of five heads).  So nothing is ever rescaled, and a thread, which holds one key of every tile, keeps its share of
// the maxima and sums in registers until a pass ends.  The weights go in as a bf16 head plus a bf16 remainder, like in the decode kernel.
// A warp brings the tiles of all passes by TMA into a ring of stages, another issues the products; these and the sixteen meet at
// mbarriers only.
// The tiles are also what the heads' pages are filled from (store): a key's 64 channels in a stage are, byte for byte, a quarter
// of an entry in a page, so another warp has TMA store them as they are.  The CTAs of a head take its tiles in turn, a tile that
// only the last one sees in full falls to that one.  (A copy kernel of its own reads the prompt again: 20 us.)
#pragma once
#include "attn_kernel.cuh"
#include "nucleus.cuh"
#include "tma.cuh"

namespace ckv {

constexpr int WA_WARPS = 16;                  // warp w: keys 32 (w % 4) .. + 31 of every tile, the (w / 4)-th quarter of the rows
constexpr int WA_THREADS = (WA_WARPS + 3) * 32;   // ... one warp brings the tiles, one issues the products, one fills the pages
constexpr int WA_KEYS = 128;                  // keys per tile
constexpr int WA_HALF = WA_KEYS * 128;        // bytes of a tile's 64 first (last) channels: 128-byte rows, 128-byte swizzle
constexpr int WA_TILE = 2 * WA_HALF;
constexpr int WA_MAX_ROWS = 160;              // rows of a CTA: 3 N <= 512 columns of tensor memory, and shared memory
constexpr int WA_TMEM = 512;
// Stages of tiles: what the rows (the swizzled layouts start on multiples of 1024), the weights and the small arrays leave room for.
__host__ __device__ constexpr int wa_stages(int rows, bool out) { return rows <= 32 ? 6 : rows <= 64 || !out ? 5 : rows <= 96 ? 4 : 3; }
constexpr int wa_smem(int rows, bool out) {
  return 1024 + wa_stages(rows, out) * WA_TILE + (out ? 3 : 1) * rows * 256 + (4 + 4 + 1 + 1) * rows * 4 + 192;
}
static_assert(wa_smem(32, true) <= 232448 && wa_smem(64, true) <= 232448 && wa_smem(96, true) <= 232448 && wa_smem(128, true) <= 232448 &&
              wa_smem(160, true) <= 232448 && wa_smem(160, false) <= 232448, "shared memory of an SM");
// Queries that a quarter of a CTA of `rows` rows takes: whole ones, so that a thread has all heads of a key's group mean.
__host__ __device__ constexpr int wa_queries(int rows, int G) { return rows / 4 / G; }

struct WindowParams {
  const unsigned char* k;      // [batch][P][H][128]
  const unsigned char* v;
  const unsigned char* q;      // [W][batch][Hq][128], from the first query of this launch
  __nv_bfloat16* out;          // the same shape
  float* pbar;                 // [U][W][Ps] group means of the probabilities
  float* logits;               // mma.sync: [U][W][G][Ps] scaled logits instead
  float* ml;                   //           [U][W][16] reference point (log2 domain) [8], normaliser [8]
  unsigned* hits;              // [U][W][words] hit bits, bit i % 32 of word i / 32
  int H, G, U, P, Ps, words;
  int W, t0;                   // queries of this launch, time of the first
  int rows;                    // rows of a CTA of the attention kernel
  int layer, store;            // store: the prompt's rows go to the heads' pages (the launch with the last query)
  float scale, scale_log2;
};

// ---- tcgen05 in the forms used here (one CTA, bf16 operands, fp32 accumulators)
// Shared memory matrix: start address, leading and stride byte offset in units of 16 bytes, swizzle (2: 128 bytes, 4: 64).
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t swizzle) {
  return (uint64_t)((addr >> 4) & 0x3fff) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46) | ((uint64_t)swizzle << 61);
}
// Instruction: fp32 accumulators, bf16 operands, M = 128, N; mn: both operands M/N-major instead of K-major.
__host__ __device__ constexpr uint32_t umma_instr(int n, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, uint32_t instr, bool add) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(instr), "r"((uint32_t)add) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// Eight columns of the warp's 32 lanes; the registers hold them after tmem_wait().
__device__ __forceinline__ void tmem_ld8(float (&r)[8], uint32_t addr) {
  __syncwarp();   // (its lanes may come from different waits)
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]) : "r"(addr));
}
__device__ __forceinline__ void tmem_wait(float (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]) :: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
template <int X>
struct Const { static constexpr int value = X; };

// v[c] over the lanes of a warp, eight columns at a time: every exchange halves the columns that a lane goes on with, so column
// c + (lane >> 2) ends up in v[c].
template <int CW, class Op>
__device__ __forceinline__ void reduce_columns(float (&v)[CW], int lane, Op op) {
#pragma unroll
  for (int c = 0; c < CW; c += 8) {
#pragma unroll
    for (int n = 4, o = 16; n >= 1; n >>= 1, o >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int x = 0; x < n; ++x) {
        const float give = up ? v[c + x] : v[c + n + x], keep = up ? v[c + n + x] : v[c + x];
        v[c + x] = op(keep, __shfl_xor_sync(0xffffffffu, give, o));
      }
    }
    v[c] = op(v[c], __shfl_xor_sync(0xffffffffu, v[c], 2));
    v[c] = op(v[c], __shfl_xor_sync(0xffffffffu, v[c], 1));
  }
}

// Causal attention of the launch's W x G (query, head) rows of every kv head over the prompt.  grid: (row blocks, U).
// CW: columns of a quarter of a CTA, p.rows = 4 CW, the first wa_queries() x G of them in use.  mk, mv: the prompt's keys and
// values, boxes of 64 channels x 128 tokens of a head; mp: the pool, boxes of a quarter of 16 entries.
// Bound: the exponentials and conversions of the second and third pass (3.3 and 3.7 thousand cycles a tile of 160 rows; the products
// take 0.6, 1.9 and 0.6 of the three passes') and the start, 5 us.  128 heads x 1024 tokens, 32 queries of 5 heads: 59 us (92 with mma.sync, twelve warps an
// SM and the logits of every head written); 2 heads x 4096 tokens, 1 query 78 (166); 1024 heads x 300 tokens, 2 queries 84 (92).
template <int CW, bool OUT>
__global__ void __launch_bounds__(WA_THREADS, 1) window_attn_kernel(const __grid_constant__ State st, const WindowParams p,
                                                                    const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                                                                    const __grid_constant__ CUtensorMap mp) {
  constexpr int N = 4 * CW, S = wa_stages(N, OUT);
  extern __shared__ unsigned char smem_raw[];
  const uint32_t s0 = (smem_u32(smem_raw) + 1023) & ~1023u;
  unsigned char* sm = smem_raw + (s0 - smem_u32(smem_raw));
  const uint32_t s_q = s0 + S * WA_TILE, s_p = s_q + N * 256;   // weights: heads, then remainders
  float* s_m = reinterpret_cast<float*>(sm + S * WA_TILE + (OUT ? 3 : 1) * N * 256);   // reference points (log2 domain)
  float* s_l = s_m + N;                                                                          // 1 / normaliser
  float2* s_ml = reinterpret_cast<float2*>(s_l + N);                                             // reference point (natural), 1 / (normaliser x query heads)
  float* s_red = reinterpret_cast<float*>(s_ml + N);                                             // [4][N]
  int* s_t = reinterpret_cast<int*>(s_red + 4 * N);                                              // times of the rows
  int* s_row = s_t + N;                                                                          // rows: query x G + head, -1 for none
  const uint32_t bar_ld = smem_u32(s_row + N);          // a load's bytes, per stage
  const uint32_t bar_e = bar_ld + 8 * S;                // a stage has been used
  const uint32_t bar_s = bar_e + 8 * S;                 // S is there, per buffer
  const uint32_t bar_free = bar_s + 16;                 // S has been read, per buffer
  const uint32_t bar_p = bar_free + 16, bar_o = bar_p + 8, tm_at = bar_o + 8;   // the weights are there; O is; the tensor memory's address
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(reinterpret_cast<unsigned char*>(s_row + N) + (tm_at - bar_ld));

  const int u = blockIdx.y, seq = u / p.H, head = u % p.H;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int qq = wa_queries(N, p.G), cols = qq * p.G;        // queries of a quarter, its columns in use
  const int q_lo = blockIdx.x * 4 * qq;                      // the CTA's first query
  auto keys_of = [&](int b) { return p.t0 + min(p.W - 1, (b + 1) * 4 * qq - 1) + 1; };   // block b's last query sees these
  const int nt = (keys_of(blockIdx.x) + WA_KEYS - 1) / WA_KEYS;
  const size_t qstride = (size_t)p.U * p.G * ROW_BYTES;      // one query of the window to the next

  // A wait gives up after about a second; from then on the thread waits for nothing, and nothing more is issued.
  bool dead = false;
  auto wait = [&](uint32_t bar, int n) { if (!dead) dead = !mbar_wait_bounded(bar, (uint32_t)n & 1u); };   // for its n-th phase
  const int uid = (seq * st.L + p.layer) * st.H + head;
  // The loads of all passes in the order in which the products use them, load i into stage i % S: the keys; the keys with every tile's
  // values behind the next tile's keys (or the keys alone); the keys once more.  (-1 - tile: values)
  const int n_mid = OUT ? 2 * nt : nt, n_loads = 2 * nt + n_mid;
  auto what = [&](int i) {
    if (i < nt) return i;
    i -= nt;
    if (i >= n_mid) return i - n_mid;
    if (!OUT) return i;
    return i == 2 * nt - 1 ? -nt : i & 1 ? (i + 1) / 2 : i ? -(i / 2) : 0;
  };
  auto load = [&](int i) {
    const int x = what(i), stage = i % S, tile = x < 0 ? -1 - x : x;
    mbar_expect_tx(bar_ld + 8 * stage, WA_TILE);
    for (int y = 0; y < 2; ++y)
      tma_tile(s0 + stage * WA_TILE + y * WA_HALF, x < 0 ? &mv : &mk, 64 * y, head, tile * WA_KEYS, seq, bar_ld + 8 * stage);
  };
  if (w == WA_WARPS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tm_at), "n"(WA_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  } else if (w == WA_WARPS + 1) {
    if (lane == 0) {
      for (int x = 0; x < S; ++x) {
        mbar_init(bar_ld + 8 * x, 1);
        mbar_init(bar_e + 8 * x, 2);   // by the products, and by the warp that fills the pages
      }
      for (int x = 0; x < 2; ++x) mbar_init(bar_s + 8 * x, 1);
      for (int x = 0; x < 3; ++x) mbar_init(bar_free + 8 * x, WA_WARPS);   // (bar_p as well)
      mbar_init(bar_o, 1);
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      for (int i = 0; i < min(S, n_loads); ++i) load(i);
    }
  } else if (w < WA_WARPS) {
    // row r of the CTA: column c of quarter x is head c % G of query q_lo + x qq + c / G; the others are zeros.
    // 64 channels per 128-byte row, 16-byte piece c of row r at c ^ (r & 7)
    constexpr int PER = N * 16 / (WA_WARPS * 32);
    if (tid < N) {
      const int c = tid % CW, q = q_lo + tid / CW * qq + c / p.G;
      const bool there = c < cols && q < p.W;
      s_row[tid] = there ? q * p.G + c % p.G : -1;
      s_t[tid] = p.t0 + (there ? q : 0);
    }
    bar_sync(1, WA_WARPS * 32);
    uint4 v[PER];
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const int i = tid + x * (WA_WARPS * 32), row = s_row[i >> 4], q = max(s_t[i >> 4] - p.t0, 0);
      const uint32_t* src = reinterpret_cast<const uint32_t*>(p.q + (size_t)q * qstride + ((size_t)u * p.G + max(row - q * p.G, 0)) * ROW_BYTES + (i & 15) * 16);
      v[x] = make_uint4(src[0], src[1], src[2], src[3]);
      if (row < 0) v[x] = make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const int i = tid + x * (WA_WARPS * 32), r = i >> 4, c = i & 15;
      *reinterpret_cast<uint4*>(sm + (s_q - s0) + (c >> 3) * (N * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = v[x];
    }
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // what was stored is read by the tensor cores
  tmem_before_sync();
  __syncthreads();
  tmem_after_sync();
  const uint32_t tm = *s_tmem;

  if (w == WA_WARPS) {
    if (lane == 0) {
      // ---- the products.  S of position i (tiles of all passes counted) goes to buffer i % 2.
      const uint64_t dk = umma_desc(s0, 16, 1024, 2), dq = umma_desc(s_q, 16, 1024, 2);
      const uint64_t dv = umma_desc(s0, WA_HALF, 1024, 2), dp = umma_desc(s_p, WA_KEYS * 64, 512, 4);
      int at = 0, stage = 0;   // the next load and its stage
      auto landed = [&] { wait(bar_ld + 8 * stage, at / S); };
      auto used = [&] {        // by the products issued so far
        umma_commit(bar_e + 8 * stage);
        ++at;
        stage = stage + 1 == S ? 0 : stage + 1;
      };
      auto issue_s = [&](int pos) {
        landed();
        if (pos > 1) wait(bar_free + 8 * (pos & 1), (pos >> 1) - 1);
        tmem_after_sync();
        if (dead) return;
        const uint64_t a = dk + stage * (WA_TILE >> 4);
#pragma unroll
        for (int x = 0; x < 8; ++x)
          umma(tm + (pos & 1) * N, a + ((x >> 2) * (WA_HALF >> 4) + (x & 3) * 2), dq + ((x >> 2) * (N * 128 >> 4) + (x & 3) * 2),
               umma_instr(N, false), x > 0);
        umma_commit(bar_s + 8 * (pos & 1));
        used();
      };
      auto issue_o = [&](int t) {
        landed();
        wait(bar_p, t);
        tmem_after_sync();
        if (dead) return;
#pragma unroll
        for (int x = 0; x < 8; ++x) {   // 16 keys at a time
          const uint64_t a = dv + (stage * (WA_TILE >> 4) + x * 128), b = dp + x * 64;
          umma(tm + 2 * N, a, b, umma_instr(N, true), t > 0 || x > 0);
          umma(tm + 2 * N, a, b + (N * 256 >> 4), umma_instr(N, true), true);
        }
        umma_commit(bar_o);
        used();
      };
#pragma unroll 1
      for (int x = 0; x < nt; ++x) issue_s(x);
      if (OUT) {   // (the next tile's S goes ahead of a tile's O: the other warps wait for it)
        issue_s(nt);
#pragma unroll 1
        for (int t = 0; t < nt; ++t) {
          if (t + 1 < nt) issue_s(nt + t + 1);
          issue_o(t);
        }
      } else {
#pragma unroll 1
        for (int x = 0; x < nt; ++x) issue_s(nt + x);
      }
#pragma unroll 1
      for (int x = 0; x < nt; ++x) issue_s(2 * nt + x);
      if (dead) atomicOr(st.errword, ERR_COPY_TIMEOUT);
    }
    __syncwarp();
  } else if (w == WA_WARPS + 1) {
    if (lane == 0) {
      // ---- the tiles
#pragma unroll 1
      for (int i = S; i < n_loads; ++i) {
        wait(bar_e + 8 * (i % S), i / S - 1);
        if (dead) break;
        load(i);
      }
      if (dead) {   // what is still on its way must land in memory that is this CTA's
        atomicOr(st.errword, ERR_COPY_TIMEOUT);
        for (int x = 0; x < S; ++x) mbar_wait_bounded(bar_ld + 8 * x, 0), mbar_wait_bounded(bar_ld + 8 * x, 1);
      }
    }
    __syncwarp();
  } else if (w == WA_WARPS + 2) {
    // ---- the prompt's rows go to the head's pages: keys in the first pass, values in the second; lane x takes the tile's page x
    // (Only here the kernel ahead, which takes the pages, has to have ended; what was queued before that one has.)
    pdl_wait();
    const bool store = OUT && p.store && st.n_cur[uid] == p.P;   // (a head that found no pages stays empty)
    const int last = gridDim.x - 1;
#pragma unroll 1
    for (int i = 0; i < n_loads; ++i) {
      const int x = what(i), tile = x < 0 ? -1 - x : x, stage = i % S, turn = tile % gridDim.x, at = tile * WA_KEYS + lane * GRP;
      const bool mine = store && (i < nt || x < 0) && blockIdx.x == ((tile + 1) * WA_KEYS <= keys_of(turn) ? turn : last) &&
                        lane < WA_KEYS / GRP && at < p.P;
      const int page = mine ? st.ptab[(size_t)uid * st.capg + at / GRP] : 0;
      wait(bar_ld + 8 * stage, i / S);
      if (mine && !dead) {   // (rows past the prompt's end are zeros and go to places without an entry)
        for (int y = 0; y < 2; ++y)
          tma_store(&mp, 0, (x < 0 ? 2 : 0) + y, ((int)(seq * st.pages_per_seq) + page) * GRP, s0 + stage * WA_TILE + y * WA_HALF + lane * GRP * 128);
        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_e + 8 * stage);
    }
    asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
    __syncwarp();
    pdl_launch();
  } else {
    const int quarter = w >> 2, c_lo = quarter * CW, key_w = (w & 3) * 32 + lane;
    const int nq = max(0, min(qq, p.W - (q_lo + quarter * qq)));   // queries of this warp's quarter
    const int t_first = p.t0 + q_lo;                               // time of the CTA's first query: keys 0 .. t take part
    const uint32_t tm_warp = tm + ((uint32_t)(w & 3) << 21) + c_lo;   // this warp's lanes and columns (lane in the upper half)
    auto s_ready = [&](int pos) {
      wait(bar_s + 8 * (pos & 1), pos >> 1);
      tmem_after_sync();
    };
    auto s_read = [&](int pos) {   // this warp has S in registers
      tmem_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_free + 8 * (pos & 1));
    };
    auto meet = [&] { bar_sync(1, WA_WARPS * 32); };
    // a column's result over the lanes of the four warps that share it
    auto put_columns = [&](const float (&v)[CW]) {
#pragma unroll
      for (int c = 0; c < CW; c += 8)
        if (!(lane & 3)) s_red[(w & 3) * N + c_lo + c + (lane >> 2)] = v[c];
    };

    // ---- first pass: every row's largest logit
    float acc[CW];   // over this thread's keys: maxima of S, then sums of weights
#pragma unroll
    for (int x = 0; x < CW; ++x) acc[x] = -INFINITY;
#pragma unroll 1
    for (int i = 0; i < nt; ++i) {
      s_ready(i);
      const int key = i * WA_KEYS + key_w;
      float s[CW / 8][8];
#pragma unroll
      for (int c = 0; c < CW / 8; ++c) tmem_ld8(s[c], tm_warp + (i & 1) * N + c * 8);
#pragma unroll
      for (int c = 0; c < CW / 8; ++c) tmem_wait(s[c]);
      s_read(i);
      if ((i + 1) * WA_KEYS - 1 <= t_first) {   // all rows see all of the tile
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[c] = fmaxf(acc[c], s[c / 8][c % 8]);
      } else {
#pragma unroll
        for (int c = 0; c < CW; ++c)
          if (key <= s_t[c_lo + c]) acc[c] = fmaxf(acc[c], s[c / 8][c % 8]);
      }
    }
    reduce_columns(acc, lane, [](float a, float b) { return fmaxf(a, b); });
    put_columns(acc);
#pragma unroll
    for (int x = 0; x < CW; ++x) acc[x] = 0.f;
    meet();
    if (tid < N)   // (key 0 takes part in every row, so the reference points are finite)
      s_m[tid] = p.scale_log2 * fmaxf(fmaxf(s_red[tid], s_red[N + tid]), fmaxf(s_red[2 * N + tid], s_red[3 * N + tid]));
    meet();

    // ---- second pass: weights, normalisers and O
#pragma unroll 1
    for (int t = 0; t < nt; ++t) {
      const int i = nt + t;
      s_ready(i);
      const int key = t * WA_KEYS + key_w;
      const bool all_see = (t + 1) * WA_KEYS - 1 <= t_first;
      float s[CW / 8][8];
#pragma unroll
      for (int c = 0; c < CW / 8; ++c) tmem_ld8(s[c], tm_warp + (i & 1) * N + c * 8);
#pragma unroll
      for (int c = 0; c < CW / 8; ++c) tmem_wait(s[c]);
      s_read(i);
      uint32_t hi[OUT ? CW / 2 : 1], lo[OUT ? CW / 2 : 1];
#pragma unroll
      for (int c = 0; c < CW; c += 8) {
        float (&e)[8] = s[c / 8];
#pragma unroll
        for (int x = 0; x < 8; x += 4) {
          const float4 m4 = *reinterpret_cast<const float4*>(s_m + c_lo + c + x);
          e[x] = ex2(fmaf(e[x], p.scale_log2, -m4.x));
          e[x + 1] = ex2(fmaf(e[x + 1], p.scale_log2, -m4.y));
          e[x + 2] = ex2(fmaf(e[x + 2], p.scale_log2, -m4.z));
          e[x + 3] = ex2(fmaf(e[x + 3], p.scale_log2, -m4.w));
        }
        if (!all_see) {
#pragma unroll
          for (int x = 0; x < 8; ++x)
            if (key > s_t[c_lo + c + x]) e[x] = 0.f;
        }
#pragma unroll
        for (int x = 0; x < 8; ++x) acc[c + x] += e[x];
        if (OUT) {
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const float a = e[2 * y], b = e[2 * y + 1];
            const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
            hi[c / 2 + y] = *reinterpret_cast<const uint32_t*>(&h);
            lo[c / 2 + y] = pack_bf16(a - __low2float(h), b - __high2float(h));
          }
        }
      }
      if (OUT) {
        if (t > 0) wait(bar_o, t - 1);   // the weights of the tile before have been used
        // 32 rows per 64-byte row of a key; 16-byte piece c of key k at c ^ (k >> 1 & 3)
#pragma unroll
        for (int c = 0; c < CW; c += 8) {
          const int col = c_lo + c, x = c / 2;
          unsigned char* to = sm + (s_p - s0) + (col >> 5) * (WA_KEYS * 64) + key_w * 64 + ((((col >> 3) & 3) ^ ((key_w >> 1) & 3)) << 4);
          *reinterpret_cast<uint4*>(to) = make_uint4(hi[x], hi[x + 1], hi[x + 2], hi[x + 3]);
          *reinterpret_cast<uint4*>(to + N * 256) = make_uint4(lo[x], lo[x + 1], lo[x + 2], lo[x + 3]);
        }
      }
      if (OUT) {
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // (the tensor cores read the weights)
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_p);
      }
    }
    reduce_columns(acc, lane, [](float a, float b) { return a + b; });
    put_columns(acc);
    meet();
    if (tid < N) {
      const float l = (s_red[tid] + s_red[N + tid]) + (s_red[2 * N + tid] + s_red[3 * N + tid]);
      s_l[tid] = 1.0f / l;
      s_ml[tid] = make_float2(to_natural(s_m[tid]), 1.0f / (l * (float)p.G));
    }
    meet();
    if (OUT) {   // a thread has a channel of the warp's rows: through the place of the weights, a warp then writes whole rows
      wait(bar_o, nt - 1);
      tmem_after_sync();
      __nv_bfloat16* so = reinterpret_cast<__nv_bfloat16*>(sm + (s_p - s0));
#pragma unroll
      for (int c = 0; c < CW; c += 8) {
        float r[8];
        tmem_ld8(r, tm_warp + 2 * N + c);
        tmem_wait(r);
#pragma unroll
        for (int x = 0; x < 8; ++x) so[(c_lo + c + x) * HD + key_w] = __float2bfloat16_rn(r[x] * s_l[c_lo + c + x]);
      }
      meet();
#pragma unroll 2
      for (int r = w; r < N; r += WA_WARPS) {
        const int c = r % CW, q = q_lo + r / CW * qq + c / p.G;
        if (c >= cols || q >= p.W || dead) continue;
        const uint32_t* from = reinterpret_cast<const uint32_t*>(so + r * HD) + lane;
        uint32_t* to = reinterpret_cast<uint32_t*>(p.out + (size_t)q * (qstride / 2) + ((size_t)u * p.G + c % p.G) * HD) + lane;
        to[0] = from[0];
        to[32] = from[32];
      }
    }

    // ---- third pass: group means, two queries at a time
    auto third = [&](auto gc) {
      constexpr int G = decltype(gc)::value;
#pragma unroll 1
      for (int t = 0; t < nt; ++t) {
        const int i = 2 * nt + t;
        s_ready(i);
        const int key = t * WA_KEYS + key_w;
        float* to = p.pbar + ((size_t)u * p.W + q_lo + quarter * qq) * p.Ps + key;
#pragma unroll 1
        for (int x = 0; x < nq; x += 2) {
          float s[2][8];   // (columns beyond G are the next query's)
          tmem_ld8(s[0], tm_warp + (i & 1) * N + x * G);
          tmem_ld8(s[1], tm_warp + (i & 1) * N + (x + 1) * G);
          tmem_wait(s[0]);
          tmem_wait(s[1]);
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            const int c = c_lo + min(x + y, nq - 1) * G;
            float sg[G], m[G], il[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
              sg[g] = __fmul_rn(s[y][g], p.scale);
              const float2 ml = s_ml[c + g];
              m[g] = ml.x;
              il[g] = ml.y;
            }
            const float pm = group_mean(sg, m, il);
            if (x + y < nq && key <= t_first + quarter * qq + x + y) to[(size_t)(x + y) * p.Ps] = pm;
          }
        }
        s_read(i);
      }
    };
    switch (p.G) {
      case 1: third(Const<1>()); break;
      case 2: third(Const<2>()); break;
      case 3: third(Const<3>()); break;
      case 4: third(Const<4>()); break;
      case 5: third(Const<5>()); break;
      case 6: third(Const<6>()); break;
      case 7: third(Const<7>()); break;
      default: third(Const<8>());
    }
    if (dead) atomicOr(st.errword, ERR_COPY_TIMEOUT);
  }
  tmem_before_sync();
  __syncthreads();
  if (w == WA_WARPS) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tm), "n"(WA_TMEM) : "memory");
}

// Row blocks of a head for W queries of G query heads: as few as there can be, or of 32 rows each if those are no more than `room`; and the
// rows of each, a multiple of 32.
inline int window_blocks(int W, int G, int room) {
  const int most = 4 * wa_queries(WA_MAX_ROWS, G), least = 4 * wa_queries(32, G);   // queries of a block
  return (W + least - 1) / least <= room ? (W + least - 1) / least : (W + most - 1) / most;
}
inline int window_rows(int W, int G, int blocks) {
  const int each = (W + blocks - 1) / blocks;   // queries of a block
  int rows = 32;
  while (4 * wa_queries(rows, G) < each) rows += 32;
  return rows;
}

using WindowAttn = void (*)(State, WindowParams, CUtensorMap, CUtensorMap, CUtensorMap);
template <bool OUT>
WindowAttn window_attn_of(int rows) {   // rows: a multiple of 32
  switch (rows) {
    case 32: return window_attn_kernel<8, OUT>;
    case 64: return window_attn_kernel<16, OUT>;
    case 96: return window_attn_kernel<24, OUT>;
    case 128: return window_attn_kernel<32, OUT>;
    default: return window_attn_kernel<40, OUT>;
  }
}
inline WindowAttn window_attn_of(int rows, bool out) { return out ? window_attn_of<true>(rows) : window_attn_of<false>(rows); }

}  // namespace ckv
