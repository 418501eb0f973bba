// Shared definitions of the Crystal-KV CUDA path (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ckv {

constexpr int HD = 128;             // head_dim
constexpr int ROW_BYTES = 256;      // one K or V row, bf16
constexpr int SLOT_BYTES = 512;     // one entry in the pool: K row followed by V row
constexpr int GRP = 16;             // entries per page = keys per streamed group (one MMA tile of keys)
constexpr int PAGE_BYTES = GRP * SLOT_BYTES;   // 8 KB: what one bulk copy brings into a ring stage
constexpr int NW = 8;               // warps per CTA
constexpr int NT = NW * 32;
constexpr int STAGES = 3;           // ring depth per warp, in pages
constexpr int RING_BYTES = NW * STAGES * PAGE_BYTES;   // 192 KB
constexpr int GMIN = 4;             // fewest groups a streaming warp is given
constexpr int GLAT = 12;            // ... raised up to this many to keep a head's pieces within the eight warps of one CTA
constexpr int QH = 8;               // query heads of a group as padded for the MMA N dimension
constexpr int MAX_UNITS_PER_CALL = 2048;   // heads of one layer launch (bounded by the planner's shared memory)
constexpr int NSETS = 16;           // logit scratch sets cycled by consecutive launches
constexpr int FIFO = 8;             // pieces a warp may have fetched ahead of the one it computes (> STAGES)

// error word bits raised by device-side consistency checks (never a trap)
constexpr int ERR_FREE_UNDERFLOW = 1;   // a head needed a page and the sequence's free list was empty
constexpr int ERR_OVER_EVICT = 2;       // a decode step found a head further over its budget than the eviction period allows
constexpr int ERR_CAPACITY = 4;         // a head's list would outgrow its capacity
constexpr int ERR_NUCLEUS = 8;          // the top-p threshold search did not find its boundary
constexpr int ERR_COPY_TIMEOUT = 16;    // a bulk copy into shared memory did not complete within a second
constexpr int ERR_PLAN = 32;            // the launch plan of a layer does not match the grid it is used with
constexpr int ERR_EMPTY = 64;           // a decode step met a head without entries

// Layout of a pool page: entry e (0..15) occupies bytes [512 e, 512 e + 512): its K row, then its
// V row, as 32 chunks of 16 bytes; chunk c is stored at chunk index c ^ (e & 7).  A page copied
// as it is into shared memory can then be read by ldmatrix (eight entries, one chunk column)
// without bank conflicts, and one bulk copy brings a whole group of keys.
__host__ __device__ __forceinline__ int chunk_offset(int e, int c) { return e * SLOT_BYTES + ((c ^ (e & 7)) << 4); }

struct State {
  // K/V pool: [batch][pages_per_seq][8192 B]
  unsigned char* pool;
  long long pages_per_seq;
  int* free_stack;   // [batch][pages_per_seq] free page ids of a sequence
  int* free_top;     // [batch] number of free pages
  // per unit (uid = (seq*L + layer)*H + head): `cap` list positions, page j backs positions 16 j .. 16 j + 15
  int* ptab;         // [units][capg] page id per 16 list positions; the first npages are owned by the unit
  int* meta_pos;     // [units][cap] token position
  int* meta_tau;     // [units][cap] last hit time
  float* meta_crf;   // [units][cap] CRF at tau
  int* n_cur;        // [units] live entries
  int* hole;         // [units] list position the next arriving entry is written to (<= n).  The live entries
                     // are the positions 0 .. n without the hole (hole == n: positions 0 .. n-1).  An entry that
                     // leaves in a decode step leaves its place to the next arrival: nothing is moved.
  int* npages;       // [units] pages owned; 16 * npages > n always (the hole is backed)
  int* budget;       // [units] == [batch][L][H]
  const float* tab;  // lambda^D, D in [0, max_context]
  int* errword;
  unsigned long long* counters;  // entries attended, hits, evictions of prompts and of evictions of several entries at once
  unsigned long long* ucount;    // [units][4] the same of decode steps, per head
  int batch, L, H, cap, capg;
};

// Launch plan of one layer, read by its next attention launch: every head cut into k pieces of
// nearly equal length, one piece per streaming warp (plan.cuh).  A piece is named by (head, j, k)
// and covers groups [g j / k, g (j + 1) / k) of the head's g groups AT LAUNCH TIME, so a plan stays
// correct when heads grow or shrink by a few entries; it is rewritten when a head's group count has
// drifted from the one it was made for by an eighth (at least two), and after every reallocation.
struct Plan {
  int4* desc;        // [pd_cap] pieces, head after head: {head index u, piece j, pieces k of the head, how they are placed}
  int4* wrange;      // [warps] pieces [x, y) of the physical warp cta * NW + w; z, w: the descriptor of piece x
                     // packed (z = head index, w = j | k << 12 | placement << 24) so that a warp starts without
                     // a second dependent read, or z = -1: read desc[x]
  int* npc;          // [U] pieces per head
  int* gplan;        // [U] groups per head the plan was made for
  int* hdr;          // [4] pieces in total, groups in total, warps the plan was made for, 1
};

// scratch of one launch pair (attention kernel, then LRFU kernel), assembled per launch: the
// logits and (m, l) come from one of NSETS cycled sets, the partials and tickets from one of two
struct Scratch {
  float* logits;     // [U][cap_s][QH] scaled logits of the step, one 32-byte row per list position
  float* pbar;       // [U][cap_s] group-mean probabilities (reused as int scratch)
  float* partials;   // [U][pmax][16 + G*128] split-K partial: m[8], l[8], O[G][128]
  float* mfin;       // [U][2][QH] per query head: merged reference point (log2 domain), then normaliser
  int* ticket;       // [U]
  int cap_s, pmax;
};

struct DecodeParams {
  State st;
  Scratch sc;
  Plan plan;                    // of this layer
  const __nv_bfloat16* q;       // [batch][Hq][128]
  const __nv_bfloat16* k_new;   // [batch][H][128]
  const __nv_bfloat16* v_new;
  __nv_bfloat16* out;           // [batch][Hq][128]
  int* done_ctr;     // LRFU kernel: [0] counts its finished CTAs, [1] set when a head's group count changed: the
                     // last CTA then writes the layer's next plan
  int* plan_len;     // [U + 1] the planner's list of lengths, per internal stream
  int layer;
  int G;          // query heads per kv head
  int t;          // time of this step
  int track;      // 1: Algorithm 1 runs (hits, CRF, eviction) in the LRFU kernel that follows
  int early;      // 1: the lists and rows of this layer are final, so the attention kernel may read them
                  //    before the kernel ahead of it in the stream has completed
  int evict_every;   // m >= 1: step 4 waits until a head is m entries over its budget, then removes them all
  int front;      // LRFU kernel: logit rows of a head requested before its length is known
  int literal;    // 1: Algorithm 1 is skipped for a head below its budget (its first line as printed)
  int plan_warps;    // warps of the attention grid the plan is made for
  int plan_grid;     // CTAs of that grid
  int cl;            // attention kernel: CTAs (a cluster) that share a head; 1: the plan places heads anywhere
  float scale;    // logit scale
  float scale_log2;
  float top_p;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

// ---- block-wide helpers (NT threads) ----
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Pieces of a head of k that the CTAs before CTA x of a cluster of cl take: k dealt evenly, longer shares
// first (the first min(k, cl) CTAs get at least one).
__host__ __device__ __forceinline__ int shared_first(int k, int x, int cl) { return k / cl * x + (x < k % cl ? x : k % cl); }

// Programmatic dependent launch: a kernel launched with the stream-serialisation attribute may
// start while the kernel before it in the stream still runs; pdl_wait() returns once that
// kernel has completed and its writes are visible, pdl_launch() lets the kernel after this
// one start.  Both are no-ops for a launch without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// ---- thread-block clusters (a launch without the attribute is a cluster of one)
__device__ __forceinline__ int cluster_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// The cluster's threads that have not exited meet; what they wrote to shared memory before arriving is visible to all.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
// The shared::cluster address of CTA `rank`'s counterpart of this CTA's shared address.
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
// Stores into another CTA's shared memory that count their bytes on an mbarrier beside the destination.
__device__ __forceinline__ void push_f32x4(uint32_t to, uint32_t bar, float4 v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1,%2,%3,%4}, [%5];\n"
               ::"r"(to), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void push_f32x2(uint32_t to, uint32_t bar, float a, float b) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1,%2}, [%3];\n"
               ::"r"(to), "f"(a), "f"(b), "r"(bar) : "memory");
}

// Exclusive scan of one int per thread across the block of NTH threads; returns this thread's
// prefix and the block total.  `red` needs NTH / 32 ints.  Contains two __syncthreads().
template <int NTH = NT>
__device__ __forceinline__ int block_excl_scan(int v, int* red, int& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  __syncthreads();
  if (lane == 31) red[w] = inc;
  __syncthreads();
  int base = 0, tot = 0;
#pragma unroll
  for (int i = 0; i < NTH / 32; ++i) {
    int x = red[i];
    if (i < w) base += x;
    tot += x;
  }
  total = tot;
  return base + inc - v;
}

// Address of chunk c (16 bytes) of the entry at list position i of a head.
__device__ __forceinline__ unsigned char* entry_chunk(const State& st, int uid, int seq, int i, int c) {
  const int page = st.ptab[(size_t)uid * st.capg + (i >> 4)];
  return st.pool + ((size_t)seq * st.pages_per_seq + page) * PAGE_BYTES + chunk_offset(i & (GRP - 1), c);
}

// Makes sure list position `need` of a head is backed by a page (a head that grew past its last
// page takes one from its sequence's free list).  One thread calls it; launches in which heads
// return pages never call it.  False: there is no page, or no room in the head's list.
__device__ __forceinline__ bool back_position(const State& st, int uid, int seq, int need) {
  const int have = st.npages[uid];
  if (need < have * GRP) return true;
  if (need >= st.cap) {
    atomicOr(st.errword, ERR_CAPACITY);
    return false;
  }
  const int idx = atomicSub(&st.free_top[seq], 1) - 1;
  if (idx < 0) {
    atomicAdd(&st.free_top[seq], 1);
    atomicOr(st.errword, ERR_FREE_UNDERFLOW);
    return false;
  }
  st.ptab[(size_t)uid * st.capg + have] = st.free_stack[(size_t)seq * st.pages_per_seq + idx];
  st.npages[uid] = have + 1;
  return true;
}

// A head keeps all n entries of a step: the next arrival goes behind them, or, when that place cannot be
// backed (the error word says so), takes the place of the last one.
__device__ __forceinline__ int keep_all(const State& st, int uid, int seq, int n) {   // (its length from now on)
  if (!back_position(st, uid, seq, n)) --n;
  st.n_cur[uid] = n;
  st.hole[uid] = n;
  return n;
}

// A decode step's counts for one head, kept per head: one launch's heads adding to the same three words held up one
// another (1024 heads of 257 entries: 0.5 us a layer).  Nothing waits for an addition: a CTA that read its head's words
// and wrote them back ended a round trip to DRAM later (64 heads of 1250 .. 3750 entries 21.65 us a layer instead of
// 21.25, 32 heads of 1025 entries 9.15 instead of 9.0).
__device__ __forceinline__ void count_unit(const State& st, int uid, int entries, int hits, int evictions) {
  unsigned long long* c = st.ucount + (size_t)uid * 4;
  atomicAdd(c, (unsigned long long)entries);
  if (hits) atomicAdd(c + 1, (unsigned long long)hits);
  if (evictions) atomicAdd(c + 2, (unsigned long long)evictions);
}

// List position of the i-th live entry of a head (i in [0, n)) given its hole.
__device__ __forceinline__ int live_pos(int i, int hole) { return i + (i >= hole ? 1 : 0); }

}  // namespace ckv
