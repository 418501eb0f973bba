// C ABI of the Crystal-KV decode hot path (see include/crystalkv.h).  Host code only
// validates, keeps the per-layer clocks and launches; every step of the path runs in the
// kernels of attn_kernel.cuh and lrfu_kernel.cuh (a decode step; its launch plan: plan.cuh),
// prefill_kernels.cuh, window_attn.cuh, window_mma.cuh and window_kernels.cuh (prompts) and aux_kernels.cuh (reallocations, exports).
//
// Stream plan of a tracked decode step of layer l: the attention kernel runs on the caller's
// stream (so `out` is ready in stream order), the LRFU kernel of the same layer on an
// internal stream behind an event, which lets it overlap the attention kernel of the next
// layer.  Before an attention kernel reuses a scratch set, or touches a layer whose LRFU
// kernel of the previous step may still run, the caller's stream waits on that kernel's
// event.  Everything else (prefill, reallocation, inspection) first joins the internal stream.
#include "../../include/crystalkv.h"

#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "attn_kernel.cuh"
#include "aux_kernels.cuh"
#include "lrfu_launch.cuh"
#include "plan.cuh"
#include "prefill_kernels.cuh"
#include "window_kernels.cuh"

using namespace ckv;

// What a handle has of its device: its memory, streams and events.
struct DeviceKit {
  void* arena = nullptr;           // the one device allocation that all arrays of the handle lie in
  size_t arena_bytes = 0;
  unsigned long long context = 0;  // the primary context that all of this belongs to (a device reset ends it); 0: another context, or unknown
  // LRFU launches are numbered; launch k uses scratch set k % NSETS and event k % EV_RING
  static constexpr int EV_RING = 32;
  // two internal streams taken in turn: the LRFU kernels of consecutive layers do not depend on
  // one another, so the second may fill SM room as the first one's CTAs finish
  cudaStream_t side[2] = {};
  cudaEvent_t evA[EV_RING] = {}, evF[EV_RING] = {};
  // host I/O: HOST_RING staging sets; inputs go up on one internal stream and results come
  // down on another, so the copies of other layers run beside the attention kernels
  static constexpr int HOST_RING = 64;
  cudaStream_t copy_in = nullptr, copy_out = nullptr;
  cudaEvent_t evIn[HOST_RING] = {}, evUse[HOST_RING] = {}, evOut[HOST_RING] = {};
};

struct crystalkv : DeviceKit {
  crystalkv_config_t cfg;
  int G = 0, U = 0, units = 0, cap = 0, num_sms = 0, grid = 0;
  long long pages_per_seq = 0;
  State st{};
  std::vector<Plan> plans;         // per layer: the launch plan of its next attention kernel
  Plan* d_plans = nullptr;
  int* done_ctr = nullptr;
  int* plan_len = nullptr;         // per internal stream: U + 1 ints for the planner of its LRFU kernels
  // scratch: logits and merged (m, l) per cycled set (the LRFU kernel reads them while later
  // attention kernels run), partials and tickets alternate between two (attention kernels do
  // not overlap one another's compute), pbar is only touched by kernels that run one at a time
  float* sc_logits[NSETS] = {};
  float* sc_mfin[NSETS] = {};
  float* sc_partials[2] = {};
  int* sc_ticket[2] = {};
  float* sc_pbar[2] = {};          // one per internal stream
  int cap_s = 0, pmax = 0;
  long long nA = 0;                // attention launches so far
  std::vector<int> t_layer;        // per layer: time of the last step
  long long kF = 0, joined = -1;   // LRFU launches so far
  std::vector<long long> lastF;    // per layer: number of its latest LRFU launch, -1 = none
  int prev_layer = -1;             // layer of the launch pair issued last, -1 after any other call
  int stage = CRYSTALKV_STAGE_THINK;
  int answer_steps = 0;
  bool uniform = true;             // no head's budget or length has been set apart from the others'
  // Per layer.  cl: CTAs (a cluster) that share a head in the attention kernel, what the layer's plan is made for;
  // len_cap: entries of a head in a decode step once it is full, of every head while uniform, else about the mean.
  std::vector<int> cl, len_cap;
  bool share_ok[MAX_CLUSTER + 1] = {};   // clusters of so many CTAs, one per head of a launch, are resident at once
  int plan_grid(int layer) const { return cl[layer] > 1 ? U * cl[layer] : grid; }   // CTAs of its launches
  // Entries of a head in a decode step of the layer (as len_cap) that brings the tokens so far to `tokens`.
  int entries(int layer, int tokens) const { return cfg.mode == CRYSTALKV_MODE_EVICT ? std::min(len_cap[layer], tokens) : tokens; }
  long long* Asum = nullptr;
  __nv_bfloat16 *dq[HOST_RING] = {}, *dk[HOST_RING] = {}, *dv[HOST_RING] = {}, *dout[HOST_RING] = {};
  long long outJoined = -1;   // newest host step whose copy back the caller's stream has waited for
  long long nHost = 0;             // host-buffer steps so far
  int* io_rec = nullptr;           // staging for export / import of one head: records, rows, count
  unsigned char* io_rows = nullptr;
  int* io_n = nullptr;
  unsigned long long* io_sum = nullptr;   // ... and for the counters
  float* tab = nullptr;
  std::string err;
  bool cuda_dead = false;
};

namespace {

thread_local std::string g_create_err;

int fail(crystalkv_t* h, int code, const std::string& msg) {
  if (h) h->err = msg;
  return code;
}

// An error that only says "not while this stream is being captured" leaves the context and the
// handle intact; every other CUDA error is sticky for the handle.
bool capture_refusal(cudaError_t e) {
  return e >= cudaErrorStreamCaptureUnsupported && e <= cudaErrorStreamCaptureWrongThread;
}

#define CK(h, call)                                                                      \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess) {                                                             \
      if ((h) && !capture_refusal(e_)) (h)->cuda_dead = true;                            \
      return fail((h), CRYSTALKV_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    }                                                                                    \
  } while (0)

// Makes the handle's device current for the duration of a call and puts the caller's back.
struct DeviceScope {
  int prev = -1;
  cudaError_t err = cudaSuccess;
  explicit DeviceScope(int dev) {
    int cur = -1;
    err = cudaGetDevice(&cur);
    if (err == cudaSuccess && cur != dev) {
      err = cudaSetDevice(dev);
      if (err == cudaSuccess) prev = cur;
    }
  }
  ~DeviceScope() {
    if (prev >= 0) cudaSetDevice(prev);
  }
  DeviceScope(const DeviceScope&) = delete;
  DeviceScope& operator=(const DeviceScope&) = delete;
};
#define ON_DEVICE(h)                       \
  DeviceScope dev_scope_((h)->cfg.device); \
  CK((h), dev_scope_.err)

// ---- what a destroyed handle leaves for the next one
// A server makes a handle for a new batch and frees it again and again.  Taking and giving back 5.5 GB costs 1.05 and 3.2 ms,
// the streams and events another half, as much as all else: a new batch of 16 prompts of 512 tokens in the 8B shape, 1.9 ms of
// kernels, took 6.7 ms and takes 1.6 to 2.0 with them kept.  So a device keeps at most one kit, of at most KEEP_BYTES, and that only
// while a quarter of its memory is free; crystalkv_trim, a handle that it does not fit and an allocation
// that fails for want of memory give it back.  (A pool of the driver's gives back by itself, but its first 5.5 GB took 34 to 280 ms.)
constexpr size_t KEEP_BYTES = size_t(8) << 30;

// The place of a device's kit.  Only kits of the device's primary context are kept, of which there is one at a time: a kit of
// another one is of a context that has ended (a device reset), and with it all that the kit names.
struct KeptKit {
  DeviceKit kit;   // (context 0: nothing is kept)
  bool empty() const { return !kit.context; }
  // Whether a kit that was made in the primary context `current` (0: the caller is in another one, or it is unknown) finds room.
  bool room_for(const DeviceKit& k, unsigned long long current) const { return k.context && k.context == current && kit.context != current; }
  bool put(const DeviceKit& k, unsigned long long current) {
    if (!room_for(k, current)) return false;
    kit = k;
    return true;
  }
  // The kit of the primary context `current`, taken out; an empty one else.
  DeviceKit take(unsigned long long current) {
    DeviceKit k;
    if (current && kit.context && kit.context != current) kit = DeviceKit{};
    if (current) std::swap(k, kit);
    return k;
  }
};
KeptKit g_kept[MAX_DEVICES];
std::mutex g_kept_mu;

template <class Fn>
Fn driver_call(const char* name) {   // a call of the CUDA driver's as of 12.0, null if there is none
  void* p = nullptr;
  cudaDriverEntryPointQueryResult r;
  if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &r) != cudaSuccess || r != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  return reinterpret_cast<Fn>(p);
}

// The id of the current context if it is the primary one of its device, else 0.
unsigned long long primary_id() {
  static const auto current = driver_call<decltype(&cuCtxGetCurrent)>("cuCtxGetCurrent");
  static const auto device_of = driver_call<decltype(&cuCtxGetDevice)>("cuCtxGetDevice");
  static const auto retain = driver_call<decltype(&cuDevicePrimaryCtxRetain)>("cuDevicePrimaryCtxRetain");
  static const auto release = driver_call<decltype(&cuDevicePrimaryCtxRelease)>("cuDevicePrimaryCtxRelease");
  static const auto state = driver_call<decltype(&cuDevicePrimaryCtxGetState)>("cuDevicePrimaryCtxGetState");
  static const auto id_of = driver_call<CUresult (*)(CUcontext, unsigned long long*)>("cuCtxGetId");
  if (!current || !device_of || !retain || !release || !state || !id_of) return 0;
  CUcontext ctx = nullptr, primary = nullptr;
  CUdevice dev = 0;
  unsigned flags = 0;
  int active = 0;
  unsigned long long id = 0;
  if (current(&ctx) != CUDA_SUCCESS || !ctx || device_of(&dev) != CUDA_SUCCESS) return 0;
  if (state(dev, &flags, &active) != CUDA_SUCCESS || !active || retain(&primary, dev) != CUDA_SUCCESS) return 0;
  release(dev);
  return primary == ctx && id_of(ctx, &id) == CUDA_SUCCESS ? id : 0;
}

void free_kit(DeviceKit& k) {
  for (cudaStream_t x : {k.side[0], k.side[1], k.copy_in, k.copy_out})
    if (x) cudaStreamDestroy(x);
  for (auto* ring : {k.evIn, k.evUse, k.evOut})
    for (int i = 0; i < DeviceKit::HOST_RING; ++i)
      if (ring[i]) cudaEventDestroy(ring[i]);
  for (auto* ring : {k.evA, k.evF})
    for (int i = 0; i < DeviceKit::EV_RING; ++i)
      if (ring[i]) cudaEventDestroy(ring[i]);
  if (k.arena) cudaFree(k.arena);
  k = DeviceKit{};
}

// The kit that the current device keeps, if it belongs to the current context, taken out; an empty one else.
DeviceKit take_kept(int device) {
  const unsigned long long ctx = primary_id();
  std::lock_guard<std::mutex> lock(g_kept_mu);
  return g_kept[device].take(ctx);
}

// Keeps a complete kit that no work on the device uses any more.  False: it is the caller's to free.
bool keep_kit(int device, const DeviceKit& kit) {
  if (!kit.arena || kit.arena_bytes > KEEP_BYTES || !kit.evF[DeviceKit::EV_RING - 1]) return false;   // (the last to be made)
  const unsigned long long ctx = primary_id();
  {
    std::lock_guard<std::mutex> lock(g_kept_mu);
    if (!g_kept[device].room_for(kit, ctx)) return false;
  }
  size_t room = 0, total = 0;
  if (cudaMemGetInfo(&room, &total) != cudaSuccess) { cudaGetLastError(); return false; }
  if (room < total / 4) return false;
  std::lock_guard<std::mutex> lock(g_kept_mu);
  return g_kept[device].put(kit, ctx);
}

// Gives back what the device keeps, whatever context is current.  True if there was something.
bool give_back(int device) {
  {
    std::lock_guard<std::mutex> lock(g_kept_mu);
    if (g_kept[device].empty()) return false;   // (a device that was never used gets no context)
  }
  static const auto current = driver_call<decltype(&cuCtxGetCurrent)>("cuCtxGetCurrent");
  static const auto make_current = driver_call<decltype(&cuCtxSetCurrent)>("cuCtxSetCurrent");
  CUcontext ctx = nullptr;
  int before = -1;
  if (!current || !make_current || current(&ctx) != CUDA_SUCCESS || cudaGetDevice(&before) != cudaSuccess) return false;
  DeviceKit kit;
  if (cudaSetDevice(device) == cudaSuccess) kit = take_kept(device);   // (the primary context is the current one now)
  const bool had = kit.arena != nullptr;
  free_kit(kit);
  if (before != device) cudaSetDevice(before);
  if (ctx) make_current(ctx);
  return had;
}

// cudaMalloc that gives back what the device keeps if there is not enough memory.
cudaError_t device_malloc(int device, void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaErrorMemoryAllocation || !give_back(device)) return e;
  cudaGetLastError();
  return cudaMalloc(p, bytes);
}

// A handle's device arrays are parts of one allocation.  Some 330 separate ones (staging sets, logit
// sets, lists) cost a handle of the 8B shape (5.5 GB) 16 ms to take and 16 ms to give back, against
// 0.5 and 2.3 ms for one of the same total size.
struct Arena {
  struct Part { void** where; size_t at; };
  std::vector<Part> parts;
  size_t bytes = 0;
  template <typename T>
  void add(T** p, size_t count) {
    parts.push_back({reinterpret_cast<void**>(p), bytes});
    bytes += (std::max<size_t>(count, 1) * sizeof(T) + 255) / 256 * 256;   // every array starts on a 256-byte boundary
  }
  // The handle's kit: the kept one if its memory is enough and at most twice as much, else a new one.
  int take(crystalkv_t* h) {
    DeviceKit& kit = *h;
    kit = take_kept(h->cfg.device);
    if (kit.arena && (kit.arena_bytes < bytes || kit.arena_bytes / 2 > bytes)) free_kit(kit);
    if (!kit.arena) {
      const cudaError_t e = device_malloc(h->cfg.device, &kit.arena, bytes);
      if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(h, e == cudaErrorMemoryAllocation ? CRYSTALKV_ENOMEM : CRYSTALKV_ECUDA,
                    std::string("cudaMalloc: ") + cudaGetErrorString(e));
      }
      kit.arena_bytes = bytes;
      kit.context = primary_id();
    }
    for (const Part& x : parts) *x.where = static_cast<unsigned char*>(kit.arena) + x.at;
    return CRYSTALKV_OK;
  }
};

// Streams and events of a kit that has none yet.
cudaError_t make_streams(DeviceKit& k) {
  if (k.side[0]) return cudaSuccess;
  // The LRFU kernels run at the highest stream priority: the attention kernel of the layer after
  // next is already queued when one of them becomes ready (it was released early and waits for
  // shared memory), and at equal priority its CTAs, which cannot be placed yet, are served first.
  int least = 0, greatest = 0;
  cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
  for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaStreamCreateWithPriority(&k.side[i], cudaStreamNonBlocking, greatest);
  for (cudaStream_t* x : {&k.copy_in, &k.copy_out})
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(x, cudaStreamNonBlocking);
  for (auto* ring : {k.evIn, k.evUse, k.evOut})
    for (int i = 0; i < DeviceKit::HOST_RING && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&ring[i], cudaEventDisableTiming);
  for (auto* ring : {k.evA, k.evF})
    for (int i = 0; i < DeviceKit::EV_RING && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&ring[i], cudaEventDisableTiming);
  return e;
}

__global__ void init_free_stack_kernel(int* stack, int* top, long long pages_per_seq, int batch) {
  const long long total = pages_per_seq * batch;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i % pages_per_seq;
    stack[i] = (int)(pages_per_seq - 1 - r);   // popping from the top hands out ascending page ids
  }
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < batch; b += blockDim.x) top[b] = (int)pages_per_seq;
}

__global__ void fill_int_kernel(int* p, long long n, int v) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    p[i] = v;
}

int validate(const crystalkv_config_t* c, std::string& why) {
  if (!c) { why = "cfg is NULL"; return CRYSTALKV_EINVAL; }
  if (c->head_dim != HD) { why = "head_dim must be 128"; return CRYSTALKV_EINVAL; }
  if (c->dtype != CRYSTALKV_BF16) { why = "dtype must be CRYSTALKV_BF16"; return CRYSTALKV_EINVAL; }
  if (c->n_layers < 1 || c->n_kv_heads < 1 || c->batch < 1) { why = "n_layers, n_kv_heads, batch must be >= 1"; return CRYSTALKV_EINVAL; }
  if (c->n_q_heads < c->n_kv_heads || c->n_q_heads % c->n_kv_heads) { why = "n_q_heads must be a multiple of n_kv_heads"; return CRYSTALKV_EINVAL; }
  if (c->n_q_heads / c->n_kv_heads > 8) { why = "group size above 8"; return CRYSTALKV_EINVAL; }
  if ((long long)c->batch * c->n_kv_heads > MAX_UNITS_PER_CALL) { why = "batch * n_kv_heads above 2048"; return CRYSTALKV_EINVAL; }
  if (c->mode != CRYSTALKV_MODE_EVICT && c->mode != CRYSTALKV_MODE_FULLKV) { why = "bad mode"; return CRYSTALKV_EINVAL; }
  if (c->max_context < 2) { why = "max_context must be >= 2"; return CRYSTALKV_EINVAL; }
  if (c->mode == CRYSTALKV_MODE_EVICT && c->budget_per_head < 1) { why = "budget_per_head must be >= 1"; return CRYSTALKV_EINVAL; }
  if (c->min_budget < 0 || c->max_budget < 0 || c->max_answer_tokens < 0) { why = "negative budget bound"; return CRYSTALKV_EINVAL; }
  if (c->max_budget && c->max_budget < c->budget_per_head) { why = "max_budget below budget_per_head"; return CRYSTALKV_EINVAL; }
  if (c->min_budget > c->budget_per_head) { why = "min_budget above budget_per_head"; return CRYSTALKV_EINVAL; }
  if (c->top_p < 0.f || c->top_p > 1.f) { why = "top_p outside (0, 1]"; return CRYSTALKV_EINVAL; }
  if (c->lambda > 1.f) { why = "lambda above 1"; return CRYSTALKV_EINVAL; }
  if (c->sm_scale < 0.f) { why = "negative sm_scale"; return CRYSTALKV_EINVAL; }
  if (c->device < 0 || c->device >= MAX_DEVICES) { why = "device ordinal outside [0, 64)"; return CRYSTALKV_EINVAL; }
  if (c->evict_every < 0 || c->evict_every > 4096) { why = "evict_every outside [0, 4096]"; return CRYSTALKV_EINVAL; }
  if (c->literal_return != 0 && c->literal_return != 1) { why = "literal_return must be 0 or 1"; return CRYSTALKV_EINVAL; }
  if (!(c->budget_ratio >= 0.f) || c->budget_ratio > 1.f) { why = "budget_ratio outside [0, 1]"; return CRYSTALKV_EINVAL; }
  return CRYSTALKV_OK;
}

// Ratio budgets: the average budget per head after `tokens` tokens, floor(r * tokens) in fp64 from
// the fp32 ratio, kept within [max(1, min_budget), budget_per_head].
int ratio_budget(const crystalkv_config_t& c, int tokens) {
  long long b = (long long)std::floor((double)c.budget_ratio * (double)tokens);
  b = std::max<long long>(b, std::max(1, c.min_budget));
  b = std::min<long long>(b, c.budget_per_head);
  return (int)b;
}

// Sets the budget of every head of one layer.
__global__ void fill_layer_budget_kernel(State st, int layer, int v) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u < st.batch * st.H) st.budget[((u / st.H) * st.L + layer) * st.H + (u % st.H)] = v;
}

int check_layer(crystalkv_t* h, int layer) {
  if (!h) return CRYSTALKV_EINVAL;
  if (h->cuda_dead) return fail(h, CRYSTALKV_ECUDA, "an earlier CUDA error is sticky for this handle");
  if (layer < 0 || layer >= h->cfg.n_layers) return fail(h, CRYSTALKV_EINVAL, "layer out of range");
  return CRYSTALKV_OK;
}

int check_unit(crystalkv_t* h, int layer, int seq, int head) {
  int rc = check_layer(h, layer);
  if (rc) return rc;
  if (seq < 0 || seq >= h->cfg.batch || head < 0 || head >= h->cfg.n_kv_heads)
    return fail(h, CRYSTALKV_EINVAL, "seq or kv_head out of range");
  return CRYSTALKV_OK;
}

DecodeParams make_params(crystalkv_t* h, int layer) {
  DecodeParams p{};
  p.st = h->st;
  p.plan = h->plans[layer];
  p.done_ctr = h->done_ctr;   // (launch_step picks the internal stream's own)
  p.plan_len = h->plan_len;
  p.sc.cap_s = h->cap_s;
  p.sc.pmax = h->pmax;
  p.sc.pbar = h->sc_pbar[0];
  p.sc.partials = h->sc_partials[h->nA & 1];
  p.sc.ticket = h->sc_ticket[h->nA & 1];
  p.sc.logits = h->sc_logits[0];
  p.sc.mfin = h->sc_mfin[0];
  h->nA++;
  p.layer = layer;
  p.G = h->G;
  p.scale = h->cfg.sm_scale;
  p.scale_log2 = h->cfg.sm_scale * 1.44269504088896340736f;
  p.top_p = h->cfg.top_p;
  p.evict_every = h->cfg.evict_every;
  p.literal = h->cfg.literal_return;
  return p;
}

// Finds out which cluster sizes give every head of a launch a cluster of its own with all clusters resident at once.
int find_clusters(crystalkv_t* h) {
  for (int cl = MAX_CLUSTER; cl > 1; cl /= 2) {
    if (h->U * cl > h->grid) continue;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(h->U * cl);
    lc.blockDim = dim3(NT);
    lc.dynamicSmemBytes = ATTN_SMEM_SHARED;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    int n = 0;
    CK(h, cudaOccupancyMaxActiveClusters(&n, attn_of(true, true), &lc));
    h->share_ok[cl] = n >= h->U;
  }
  return CRYSTALKV_OK;
}

// CTAs that share a head of `entries` entries, where there is room for a cluster per head (find_clusters): a launch bound by
// its chain of dependent steps (pieces of at most GLAT groups) gains what its warps stream less, a group being worth
// about 0.4 us and the wider merge as much, and loses where the clusters leave Algorithm 1's kernels no SM without an attention CTA.
//
// Two CTAs, by the groups a warp streams without sharing.  us a layer on one CTA and on two (24 layers where nothing else is said):
//  * one layer, whose launches cannot start early: from two.  2 heads of 17 groups 17.8 and 16.3, 64 of 33 20.5 and 18.4; 1 head of 12 16.4
//    and 15.0, 74 of 16 18.8 and 17.7 (of 9 groups 17.0 and 17.4).
//  * two layers: from four groups less with sharing than without.  The line is older than these figures and higher than it need be.
//  * from three while two CTAs a head fill half of the SMs at most: 1 head of 17 groups 5.95 and 5.15, 16 of 17 6.3 and 5.55, 32 of 17 6.35 and 5.75 (on
//    four, which make pieces of two groups as well, 6.85); of 24 6.8 and 5.8.
//  * else from four: 50 heads of 41 groups 8.4 and 7.0, 60 of 33 7.6 and 7.2, 64 of 25 6.7 and 6.75, of 30 7.05 and 6.9, of 33 7.75 and 7.5;
//    68 of 30 7.3 and 7.4, of 33 8.0 and 7.85; three layers, 70 of 25 10.25 and 9.05.
//  * from five where fewer than twelve SMs are left (70 of 25 6.9 and 7.2, of 33 8.1 and 8.0, of 40 8.8 and 8.5; 72 of 30 7.4 and 7.75),
//    from six for heads of one length where fewer than four are (74 of 25 7.1 and 7.8, of 33 8.25 and 8.75, of 40 9.05 and 9.15, of 41 9.55 and 9.3; with unequal budgets of
//    33 groups on average 8.85 and 8.85, of 40 10.15 and 9.3).  Not with three layers: 74 of 25 10.3 and 8.95 (but of 40 11.4 and 12.1).
// Four CTAs where their pieces are two groups shorter again, and from four groups a warp without sharing on while they fill half of the SMs at
// most (below, the plan makes pieces of two groups either way): 32 heads of 41 groups 6.5 on two and 6.95 on four, of 50 7.5 and 7.4, of 65 8.5 and
// 8.3; 16 of 17 5.55 and 5.7, of 30 5.75 and 5.75, of 33 6.15 and 5.7, of 41 6.3 and 5.85; three layers with unequal budgets, 4 of 30 on average 9.35 and 8.25.
//
// Longer heads of one length (from 193 groups, where they no longer fit a CTA in pieces of 2 GLAT) gain from two CTAs where their
// other choice is more than eight pieces and a merge through global memory at the end of the launch.  The longer the pieces,
// the more the CTAs that then have nothing to stream count: up to 14 groups a piece from 45 heads on, up to 24 from 52.  us a
// layer, not shared and shared, of 194, 226, 257, 313 and 376 groups: 48 heads 21.7 21.4 23.3 27.5 37.1 and 18.2 20.6 22.8 26.5 31.6; 52 heads 22.2
// 22.4 25.0 29.4 37.4 and 18.5 21.1 23.5 27.6 35.1; 64 heads of 257 28.2 and 27.1.  (These lines, too, are older than the figures, by which 40 heads of
// 194 groups, 20.7 and 17.7, and 48 of 376 would share as well.)
int share_heads(crystalkv_t* h, int entries) {
  const int g = (entries + GRP - 1) / GRP, alone = (g + NW - 1) / NW;
  const int layers = h->cfg.n_layers, left = h->num_sms - 2 * h->U;   // SMs that two CTAs a head leave
  auto per = [&](int cl) { return (g + NW * cl - 1) / (NW * cl); };
  const bool merge = h->uniform && 10 * h->U >= 3 * h->num_sms && alone > 2 * GLAT &&
                     per(2) <= (20 * h->U >= 7 * h->num_sms ? 2 * GLAT : GLAT + 2);
  const int from = layers == 1 ? 2 : 4 * h->U <= h->num_sms ? 3 : layers == 3 || left >= 12 ? 4 : left >= 4 || !h->uniform ? 5 : 6;
  auto pays = [&](int cl) {
    return h->share_ok[cl] && (per(cl) <= GLAT || (cl == 2 && merge)) && (layers == 2 ? alone - per(cl) >= 4 : alone >= from);
  };
  if (pays(4) && (!pays(2) || (8 * h->U <= h->num_sms ? alone >= 4 : per(2) - per(4) >= 2))) return 4;
  return pays(2) ? 2 : 1;
}
static_assert(MAX_CLUSTER == 4, "share_heads weighs two CTAs and four");

// Writes the launch plans of `count` layers from their heads' current lengths, on `s`; the layers share heads alike.
int replan(crystalkv_t* h, int layer0, int count, cudaStream_t s) {
  plan_kernel<<<count, NT, 0, s>>>(h->st, h->d_plans, layer0, h->plan_grid(layer0) * NW, h->plan_grid(layer0), h->cl[layer0]);
  CK(h, cudaGetLastError());
  return CRYSTALKV_OK;
}

// The caller sets heads apart by hand: their lengths may have nothing to do with the mean any more, so
// plans place heads anywhere from now on.  On `s`, which has joined the internal streams.
int leave_clusters(crystalkv_t* h, cudaStream_t s) {
  h->uniform = false;
  for (bool& x : h->share_ok) x = false;
  for (int l = 0; l < h->cfg.n_layers; ++l) {
    if (h->cl[l] == 1) continue;
    h->cl[l] = 1;
    if (int rc = replan(h, l, 1, s)) return rc;
  }
  return CRYSTALKV_OK;
}

// Brings the heads of `count` layers down to their budgets, on `s`, which has joined the internal
// streams (no launch uses a logit set meanwhile).
int shrink_layers(crystalkv_t* h, int layer0, int count, int t_last, cudaStream_t s) {
  ShrinkScratch sc;
  for (int i = 0; i < NSETS; ++i) sc.area[i] = reinterpret_cast<int*>(h->sc_logits[i]);
  sc.cap_s = h->cap_s;
  for (int l = 0; l < count; l += SHRINK_LAYERS) {
    shrink_kernel<<<dim3(h->U, std::min(SHRINK_LAYERS, count - l)), NT, 0, s>>>(h->st, layer0 + l, t_last, sc);
    CK(h, cudaGetLastError());
  }
  return CRYSTALKV_OK;
}

// Makes `s` wait for every LRFU kernel launched so far.
int join_side(crystalkv_t* h, cudaStream_t s) {
  h->prev_layer = -1;
  if (h->kF > 0) CK(h, cudaStreamWaitEvent(s, h->evF[(h->kF - 1) % crystalkv::EV_RING], 0));
  if (h->kF > 1) CK(h, cudaStreamWaitEvent(s, h->evF[(h->kF - 2) % crystalkv::EV_RING], 0));   // the other internal stream
  h->joined = h->kF - 1;
  if (h->nHost > 0) CK(h, cudaStreamWaitEvent(s, h->evOut[(h->nHost - 1) % crystalkv::HOST_RING], 0));   // copies back run in order
  return CRYSTALKV_OK;
}

// A launch that may start before the kernel ahead of it in the stream has ended; the kernel waits for that (griddepcontrol.wait).
// The kernels of a prompt let the next one start once they have themselves waited, so everything before the kernel ahead has ended by then;
// what the kernel ahead writes is read with ordinary loads, after the wait.  The last one lets nothing start: what follows it is none of them.
// Ordinary launches leave 1 to 2 us between two of them: a new batch of 16 prompts of 512 tokens 1.75 ms and 1.62, windows of 32 queries 6.1 and 5.8.
template <class... P, class... A>
cudaError_t launch_next(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid;
  lc.blockDim = dim3(threads);
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kernel, static_cast<P>(args)...);
}

// A tensor map of bf16 in boxes of `box`, zeros beyond the ends.
bool tensor_map(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box,
                CUtensorMapSwizzle swizzle) {
  static const auto encode = driver_call<decltype(&cuTensorMapEncodeTiled)>("cuTensorMapEncodeTiled");
  const cuuint32_t step[4] = {1, 1, 1, 1};
  return encode && encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// The tokens of a prompt as tiles: [batch][P][H][128] in boxes of 64 channels x `tokens` tokens of one head.
bool tile_map(CUtensorMap* m, const void* base, int batch, int P, int H, int tokens) {
  const cuuint64_t dims[4] = {HD, (cuuint64_t)H, (cuuint64_t)P, (cuuint64_t)batch};
  const cuuint64_t strides[3] = {ROW_BYTES, (cuuint64_t)H * ROW_BYTES, (cuuint64_t)P * H * ROW_BYTES};
  const cuuint32_t box[4] = {HD / 2, 1, (cuuint32_t)tokens, 1};
  return tensor_map(m, base, 4, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}
// The pool as quarters of entries, in boxes of a page's.
bool pool_map(CUtensorMap* m, const crystalkv_t* h) {
  const cuuint64_t dims[3] = {HD / 2, 4, (cuuint64_t)h->cfg.batch * h->pages_per_seq * GRP}, strides[2] = {SLOT_BYTES / 4, SLOT_BYTES};
  const cuuint32_t box[3] = {HD / 2, 1, GRP};
  return tensor_map(m, h->st.pool, 3, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

// One attention launch on `s` and its follow-up (Algorithm 1 when it runs, the heads' new lengths
// and the layer's next plan) on the internal stream.
int launch_step(crystalkv_t* h, DecodeParams& p, int layer, cudaStream_t s) {
  const int entries = h->entries(layer, p.t + 1), share = share_heads(h, entries);
  if (share != h->cl[layer]) {   // the heads have filled so far: once or twice in a layer's life
    if (int rc = join_side(h, s)) return rc;
    h->cl[layer] = share;
    if (int rc = replan(h, layer, 1, s)) return rc;
  }
  p.cl = h->cl[layer];
  p.plan_grid = h->plan_grid(layer);
  p.plan_warps = p.plan_grid * NW;
  const long long k = h->kF;
  {
    // launch k reuses the scratch of launch k - NSETS and continues the state its layer's
    // previous LRFU launch wrote; each internal stream runs in order, so the events of two
    // consecutive launches cover everything before them
    // A wait on the caller's stream costs several microseconds (the attention kernel behind it
    // no longer starts early), so one wait covers as many launches as the sets allow: it targets
    // the newest LRFU launch that has had two attention kernels' time to finish.
    const long long need = std::max(k - NSETS, h->lastF[layer]);
    if (need >= 0 && need > h->joined) {
      const long long target = std::max(need, k - 3);
      CK(h, cudaStreamWaitEvent(s, h->evF[target % crystalkv::EV_RING], 0));
      if (target > 0) CK(h, cudaStreamWaitEvent(s, h->evF[(target - 1) % crystalkv::EV_RING], 0));   // the other internal stream
      h->joined = target;
    }
    p.sc.logits = h->sc_logits[k % NSETS];
    p.sc.mfin = h->sc_mfin[k % NSETS];
  }
  // The attention kernel may start while the kernel ahead of it still runs: it first fills its
  // pipeline from the cache and waits for that kernel before it touches the call's inputs.
  // That is only sound if the kernel ahead cannot be writing this layer's lists or plan, which holds
  // when it is the attention kernel of another layer.  Else the launch is an ordinary one: it is not enough to wait
  // inside, because the kernel reads them through the read-only path, which wants them final when it starts.
  p.early = (h->prev_layer >= 0 && h->prev_layer != layer) ? 1 : 0;
  {
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(p.plan_grid);
    lc.blockDim = dim3(NT);
    lc.dynamicSmemBytes = p.cl > 1 ? ATTN_SMEM_SHARED : ATTN_SMEM;
    lc.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = p.early;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = p.cl;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = p.cl > 1 ? 2 : 1;
    CK(h, cudaLaunchKernelEx(&lc, attn_of(p.cl > 1, p.track != 0), p));
  }
  h->prev_layer = layer;
  {
    const int si = (int)(k & 1);
    cudaEvent_t ea = h->evA[k % crystalkv::EV_RING];
    p.sc.pbar = h->sc_pbar[si];
    p.done_ctr = h->done_ctr + 2 * si;
    p.plan_len = h->plan_len + si * (h->U + 1);
    CK(h, cudaEventRecord(ea, s));
    CK(h, cudaStreamWaitEvent(h->side[si], ea, 0));
    const int threads = p.track ? lrfu_threads(h->U, entries, h->uniform, h->num_sms) : LRFU_SMALL;
    p.front = std::min(h->cap_s, h->uniform ? entries : std::min(p.t + 1, FRONT * threads));
    const int npb = std::min(std::min(h->cap, p.t + 1), pbar_room(threads, h->U, entries, h->num_sms, p.cl > 1));
    CK(h, lrfu_launch(threads, npb, h->G, p, h->U, h->side[si]));
    CK(h, cudaEventRecord(h->evF[k % crystalkv::EV_RING], h->side[si]));
    h->lastF[layer] = k;
    h->kF = k + 1;
  }
  return CRYSTALKV_OK;
}

}  // namespace

extern "C" {

const char* crystalkv_strerror(int code) {
  switch (code) {
    case CRYSTALKV_OK: return "ok";
    case CRYSTALKV_EINVAL: return "invalid argument";
    case CRYSTALKV_ESTATE: return "call out of order or capacity exhausted";
    case CRYSTALKV_ENOMEM: return "device allocation failed";
    case CRYSTALKV_ECUDA: return "CUDA runtime error";
    case CRYSTALKV_ECHECK: return "device-side consistency check failed";
  }
  return "unknown error";
}

const char* crystalkv_last_error(crystalkv_t* h) { return h ? h->err.c_str() : g_create_err.c_str(); }

int crystalkv_destroy(crystalkv_t* h) {
  if (!h) return CRYSTALKV_OK;
  DeviceScope scope(h->cfg.device);
  const bool idle = cudaDeviceSynchronize() == cudaSuccess && !h->cuda_dead;
  if (!idle || !keep_kit(h->cfg.device, *h)) free_kit(*h);
  delete h;
  return CRYSTALKV_OK;
}

int crystalkv_trim(int device) {
  if (device < 0 || device >= MAX_DEVICES) return CRYSTALKV_EINVAL;
  give_back(device);
  std::lock_guard<std::mutex> lock(g_kept_mu);
  return g_kept[device].empty() ? CRYSTALKV_OK : CRYSTALKV_ECUDA;
}

int crystalkv_debug_kept_kit(const int32_t* ops, int32_t n, int32_t* found) {
  if (!ops || !found || n < 0) return CRYSTALKV_EINVAL;
  KeptKit place;
  for (int i = 0; i < n; ++i) {
    const int32_t* op = ops + 4 * i;   // what, current context, the kit's context, the kit's number
    DeviceKit k;
    if (op[0] == 0) {
      k.context = (unsigned long long)op[2];
      k.arena_bytes = (size_t)op[3];
      found[i] = place.put(k, (unsigned long long)op[1]);
    } else if (op[0] == 1) {
      found[i] = (int32_t)place.take((unsigned long long)op[1]).arena_bytes;
    } else {
      return CRYSTALKV_EINVAL;
    }
  }
  return place.empty() ? 0 : 1;
}

int crystalkv_create(const crystalkv_config_t* cfg, crystalkv_t** out) {
  std::string why;
  int rc = validate(cfg, why);
  if (rc) { g_create_err = why; return rc; }
  if (!out) { g_create_err = "out is NULL"; return CRYSTALKV_EINVAL; }
  crystalkv_t* h = new (std::nothrow) crystalkv();
  if (!h) return CRYSTALKV_ENOMEM;
  h->cfg = *cfg;
  crystalkv_config_t& c = h->cfg;
  if (c.top_p == 0.f) c.top_p = 0.9f;
  if (c.lambda < 0.f) c.lambda = 0.6f;
  if (c.sm_scale == 0.f) c.sm_scale = (float)(1.0 / std::sqrt((double)c.head_dim));
  if (c.min_budget == 0) c.min_budget = std::min(c.budget_per_head, std::max(16, c.budget_per_head / 8));
  if (c.max_budget == 0) c.max_budget = 4 * c.budget_per_head;
  if (c.evict_every < 1) c.evict_every = 1;
  const bool evict = c.mode == CRYSTALKV_MODE_EVICT;
  h->G = c.n_q_heads / c.n_kv_heads;
  h->U = c.batch * c.n_kv_heads;
  h->units = h->U * c.n_layers;
  // list positions per head: entries up to the largest budget plus those that arrive before the
  // next eviction and the answer-stage tail, plus the place of the next arrival; FullKV keeps
  // every token.  Whole pages of 16.
  h->cap = evict ? c.max_budget + c.evict_every + c.max_answer_tokens + 1 : c.max_context + 1;
  h->cap = (h->cap + GRP - 1) / GRP * GRP;
  // pages per sequence: the entries all heads may hold together (B_total, what arrives before an
  // eviction, the answer tail, the hole), and one page per head for lists that end inside a page
  {
    const long long N = (long long)c.n_layers * c.n_kv_heads;
    const long long per_head = evict ? (long long)c.budget_per_head + c.evict_every + c.max_answer_tokens + 1
                                     : (long long)c.max_context + 1;
    h->pages_per_seq = (N * per_head + GRP - 1) / GRP + N;
  }
  if (h->pages_per_seq > 0x7fffffffLL) { g_create_err = "more than 2^31 pages per sequence"; delete h; return CRYSTALKV_EINVAL; }

#define CREATE_FAIL(code_)                    \
  do {                                        \
    int c_ = (code_);                         \
    g_create_err = h->err;                    \
    crystalkv_destroy(h);                     \
    return c_;                                \
  } while (0)
#define CKC(call)                                                              \
  do {                                                                         \
    cudaError_t e_ = (call);                                                   \
    if (e_ != cudaSuccess) {                                                   \
      h->err = std::string(#call) + ": " + cudaGetErrorString(e_);             \
      CREATE_FAIL(CRYSTALKV_ECUDA);                                            \
    }                                                                          \
  } while (0)
  DeviceScope scope(c.device);
  CKC(scope.err);
  CKC(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, c.device));
  int bps = 0;
  for (int x = 0; x < 4; ++x) {
    // (the same for every handle: the attribute belongs to the function, so no handle may lower it under another)
    const bool shared = x & 1;
    const AttnKernel attn = attn_of(shared, x >> 1);
    CKC(cudaFuncSetAttribute(attn, cudaFuncAttributeMaxDynamicSharedMemorySize, shared ? ATTN_SMEM_SHARED : ATTN_SMEM));
    // The largest shared-memory carve-out, although the ring alone would fit a smaller one: the CTAs
    // of the LRFU kernel have to find room beside an attention CTA on the same SM.
    CKC(cudaFuncSetAttribute(attn, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared));
  }
  CKC(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, attn_of(false, true), NT, ATTN_SMEM));
  if (bps < 1) { h->err = "attention kernel does not fit on an SM"; CREATE_FAIL(CRYSTALKV_ECUDA); }
  h->grid = h->num_sms * bps;
  h->cl.assign(c.n_layers, 1);
  h->len_cap.assign(c.n_layers, c.budget_per_head + c.evict_every);
  if (int r = find_clusters(h)) CREATE_FAIL(r);
  State& st = h->st;
  st.batch = c.batch; st.L = c.n_layers; st.H = c.n_kv_heads; st.cap = h->cap; st.capg = h->cap / GRP;
  st.pages_per_seq = h->pages_per_seq;
  // launch plans, one per layer: at most one piece per warp and one more per head
  const int nWarps = h->grid * NW, pd_cap = nWarps + h->U;
  int4 *desc = nullptr, *wr = nullptr;
  int *npc = nullptr, *gpl = nullptr, *hdr = nullptr;
  const int capgroups = (h->cap + GRP - 1) / GRP;
  h->cap_s = evict ? h->cap : 4;   // whole 128-byte lines of logit rows per unit (cap is a multiple of 16)
  h->pmax = capgroups / GMIN + 2;
  const size_t qn = (size_t)c.batch * c.n_q_heads * HD, kn = (size_t)c.batch * c.n_kv_heads * HD;
  {
    Arena a;
    a.add(&st.pool, (size_t)c.batch * h->pages_per_seq * PAGE_BYTES);
    a.add(&st.free_stack, (size_t)c.batch * h->pages_per_seq);
    a.add(&st.free_top, c.batch);
    a.add(&st.ptab, (size_t)h->units * st.capg);
    a.add(&st.meta_pos, (size_t)h->units * h->cap);
    a.add(&st.meta_tau, (size_t)h->units * h->cap);
    a.add(&st.meta_crf, (size_t)h->units * h->cap);
    a.add(&st.n_cur, h->units);
    a.add(&st.hole, h->units);
    a.add(&st.npages, h->units);
    a.add(&st.budget, h->units);
    a.add(&desc, (size_t)c.n_layers * pd_cap);
    a.add(&wr, (size_t)c.n_layers * nWarps);
    a.add(&npc, (size_t)c.n_layers * h->U);
    a.add(&gpl, (size_t)c.n_layers * h->U);
    a.add(&hdr, (size_t)c.n_layers * 4);
    a.add(&h->d_plans, c.n_layers);
    a.add(&h->done_ctr, 4);   // per internal stream: finished CTAs of its running LRFU kernel; whether the layer's plan went stale
    a.add(&h->plan_len, (size_t)2 * (h->U + 1));
    a.add(&h->tab, (size_t)c.max_context + 1);
    a.add(&st.errword, 1);
    a.add(&st.counters, 4);
    a.add(&st.ucount, (size_t)h->units * 4);
    a.add(&h->Asum, h->units);
    for (int i = 0; i < NSETS; ++i) a.add(&h->sc_logits[i], (size_t)h->U * h->cap_s * QH);   // one block: no padding between sets
    for (int i = 0; i < NSETS; ++i) a.add(&h->sc_mfin[i], (size_t)h->U * 2 * QH);
    for (int i = 0; i < 2; ++i) {
      a.add(&h->sc_partials[i], (size_t)h->U * h->pmax * (16 + h->G * HD));
      a.add(&h->sc_ticket[i], h->U);
      a.add(&h->sc_pbar[i], (size_t)h->U * h->cap_s);
    }
    for (int i = 0; i < crystalkv::HOST_RING; ++i) {
      a.add(&h->dq[i], qn); a.add(&h->dout[i], qn); a.add(&h->dk[i], kn); a.add(&h->dv[i], kn);
    }
    a.add(&h->io_rec, (size_t)3 * h->cap);
    a.add(&h->io_rows, (size_t)2 * h->cap * ROW_BYTES);
    a.add(&h->io_n, 1);
    a.add(&h->io_sum, 4);
    if (int r = a.take(h)) CREATE_FAIL(r);
    CKC(make_streams(*h));
  }
  st.tab = h->tab;
  CKC(cudaMemset(hdr, 0, (size_t)c.n_layers * 4 * sizeof(int)));
  CKC(cudaMemset(h->done_ctr, 0, 4 * sizeof(int)));
  for (int i = 0; i < 2; ++i) CKC(cudaMemset(h->sc_ticket[i], 0, (size_t)h->U * sizeof(int)));
  h->plans.resize(c.n_layers);
  for (int l = 0; l < c.n_layers; ++l)
    h->plans[l] = Plan{desc + (size_t)l * pd_cap, wr + (size_t)l * nWarps, npc + (size_t)l * h->U, gpl + (size_t)l * h->U,
                       hdr + (size_t)l * 4};
  CKC(cudaMemcpy(h->d_plans, h->plans.data(), (size_t)c.n_layers * sizeof(Plan), cudaMemcpyHostToDevice));

  // lambda^D as fp32 from an fp64 pow; pow(0, 0) = 1 keeps same-step hits when lambda = 0
  {
    std::vector<float> tab((size_t)c.max_context + 1);
    for (int D = 0; D <= c.max_context; ++D) {
      tab[D] = (float)std::pow((double)c.lambda, (double)D);
      if (tab[D] == 0.0f && D > 0) break;   // powers of lambda < 1 do not grow again: the rest is 0
    }
    CKC(cudaMemcpy(h->tab, tab.data(), tab.size() * sizeof(float), cudaMemcpyHostToDevice));
  }
  init_free_stack_kernel<<<1024, 256>>>(st.free_stack, st.free_top, h->pages_per_seq, c.batch);
  fill_int_kernel<<<256, 256>>>(st.budget, h->units, c.budget_per_head);
  CKC(cudaMemset(st.n_cur, 0, (size_t)h->units * sizeof(int)));
  CKC(cudaMemset(st.hole, 0, (size_t)h->units * sizeof(int)));
  CKC(cudaMemset(st.npages, 0, (size_t)h->units * sizeof(int)));
  CKC(cudaMemset(st.errword, 0, sizeof(int)));
  CKC(cudaMemset(st.counters, 0, 4 * sizeof(unsigned long long)));
  CKC(cudaMemset(st.ucount, 0, (size_t)h->units * 4 * sizeof(unsigned long long)));
  CKC(cudaGetLastError());
  CKC(cudaDeviceSynchronize());
  h->t_layer.assign(c.n_layers, -1);
  h->lastF.assign(c.n_layers, -1);
  *out = h;
  return CRYSTALKV_OK;
#undef CREATE_FAIL
#undef CKC
}

int crystalkv_set_stage(crystalkv_t* h, int stage) {
  if (!h) return CRYSTALKV_EINVAL;
  if (stage != CRYSTALKV_STAGE_THINK && stage != CRYSTALKV_STAGE_ANSWER) return fail(h, CRYSTALKV_EINVAL, "bad stage");
  if (stage == CRYSTALKV_STAGE_THINK && h->answer_steps > 0)
    return fail(h, CRYSTALKV_ESTATE, "answer tokens were appended; the think stage cannot resume");
  ON_DEVICE(h);
  if (stage != h->stage)   // no LRFU kernel is left behind the switch
    for (cudaStream_t x : h->side) CK(h, cudaStreamSynchronize(x));
  h->prev_layer = -1;
  h->stage = stage;
  return CRYSTALKV_OK;
}

int crystalkv_time(crystalkv_t* h, int layer) {
  if (!h || layer < 0 || layer >= h->cfg.n_layers) return -1;
  return h->t_layer[layer];
}

// Queries of a window over P tokens that one launch replays: what the logit sets, the pbar area and, for mma.sync, which keeps the logits
// of every query head, the partials have room for.
static int window_queries(const crystalkv_t* h, int P, bool tc) {
  const long long rows = (P + 7) / 8 * 8, words = (P + 31) / 32;
  return (int)std::max<long long>(1, std::min({(long long)NSETS * h->cap_s * QH / (tc ? rows : h->G * rows),
                                               tc ? 1ll << 30 : (long long)h->pmax * (16 + h->G * HD) / 16, h->cap_s / words, 1ll << 30}));
}

// Whether the attention of a window runs on tcgen05 (window_attn.cuh: one CTA an SM, three passes over the keys) or on mma.sync
// (window_mma.cuh: three CTAs an SM, one pass).  us a layer, all kernels of the window, on tcgen05 and on mma.sync:
//  * With outputs the products decide, except for prompts of one tile, whose CTAs are all start and end, with more heads than SMs (8 queries
//    of 5 heads: 1024 heads x 40 tokens 100 and 79; 1 query of 5: 512 x 64 50 and 45; but 160 x 100 33 and 37) or more than 128 rows (32 of 5: 48 x 64 36 and 31), and for
//    very many heads with many queries over little more (64 of 1: 1024 x 129 292 and 271; but 64 of 5: 512 x 300 307 and 412).
//  * Without outputs there is half the work for the tensor cores, and the three passes show: with more heads than SMs (1 query of 5: 1024 x 300 159 and
//    134; 8 of 2: 256 x 1000 126 and 117) unless the logits of all heads, which mma.sync leaves in memory, cost more (32 of 5: 256 x 1000 182
//    and 249), and with one query head over long prompts (64 of 1: 32 x 2048 163 and 153, 8 of 1: 128 x 4096 222 and 207; but 64 of 1: 16 x 129 47 and 55).
//  * Where the scratch holds the logits of all heads of fewer queries than it holds means, another launch costs more than all of this (64 of 8
//    with outputs: 32 x 64 50 and 78), but for very many heads.
static bool window_tcgen05(const crystalkv_t* h, int P, int W, bool out) {
  auto launches = [&](bool tc) { return (W - 1) / window_queries(h, P, tc); };
  const bool very = h->U > 4 * h->num_sms, once = launches(false) == launches(true), many = h->U > h->num_sms && (once || very);
  if (out) return !(P <= 64 && (many || (once && (long long)W * h->G > 128))) && !(very && P <= 192 && W >= 32);
  return !(many && !(h->G >= 5 && W >= 16 && P >= 256)) && !(h->G == 1 && W >= 8 && P >= 1000);
}
// Row blocks of a head on tcgen05.  Without outputs small ones for few heads, from 512 tokens on: 16 heads x 4096 tokens, 16 queries of 8 heads
// 104 us a layer instead of 128; but 32 heads x 300, 16 of 5 34 and 32.
static int window_blocks_of(const crystalkv_t* h, int P, int W, bool out) { return window_blocks(W, h->G, out || P < 512 ? 0 : h->num_sms / h->U); }

// Whether a window's attention kernel also fills the pages, from the tiles it reads: a tile's pages hold up one of a head's
// CTAs, which take the tiles in turn, 0.6 us, a copy kernel over the whole chip takes 4.5 us and the time of the bytes.  The window's kernels of a layer,
// pages from the tiles and copied: 2 heads x 4096 tokens, 1 query 120 us and 105; 16 heads x 4096, 6 queries 140 and 133, x 12000, 8 queries 416
// and 380, x 1024, 8 queries 43.5 and 45; 32 heads x 2048, 8 queries 79 and 82; 40 heads x 1024, 32 queries 75 and 82; 64 heads x
// 1024, 2 queries 43 and 50, x 4096, 6 queries 141 and 161.
static bool window_fills_pages(const crystalkv_t* h, int P, int W, bool tc) {
  if (!tc) return true;   // (short prompts, for which a launch more costs what it saves)
  const long long blocks = window_blocks_of(h, P, (W - 1) % window_queries(h, P, tc) + 1, true);   // of the last launch
  return 470ll * P < blocks * (450000 + 17ll * h->U * P);
}

// Algorithm 1 with the queries of the prompt's last W tokens, in as many launches as the scratch
// asks for (usually one): steps 1-3 for every query, step 4 after the last one.  Everything runs on
// `s`, which has joined the internal streams: the logit sets, one block of the arena, hold the
// window's group means, the first pbar area the hit bits.
// mk, mv, mp: tiles of the prompt's keys and values, the pool.
static int replay_window(crystalkv_t* h, int layer, const unsigned char* k, const unsigned char* v, const unsigned char* q, int P, int W,
                         __nv_bfloat16* out, bool tc, bool fill_pages, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mp, cudaStream_t s) {
  const crystalkv_config_t& c = h->cfg;
  WindowParams p{};
  p.k = k; p.v = v;
  p.pbar = p.logits = h->sc_logits[0];
  p.ml = h->sc_partials[0];
  p.hits = reinterpret_cast<unsigned*>(h->sc_pbar[0]);
  p.H = c.n_kv_heads; p.G = h->G; p.U = h->U; p.P = P; p.layer = layer;
  p.Ps = (P + 7) / 8 * 8;   // rows of group means start on 32-byte sectors
  p.words = (P + 31) / 32;
  p.scale = c.sm_scale;
  p.scale_log2 = c.sm_scale * 1.44269504088896340736f;
  const int fit = window_queries(h, P, tc);
  const size_t sm = (size_t)P * sizeof(float) <= WIN_SMEM ? (size_t)P * sizeof(float) : 0;
  const int plan_grid = h->plan_grid(layer);
  const size_t qn = (size_t)c.batch * c.n_q_heads * HD;
  for (int w0 = 0; w0 < W; w0 += p.W) {
    p.W = std::min(W - w0, fit);
    p.t0 = P - W + w0;
    p.q = q + (size_t)w0 * qn * sizeof(__nv_bfloat16);
    p.out = out ? out + (size_t)w0 * qn : nullptr;
    const bool last = w0 + p.W == W;
    p.store = last && fill_pages;
    if (tc) {
      const int blocks = window_blocks_of(h, P, p.W, out != nullptr);
      p.rows = window_rows(p.W, p.G, blocks);
      const auto attn = window_attn_of(p.rows, out != nullptr);
      const int smem = wa_smem(p.rows, out != nullptr);
      CK(h, cudaFuncSetAttribute(attn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      CK(h, launch_next(attn, dim3(blocks, h->U), WA_THREADS, smem, s, h->st, p, mk, mv, mp));
    } else {
      const auto attn = out ? window_mma_kernel<true> : window_mma_kernel<false>;
      CK(h, cudaFuncSetAttribute(attn, cudaFuncAttributeMaxDynamicSharedMemorySize, WM_SMEM));
      // (An ordinary launch: early CTAs gather, three to an SM, on the SMs that are free first.  32 heads x 2048 tokens, 32 queries of 2 heads 133 us
      // a layer instead of 89.)
      attn<<<dim3((p.W * p.G + WM_ROWS - 1) / WM_ROWS, h->U), WM_WARPS * 32, WM_SMEM, s>>>(h->st, p);
      CK(h, cudaGetLastError());
    }
    const bool small = P <= WH_SMALL && (long long)p.W * h->U >= P + h->num_sms;
    CK(h, launch_next(small ? window_hits_of<64>(tc ? 0 : p.G) : window_hits_of<NT>(tc ? 0 : p.G), dim3(p.W, h->U), small ? 64 : NT, sm, s,
                      h->st, p, c.top_p, c.literal_return, sm > 0));
    const bool wide = P > APPLY_LINE && 2 * h->U <= h->num_sms;
    CK(h, launch_next(wide ? window_apply_kernel<APPLY_WIDE> : window_apply_kernel<NT>, dim3(1 + h->U), wide ? APPLY_WIDE : NT, 0, s, h->st, p,
                      last, c.evict_every, reinterpret_cast<int*>(h->sc_pbar[1]), h->cap_s, h->plans[layer], plan_grid, h->cl[layer], h->plan_len));
  }
  return CRYSTALKV_OK;
}

// Prompt insertion and the Algorithm 1 passes that seed CRF/tau: one pass with the last query
// (W = 0) or a replay of the last W queries, each over the tokens up to its own.
static int prefill_common(crystalkv_t* h, int layer, const void* k, const void* v, const void* q,
                          int P, int W, void* out_window, void* stream) {
  int rc = check_layer(h, layer);
  if (rc) return rc;
  if (!k || !v || !q) return fail(h, CRYSTALKV_EINVAL, "null tensor");
  const crystalkv_config_t& c = h->cfg;
  const bool evict = c.mode == CRYSTALKV_MODE_EVICT;
  if (P < 1) return fail(h, CRYSTALKV_EINVAL, "P must be >= 1");
  // With a last query only, a prompt is scored from the caller's tensors and only its survivors are
  // stored; with an observation window the whole prompt must fit the pool for a moment (the
  // window's attention outputs need the values).
  if (evict && W > 0 && P > c.budget_per_head + c.max_answer_tokens)
    return fail(h, CRYSTALKV_EINVAL, "prompt with an observation window longer than budget_per_head + max_answer_tokens");
  if (evict && P + 1 > h->cap) return fail(h, CRYSTALKV_EINVAL, "prompt longer than the heads' list capacity (max_budget + evict_every + max_answer_tokens)");
  if (P >= c.max_context) return fail(h, CRYSTALKV_EINVAL, "prompt reaches max_context");
  const auto misaligned = [](const void* x, uintptr_t bytes) { return reinterpret_cast<uintptr_t>(x) % bytes != 0; };
  if (misaligned(k, 16) || misaligned(v, 16)) return fail(h, CRYSTALKV_EINVAL, "k and v must be 16-byte aligned");
  if (evict && W > 0 && (misaligned(q, 4) || misaligned(out_window, 4)))
    return fail(h, CRYSTALKV_EINVAL, "q_window and out_window must be 4-byte aligned");
  if (h->t_layer[layer] >= 0) return fail(h, CRYSTALKV_ESTATE, "layer already prefilled");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // All that a call may be refused for comes before the first launch and the first change: a refused layer is still to be loaded.
  CUtensorMap mk{}, mv{}, mp{};
  if (evict) {
    bool ok = tile_map(&mk, k, c.batch, P, c.n_kv_heads, W > 0 ? WA_KEYS : SCORE_KEYS);
    if (W > 0) ok = ok && tile_map(&mv, v, c.batch, P, c.n_kv_heads, WA_KEYS) && pool_map(&mp, h);
    if (!ok) return fail(h, CRYSTALKV_ECUDA, "the driver makes no tensor maps (cuTensorMapEncodeTiled)");
  }
  rc = join_side(h, s);   // the insertion takes pages; no LRFU kernel may take or return any meanwhile
  if (rc) return rc;
  const auto* kb = static_cast<const unsigned char*>(k);
  const auto* vb = static_cast<const unsigned char*>(v);
  // CTAs per head of the row copy: a page per warp and turn, up to eight CTAs per SM in all
  const int per_head = std::max(1, std::min((P / GRP + NW) / NW, (8 * h->num_sms + h->U - 1) / h->U));
  h->prev_layer = -1;
  if (evict && c.budget_ratio > 0.f) h->len_cap[layer] = ratio_budget(c, P) + c.evict_every;
  h->cl[layer] = share_heads(h, h->entries(layer, P + 1));
  const int plan_grid = h->plan_grid(layer);
  if (evict && W == 0) {
    // Algorithm 1 with the last query over scores and metadata only, then the survivors' rows; every
    // kernel on `s`, which has joined the internal streams, so any scratch set is free
    DecodeParams p = make_params(h, layer);
    const int chunks = (P + SCORE_KEYS - 1) / SCORE_KEYS;
    const size_t sm = (size_t)P * sizeof(float) <= SEL_SMEM ? (size_t)P * sizeof(float) : 0;
    if (sm > 32 * 1024)
      CK(h, cudaFuncSetAttribute(prefill_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SEL_SMEM));
    const long long items = (long long)c.batch * chunks * c.n_kv_heads;
    const int ctas = (int)std::min<long long>(h->num_sms, (items + NW - 1) / NW);
    const int warps = ctas * NW < c.n_kv_heads ? ctas * NW : ctas * NW / c.n_kv_heads * c.n_kv_heads;
    CK(h, cudaFuncSetAttribute(prefill_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM));
    prefill_score_kernel<<<ctas, NT, SCORE_SMEM, s>>>(p.sc, mk, static_cast<const __nv_bfloat16*>(q), c.batch, c.n_kv_heads, h->G, P, warps,
                                                      p.scale, p.scale_log2, h->st.errword);
    CK(h, cudaGetLastError());
    CK(h, launch_next(prefill_select_kernel, dim3(h->U), SEL_NT, sm, s, h->st, p.sc, layer, P, h->G, chunks, c.top_p,
                      c.evict_every, c.literal_return, c.budget_ratio > 0.f ? ratio_budget(c, P) : 0, sm > 0));
    CK(h, launch_next(prefill_rows_kernel, dim3(1 + h->U * per_head), NT, 0, s, h->st, h->plans[layer], layer, kb, vb, P, ROWS_SURVIVORS,
                      per_head, plan_grid * NW, plan_grid, h->cl[layer]));
    h->t_layer[layer] = P - 1;
    return CRYSTALKV_OK;
  }
  if (evict && c.budget_ratio > 0.f) {   // the prompt's share of the context
    fill_layer_budget_kernel<<<(h->U + NT - 1) / NT, NT, 0, s>>>(h->st, layer, ratio_budget(c, P));
    CK(h, cudaGetLastError());
  }
  // the whole prompt is stored; in full-cache mode the first step's plan is written beside the copy, and a replayed window
  // copies the rows in its attention kernel where that reads all of them (it has outputs) and is wide enough
  const bool tc = evict && window_tcgen05(h, P, W, out_window != nullptr), fill_pages = evict && out_window && window_fills_pages(h, P, W, tc);
  prefill_take_kernel<<<h->U, NT, 0, s>>>(h->st, layer, P, W > 0 ? 1 : 0);
  CK(h, cudaGetLastError());
  if (!fill_pages) {
    CK(h, launch_next(prefill_rows_kernel, dim3(1 + h->U * per_head), NT, 0, s, h->st, h->plans[layer], layer, kb, vb, P,
                      W > 0 ? ROWS_ALL : ROWS_ALL_LAST, per_head, evict ? 0 : plan_grid * NW, plan_grid, h->cl[layer]));
  }
  if (evict) {
    rc = replay_window(h, layer, kb, vb, static_cast<const unsigned char*>(q), P, W, static_cast<__nv_bfloat16*>(out_window), tc, fill_pages,
                       mk, mv, mp, s);
    if (rc) return rc;
  }
  h->t_layer[layer] = P - 1;
  return CRYSTALKV_OK;
}

int crystalkv_prefill(crystalkv_t* h, int layer, const void* k, const void* v, const void* q_last,
                      int P, void* stream) {
  return prefill_common(h, layer, k, v, q_last, P, 0, nullptr, stream);
}

int crystalkv_prefill_window(crystalkv_t* h, int layer, const void* k, const void* v,
                             const void* q_window, int P, int W, void* out_window, void* stream) {
  if (h && (W < 1 || W > P)) return fail(h, CRYSTALKV_EINVAL, "W must be in [1, P]");
  return prefill_common(h, layer, k, v, q_window, P, W, out_window, stream);
}

int crystalkv_decode_step(crystalkv_t* h, int layer, const void* q, const void* k_new,
                          const void* v_new, void* out, void* stream) {
  int rc = check_layer(h, layer);
  if (rc) return rc;
  if (!q || !k_new || !v_new || !out) return fail(h, CRYSTALKV_EINVAL, "null tensor");
  const crystalkv_config_t& c = h->cfg;
  if (h->t_layer[layer] < 0) return fail(h, CRYSTALKV_ESTATE, "decode before prefill");
  const int t = h->t_layer[layer] + 1;
  ON_DEVICE(h);
  if (t >= c.max_context) return fail(h, CRYSTALKV_ESTATE, "max_context reached");
  const bool track = c.mode == CRYSTALKV_MODE_EVICT && h->stage == CRYSTALKV_STAGE_THINK;
  if (c.mode == CRYSTALKV_MODE_EVICT && h->stage == CRYSTALKV_STAGE_ANSWER) {
    // every layer appends once per answer token; count tokens by layer 0's clock
    const int used = h->answer_steps / c.n_layers;
    if (used >= c.max_answer_tokens) return fail(h, CRYSTALKV_ESTATE, "max_answer_tokens reached");
  }
  DecodeParams p = make_params(h, layer);
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.k_new = static_cast<const __nv_bfloat16*>(k_new);
  p.v_new = static_cast<const __nv_bfloat16*>(v_new);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.t = t;
  p.track = track ? 1 : 0;
  rc = launch_step(h, p, layer, static_cast<cudaStream_t>(stream));
  if (rc) return rc;
  h->t_layer[layer] = t;
  if (!track && c.mode == CRYSTALKV_MODE_EVICT) h->answer_steps++;
  return CRYSTALKV_OK;
}

int crystalkv_decode_step_host(crystalkv_t* h, int layer, const void* q_host, const void* k_new_host,
                               const void* v_new_host, void* out_host, void* stream) {
  int rc = check_layer(h, layer);
  if (rc) return rc;
  if (!q_host || !k_new_host || !v_new_host || !out_host) return fail(h, CRYSTALKV_EINVAL, "null tensor");
  ON_DEVICE(h);
  const crystalkv_config_t& c = h->cfg;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t qb = (size_t)c.batch * c.n_q_heads * HD * 2, kb = (size_t)c.batch * c.n_kv_heads * HD * 2;
  if (h->t_layer[layer] < 0) return fail(h, CRYSTALKV_ESTATE, "decode before prefill");
  // Staging set j was last used HOST_RING host steps ago.  Page-locked inputs that the GPU can
  // address are fetched by one small kernel in the caller's stream; anything else (pageable
  // memory, 16-byte misalignment) goes up by three copies on the copy-in stream, for which the
  // caller's stream then waits.  The result comes down on the copy-out stream behind the
  // attention kernel.
  const int j = (int)(h->nHost % crystalkv::HOST_RING);
  const void* dev_view[3] = {nullptr, nullptr, nullptr};
  const void* host_in[3] = {q_host, k_new_host, v_new_host};
  bool mapped = true;
  for (int i = 0; i < 3 && mapped; ++i) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, host_in[i]) != cudaSuccess) { cudaGetLastError(); mapped = false; break; }
    mapped = at.type == cudaMemoryTypeHost && at.devicePointer != nullptr &&
             (reinterpret_cast<uintptr_t>(at.devicePointer) & 15) == 0;
    dev_view[i] = at.devicePointer;
  }
  if (mapped) {
    // The set's staged inputs were read by an attention kernel HOST_RING launches back in this
    // stream, which is complete before this kernel may start.  Its result buffer must have been
    // copied down as well; a wait in the caller's stream costs several microseconds, so one wait
    // on a much newer copy covers the steps until the ring comes round again.
    const long long n = h->nHost;
    if (n >= crystalkv::HOST_RING && n - crystalkv::HOST_RING > h->outJoined) {
      const long long target = n - 4;   // a copy that has long run by the time the stream gets here
      CK(h, cudaStreamWaitEvent(s, h->evOut[target % crystalkv::HOST_RING], 0));
      h->outJoined = target;
    }
    const int nq = (int)(qb / 16), nk = (int)(kb / 16);
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((nq + 2 * nk + NT - 1) / NT);
    lc.blockDim = dim3(NT);
    lc.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    CK(h, cudaLaunchKernelEx(&lc, stage_in_kernel, reinterpret_cast<uint4*>(h->dq[j]), reinterpret_cast<uint4*>(h->dk[j]),
                             reinterpret_cast<uint4*>(h->dv[j]), static_cast<const uint4*>(dev_view[0]),
                             static_cast<const uint4*>(dev_view[1]), static_cast<const uint4*>(dev_view[2]), nq, nk));
  } else {
    // the copy back of the step that used the set before ran behind that step's attention
    // kernel, so its event covers both
    if (h->nHost >= crystalkv::HOST_RING) CK(h, cudaStreamWaitEvent(h->copy_in, h->evOut[j], 0));
    CK(h, cudaMemcpyAsync(h->dq[j], q_host, qb, cudaMemcpyHostToDevice, h->copy_in));
    CK(h, cudaMemcpyAsync(h->dk[j], k_new_host, kb, cudaMemcpyHostToDevice, h->copy_in));
    CK(h, cudaMemcpyAsync(h->dv[j], v_new_host, kb, cudaMemcpyHostToDevice, h->copy_in));
    CK(h, cudaEventRecord(h->evIn[j], h->copy_in));
    CK(h, cudaStreamWaitEvent(s, h->evIn[j], 0));
  }
  rc = crystalkv_decode_step(h, layer, h->dq[j], h->dk[j], h->dv[j], h->dout[j], stream);
  if (rc) return rc;
  CK(h, cudaEventRecord(h->evUse[j], s));
  CK(h, cudaStreamWaitEvent(h->copy_out, h->evUse[j], 0));
  CK(h, cudaMemcpyAsync(out_host, h->dout[j], qb, cudaMemcpyDeviceToHost, h->copy_out));
  CK(h, cudaEventRecord(h->evOut[j], h->copy_out));
  h->nHost++;
  return CRYSTALKV_OK;
}

int crystalkv_rebudget(crystalkv_t* h, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  if (h->cuda_dead) return fail(h, CRYSTALKV_ECUDA, "an earlier CUDA error is sticky for this handle");
  const crystalkv_config_t& c = h->cfg;
  if (c.mode != CRYSTALKV_MODE_EVICT) return fail(h, CRYSTALKV_ESTATE, "rebudget in FullKV mode");
  ON_DEVICE(h);
  const int t_last = h->t_layer[0];
  if (t_last < 0) return fail(h, CRYSTALKV_ESTATE, "rebudget before prefill");
  for (int l = 1; l < c.n_layers; ++l)
    if (h->t_layer[l] != t_last) return fail(h, CRYSTALKV_ESTATE, "layers are at different time steps");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  crf_sum_kernel<<<h->units, NT, 0, s>>>(h->st, t_last, h->Asum);
  CK(h, cudaGetLastError());
  const int N = c.n_layers * c.n_kv_heads;
  const size_t sm = (size_t)N * (3 * sizeof(double) + sizeof(long long) + 2 * sizeof(int)) + (size_t)c.n_layers * 2 * sizeof(double);
  if (sm > 48 * 1024) CK(h, cudaFuncSetAttribute(alg2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  const long long B_total = (long long)(c.budget_ratio > 0.f ? ratio_budget(c, t_last + 1) : c.budget_per_head) * N;
  alg2_kernel<<<c.batch, NT, sm, s>>>(h->Asum, h->st.budget, c.n_layers, c.n_kv_heads, B_total, c.min_budget, c.max_budget);
  CK(h, cudaGetLastError());
  h->uniform = false;
  h->len_cap.assign(c.n_layers, (int)(B_total / N) + c.evict_every);
  if (int sr = shrink_layers(h, 0, c.n_layers, t_last, s)) return sr;
  // heads changed length: every layer's next decode step needs a new plan (all layers are at the same time)
  h->cl.assign(c.n_layers, share_heads(h, h->entries(0, t_last + 2)));
  return replan(h, 0, c.n_layers, s);
}

int crystalkv_set_budget(crystalkv_t* h, int layer, int seq, int kv_head, int32_t budget, void* stream) {
  int rc = check_unit(h, layer, seq, kv_head);
  if (rc) return rc;
  const crystalkv_config_t& c = h->cfg;
  if (c.mode != CRYSTALKV_MODE_EVICT) return fail(h, CRYSTALKV_ESTATE, "set_budget in FullKV mode");
  if (budget < 1 || budget > c.max_budget) return fail(h, CRYSTALKV_EINVAL, "budget outside [1, max_budget]");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  if (int lr = leave_clusters(h, s)) return lr;
  const int uid = (seq * c.n_layers + layer) * c.n_kv_heads + kv_head;
  CK(h, cudaMemcpyAsync(h->st.budget + uid, &budget, sizeof(int), cudaMemcpyHostToDevice, s));
  CK(h, cudaStreamSynchronize(s));
  if (h->t_layer[layer] >= 0) {
    if (int sr = shrink_layers(h, layer, 1, h->t_layer[layer], s)) return sr;
    return replan(h, layer, 1, s);
  }
  return CRYSTALKV_OK;
}

int crystalkv_get_budgets(crystalkv_t* h, int32_t* out_host, void* stream) {
  if (!h || !out_host) return fail(h, CRYSTALKV_EINVAL, "null argument");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  CK(h, cudaMemcpyAsync(out_host, h->st.budget, (size_t)h->units * sizeof(int), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  return CRYSTALKV_OK;
}

// Copies one head's entries to the host, sorted by token position: records and, if asked for, rows.
static int fetch_unit(crystalkv_t* h, int layer, int seq, int kv_head, std::vector<int32_t>& rec,
                      std::vector<unsigned char>* krows, std::vector<unsigned char>* vrows, cudaStream_t s) {
  const crystalkv_config_t& c = h->cfg;
  if (int jr = join_side(h, s)) return jr;
  const int uid = (seq * c.n_layers + layer) * c.n_kv_heads + kv_head;
  export_unit_kernel<<<1, NT, 0, s>>>(h->st, uid, seq, h->io_rec, krows ? h->io_rows : nullptr,
                                      krows ? h->io_rows + (size_t)h->cap * ROW_BYTES : nullptr, h->io_n);
  CK(h, cudaGetLastError());
  int n = 0;
  CK(h, cudaMemcpyAsync(&n, h->io_n, sizeof(int), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  std::vector<int32_t> raw((size_t)3 * n);
  std::vector<unsigned char> kr, vr;
  CK(h, cudaMemcpyAsync(raw.data(), h->io_rec, raw.size() * 4, cudaMemcpyDeviceToHost, s));
  if (krows) {
    kr.resize((size_t)n * ROW_BYTES); vr.resize((size_t)n * ROW_BYTES);
    CK(h, cudaMemcpyAsync(kr.data(), h->io_rows, kr.size(), cudaMemcpyDeviceToHost, s));
    CK(h, cudaMemcpyAsync(vr.data(), h->io_rows + (size_t)h->cap * ROW_BYTES, vr.size(), cudaMemcpyDeviceToHost, s));
  }
  CK(h, cudaStreamSynchronize(s));
  std::vector<int> idx(n);
  for (int i = 0; i < n; ++i) idx[i] = i;
  std::sort(idx.begin(), idx.end(), [&](int a, int b) { return raw[3 * a] < raw[3 * b]; });
  rec.resize((size_t)3 * n);
  if (krows) { krows->resize((size_t)n * ROW_BYTES); vrows->resize((size_t)n * ROW_BYTES); }
  for (int i = 0; i < n; ++i) {
    std::memcpy(&rec[3 * i], &raw[3 * idx[i]], 12);
    if (krows) {
      std::memcpy(krows->data() + (size_t)i * ROW_BYTES, kr.data() + (size_t)idx[i] * ROW_BYTES, ROW_BYTES);
      std::memcpy(vrows->data() + (size_t)i * ROW_BYTES, vr.data() + (size_t)idx[i] * ROW_BYTES, ROW_BYTES);
    }
  }
  return CRYSTALKV_OK;
}

int crystalkv_export_state(crystalkv_t* h, int layer, int seq, int kv_head, int32_t* host_buf,
                           int32_t cap, int32_t* n_out, void* stream) {
  int rc = check_unit(h, layer, seq, kv_head);
  if (rc) return rc;
  if (!host_buf || !n_out) return fail(h, CRYSTALKV_EINVAL, "null argument");
  ON_DEVICE(h);
  std::vector<int32_t> rec;
  rc = fetch_unit(h, layer, seq, kv_head, rec, nullptr, nullptr, static_cast<cudaStream_t>(stream));
  if (rc) return rc;
  const int n = (int)(rec.size() / 3);
  *n_out = n;
  if (n > cap) return fail(h, CRYSTALKV_ESTATE, "buffer too small");
  std::memcpy(host_buf, rec.data(), rec.size() * 4);
  return CRYSTALKV_OK;
}

int crystalkv_export_kv(crystalkv_t* h, int layer, int seq, int kv_head, void* k_rows_host, void* v_rows_host,
                        int32_t cap, int32_t* n_out, void* stream) {
  int rc = check_unit(h, layer, seq, kv_head);
  if (rc) return rc;
  if (!k_rows_host || !v_rows_host || !n_out) return fail(h, CRYSTALKV_EINVAL, "null argument");
  ON_DEVICE(h);
  std::vector<int32_t> rec;
  std::vector<unsigned char> kr, vr;
  rc = fetch_unit(h, layer, seq, kv_head, rec, &kr, &vr, static_cast<cudaStream_t>(stream));
  if (rc) return rc;
  const int n = (int)(rec.size() / 3);
  *n_out = n;
  if (n > cap) return fail(h, CRYSTALKV_ESTATE, "buffer too small");
  std::memcpy(k_rows_host, kr.data(), kr.size());
  std::memcpy(v_rows_host, vr.data(), vr.size());
  return CRYSTALKV_OK;
}

int crystalkv_get_retained(crystalkv_t* h, int layer, int seq, int kv_head, int32_t* pos_out_host,
                           int32_t cap, int32_t* n_out, void* stream) {
  int rc = check_unit(h, layer, seq, kv_head);
  if (rc) return rc;
  if (!pos_out_host || !n_out) return fail(h, CRYSTALKV_EINVAL, "null argument");
  ON_DEVICE(h);
  std::vector<int32_t> rec;
  rc = fetch_unit(h, layer, seq, kv_head, rec, nullptr, nullptr, static_cast<cudaStream_t>(stream));
  if (rc) return rc;
  const int n = (int)(rec.size() / 3);
  *n_out = n;
  if (n > cap) return fail(h, CRYSTALKV_ESTATE, "buffer too small");
  for (int i = 0; i < n; ++i) pos_out_host[i] = rec[3 * i];
  return CRYSTALKV_OK;
}

int crystalkv_import_state(crystalkv_t* h, int layer, int seq, int kv_head, const int32_t* host_buf,
                           int32_t n_rec, const void* k_rows_host, const void* v_rows_host, int32_t budget,
                           int32_t t, void* stream) {
  int rc = check_unit(h, layer, seq, kv_head);
  if (rc) return rc;
  if (!host_buf || !k_rows_host || !v_rows_host) return fail(h, CRYSTALKV_EINVAL, "null argument");
  const crystalkv_config_t& c = h->cfg;
  if (n_rec < 1 || n_rec + 1 > h->cap) return fail(h, CRYSTALKV_EINVAL, "entry count outside [1, list capacity)");
  if (budget < 0 || (c.mode == CRYSTALKV_MODE_EVICT && budget > c.max_budget)) return fail(h, CRYSTALKV_EINVAL, "budget outside [0, max_budget]");
  if (t < 0 || t >= c.max_context) return fail(h, CRYSTALKV_EINVAL, "time outside [0, max_context)");
  if (h->t_layer[layer] >= 0 && h->t_layer[layer] != t) return fail(h, CRYSTALKV_ESTATE, "the layer is at another time step");
  for (int i = 0; i < n_rec; ++i)
    if (host_buf[3 * i] < 0 || host_buf[3 * i] > t || host_buf[3 * i + 2] < 0 || host_buf[3 * i + 2] > t)
      return fail(h, CRYSTALKV_EINVAL, "a record's position or last hit time lies after the layer's time");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  if (int lr = leave_clusters(h, s)) return lr;
  const int uid = (seq * c.n_layers + layer) * c.n_kv_heads + kv_head;
  CK(h, cudaMemcpyAsync(h->io_rec, host_buf, (size_t)n_rec * 12, cudaMemcpyHostToDevice, s));
  CK(h, cudaMemcpyAsync(h->io_rows, k_rows_host, (size_t)n_rec * ROW_BYTES, cudaMemcpyHostToDevice, s));
  CK(h, cudaMemcpyAsync(h->io_rows + (size_t)h->cap * ROW_BYTES, v_rows_host, (size_t)n_rec * ROW_BYTES, cudaMemcpyHostToDevice, s));
  int b = budget;
  if (b == 0) {
    CK(h, cudaMemcpyAsync(&b, h->st.budget + uid, sizeof(int), cudaMemcpyDeviceToHost, s));
    CK(h, cudaStreamSynchronize(s));
  }
  import_unit_kernel<<<1, NT, 0, s>>>(h->st, uid, seq, h->io_rec, h->io_rows, h->io_rows + (size_t)h->cap * ROW_BYTES, n_rec, b);
  CK(h, cudaGetLastError());
  CK(h, cudaStreamSynchronize(s));   // the host buffers and the staging area are free again
  h->t_layer[layer] = t;
  h->prev_layer = -1;
  return replan(h, layer, 1, s);
}

int crystalkv_get_counters(crystalkv_t* h, uint64_t* entries_attended, uint64_t* hits,
                           uint64_t* evictions, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  unsigned long long v[3];
  sum_counters_kernel<<<1, 1024, 0, s>>>(h->st, h->units, h->io_sum);
  CK(h, cudaGetLastError());
  CK(h, cudaMemcpyAsync(v, h->io_sum, sizeof(v), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  if (entries_attended) *entries_attended = v[0];
  if (hits) *hits = v[1];
  if (evictions) *evictions = v[2];
  return CRYSTALKV_OK;
}

int crystalkv_validate(crystalkv_t* h, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  if (h->cuda_dead) return fail(h, CRYSTALKV_ECUDA, "an earlier CUDA error is sticky for this handle");
  const crystalkv_config_t& c = h->cfg;
  for (int l = 0; l < c.n_layers; ++l)
    if (h->t_layer[l] < 0) return fail(h, CRYSTALKV_ESTATE, "validate before every layer is prefilled");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  const long long total = (long long)c.batch * h->pages_per_seq;
  int* seen = nullptr;
  CK(h, device_malloc(c.device, reinterpret_cast<void**>(&seen), (size_t)(total + 2) * sizeof(int)));
  cudaError_t e = cudaMemsetAsync(seen, 0, (size_t)(total + 2) * sizeof(int), s);
  if (e == cudaSuccess) {
    mark_free_kernel<<<dim3(256, c.batch), 256, 0, s>>>(h->st, seen);
    for (int l = 0; l < c.n_layers; ++l)
      mark_owned_kernel<<<h->U, 128, 0, s>>>(h->st, l, seen);
    count_bad_kernel<<<1024, 256, 0, s>>>(seen, total, seen + total + 1);
    e = cudaGetLastError();
  }
  int res[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(res, seen + total, 2 * sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(seen);
  CK(h, e);
  if (res[0] || res[1])
    return fail(h, CRYSTALKV_ECHECK, "page ownership broken: " + std::to_string(res[0]) + " ids or counts out of range, " +
                                         std::to_string(res[1]) + " pages not owned exactly once");
  return CRYSTALKV_OK;
}

// ---- the page-ownership check for callers that cannot allocate device memory
// The per-page counters live in this file-scope device array instead of a temporary from
// cudaMalloc.  Every GPU that loads the library holds the array (512 KB) until the process exits.
constexpr long long STATIC_SEEN_PAGES = 1ll << 17;
static __device__ __align__(256) int g_seen_static[STATIC_SEEN_PAGES + 2];
constexpr int STATIC_MAX_DEVICES = 64;
static int* g_seen_addr[STATIC_MAX_DEVICES] = {};   // device address of the array, per device ordinal
static std::mutex g_seen_mu;                        // guards the look-up above

int crystalkv_validate_static(crystalkv_t* h, int32_t* counts_out_host, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  if (h->cuda_dead) return fail(h, CRYSTALKV_ECUDA, "an earlier CUDA error is sticky for this handle");
  const crystalkv_config_t& c = h->cfg;
  for (int l = 0; l < c.n_layers; ++l)
    if (h->t_layer[l] < 0) return fail(h, CRYSTALKV_ESTATE, "validate before every layer is prefilled");
  const long long total = (long long)c.batch * h->pages_per_seq;
  if (total > STATIC_SEEN_PAGES)
    return fail(h, CRYSTALKV_EINVAL,
                "crystalkv_validate_static: the handle has " + std::to_string(total) + " pool pages, the built-in "
                "scratch covers " + std::to_string(STATIC_SEEN_PAGES) + "; use crystalkv_validate");
  if (c.device >= STATIC_MAX_DEVICES) return fail(h, CRYSTALKV_EINVAL, "crystalkv_validate_static: device ordinal above 63");
  ON_DEVICE(h);
  int* seen = nullptr;
  {
    // In host code the array's name is only a handle for the runtime; its device address has
    // to be asked for, once per device and with that device current.
    std::lock_guard<std::mutex> lock(g_seen_mu);
    if (!g_seen_addr[c.device]) {
      int* addr = nullptr;
      CK(h, cudaGetSymbolAddress(reinterpret_cast<void**>(&addr), g_seen_static));
      g_seen_addr[c.device] = addr;
    }
    seen = g_seen_addr[c.device];
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  // the array keeps what the last call left: everything this call reads starts from zero
  CK(h, cudaMemsetAsync(seen, 0, (size_t)(total + 2) * sizeof(int), s));
  mark_free_kernel<<<dim3(256, c.batch), 256, 0, s>>>(h->st, seen);
  for (int l = 0; l < c.n_layers; ++l)
    mark_owned_kernel<<<h->U, 128, 0, s>>>(h->st, l, seen);
  count_bad_kernel<<<1024, 256, 0, s>>>(seen, total, seen + total + 1);
  CK(h, cudaGetLastError());
  int res[2] = {0, 0};
  CK(h, cudaMemcpyAsync(res, seen + total, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  if (counts_out_host) { counts_out_host[0] = res[0]; counts_out_host[1] = res[1]; }
  if (res[0] || res[1])
    return fail(h, CRYSTALKV_ECHECK, "page ownership broken: " + std::to_string(res[0]) + " ids or counts out of range, " +
                                         std::to_string(res[1]) + " pages not owned exactly once");
  return CRYSTALKV_OK;
}

int crystalkv_debug_set_page(crystalkv_t* h, int layer, int seq, int kv_head, int32_t index, int32_t page, void* stream) {
  int rc = check_unit(h, layer, seq, kv_head);
  if (rc) return rc;
  if (index < 0 || index >= h->st.capg || page < 0 || page >= h->pages_per_seq)
    return fail(h, CRYSTALKV_EINVAL, "page table index or page id out of range");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  const int uid = (seq * h->cfg.n_layers + layer) * h->cfg.n_kv_heads + kv_head;
  CK(h, cudaMemcpyAsync(h->st.ptab + (size_t)uid * h->st.capg + index, &page, sizeof(int), cudaMemcpyHostToDevice, s));
  CK(h, cudaStreamSynchronize(s));
  return CRYSTALKV_OK;
}

int crystalkv_debug_ctas_needed(int32_t whole_ctas, const int32_t* runs_by_length) {
  if (!runs_by_length || whole_ctas < 0) return CRYSTALKV_EINVAL;
  int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int s = 1; s < 8; ++s) {
    if (runs_by_length[s] < 0) return CRYSTALKV_EINVAL;
    cnt[s] = runs_by_length[s];
  }
  return ctas_needed(whole_ctas, cnt);
}

static int place_runs_hook(int32_t whole_ctas, const int32_t* runs_by_length, int32_t grid, int32_t spread, int32_t* first_warp, int32_t cap) {
  if (!runs_by_length || !first_warp || whole_ctas < 0 || grid < 0) return CRYSTALKV_EINVAL;
  int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  long long total = 0;
  for (int s = 1; s < 8; ++s) {
    if (runs_by_length[s] < 0) return CRYSTALKV_EINVAL;
    cnt[s] = runs_by_length[s];
    total += cnt[s];
  }
  if (total > cap) return CRYSTALKV_EINVAL;
  Placement p{};
  if (whole_ctas > grid || !place_runs(whole_ctas, cnt, grid, spread != 0, p)) return CRYSTALKV_ESTATE;
  int at = 0;
  for (int s = 7; s >= 1; --s)
    for (int r = 0; r < cnt[s]; ++r) first_warp[at++] = run_warp(p, s, r);
  return at;
}

int crystalkv_debug_place_runs(int32_t whole_ctas, const int32_t* runs_by_length, int32_t grid, int32_t* first_warp, int32_t cap) {
  return place_runs_hook(whole_ctas, runs_by_length, grid, 0, first_warp, cap);
}

int crystalkv_debug_spread_runs(int32_t whole_ctas, const int32_t* runs_by_length, int32_t grid, int32_t* first_warp, int32_t cap) {
  return place_runs_hook(whole_ctas, runs_by_length, grid, 1, first_warp, cap);
}

int crystalkv_debug_get_plan(crystalkv_t* h, int layer, int32_t* hdr_host, int32_t* wrange_host, int32_t warps_cap,
                             int32_t* desc_host, int32_t pieces_cap, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  if (h->cuda_dead) return fail(h, CRYSTALKV_ECUDA, "an earlier CUDA error is sticky for this handle");
  if (layer < 0 || layer >= h->cfg.n_layers || !hdr_host || !wrange_host || !desc_host)
    return fail(h, CRYSTALKV_EINVAL, "layer out of range or a NULL output");
  const int nWarps = h->grid * NW;
  if (warps_cap < nWarps || pieces_cap < nWarps + h->U) return fail(h, CRYSTALKV_EINVAL, "output arrays too small for the plan");
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  const Plan& pl = h->plans[layer];
  CK(h, cudaMemcpyAsync(hdr_host, pl.hdr, 4 * sizeof(int), cudaMemcpyDeviceToHost, s));
  // (a plan for shared heads names only the warps of their clusters: the others have nothing to stream)
  std::vector<int4> wr((size_t)nWarps, make_int4(0, 0, -1, 0));
  CK(h, cudaMemcpyAsync(wr.data(), pl.wrange, (size_t)std::min(nWarps, h->plan_grid(layer) * NW) * sizeof(int4), cudaMemcpyDeviceToHost, s));
  CK(h, cudaMemcpyAsync(desc_host, pl.desc, (size_t)(nWarps + h->U) * sizeof(int4), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  for (int w = 0; w < nWarps; ++w) { wrange_host[2 * w] = wr[w].x; wrange_host[2 * w + 1] = wr[w].y; }
  return CRYSTALKV_OK;
}

int crystalkv_join(crystalkv_t* h, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  if (h->cuda_dead) return fail(h, CRYSTALKV_ECUDA, "an earlier CUDA error is sticky for this handle");
  ON_DEVICE(h);
  return join_side(h, static_cast<cudaStream_t>(stream));
}

int crystalkv_check(crystalkv_t* h, void* stream) {
  if (!h) return CRYSTALKV_EINVAL;
  ON_DEVICE(h);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (int jr = join_side(h, s)) return jr;
  int w = 0;
  CK(h, cudaMemcpyAsync(&w, h->st.errword, sizeof(int), cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  if (w == 0) return CRYSTALKV_OK;
  CK(h, cudaMemsetAsync(h->st.errword, 0, sizeof(int), s));
  std::string msg = "device error word:";
  if (w & ERR_FREE_UNDERFLOW) msg += " free page list underflow;";
  if (w & ERR_OVER_EVICT) msg += " head further over its budget than the eviction period in a decode step;";
  if (w & ERR_CAPACITY) msg += " head list capacity exceeded;";
  if (w & ERR_NUCLEUS) msg += " top-p boundary not found;";
  if (w & ERR_COPY_TIMEOUT) msg += " a bulk copy into shared memory timed out;";
  if (w & ERR_PLAN) msg += " a layer's launch plan did not fit the launch;";
  if (w & ERR_EMPTY) msg += " a decode step met a head without entries;";
  return fail(h, CRYSTALKV_ECHECK, msg);
}

}  // extern "C"
