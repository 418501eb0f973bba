// Attention of an observation window's queries over a prompt on mma.sync: for launches that the kernel on tcgen05 (window_attn.cuh) is
// too large for (window_tcgen05() in crystalkv.cu).  A CTA of four warps takes 64 (query, head) rows, three fit an SM, and the keys are passed once.
#pragma once
#include "window_attn.cuh"

namespace ckv {

constexpr int WM_WARPS = 4;                   // warps of a CTA, 16 (query, head) rows each
constexpr int WM_ROWS = WM_WARPS * 16;
constexpr int WM_KEYS = 64;                   // keys per tile
constexpr int WM_TILE = WM_KEYS * ROW_BYTES;  // bytes of a K (or V) tile
constexpr int WM_SMEM = 4 * WM_TILE;          // K and V, two stages

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
__global__ void __launch_bounds__(WM_WARPS * 32, 3) window_mma_kernel(const __grid_constant__ State st, const WindowParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  pdl_launch();   // (an ordinary launch)
  const int u = blockIdx.y, seq = u / p.H, head = u % p.H;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int R = p.W * p.G, r_lo = blockIdx.x * WM_ROWS;
  const int ra = r_lo + w * 16 + gid, rb = ra + 8;          // this lane's two rows
  const bool va = ra < R, vb = rb < R;
  const int wa = min(ra, R - 1) / p.G, ga = min(ra, R - 1) % p.G, wb = min(rb, R - 1) / p.G, gb = min(rb, R - 1) % p.G;
  const int ta = p.t0 + wa, tb = p.t0 + wb;                 // times: keys 0 .. t take part
  auto keys_of = [&](int b) { return p.t0 + min(R - 1, (b + 1) * WM_ROWS - 1) / p.G + 1; };   // block b's last query sees these
  const int n_keys = keys_of(blockIdx.x);
  const int ntiles = (n_keys + WM_KEYS - 1) / WM_KEYS;
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
    const uint32_t ks = s0 + stage * 2 * WM_TILE, vs = ks + WM_TILE;
    const int c = tid & 15;
#pragma unroll
    for (int x = 0; x < WM_KEYS / 8; ++x) {
      const int key = (tid >> 4) + 8 * x;
      const size_t off = (size_t)min(tile * WM_KEYS + key, p.P - 1) * row;   // (keys past the prompt are masked)
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
    const uint32_t ks = s0 + stage * 2 * WM_TILE, vs = ks + WM_TILE;
    if (store) {
      const int last = gridDim.x - 1, turn = tile % gridDim.x;
      if (blockIdx.x == ((tile + 1) * WM_KEYS <= keys_of(turn) ? turn : last)) {   // an entry per warp and turn, lane c its chunk c
        const int* pt = st.ptab + (size_t)uid * st.capg + tile * (WM_KEYS / GRP);
        unsigned char* pool = st.pool + (size_t)seq * st.pages_per_seq * PAGE_BYTES;
#pragma unroll 4
        for (int key = w; key < min(WM_KEYS, p.P - tile * WM_KEYS); key += WM_WARPS) {
          const uint32_t at = lane < 16 ? ks + key * ROW_BYTES + ((lane ^ ((key & 1) << 2)) << 4)
                                        : vs + key * ROW_BYTES + (((lane - 16) ^ (key & 7)) << 4);
          uint4 x;
          asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];\n" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "r"(at));
          *reinterpret_cast<uint4*>(pool + (size_t)pt[key / GRP] * PAGE_BYTES + chunk_offset(key & (GRP - 1), lane)) = x;
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
    const int k0 = tile * WM_KEYS + 2 * tig;
    float ca = -INFINITY, cb = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int key = k0 + nt * 8;
      if (va && key <= ta) *reinterpret_cast<float2*>(lga + tile * WM_KEYS + nt * 8) = make_float2(__fmul_rn(s[nt][0], p.scale), __fmul_rn(s[nt][1], p.scale));
      if (vb && key <= tb) *reinterpret_cast<float2*>(lgb + tile * WM_KEYS + nt * 8) = make_float2(__fmul_rn(s[nt][2], p.scale), __fmul_rn(s[nt][3], p.scale));
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

}  // namespace ckv
