// Launching Algorithm 1's kernel (lrfu_kernel.cuh): its launch shape, and the instantiations by group
// size, which are compiled in units of their own.
#pragma once
#include "common.cuh"

namespace ckv {

constexpr int MAX_DEVICES = 64;   // device ordinals this library keeps per-device state for
constexpr int FRONT = 5;   // entries per thread whose logit rows are requested before n is known
constexpr int LRFU_SMALL = 64;   // threads of the CTAs for short heads

// Threads of a head's CTA.  hint: entries of a head in this step if all are alike (uniform), else about
// the mean (crystalkv::entries; it follows heads that fill).
//  * Heads of at most 5 x 64 entries take CTAs of two warps once there are more heads than SMs: six
//    of them fit beside an attention CTA instead of two of eight warps, most of which idle in the
//    block-wide steps.  128 sequences of 8 heads of 257 entries: 27.8 us a layer instead of 38.7.
//  * All other heads take CTAs of eight warps, two of which fit beside an attention CTA.  (Sixteen for heads of more than
//    1280 entries where every head finds an SM make the kernel shorter and the layer longer: what counts is how hard a CTA
//    presses on the attention warps of its SM.  us a layer with sixteen and with eight, heads of 4097 entries: 16 heads 13.8 and
//    13.7, 32 17.4 and 18.2, 44 23.1 and 22.4, 48 24.0 and 23.4, 64 29.9 and 28.2, 72 31.4 and 30.3, 96 43.1 and 42.4; 128 heads of 1024 ..
//    3072 27.7 and 27.0, 64 of 1300 .. 3900 21.9 and 20.4, 32 of 2049 12.0 and 11.5.)
inline int lrfu_threads(int U, int hint, bool uniform, int num_sms) {
  return uniform && hint <= FRONT * LRFU_SMALL && U > num_sms ? LRFU_SMALL : NT;
}

// Entries whose pbar a CTA keeps in shared memory (longer heads use the global scratch).  Beside an attention CTA an SM
// has 34 KB left, 30 KB beside one that shares heads: room for six CTAs of LRFU_SMALL, two of NT, or one of NT for long heads
// that find an SM each.
// (One of NT for few heads of any length: 64 heads of 128 .. 2000 entries 11.55 us a layer instead of 11.3.)
inline int pbar_room(int threads, int U, int hint, int num_sms, bool shared) {
  if (threads == LRFU_SMALL) return FRONT * LRFU_SMALL;
  const int two = shared ? 1440 : 1856, one = shared ? 5248 : 5632;
  return hint > two && U <= num_sms ? one : two;
}

// Launches the kernel for `heads` heads; threads: LRFU_SMALL or NT; npb: entries whose pbar fits shared memory.
cudaError_t lrfu_launch_small(int G, const DecodeParams& p, int npb, int heads, cudaStream_t s);
cudaError_t lrfu_launch_mid(int G, const DecodeParams& p, int npb, int heads, cudaStream_t s);
inline cudaError_t lrfu_launch(int threads, int npb, int G, const DecodeParams& p, int heads, cudaStream_t s) {
  return threads == LRFU_SMALL ? lrfu_launch_small(G, p, npb, heads, s) : lrfu_launch_mid(G, p, npb, heads, s);
}

}  // namespace ckv
