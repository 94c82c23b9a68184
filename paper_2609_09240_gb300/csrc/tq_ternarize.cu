// tq_ternarize.cu - E2M-ATQ ternarization of fp16 weights straight into the
// packed format (paper "Conversion Pipeline", subsection "E2M-ATQ"; the
// representation of "Model and Representation", eq. for W-hat, read per
// (row, group of 128) block).
//
// Per block w (128 fp16 weights of one row and group):
//   mu = mean(w), c = w - mu, Delta0 = 0.75 mean|c|, T0 = sign(c) where
//   |c| > Delta0, alpha0 = least-squares scale of c on T0; residual
//   r = c - alpha0 T0 with energy E = sum r^2.  The projection's nnz blocks
//   of largest E (ties: lower block id) are salient: their residual gets a
//   second support T1 by the same threshold rule and its least-squares
//   scale alpha1.  Then `sweeps` alternating refinements of mu, alpha0,
//   alpha1 with the supports fixed.  Stored: offset = fp16(mu), scale1 =
//   fp16(alpha0), scale2 = fp16(alpha1), plane 1 = T0, plane 2 = T1.
//
// The supports, thresholds and the salience are integer decisions taken from
// floats, so their arithmetic is fixed: IEEE float32 with explicit
// round-to-nearest operations (never contracted into fused multiply-adds),
// every sum over a block in index order 0..127 from +0, means as sums times
// 1/128.  One thread owns one block, which makes index order its natural
// order.  The refinement decides nothing and runs on per-block moments (see
// plane2_blocks); its fp16 outputs agree with in-order passes to one ulp.
//
// Kernels, in launch order:
//   tern_stats_kernel   per block: mu, Delta0, alpha0 and E (key = E's bits)
//   tern_select_kernel  four passes of an 8-bit radix select of the nnz-th
//                       largest key, the salience words (keys above the
//                       selected key, and the first `need` equal keys in
//                       block-id order) and rowptr, in one cluster; if the
//                       keys exceed its shared memory or the device holds no
//                       such cluster, instead, over the whole chip,
//                       tern_hist_kernel (a pass each; the last CTA to finish
//                       picks the digit, no CTA waits for another),
//                       tern_count_kernel (keys equal to the selected one, per
//                       chunk of salience words), tern_mark_kernel and rowptr
//                       (tq_codec.cu); then
//   tern_planes_kernel  per block: supports, second plane, refinement, and
//                       the packed bytes and fp16 parameters (salient blocks
//                       by record, in CTAs of their own).
// Each is launched while its predecessor still runs (programmatic dependent
// launch) and waits for it before it reads anything (rowptr of many rows, after
// its end).
#include <algorithm>

#include "tq_common.cuh"
#include "tq_launch.cuh"
#include "tq_sm100.cuh"

namespace tq {

cudaError_t launch_rowptr(int N, int K, const uint32_t *sal, int32_t *rowptr, uint32_t *status, bool behind_smem,
                          cudaStream_t s);

namespace tz {

constexpr int kBlockThreads = 128;  // per-block kernels: one thread per (row, group)
constexpr int kSelThreads = 1024;   // histogram kernels
constexpr int kMarkWords = 128;     // count / mark kernels: salience words per CTA,
constexpr int kWarpWords = 8;       // per warp (with 32 per warp 9 to 10 us a kernel, this 5.3 and 6.6)
constexpr int kMarkThreads = 32 * kMarkWords / kWarpWords;
constexpr float kInvGroup = 0.0078125f;  // 1 / 128, exact
constexpr float kThresh = 0.75f;         // E2M-ATQ threshold factor

// Radix-select state after each pass: bits of the selected key fixed so far,
// and how many keys with that prefix are still to take.
struct SelState {
  uint32_t prefix[5];
  uint32_t pad_;
  int64_t need[5];
};

struct SelWork {
  uint32_t hist[4][256];
  uint32_t done[4];  // CTAs finished per pass
  uint32_t pad_[4];
  SelState st;
};

// A block's 128 fp16 weights, staged in shared memory by the warp of the
// thread that owns the block, 16 bytes of padding behind its 256, so that a
// warp's 16-byte loads (eight weights of each of its blocks) are free of bank
// conflicts.  Every pass re-reads the block with volatile loads, which the
// compiler can neither merge nor hoist, so a thread's registers hold only
// scalars (a block's 128 floats and its supports exceed the register file).
constexpr int kBlkStride = 2 * kGroup + 16;
constexpr int kBlkShared = kBlockThreads * kBlkStride;
struct Blk {
  uint32_t base;  // shared address of the thread's block
  // weights 8 j .. 8 j + 7
  __device__ __forceinline__ void oct(int j, float (&x)[8]) const {
    uint32_t w[4];
    asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                 : "r"(base + 16u * (uint32_t)j));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
      x[2 * i] = v.x, x[2 * i + 1] = v.y;
    }
  }
  // fn(x) for the weights in index order.
  template <class Fn>
  __device__ __forceinline__ void all(Fn fn) const {
#pragma unroll 4
    for (int j = 0; j < 16; ++j) {
      float x[8];
      oct(j, x);
#pragma unroll
      for (int i = 0; i < 8; ++i) fn(x[i]);
    }
  }
  // The 26 packed bytes of the trits fn(x) of the weights in index order, as
  // 13 halfwords at dst: a trit adds its power of 3 to a byte that starts
  // with every digit 1 (digit = trit + 1, first trit least significant; the
  // tail byte holds trits 125..127 and two pad digits 1).
  template <class Fn>
  __device__ __forceinline__ void pack(uint16_t *dst, Fn fn) const {
#pragma unroll 1
    for (int h = 0; h < 4; ++h) {  // weights 40 h .. 40 h + 39: bytes 8 h .. 8 h + 7 (the last round: 24 and the tail)
      constexpr int pw[5] = {1, 3, 9, 27, 81};
      int v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = kZeroByte;
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        if (j == 0 || h < 3) {
          float x[8];
          oct(5 * h + j, x);
#pragma unroll
          for (int i = 0; i < 8; ++i) v[(8 * j + i) / 5] += pw[(8 * j + i) % 5] * fn(x[i]);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k == 0 || h < 3) dst[4 * h + k] = (uint16_t)(v[2 * k] | v[2 * k + 1] << 8);
    }
  }
};

// The trit of c at threshold d >= 0: +1 above d, -1 below -d.
__device__ __forceinline__ int trit_of(float c, float d) { return (c > d ? 1 : 0) - (c < -d ? 1 : 0); }
// a * t for a trit t as the sums take it: +a, -a or +0.
__device__ __forceinline__ float times_trit(float a, int t) { return t > 0 ? a : t < 0 ? -a : 0.f; }

// The whole warp: stages every lane's block b (none if negative), two blocks'
// 512 bytes per coalesced load (a thread loading its own block touched 32
// cache lines with each).
__device__ __forceinline__ Blk stage_block(const uint16_t *W, int64_t b, unsigned char *sx) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char *mine = sx + warp * 32 * kBlkStride;
  uint4 v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int64_t bb = __shfl_sync(0xffffffffu, b, 2 * i + (lane >> 4));
    v[i] = bb >= 0 ? __ldg(reinterpret_cast<const uint4 *>(W + bb * kGroup) + (lane & 15)) : make_uint4(0u, 0u, 0u, 0u);
  }
  __syncwarp();  // the previous blocks' reads are done
#pragma unroll
  for (int i = 0; i < 16; ++i)
    *reinterpret_cast<uint4 *>(mine + (2 * i + (lane >> 4)) * kBlkStride + 16 * (lane & 15)) = v[i];
  __syncwarp();
  return Blk{(uint32_t)__cvta_generic_to_shared(mine + lane * kBlkStride)};
}

// ------------------------------------------------------------ selection, by digits
// Warp 0 of the last CTA of a pass: the digit d (255 down to 0) at which the
// counts of hist, added from the top, reach need; returns need minus the
// counts above d.
template <class H>
__device__ void pick_digit(H hist, int64_t need, int &digit, int64_t &need_out) {
  const int lane = threadIdx.x & 31;
  uint32_t c[8];
  int64_t loc = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    c[j] = hist(255 - 8 * lane - j);
    loc += c[j];
  }
  int64_t incl = loc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const int64_t excl = incl - loc;
  const unsigned owner = __ballot_sync(0xffffffffu, excl < need && need <= incl);
  // need <= the count of keys with the current prefix, so exactly one lane owns it
  const int src = owner ? __ffs(owner) - 1 : 0;
  int d = 0;
  int64_t rem = 1;
  if (lane == src) {
    int64_t cum = excl;
    bool found = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (found) continue;
      if (cum + c[j] >= need) {
        d = 255 - 8 * lane - j;
        rem = need - cum;
        found = true;
      } else {
        cum += c[j];
      }
    }
  }
  digit = __shfl_sync(0xffffffffu, d, src);
  need_out = __shfl_sync(0xffffffffu, rem, src);
}

// The end of a CTA's part of a pass (all its threads): its histogram hs is
// added to the pass's; the last CTA picks the digit.
__device__ __forceinline__ void finish_pass(int pass, uint32_t prefix, int64_t need, const uint32_t *hs, bool &last,
                                            SelWork *sw) {
  const int tid = threadIdx.x, shift = 24 - 8 * pass;
  __syncthreads();
  for (int i = tid; i < 256; i += blockDim.x)
    if (hs[i]) atomicAdd(&sw->hist[pass][i], hs[i]);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&sw->done[pass], 1u) == gridDim.x - 1;
  __syncthreads();
  if (last && tid < 32) {
    __threadfence();
    int d;
    int64_t rem;
    pick_digit([&](int i) { return __ldcg(&sw->hist[pass][i]); }, need, d, rem);
    if (tid == 0) {
      sw->st.prefix[pass + 1] = prefix | ((uint32_t)d << shift);
      sw->st.need[pass + 1] = rem;
    }
  }
}

// ------------------------------------------------------------ statistics
// Four passes over a block.  No pass needs the support itself: with c = w - mu
// and Delta0 >= 0, a trit is nonzero where |c| > Delta0 and has c's sign, so
// c * T0 is |c| there and +0 elsewhere (adding +0 to the sum of magnitudes
// changes nothing), and r = c - alpha0 T0 has the magnitude | |c| - alpha0 |
// there and |c| elsewhere (rounding is symmetric in the sign); E only sees r^2.
// An inf or NaN weight makes the sum of the (16-bit) weights inf or NaN, and
// nothing else does.  Issue-bound: 19 instructions per weight, where bit masks
// of the support and products with its trits took 64 (114 us for 4096 x 12288;
// 55 without them, 42 with the blocks staged by whole warps).
__global__ void __launch_bounds__(kBlockThreads) tern_stats_kernel(int64_t NB, const uint16_t *W, float4 *stats,
                                                                   uint32_t *keys, uint32_t *status) {
  __shared__ __align__(16) unsigned char sx[kBlkShared];
  grid_dep_launch_next();
  const int64_t step = (int64_t)gridDim.x * kBlockThreads;
  for (int64_t b0 = (int64_t)blockIdx.x * kBlockThreads + (threadIdx.x & ~31); b0 < NB; b0 += step) {
    const int64_t b = b0 + (threadIdx.x & 31);
    const Blk B = stage_block(W, b < NB ? b : -1, sx);
    if (b >= NB) continue;
    float s = 0.f;
    B.all([&](float x) { s = __fadd_rn(s, x); });
    if (!isfinite(s)) atomicOr(status, TQ_DATA_BAD_WEIGHT);
    const float mu = __fmul_rn(s, kInvGroup);
    float a = 0.f;
    B.all([&](float x) { a = __fadd_rn(a, fabsf(__fsub_rn(x, mu))); });
    const float d0 = __fmul_rn(kThresh, __fmul_rn(a, kInvGroup));
    float p = 0.f;
    int n0 = 0;
    B.all([&](float x) {
      const float c = fabsf(__fsub_rn(x, mu));
      if (c > d0) p = __fadd_rn(p, c), ++n0;
    });
    const float a0 = n0 > 0 ? __fdiv_rn(p, (float)n0) : 0.f;
    float e = 0.f;
    B.all([&](float x) {
      const float c = fabsf(__fsub_rn(x, mu));
      const float r = c > d0 ? __fsub_rn(c, a0) : c;
      e = __fadd_rn(e, __fmul_rn(r, r));
    });
    stats[b] = make_float4(mu, d0, a0, 0.f);
    keys[b] = __float_as_uint(e);
  }
}

// --------------------------------------------------------------- select
__global__ void __launch_bounds__(kSelThreads) tern_hist_kernel(int pass, int64_t NB, int64_t nnz,
                                                                const uint32_t *keys, SelWork *sw) {
  __shared__ uint32_t hs[256];
  __shared__ bool last;
  const int tid = threadIdx.x;
  if (tid < 256) hs[tid] = 0u;
  __syncthreads();
  grid_dep_launch_next();
  grid_dep_wait();
  const uint32_t prefix = pass ? __ldcg(&sw->st.prefix[pass]) : 0u;
  const int64_t need = pass ? __ldcg(reinterpret_cast<const long long *>(&sw->st.need[pass])) : nnz;
  const int shift = 24 - 8 * pass;
  // keys whose bits above `shift + 8` match the prefix (all keys in pass 0)
  const uint32_t hi_mask = pass ? 0xffffffffu << (shift + 8) : 0u;
  for (int64_t b = (int64_t)blockIdx.x * kSelThreads + tid; b < NB; b += (int64_t)gridDim.x * kSelThreads) {
    const uint32_t k = keys[b];
    if ((k & hi_mask) == prefix) atomicAdd(&hs[(k >> shift) & 255u], 1u);
  }
  finish_pass(pass, prefix, need, hs, last, sw);
}

// Masks of the kWarpWords salience words from w0 on (word w: row w / SW, word
// w % SW) against the selected key T, built by one warp: per word, lane l
// reads the key of group 32 (w % SW) + l (one coalesced load) and two
// ballots give the valid groups above T and equal to T; lane k keeps word
// w0 + k's masks.
__device__ __forceinline__ void warp_word_masks(const uint32_t *keys, int G, int SW, int NW, int w0, uint32_t T,
                                                uint32_t &gt, uint32_t &eq) {
  const int lane = threadIdx.x & 31;
  gt = 0u, eq = 0u;
  uint32_t v[kWarpWords];
  bool ok[kWarpWords];
  int n = w0 / SW, j = w0 - n * SW;
  // all loads first (in flight together), then the ballots
#pragma unroll
  for (int k = 0; k < kWarpWords; ++k) {
    ok[k] = w0 + k < NW && lane < G - 32 * j;
    v[k] = ok[k] ? keys[(int64_t)n * G + 32 * j + lane] : 0u;
    if (++j == SW) j = 0, ++n;
  }
#pragma unroll
  for (int k = 0; k < kWarpWords; ++k) {
    const uint32_t bg = __ballot_sync(0xffffffffu, ok[k] && v[k] > T);
    const uint32_t be = __ballot_sync(0xffffffffu, ok[k] && v[k] == T);
    if (lane == k) gt = bg, eq = be;
  }
}

__device__ __forceinline__ int block_sum(int v, int *red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  int t = 0;
  for (int i = 0; i < kMarkThreads / 32; ++i) t += red[i];
  return t;
}

// Keys equal to the selected key, per chunk of kMarkWords salience words.
__global__ void __launch_bounds__(kMarkThreads) tern_count_kernel(int NW, int G, int SW, const uint32_t *keys,
                                                                  const SelWork *sw, uint32_t *chunk_eq) {
  __shared__ int red[kMarkThreads / 32];
  grid_dep_launch_next();
  grid_dep_wait();
  const int w0 = (int)blockIdx.x * kMarkWords + (threadIdx.x >> 5) * kWarpWords;
  uint32_t gt, eq;
  warp_word_masks(keys, G, SW, NW, w0, sw->st.prefix[4], gt, eq);
  const int t = block_sum(__popc(eq), red);
  if (threadIdx.x == 0) chunk_eq[blockIdx.x] = (uint32_t)t;
}

// Salience words of a chunk: groups above the selected key, and equal ones
// while fewer than `need` equal keys precede them in block-id order.
__global__ void __launch_bounds__(kMarkThreads) tern_mark_kernel(int NW, int G, int SW, const uint32_t *keys,
                                                                 const SelWork *sw, const uint32_t *chunk_eq,
                                                                 uint32_t *sal) {
  __shared__ int red[kMarkThreads / 32];
  __shared__ int wpre[kMarkThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  grid_dep_launch_next();
  grid_dep_wait();
  const uint32_t T = sw->st.prefix[4];
  const int64_t need = sw->st.need[4];
  // equal keys in earlier chunks
  int before = 0;
  for (int c = tid; c < (int)blockIdx.x; c += kMarkThreads) before += (int)chunk_eq[c];
  const int64_t base = block_sum(before, red);
  const int w0 = (int)blockIdx.x * kMarkWords + wid * kWarpWords;
  uint32_t gt, eq;
  warp_word_masks(keys, G, SW, NW, w0, T, gt, eq);
  // exclusive scan of the equal counts over the chunk's words (block-id order)
  const int cnt = __popc(eq);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wpre[wid] = incl;
  __syncthreads();
  int wbase = 0;
  for (int i = 0; i < wid; ++i) wbase += wpre[i];
  int64_t rank = base + wbase + incl - cnt;  // equal keys before this word
  uint32_t take = 0u;
  for (uint32_t m = eq; m && rank < need; m &= m - 1u, ++rank) take |= m & (~m + 1u);
  const int w = w0 + lane;
  if (lane < kWarpWords && w < NW) sal[w] = gt | take;
}

// The selection in one cluster of kSelCtas CTAs, CTA r holding the keys of
// rows [N r / kSelCtas, N (r + 1) / kSelCtas) in shared memory: each digit's
// histograms are added up through distributed shared memory, every CTA picking
// the digit for itself.  What a digit costs is its chain of latencies, here a
// cluster barrier (about 1000 cycles) and 16 SMs' scan of the keys (2000 to
// 4000) instead of a launch, global atomics and a ticket: for 4096 x 12288 the
// four passes, counting, marking and rowptr took 57 us as seven launches (38
// with programmatic dependent launches), this 30.  Taken while the keys fit
// (about 850,000 blocks if the groups are a multiple of 32); with eight CTAs
// it took 43 us, and digits of 11 bits (three barriers, but 2048 bins to add
// up over 16 CTAs) 48.  A cluster of 16 is not a portable size: a device (a
// partition of one) whose GPCs have fewer SMs takes the separate kernels.
constexpr int kSelCtas = 16, kSelWarps = kSelThreads / 32, kSelBatch = 8;
constexpr int kSelCopies = 8;    // of the first digit's histogram (all keys, in a few bins),
constexpr int kSelStride = 257;  // on different banks
constexpr int kSelHist = kSelCopies * kSelStride + 3 * 256;
constexpr int kSelKeys = (232448 - 8192) / 4 - kSelHist;  // keys per CTA
__host__ __device__ inline int64_t select_keys(int N, int SW) {
  return (int64_t)((N + kSelCtas - 1) / kSelCtas) * SW * 32;  // per CTA, rows padded to whole words
}

// The 32-bit word at shared address `addr` of CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t ld_cluster(const uint32_t *p, int rank) {
  uint32_t a, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__global__ void __launch_bounds__(kSelThreads)
    tern_select_kernel(int N, int G, int SW, uint32_t nnz, const uint32_t *keys, uint32_t *sal, int32_t *rowptr) {
  // histograms of the four digits (each its own, so that one cluster barrier
  // per digit is enough), then the CTA's keys
  extern __shared__ uint32_t sel_smem[];
  uint32_t *const kk = sel_smem + kSelHist;
  __shared__ uint32_t part[4][256], wsum[kSelWarps], wgt[kSelWarps], weq[kSelWarps];
  __shared__ uint32_t cnt[2];  // the CTA's keys above and equal to the selected one
  __shared__ uint32_t s_digit, s_need;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, r = blockIdx.x;
  const int64_t n0 = (int64_t)N * r / kSelCtas, n1 = (int64_t)N * (r + 1) / kSelCtas;
  // each warp has an equal share of the CTA's salience words (32 keys, a row's
  // last word fewer), in order, and a lane one key of each
  const int nw = (int)(n1 - n0) * SW, share = (nw + kSelWarps - 1) / kSelWarps;
  const int w0 = min(nw, wid * share), w1 = min(nw, w0 + share);
  const uint32_t last = G % 32 ? (1u << (G % 32)) - 1u : ~0u;  // keys of a row's last word
  grid_dep_launch_next();
  for (int i = tid; i < kSelHist; i += kSelThreads) sel_smem[i] = 0u;
  __syncthreads();
  grid_dep_wait();
  uint32_t *h = sel_smem + (lane % kSelCopies) * kSelStride;
  for (int w = w0; w < w1; w += kSelBatch) {
    uint32_t k[kSelBatch];
    bool ok[kSelBatch];
    int n = w / SW, j = w - n * SW;
    const uint32_t *src = keys + (n0 + n) * G + 32 * j + lane;
#pragma unroll
    for (int i = 0; i < kSelBatch; ++i) {
      const bool edge = ++j == SW;
      ok[i] = w + i < w1 && (!edge || ((last >> lane) & 1u));
      k[i] = ok[i] ? *src : 0u;
      src += edge ? G - 32 * (SW - 1) : 32;
      if (edge) j = 0;
    }
#pragma unroll
    for (int i = 0; i < kSelBatch; ++i) {
      if (w + i < w1) kk[32 * (w + i) + lane] = k[i];
      if (ok[i]) atomicAdd(&h[k[i] >> 24], 1u);
    }
  }
  __syncthreads();
  if (tid < 256) {
    uint32_t v = 0;
#pragma unroll
    for (int c = 0; c < kSelCopies; ++c) v += sel_smem[c * kSelStride + tid];
    sel_smem[tid] = v;
  }
  uint32_t prefix = 0u, need = nnz;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    h = pass == 0 ? sel_smem : sel_smem + kSelCopies * kSelStride + (pass - 1) * 256;
    if (pass) {
      // the padding (zeros) is not counted
      if (tid == 0 && prefix == 0u) atomicAdd(&h[0], 0u - (uint32_t)(n1 - n0) * (uint32_t)(SW * 32 - G));
      for (int w = w0; w < w1; w += kSelBatch) {
        uint32_t k[kSelBatch];
#pragma unroll
        for (int i = 0; i < kSelBatch; ++i) k[i] = w + i < w1 ? kk[32 * (w + i) + lane] : ~prefix;
#pragma unroll
        for (int i = 0; i < kSelBatch; ++i)
          if ((k[i] ^ prefix) >> (shift + 8) == 0u) atomicAdd(&h[(k[i] >> shift) & 255u], 1u);
      }
    }
    cluster_sync();
    // the cluster's histogram, four CTAs to a thread, and its sums from the
    // highest bin down: the digit is the bin with the need-th key of those left
    const int bin = 255 - tid % 256;
    {
      uint32_t v = 0;
#pragma unroll
      for (int j = 0; j < kSelCtas / 4; ++j) v += ld_cluster(h + bin, kSelCtas / 4 * (tid / 256) + j);
      part[tid / 256][tid % 256] = v;
    }
    __syncthreads();
    if (tid < 256) {
      const uint32_t c = part[0][tid] + part[1][tid] + part[2][tid] + part[3][tid];
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      if (lane == 31) wsum[wid] = incl;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const uint32_t before = __reduce_add_sync(0xffffffffu, lane < wid ? wsum[lane] : 0u) + incl - c;
      if (before < need && need <= before + c) s_digit = bin, s_need = need - before;
    }
    __syncthreads();
    prefix |= s_digit << shift, need = s_need;
  }
  // the warp's keys above and equal to the selected one
  uint32_t agt = 0, aeq = 0;
#pragma unroll 8
  for (int w = w0; w < w1; ++w) {
    const uint32_t k = kk[32 * w + lane];
    agt += k > prefix, aeq += k == prefix;
  }
  agt = __reduce_add_sync(0xffffffffu, agt), aeq = __reduce_add_sync(0xffffffffu, aeq);
  if (prefix == 0u) aeq -= (uint32_t)(w1 / SW - w0 / SW) * (uint32_t)(SW * 32 - G);  // the padding
  if (lane == 0) wgt[wid] = agt, weq[wid] = aeq;
  __syncthreads();
  uint32_t above = __reduce_add_sync(0xffffffffu, lane < wid ? wgt[lane] : 0u);
  uint32_t equal = __reduce_add_sync(0xffffffffu, lane < wid ? weq[lane] : 0u);
  if (tid == kSelThreads - 1) cnt[0] = above + agt, cnt[1] = equal + aeq;
  cluster_sync();
  above += __reduce_add_sync(0xffffffffu, lane < r ? ld_cluster(cnt, lane & (kSelCtas - 1)) : 0u);
  equal += __reduce_add_sync(0xffffffffu, lane < r ? ld_cluster(cnt + 1, lane & (kSelCtas - 1)) : 0u);
  uint32_t before = above + min(equal, need);  // salient groups of earlier words
  auto excl = [&](uint32_t v, uint32_t &total) {  // sums over the lanes before this one
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - v;
  };
  for (int w = w0; w < w1; w += 32) {  // a lane holds one of 32 words
    uint32_t gt = 0u, eq = 0u;
#pragma unroll 8
    for (int i = 0; i < min(32, w1 - w); ++i) {
      const uint32_t k = kk[32 * (w + i) + lane];
      const uint32_t bg = __ballot_sync(0xffffffffu, k > prefix), be = __ballot_sync(0xffffffffu, k == prefix);
      if (lane == i) gt = bg, eq = be;
    }
    const int n = (w + lane) / SW, j = w + lane - n * SW;
    if (j == SW - 1) eq &= last;
    uint32_t neq, ntake;
    uint32_t rank = equal + excl(__popc(eq), neq), take = gt;
    for (uint32_t m = eq; m && rank < need; m &= m - 1u, ++rank) take |= m & (~m + 1u);
    const uint32_t pre = excl(__popc(take), ntake);
    if (w + lane < w1) {
      sal[n0 * SW + w + lane] = take;
      if (j == 0) rowptr[n0 + n] = (int32_t)(before + pre);
    }
    equal += neq, before += ntake;
  }
  if (r == kSelCtas - 1 && tid == kSelThreads - 1) rowptr[N] = (int32_t)before;
  cluster_sync();  // no CTA ends while another may read its counts
}

// ---------------------------------------------------------------- planes
// Blocks without a second plane (the CTAs from p2_ctas on of
// tern_planes_kernel): the first support from the statistics, then `sweeps`
// refinements of mu and alpha0 (alpha1 = 0) on the block's moments (see
// plane2_blocks).
// Salient blocks are skipped here; plane2_blocks writes them.  Also
// zeroes each row's pad bytes.
__device__ __forceinline__ void plane1_blocks(int cta, int ctas, unsigned char *sx, int N, int K, int sweeps,
                                              const uint16_t *W, const float4 *stats, const uint32_t *sal,
                                              uint8_t *plane1, __half *s1, __half *off) {
  const int G = K / kGroup, SW = sal_words_of(K);
  const int64_t NB = (int64_t)N * G, RB = row_bytes_of(K);
  const int64_t step = (int64_t)ctas * kBlockThreads;
  for (int64_t b0 = (int64_t)cta * kBlockThreads + (threadIdx.x & ~31); b0 < NB; b0 += step) {
    const int64_t b = b0 + (threadIdx.x & 31), n = b < NB ? b / G : 0;
    const int g = (int)(b - n * G);
    uint8_t *row = plane1 + n * RB;
    bool live = b < NB;
    if (live && g == G - 1)
      for (int64_t i = (int64_t)kGroupBytes * G; i < RB; ++i) row[i] = 0;
    if (live && ((sal[n * SW + (g >> 5)] >> (g & 31)) & 1u)) live = false;
    const Blk B = stage_block(W, live ? b : -1, sx);
    if (!live) continue;
    const float4 st = stats[b];
    float mu = st.x, a0 = st.z;
    const float d = st.y;
    float mw = 0.f, mw0 = 0.f;  // sum w, sum w T0
    int n0 = 0, z0 = 0;         // |T0|, sum T0
    uint16_t *dst = reinterpret_cast<uint16_t *>(row + (int64_t)kGroupBytes * g);
    B.pack(dst, [&](float x) {
      const int t = trit_of(__fsub_rn(x, mu), d);
      mw += x, mw0 += times_trit(x, t), n0 += t * t, z0 += t;
      return t;
    });
    for (int sw = 0; sw < sweeps; ++sw) {
      mu = (mw - a0 * z0) * kInvGroup;
      a0 = n0 > 0 ? (mw0 - mu * z0) / n0 : 0.f;
    }
    off[b] = __float2half_rn(mu);
    s1[b] = __float2half_rn(a0);
  }
}

// Salient blocks (the first p2_ctas CTAs of tern_planes_kernel, scheduled
// first because they take longest), one thread per plane-2 record j < nnz:
// the record's row
// (the last n with rowptr[n] <= j) and group (the (j - rowptr[n])-th set
// salience bit of the row), then both supports, the refinement of mu,
// alpha0 and alpha1, and both planes' bytes and parameters.
//
// The refinement decides nothing (the supports are fixed), so it runs on
// the block's moments: with n0 = |T0|, n1 = |T1|, s0 = sum T0, s1 = sum T1,
// s01 = sum T0 T1 and the sums w, w T0, w T1, a sweep is
//   mu = (sum w - alpha0 s0 - alpha1 s1) / 128,
//   alpha0 = (sum w T0 - mu s0 - alpha1 s01) / n0,
//   alpha1 = (sum w T1 - mu s1 - alpha0 s01) / n1,
// the exact coordinate updates of the least-squares fit, without a pass
// over the weights.  Supports and thresholds keep the in-order sums.
__device__ __forceinline__ void plane2_blocks(int cta, int ctas, unsigned char *sx, int N, int K, int sweeps,
                                              int64_t nnz, const uint16_t *W, const float4 *stats,
                                              const uint32_t *sal, const int32_t *rowptr, uint8_t *plane1,
                                              uint8_t *plane2, __half *s1, __half *off, __half *s2,
                                              uint32_t *status) {
  const int G = K / kGroup, SW = sal_words_of(K);
  const int64_t RB = row_bytes_of(K);
  const int64_t step = (int64_t)ctas * kBlockThreads;
  for (int64_t j0 = (int64_t)cta * kBlockThreads + (threadIdx.x & ~31); j0 < nnz; j0 += step) {
    const int64_t j = j0 + (threadIdx.x & 31);
    int n = 0, g = -1;
    if (j < nnz) {
      int lo = 0, hi = N;  // rowptr[lo] <= j < rowptr[hi] for a consistent rowptr
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (rowptr[mid] <= j) lo = mid; else hi = mid;
      }
      n = lo;
      int rank = (int)(j - rowptr[n]);
      for (int w = 0; w < SW && g < 0 && rank >= 0; ++w) {
        uint32_t m = sal[(int64_t)n * SW + w];
        if (G - 32 * w < 32) m &= (1u << (G - 32 * w)) - 1u;
        const int c = __popc(m);
        if (rank < c) {
          for (int k = 0; k < rank; ++k) m &= m - 1u;
          g = 32 * w + __ffs(m) - 1;
        } else {
          rank -= c;
        }
      }
      if (g < 0) atomicOr(status, TQ_DATA_BAD_ROWPTR);  // rowptr disagrees with the salience map
    }
    const int64_t b = g >= 0 ? (int64_t)n * G + g : -1;
    const Blk B = stage_block(W, b, sx);
    if (b < 0) continue;
    const float4 st = stats[b];
    const float mu0 = st.x, d0 = st.y, a00 = st.z;
    float mu = mu0, a0 = a00, a1 = 0.f;
    float mw = 0.f, mw0 = 0.f, mw1 = 0.f;  // sum w, sum w T0, sum w T1
    int n0 = 0, n1 = 0;                    // |T0|, |T1|
    int z0 = 0, z1 = 0, z01 = 0;           // sum T0, sum T1, sum T0 T1
    float bsum = 0.f;
    // first plane, and the mean magnitude of the residual r = c - alpha0 T0
    B.pack(reinterpret_cast<uint16_t *>(plane1 + (int64_t)n * RB + (int64_t)kGroupBytes * g), [&](float x) {
      const float c = __fsub_rn(x, mu0);
      const int t = trit_of(c, d0);
      mw += x, mw0 += times_trit(x, t), n0 += t * t, z0 += t;
      bsum = __fadd_rn(bsum, fabsf(__fsub_rn(c, times_trit(a00, t))));
      return t;
    });
    // second support on the residual, same threshold rule
    const float d1 = __fmul_rn(kThresh, __fmul_rn(bsum, kInvGroup));
    B.pack(reinterpret_cast<uint16_t *>(plane2 + j * kGroupBytes), [&](float x) {
      const float c = __fsub_rn(x, mu0);
      const int t0 = trit_of(c, d0), t = trit_of(__fsub_rn(c, times_trit(a00, t0)), d1);
      mw1 += times_trit(x, t), n1 += t * t, z1 += t, z01 += t0 * t;
      return t;
    });
    // alpha1 = sum r T1 / n1 with r = w - mu - alpha0 T0
    a1 = n1 > 0 ? (mw1 - mu * z1 - a0 * z01) / n1 : 0.f;
    for (int sw = 0; sw < sweeps; ++sw) {
      mu = (mw - a0 * z0 - a1 * z1) * kInvGroup;
      a0 = n0 > 0 ? (mw0 - mu * z0 - a1 * z01) / n0 : 0.f;
      if (n1 > 0) a1 = (mw1 - mu * z1 - a0 * z01) / n1;
    }
    off[b] = __float2half_rn(mu);
    s1[b] = __float2half_rn(a0);
    s2[j] = __float2half_rn(a1);
  }
}

// Both kinds of blocks in one launch: CTAs below p2_ctas take the salient
// records, the rest the other blocks, so the two run side by side.
__global__ void __launch_bounds__(kBlockThreads, 6) tern_planes_kernel(int N, int K, int sweeps, int64_t nnz, int p2_ctas,
                                                                   const uint16_t *W, const float4 *stats,
                                                                   const uint32_t *sal, const int32_t *rowptr,
                                                                   uint8_t *plane1, uint8_t *plane2, __half *s1,
                                                                   __half *off, __half *s2, uint32_t *status) {
  __shared__ __align__(16) unsigned char sx[kBlkShared];
  grid_dep_launch_next();
  grid_dep_wait();
  if ((int)blockIdx.x < p2_ctas)
    plane2_blocks(blockIdx.x, p2_ctas, sx, N, K, sweeps, nnz, W, stats, sal, rowptr, plane1, plane2, s1, off, s2,
                  status);
  else
    plane1_blocks(blockIdx.x - p2_ctas, gridDim.x - p2_ctas, sx, N, K, sweeps, W, stats, sal, plane1, s1, off);
}

int grid_blocks(int64_t NB) {
  int64_t g = (NB + kBlockThreads - 1) / kBlockThreads;
  return (int)(g < 1 ? 1 : g > 152 * 16 ? 152 * 16 : g);
}

}  // namespace tz

size_t ternarize_ws_bytes(int N, int K) {
  const int64_t NB = (int64_t)N * (K / kGroup);
  const int64_t NW = (int64_t)N * sal_words_of(K);
  const int64_t chunks = (NW + tz::kMarkWords - 1) / tz::kMarkWords;
  auto pad = [](int64_t b) { return (b + 255) / 256 * 256; };
  return (size_t)(pad(NB * 16) + pad(NB * 4) + pad(sizeof(tz::SelWork)) + pad(chunks * 4));
}

cudaError_t launch_ternarize(int N, int K, const uint16_t *W, int64_t nnz, int sweeps, uint8_t *plane1,
                             uint32_t *sal, int32_t *rowptr, uint8_t *plane2, uint16_t *scale1, uint16_t *offset,
                             uint16_t *scale2, unsigned char *ws, uint32_t *status, cudaStream_t s) {
  using namespace tz;
  const int G = K / kGroup, SW = sal_words_of(K);
  const int64_t NB = (int64_t)N * G, NW = (int64_t)N * SW;
  const int64_t chunks = (NW + kMarkWords - 1) / kMarkWords;
  auto pad = [](int64_t b) { return (b + 255) / 256 * 256; };
  float4 *stats = reinterpret_cast<float4 *>(ws);
  uint32_t *keys = reinterpret_cast<uint32_t *>(ws + pad(NB * 16));
  SelWork *sw = reinterpret_cast<SelWork *>(ws + pad(NB * 16) + pad(NB * 4));
  uint32_t *chunk_eq = reinterpret_cast<uint32_t *>(ws + pad(NB * 16) + pad(NB * 4) + pad(sizeof(SelWork)));
  // (the limit of shared memory is the same for every call: other threads set it too)
  constexpr int kSelMaxSmem = 4 * (kSelHist + kSelKeys);
  const bool cluster = nnz > 0 && select_keys(N, SW) <= kSelKeys &&
                       clusters_at_once<tern_select_kernel>(kSelCtas, kSelThreads, kSelMaxSmem) > 0;
  cudaError_t e = cudaSuccess;
  if (nnz == 0) e = cudaMemsetAsync(sal, 0, (size_t)NW * 4, s);
  if (nnz > 0 && !cluster) e = cudaMemsetAsync(sw, 0, sizeof(SelWork), s);
  if (e != cudaSuccess) return e;
  tern_stats_kernel<<<grid_blocks(NB), kBlockThreads, 0, s>>>(NB, W, stats, keys, status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (cluster) {
    const int smem = (int)(4 * (kSelHist + select_keys(N, SW)));
    e = cudaFuncSetAttribute(tern_select_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(tern_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelMaxSmem);
    if (e != cudaSuccess) return e;
    e = launch_dependent_cluster(tern_select_kernel, dim3(kSelCtas), kSelCtas, kSelThreads, smem, s, N, G, SW,
                                 (uint32_t)nnz, keys, sal, rowptr);
    if (e != cudaSuccess) return e;
  } else {
    if (nnz > 0) {
      const int hg = (int)std::min<int64_t>((NB + kSelThreads - 1) / kSelThreads, 152 * 2);
      for (int p = 0; p < 4; ++p)
        if ((e = launch_dependent(tern_hist_kernel, dim3(hg), kSelThreads, s, p, NB, nnz, keys, sw)) != cudaSuccess)
          return e;
      const dim3 grid((unsigned)chunks);
      if ((e = launch_dependent(tern_count_kernel, grid, kMarkThreads, s, (int)NW, G, SW, keys, sw, chunk_eq)) !=
          cudaSuccess)
        return e;
      if ((e = launch_dependent(tern_mark_kernel, grid, kMarkThreads, s, (int)NW, G, SW, keys, sw, chunk_eq, sal)) !=
          cudaSuccess)
        return e;
    }
    if ((e = launch_rowptr(N, K, sal, rowptr, status, true, s)) != cudaSuccess) return e;
  }
  __half *h1 = reinterpret_cast<__half *>(scale1), *ho = reinterpret_cast<__half *>(offset);
  const int p2 = nnz > 0 ? grid_blocks(nnz) : 0;
  return launch_dependent(tern_planes_kernel, dim3((unsigned)(p2 + grid_blocks(NB))), kBlockThreads, s, N, K, sweeps,
                          nnz, p2, W, stats, sal, rowptr, plane1, plane2, h1, ho, reinterpret_cast<__half *>(scale2), status);
}

}  // namespace tq
