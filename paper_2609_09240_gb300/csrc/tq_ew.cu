// tq_ew.cu - the linear layer of the element-wise four-mask representation
// (paper "Model and Representation": four disjoint salience masks with
// orders [2, 2, 1, 1], W-hat = (mu + alpha0 T0 + alpha1 T1) (.) M, one mu /
// alpha0 per row and mask, alpha1 for the two order-2 masks).
//
// With mask 3 the largest (86.5 % of a recorded projection), the layer is
//   y[m][n] = mu3 S[m] + alpha0_3 P0[m][n]
//           + sum over the elements k of the row's other masks q of
//             x[m][k] ((mu_q - mu3) + (alpha0_q - alpha0_3) T0[n,k] + alpha1_q T1[n,k]),
// S = sum_k x, P0 = sum_k T0 x.  The first line is the group format's
// linear over plane 1 with s1 = alpha0_3 and off = mu3 in every group and no
// second plane: the library's decode or prefill path runs it, through
// per-call views of s1 / off in the workspace (views_kernel), into an fp32
// buffer.  correct_kernel then adds the second line and writes y.
#include <algorithm>
#include <type_traits>

#include "tq_common.cuh"
#include "tq_ew_pairs.cuh"
#include "tq_launch.cuh"
#include "tq_sm100.cuh"

namespace tq {
namespace ew {

constexpr int kWarps = 8;  // warps per block of correct_kernel

// One problem of a batched call, as the views kernel sees it ...
struct ViewProb {
  const __half *mu, *a0;  // [N][4]
  __half *s1v, *offv;     // views [N][G]
  uint32_t *salv;         // [N][sal_words] (zero)
  int32_t *rpv;           // [N+1] (zero)
  int32_t N, K;
};
// ... and as correct_kernel sees it: its weight, x, the fp32 plane-1
// result and y; S warps per row and the kernel's blocks for it.
struct Prob {
  const uint32_t *mask;     // [N][K/16]
  const uint8_t *plane1;    // [N][row_bytes]
  const int32_t *p2rowptr;  // [N+1]
  const uint8_t *plane2;
  const __half *mu, *a0, *a1;  // [N][4], [N][4], [N][2]
  const int32_t *idx_off;      // correction index (or null): offsets [N nb + 1]
  const uint16_t *idx;         //   and entries
  const __half *x;             // [M][K]
  float *ydense;               // [M][N]
  void *y;                     // [M][N], fp16 or fp32
  int32_t N, K, S, blocks;     // blocks = 0: the problem is the other kernel's
  int64_t w_begin;             // N G of the index kernel's problems before it
};
template <typename T, int CAP = TQ_MAX_BATCH>
struct Batch {
  int32_t count;
  T prob[CAP];
};
static_assert(sizeof(Batch<Prob>) <= 32764 && sizeof(Batch<ViewProb>) <= 32764, "launch parameters");

// fn with the smallest launch parameters that hold bt (31 KB of them cost
// 1 us more per launch than those of eight problems).
template <typename T, class Fn>
cudaError_t with_batch(const Batch<T> &bt, Fn fn) {
  if (bt.count > kFewProblems) return fn(bt);
  Batch<T, kFewProblems> few;
  few.count = bt.count;
  std::copy(bt.prob, bt.prob + bt.count, few.prob);
  return fn(few);
}

constexpr int kViewThreads = 256, kViewUnits = 2;  // views_kernel: 16-byte units of each view per thread

// Block row blockIdx.y = problem: s1 view = alpha0 of mask 3, off view =
// mu of mask 3 in every group of the row, eight groups per 16-byte store
// wherever the rows begin; the views' salience words and rowptr are zero (no
// second plane).  A small kernel between two launches: it starts while the
// stream's previous kernel ends, and the prep kernel while it runs.
template <class BT>
__global__ void __launch_bounds__(kViewThreads) views_kernel(const __grid_constant__ BT bt) {
  grid_dep_launch_next();
  grid_dep_wait();  // the last call's kernels may read these views
  const ViewProb &P = bt.prob[blockIdx.y];
  const int N = P.N, G = P.K / kGroup, W = sal_words_of(P.K);
  const int i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  const unsigned short *mu = reinterpret_cast<const unsigned short *>(P.mu);
  const unsigned short *a0 = reinterpret_cast<const unsigned short *>(P.a0);
  const int total = N * G, units = (total + 7) / 8;
  for (int i = i0; i < units; i += step) {
    int n = 8 * i / G, g = 8 * i - n * G;
    uint32_t a = __ldg(a0 + (int64_t)n * 4 + 3), m = __ldg(mu + (int64_t)n * 4 + 3);
    uint32_t av[4], mv[4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j > 0 && ++g == G) {
        g = 0;
        if (++n < N) a = __ldg(a0 + (int64_t)n * 4 + 3), m = __ldg(mu + (int64_t)n * 4 + 3);
      }
      av[j / 2] = j & 1 ? av[j / 2] | a << 16 : a;
      mv[j / 2] = j & 1 ? mv[j / 2] | m << 16 : m;
    }
    if (8 * i + 8 <= total) {
      reinterpret_cast<uint4 *>(P.s1v)[i] = make_uint4(av[0], av[1], av[2], av[3]);
      reinterpret_cast<uint4 *>(P.offv)[i] = make_uint4(mv[0], mv[1], mv[2], mv[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (8 * i + j < total) {
          P.s1v[8 * i + j] = __ushort_as_half((unsigned short)(av[j / 2] >> (16 * (j & 1))));
          P.offv[8 * i + j] = __ushort_as_half((unsigned short)(mv[j / 2] >> (16 * (j & 1))));
        }
    }
  }
  for (int i = i0; i < N * W; i += step) P.salv[i] = 0u;
  for (int i = i0; i <= N; i += step) P.rpv[i] = 0;
}

// The five base-3 digits of a byte (values above 242 read as 242), two bits
// each, first digit in bits 0..1.
__device__ __forceinline__ uint32_t digit_code(int v) {
  v = v > 242 ? 242 : v;
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    c |= (uint32_t)(v % 3) << (2 * i);
    v /= 3;
  }
  return c;
}

__device__ __forceinline__ float ldx(const __half *p) {
  return __half2float(__ushort_as_half(__ldg(reinterpret_cast<const unsigned short *>(p))));
}

// Four 2-bit fields (bits 0..15 hold eight) spread to 4-bit spacing: field
// j of x at bits 2j..2j+1 -> bits 4j..4j+1.
__device__ __forceinline__ uint32_t spread2(uint32_t x) {
  x &= 0xffffu;
  x = (x | (x << 8)) & 0x00ff00ffu;
  x = (x | (x << 4)) & 0x0f0f0f0fu;
  x = (x | (x << 2)) & 0x33333333u;
  return x;
}

// Adds the elements of masks 0..2 to the dense fp32 result of tokens
// [m0, m0 + mt) (mt <= MT) and writes y.  S warps share a row, warp s taking
// a contiguous range of the row's 512-element chunks.
//
// Per chunk a lane owns one mask word (16 elements) and its 16 activations
// per token.  The chunk's plane-1 bytes (four groups of 26) are read as
// 32-bit words by the first lanes and each lane takes the four bytes
// holding its 16 trits by two shuffles and a funnel shift; a shared table
// turns each byte into five two-bit digits, so the word's T0 digits line up
// with its mask fields.  Each element's mask q and digit d0 form a 4-bit
// code (q << 2 | d0); two neighbouring elements' codes form a byte, and the
// row's 256-entry pair table gives both elements' weights
// (mu_q - mu_3) + (alpha0_q - alpha0_3) (d0 - 1) in one 8-byte load (mask-3
// codes give 0), so the sixteen elements cost eight loads and no branch.
// The order-2 elements (masks 0, 1; 3.6 % of a recorded projection) add
// alpha1_q T1 x in a loop over their bits: the T1 trit is plane 2's trit at
// the element's rank among the row's order-2 elements, the warp's exclusive
// scan of the words' order-2 counts plus the count of the row's earlier
// warps (a first pass over the mask words gives each warp its count).
template <bool F32, int MT>
__global__ void __launch_bounds__(32 * kWarps) correct_kernel(const __grid_constant__ Batch<Prob> bt, int m0, int mt) {
  const Prob &w = bt.prob[blockIdx.y];
  if ((int)blockIdx.x >= w.blocks) return;
  const int N = w.N, K = w.K, S = w.S;
  __shared__ uint32_t dig[256];
  __shared__ float2 ptab[kWarps][256];
  __shared__ int cnt[kWarps];
  __shared__ float part[kWarps][MT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < 256; i += blockDim.x) dig[i] = digit_code(i);
  const int r_in = warp / S, seg = warp - r_in * S;
  const int n = blockIdx.x * (kWarps / S) + r_in;
  const bool live = n < N;
  const int WK = K / 16, C = (WK + 31) / 32, G = K / kGroup;
  const int c_lo = (int)((int64_t)seg * C / S), c_hi = (int)((int64_t)(seg + 1) * C / S);
  const int64_t nr = live ? n : 0;
  const uint32_t *mrow = w.mask + nr * WK;
  {
    // code q << 2 | d0 -> weight (zero for mask 3 and the unused d0 = 3)
    float v = 0.f;
    const int q = lane >> 2, d0 = lane & 3;
    if (live && lane < 12 && d0 < 3) {
      const float mu3 = __half2float(w.mu[nr * 4 + 3]), a03 = __half2float(w.a0[nr * 4 + 3]);
      v = (__half2float(w.mu[nr * 4 + q]) - mu3) + (__half2float(w.a0[nr * 4 + q]) - a03) * (float)(d0 - 1);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = lane + 32 * i;
      const float wa = __shfl_sync(0xffffffffu, v, e & 15), wb = __shfl_sync(0xffffffffu, v, e >> 4);
      ptab[warp][e] = make_float2(wa, wb);
    }
  }
  int mine = 0;
  if (live)
    for (int c = c_lo; c < c_hi; ++c) {
      const int wi = c * 32 + lane;
      if (wi < WK) mine += __popc(~__ldg(mrow + wi) & 0xaaaaaaaau);
    }
#pragma unroll
  for (int o = 16; o; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if (lane == 0) cnt[warp] = mine;
  __syncthreads();
  float acc[MT];
#pragma unroll
  for (int t = 0; t < MT; ++t) acc[t] = 0.f;
  if (live) {
    int base = 0;  // order-2 elements of the row before this warp's chunk
    for (int s = 0; s < seg; ++s) base += cnt[r_in * S + s];
    const uint8_t *p1 = w.plane1 + nr * row_bytes_of(K);
    const uint8_t *p2 = w.plane2 + w.p2rowptr[nr];
    const __half *xm = w.x + (int64_t)m0 * K;
    const int e0 = 16 * (lane & 7), s2 = 2 * (e0 % 5);
    const int B = (lane >> 3) * kGroupBytes + e0 / 5;  // first plane-1 byte of the lane's word in its chunk
    const float2 *pt = ptab[warp];
    const float a1_0 = __half2float(w.a1[nr * 2]), a1_1 = __half2float(w.a1[nr * 2 + 1]);
    for (int c = c_lo; c < c_hi; ++c) {
      const int wi = c * 32 + lane;
      const bool in = wi < WK;
      const uint32_t mw = in ? __ldg(mrow + wi) : 0xffffffffu;  // absent words read as all mask 3
      const int nw = (min(4, G - 4 * c) * kGroupBytes + 3) / 4;
      const uint32_t pw = lane < nw ? __ldg(reinterpret_cast<const uint32_t *>(p1 + (int64_t)c * 4 * kGroupBytes) + lane) : 0u;
      const uint32_t lo = __shfl_sync(0xffffffffu, pw, B >> 2), hi = __shfl_sync(0xffffffffu, pw, (B >> 2) + 1);
      uint4 xv[MT][2];
#pragma unroll
      for (int t = 0; t < MT; ++t) {
        const uint4 *xp = reinterpret_cast<const uint4 *>(xm + (int64_t)t * K + wi * 16);
        const bool ok = in && t < mt;
        xv[t][0] = ok ? __ldg(xp) : make_uint4(0u, 0u, 0u, 0u);
        xv[t][1] = ok ? __ldg(xp + 1) : make_uint4(0u, 0u, 0u, 0u);
      }
      const uint32_t o2 = ~mw & 0xaaaaaaaau;  // high bit of each order-2 field (mask 0, 1)
      const int c2 = __popc(o2);
      int incl = c2;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const uint32_t rank0 = (uint32_t)(base + incl - c2);
      base += __shfl_sync(0xffffffffu, incl, 31);
      const uint32_t v = __funnelshift_r(lo, hi, 8 * (B & 3));
      const uint64_t code = (uint64_t)dig[v & 255u] | (uint64_t)dig[(v >> 8) & 255u] << 10 |
                            (uint64_t)dig[(v >> 16) & 255u] << 20 | (uint64_t)dig[v >> 24] << 30;
      const uint32_t T = (uint32_t)(code >> s2);  // T0 digit of field j in bits 2j..2j+1
      const uint32_t nib[2] = {spread2(mw) << 2 | spread2(T), spread2(mw >> 16) << 2 | spread2(T >> 16)};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float2 wp = pt[(nib[k >> 2] >> (8 * (k & 3))) & 255u];
#pragma unroll
        for (int t = 0; t < MT; ++t) {
          const uint4 &q4 = xv[t][k >> 2];
          const uint32_t hw = (k & 3) == 0 ? q4.x : (k & 3) == 1 ? q4.y : (k & 3) == 2 ? q4.z : q4.w;
          const float2 xf = __half22float2(*reinterpret_cast<const __half2 *>(&hw));
          acc[t] = fmaf(wp.x, xf.x, fmaf(wp.y, xf.y, acc[t]));
        }
      }
      for (uint32_t bits = o2; bits; bits &= bits - 1) {
        const int jb = __ffs(bits) - 1;  // 2 j + 1
        const uint32_t r = rank0 + __popc(o2 & ((1u << jb) - 1u));
        const uint32_t rb = r / 5u;
        const int t1 = (int)((dig[__ldg(p2 + rb)] >> (2u * (r - 5u * rb))) & 3u) - 1;
        if (t1 == 0) continue;
        const float a1 = ((mw >> (jb - 1)) & 1u) ? a1_1 : a1_0;
        const float wc = t1 > 0 ? a1 : -a1;
        const __half *xk = xm + wi * 16 + (jb >> 1);
#pragma unroll
        for (int t = 0; t < MT; ++t)
          if (t < mt) acc[t] = fmaf(wc, ldx(xk + (int64_t)t * K), acc[t]);
      }
    }
  }
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    float v = acc[t];
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == t) part[warp][t] = v;
  }
  __syncthreads();
  if (live && seg == 0 && lane < mt) {
    float v = 0.f;
    for (int s = 0; s < S; ++s) v += part[r_in * S + s][lane];
    const int64_t i = (int64_t)(m0 + lane) * N + n;
    v += w.ydense[i];
    if (F32)
      static_cast<float *>(w.y)[i] = v;
    else
      static_cast<__half *>(w.y)[i] = __float2half_rn(v);
  }
}

constexpr int kIdxBlock = 2048, kIdxShift = 11;  // the correction index's blocks and code position
constexpr int kIdxWarps = 16, kIdxThreads = 32 * kIdxWarps;
constexpr int kIdxAhead = 5;  // pairs of entries per lane loaded one block ahead
constexpr int kIdxTabBytes = kIdxWarps * 32 * 4;
constexpr int kIdxMaxSmem = 227 * 1024, kSmSmem = 228 * 1024;  // shared memory of a block, of an SM

// Staged bytes per element: one token as fp32, more side by side as fp16.
__host__ __device__ constexpr int elem_bytes(int MT) { return MT == 1 ? 4 : 2 * MT; }
// correct_idx_kernel's dynamic shared memory: the warps' tables, then the
// activations from the next multiple of a block's bytes on.
constexpr int64_t idx_smem_bytes(int K, int MT) {
  return (int64_t)((K + kIdxBlock - 1) / kIdxBlock + 1) * kIdxBlock * elem_bytes(MT);
}

__device__ __forceinline__ float half_at(uint32_t w, int hi) {
  return __half2float(__ushort_as_half((unsigned short)(hi ? w >> 16 : w & 0xffffu)));
}
__device__ __forceinline__ float lds_f32(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
// The MT activations of the element staged at shared address a.
template <int MT>
__device__ __forceinline__ void staged_acts(uint32_t a, float (&x)[MT]) {
  if constexpr (MT == 1) {
    x[0] = lds_f32(a);
  } else {
    uint32_t w[MT / 2];
    if constexpr (MT == 2)
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[0]) : "r"(a));
    else if constexpr (MT == 4)
      asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(a));
    else
      asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                   : "r"(a));
#pragma unroll
    for (int t = 0; t < MT; ++t) x[t] = half_at(w[t / 2], t & 1);
  }
}

// Adds those of the index's first and last entries that are read alone
// (tq_ew_pairs.cuh) and lie in rows [r_lo, r_hi) to the plane-1 result y [N] of
// the token whose activations x are (the warp that has the rows, before it
// reads their y).
__device__ __forceinline__ void add_alone(const Prob &w, const unsigned short *x, float *y, int r_lo, int r_hi) {
  const int nb = (w.K + kIdxBlock - 1) / kIdxBlock, odd = (int)(((uintptr_t)w.idx >> 1) & 1u);
  const int entries = __ldg(w.idx_off + (int64_t)w.N * nb);
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const int i = side ? entries - 1 : 0;
    const int64_t lo = (int64_t)r_lo * nb, hi = (int64_t)r_hi * nb;
    if (!read_alone(side, odd, entries) || i < __ldg(w.idx_off + lo) || i >= __ldg(w.idx_off + hi)) continue;
    int64_t f = lo, end = hi;  // the entry's block: the last that begins at or before it
    while (end - f > 1) {
      const int64_t mid = (f + end) / 2;
      if (__ldg(w.idx_off + mid) <= i) f = mid; else end = mid;
    }
    const int n = (int)(f / nb), b = (int)(f - (int64_t)n * nb);
    const int en = __ldg(w.idx + i), code = en >> kIdxShift, q = code / 9;
    if (code >= 27) continue;
    const __half *mu = w.mu + (int64_t)n * 4, *a0 = w.a0 + (int64_t)n * 4;
    float wt = (__half2float(mu[q]) - __half2float(mu[3])) +
               (__half2float(a0[q]) - __half2float(a0[3])) * (float)(code / 3 % 3 - 1);
    if (q < 2) wt += __half2float(w.a1[(int64_t)n * 2 + q]) * (float)(code % 3 - 1);
    const int k = min(b * kIdxBlock + (en & (kIdxBlock - 1)), w.K - 1);
    y[n] = fmaf(wt, __half2float(__ushort_as_half(__ldg(x + k))), y[n]);
  }
}

// The same correction from the correction index.  An entry names its element
// k (within its block of 2048) and code = 9 q + 3 d0 + d1 (digits d = trit +
// 1), whose weight (mu_q - mu_3) + (alpha0_q - alpha0_3) T0 + alpha1_q T1 is
// read from the row's 27-entry table.  Only the entries and x are read: no
// mask plane, plane-1 or plane-2 bytes.
//
// The rows of every indexed problem of the call, one after the other and
// weighted with their length, are cut into one run per block, and the block's
// rows of a problem into one run per warp.  A block stages x[tokens][K]
// whenever its run enters another problem, the tokens of an element side by
// side: a gather from global memory touches some 20 cache lines per warp
// load, the same 32 words of shared memory take three to four bank cycles.
// Entries, offsets, table values and the plane-1 result are loaded ahead of
// their use (the rows of a warp are contiguous, and so are their entries):
// a lane has its ten entries of the next block (320 per warp; 13.6 % coverage
// has 279) in registers while it works on this one; fuller blocks finish
// in a loop.  What binds is the instructions per entry, so entries come in pairs, a table
// or activation address is one shift and one three-input AND-OR (tables and
// blocks lie at multiples of their size), one token is staged as fp32, and
// entries past a block's end are cut by predicates: 20
// warp-instructions per 32 entries with all that surrounds them, 19.4 M for
// one Qwen3-8B layer in 27.8 us (66 % of the issue slots; 54 MB, whose floor
// is 8 us), against 31.6 M in 39.5 us with one guarded entry per lane and
// step, and 48 us with gathers from global memory.
// STAGED = false reads x from global memory: K x tokens beyond a block's
// shared memory.  What binds is then the latency of the gathers, so a lane has
// ten under way (each loaded whether or not its entry is one), and one or two
// tokens take 64 registers, so that an SM holds 32 warps, since a long call is
// faster for it (16384 x 57344, one token, 13.6 and 60 % coverage: 212 and
// 683 us, with 128 registers 234 and 1018, with a gather at a time for eight
// tokens, whatever the call's, 625 and 2712, from warps of a row each 285 and
// 725; 300 x 57344 with 13.6 %: 38, 34, 91 and 79).
template <bool F32, int MT, bool STAGED, class BT>
__global__ void __launch_bounds__(kIdxThreads, MT == 8 || (!STAGED && MT > 2) ? 1 : 2)
    correct_idx_kernel(const __grid_constant__ BT bt, int64_t total, int m0, int mt) {
  constexpr int kES = elem_bytes(MT), kBlockBytes = kIdxBlock * kES;
  constexpr int kESLog = MT == 8 ? 4 : MT == 4 ? 3 : 2;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t base = smem_u32(smem);
  float *tab = reinterpret_cast<float *>(smem) + warp * 32;
  const uint32_t tab_a = base + (uint32_t)warp * 128u;
  const uint32_t xs_a = (base + kIdxTabBytes + kBlockBytes - 1) / kBlockBytes * kBlockBytes;
  unsigned char *xs = smem + (xs_a - base);
  // the block's run: row r of problem p lies in it if its first weight unit
  // (w_begin + r G) does
  const int64_t u_lo = total * blockIdx.x / gridDim.x, u_hi = total * (blockIdx.x + 1) / gridDim.x;
  int p = 0;
  for (int step = 1 << (31 - __clz(max(bt.count, 1))); step >= 1; step >>= 1)
    if (p + step < bt.count && bt.prob[p + step].w_begin <= u_lo) p += step;
  for (; p < bt.count; ++p) {
    const Prob &w = bt.prob[p];
    if (w.w_begin >= u_hi) break;
    if (!w.idx) continue;  // the other kernel's
    const int N = w.N, K = w.K, G = K / kGroup;
    const int b_lo = (int)min((int64_t)N, (max(u_lo - w.w_begin, (int64_t)0) + G - 1) / G);
    const int b_hi = (int)min((int64_t)N, (u_hi - w.w_begin + G - 1) / G);
    if (b_lo >= b_hi) continue;
    const unsigned short *xm = reinterpret_cast<const unsigned short *>(w.x) + (int64_t)m0 * K;
    const int nb = (K + kIdxBlock - 1) / kIdxBlock;
    // the warp's rows, their first and last offsets and the index's last one, on
    // the way while x is staged (waited for after it, the last one, which every
    // warp reads, cost a Qwen3-8B layer 1.2 us)
    const int r_lo = b_lo + (b_hi - b_lo) * warp / kIdxWarps, r_hi = b_lo + (b_hi - b_lo) * (warp + 1) / kIdxWarps;
    const int blocks = (r_hi - r_lo) * nb;
    const int32_t *offs = w.idx_off + (int64_t)r_lo * nb;
    const int entries = __ldg(w.idx_off + (int64_t)N * nb), o0 = __ldg(offs), o1 = __ldg(offs + min(1, blocks)),
              o2 = __ldg(offs + min(2, blocks)), oN = __ldg(offs + blocks);
    if (STAGED) {
      __syncthreads();  // the warps are done with the problem before
      for (int i = threadIdx.x; i < nb * (kIdxBlock / 8); i += kIdxThreads) {
        uint4 v[MT];
#pragma unroll
        for (int t = 0; t < MT; ++t)  // zeros past K
          v[t] = t < mt && 8 * i < K ? __ldg(reinterpret_cast<const uint4 *>(xm + (int64_t)t * K) + i)
                                     : make_uint4(0u, 0u, 0u, 0u);
        if constexpr (MT == 1) {
          float4 *d = reinterpret_cast<float4 *>(xs) + 2 * i;
          d[0] = make_float4(half_at(v[0].x, 0), half_at(v[0].x, 1), half_at(v[0].y, 0), half_at(v[0].y, 1));
          d[1] = make_float4(half_at(v[0].z, 0), half_at(v[0].z, 1), half_at(v[0].w, 0), half_at(v[0].w, 1));
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            uint32_t *d = reinterpret_cast<uint32_t *>(xs + (8 * i + j) * kES);
#pragma unroll
            for (int t = 0; t < MT; t += 2) {
              const uint4 &a = v[t], &b = v[t + 1];
              const uint32_t wa = (j >> 1) == 0 ? a.x : (j >> 1) == 1 ? a.y : (j >> 1) == 2 ? a.z : a.w;
              const uint32_t wb = (j >> 1) == 0 ? b.x : (j >> 1) == 1 ? b.y : (j >> 1) == 2 ? b.z : b.w;
              d[t / 2] = __byte_perm(wa, wb, j & 1 ? 0x7632 : 0x5410);
            }
          }
        }
      }
      __syncthreads();
    }
    grid_dep_wait();  // the plane-1 pass (returns at once from the second time on)
    if (r_lo >= r_hi) continue;
    // entries as aligned pairs, but for the index's first and last where a word
    // of theirs reaches beyond it (tq_ew_pairs.cuh): these go into ydense
    const int odd = (int)(((uintptr_t)w.idx >> 1) & 1u);
    const uint32_t *iw = reinterpret_cast<const uint32_t *>(w.idx - odd);
    const int last = pairs_end(odd, entries);
    auto off_at = [&](int i) { return pairs_clamp(__ldg(offs + i), odd, last); };
    auto load_pairs = [&](uint32_t (&v)[kIdxAhead], int e, int e1) {
      const int first = (e + odd) >> 1, c = ((e1 + odd + 1) >> 1) - first;
      const uint32_t *q = iw + first + lane;
#pragma unroll
      for (int j = 0; j < kIdxAhead; ++j) v[j] = lane + 32 * j < c && e < e1 ? __ldg(q + 32 * j) : 0u;
    };
    // this lane's table entry of row n: codes 27..31 (none in a valid index) weigh nothing
    const int q = min(lane / 9, 2), d0 = (lane / 3) % 3, d1 = lane % 3;
    unsigned short h[5];
    auto load_params = [&](int n) {
      const unsigned short *mu = reinterpret_cast<const unsigned short *>(w.mu) + (int64_t)n * 4;
      const unsigned short *a0 = reinterpret_cast<const unsigned short *>(w.a0) + (int64_t)n * 4;
      h[0] = __ldg(mu + q), h[1] = __ldg(mu + 3), h[2] = __ldg(a0 + q), h[3] = __ldg(a0 + 3);
      h[4] = q < 2 ? __ldg(reinterpret_cast<const unsigned short *>(w.a1) + (int64_t)n * 2 + q) : (unsigned short)0;
    };
    auto h2f = [](unsigned short v) { return __half2float(__ushort_as_half(v)); };
    load_params(r_lo);
    int e = pairs_clamp(o0, odd, last), e1 = pairs_clamp(o1, odd, last);
    int e2 = pairs_clamp(o2, odd, last);  // the next block's end
    uint32_t v[kIdxAhead];
    load_pairs(v, e, e1);
    if ((o0 == 0 && read_alone(false, odd, entries)) || (oN == entries && read_alone(true, odd, entries)))
      if (lane < mt && lane < MT) add_alone(w, xm + (int64_t)lane * K, w.ydense + (int64_t)(m0 + lane) * N, r_lo, r_hi);
    int f = 0;  // the block among the run's
    for (int n = r_lo; n < r_hi; ++n) {
      float a = (h2f(h[0]) - h2f(h[1])) + (h2f(h[2]) - h2f(h[3])) * (float)(d0 - 1);
      if (q < 2) a += h2f(h[4]) * (float)(d1 - 1);
      __syncwarp();  // the row before is done with the table
      tab[lane] = lane < 27 ? a : 0.f;
      __syncwarp();
      if (n + 1 < r_hi) load_params(n + 1);
      const int64_t yi = (int64_t)(m0 + lane) * N + n;
      const float yd = lane < mt && lane < MT ? w.ydense[yi] : 0.f;
      float acc[MT];
#pragma unroll
      for (int t = 0; t < MT; ++t) acc[t] = 0.f;
      auto add_at = [&](uint32_t en, bool in, int b) {  // en: the entry (of block b) in bits 0..15
        if constexpr (STAGED) {
          const float wt = lds_f32((en >> 9 & 0x7cu) | tab_a);
          float x[MT];
          staged_acts<MT>((en << kESLog & ((kIdxBlock - 1) << kESLog)) | (xs_a + (uint32_t)b * kBlockBytes), x);
          if (in) {
#pragma unroll
            for (int t = 0; t < MT; ++t) acc[t] = fmaf(wt, x[t], acc[t]);
          }
        } else {
          // (loaded whether or not `in`: the gathers of a lane's entries are
          // then under way together)
          const float wt = tab[en >> kIdxShift & 31u];
          const unsigned short *xk = xm + min(b * kIdxBlock + (int)(en & (kIdxBlock - 1)), K - 1);
          unsigned short x[MT];
#pragma unroll
          for (int t = 0; t < MT; ++t) x[t] = __ldg(xk + (int64_t)min(t, mt - 1) * K);
          if (in) {
#pragma unroll
            for (int t = 0; t < MT; ++t) acc[t] = fmaf(wt, h2f(x[t]), acc[t]);
          }
        }
      };
      for (int b = 0; b < nb; ++b, ++f) {
        const int e3 = f + 2 < blocks ? off_at(f + 3) : e2;
        uint32_t u[kIdxAhead];  // the next block's entries
        load_pairs(u, e1, e2);
        auto add = [&](uint32_t en, bool in) { add_at(en, in, b); };
        const int front = (e + odd) & 1, c = e1 - e + front;  // entries from the first word on, the first `front` not ours
        const int i0 = 2 * lane;
        add(v[0], i0 < c && i0 >= front);
        add(v[0] >> 16, i0 + 1 < c);
        if (STAGED || c > 64) {  // (a block of few entries gathers for these only)
#pragma unroll
          for (int j = 1; j < kIdxAhead; ++j) {
            const int i = i0 + 64 * j;
            add(v[j], i < c);
            add(v[j] >> 16, i + 1 < c);
          }
        }
        if constexpr (STAGED) {
          const int i0t = 2 * (lane + 32 * kIdxAhead);
          auto tail = [&](int i) {
            const uint32_t r = __ldg(iw + ((e + odd) >> 1) + (i >> 1));
            add(r, true);
            add(r >> 16, i + 1 < c);
          };
          // (two steps at once for four and eight tokens: the compiler's own
          // choice, faster for one and two, is 15 % slower for four with every
          // element indexed)
          if constexpr (MT >= 4) {
#pragma unroll 2
            for (int i = i0t; i < c; i += 64) tail(i);
          } else {
            for (int i = i0t; i < c; i += 64) tail(i);
          }
        } else {  // as many gathers under way as for the first entries
          for (int i1 = i0 + 64 * kIdxAhead; i1 - i0 < c; i1 += 64 * kIdxAhead) {
            uint32_t r[kIdxAhead];
#pragma unroll
            for (int j = 0; j < kIdxAhead; ++j)
              r[j] = i1 + 64 * j < c ? __ldg(iw + ((e + odd) >> 1) + (i1 >> 1) + 32 * j) : 0u;
#pragma unroll
            for (int j = 0; j < kIdxAhead; ++j) {
              add(r[j], i1 + 64 * j < c);
              add(r[j] >> 16, i1 + 64 * j + 1 < c);
            }
          }
        }
        e = e1, e1 = e2, e2 = e3;
#pragma unroll
        for (int j = 0; j < kIdxAhead; ++j) v[j] = u[j];
      }
      float mine = 0.f;
#pragma unroll
      for (int t = 0; t < MT; ++t) {
        float s = acc[t];
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == t) mine = s;
      }
      if (lane < mt && lane < MT) {
        mine += yd;
        if (F32)
          static_cast<float *>(w.y)[yi] = mine;
        else
          static_cast<__half *>(w.y)[yi] = __float2half_rn(mine);
      }
    }
  }
}

// Warps per row: the largest power of two up to 8 that leaves each warp at
// least three chunks, raised (up to one chunk per warp) while the grid holds
// fewer than four blocks per SM.
int warps_per_row(int N, int K, int num_sms) {
  const int C = (K / 16 + 31) / 32;
  int S = 1;
  while (S < kWarps && C / (2 * S) >= 3) S *= 2;
  while (S < kWarps && 2 * S <= C && (int64_t)N * S / kWarps < 4LL * num_sms) S *= 2;
  return S;
}

template <bool F32, int MT>
cudaError_t launch_correct(int M, const Batch<Prob> &bt, int grid, cudaStream_t s) {
  for (int m0 = 0; m0 < M; m0 += MT) {
    correct_kernel<F32, MT><<<dim3(grid, bt.count), 32 * kWarps, 0, s>>>(bt, m0, std::min(MT, M - m0));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// grid: blocks for the call's indexed rows at one row per warp (at two warps
// per row where x is gathered: few rows are then on more SMs), capped at what
// the chip holds.
template <bool F32, int MT, bool STAGED>
cudaError_t launch_correct_idx(int M, const Batch<Prob> &bt, int64_t total, int rows, int Kmax, int num_sms,
                               cudaStream_t s) {
  const int smem = STAGED ? (int)idx_smem_bytes(Kmax, MT) : kIdxTabBytes;
  const int per_sm = MT < 8 && (STAGED || MT <= 2) && 2 * (smem + 1024) <= kSmSmem ? 2 : 1;
  constexpr int kRowsPerBlock = STAGED ? kIdxWarps : kIdxWarps / 2;
  const int grid = std::max(1, std::min((rows + kRowsPerBlock - 1) / kRowsPerBlock, per_sm * num_sms));
  return with_batch(bt, [&](const auto &b) {
    const auto kern = correct_idx_kernel<F32, MT, STAGED, std::decay_t<decltype(b)>>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kIdxMaxSmem);
    for (int m0 = 0; m0 < M && e == cudaSuccess; m0 += MT)
      e = launch_dependent_cluster(kern, dim3(grid), 1, kIdxThreads, smem, s, b, total, m0, std::min(MT, M - m0));
    return e;
  });
}

template <bool F32>
cudaError_t launch_correct_mt(int M, const Batch<Prob> &bt, int grid, cudaStream_t s) {
  if (M == 1) return launch_correct<F32, 1>(M, bt, grid, s);
  if (M == 2) return launch_correct<F32, 2>(M, bt, grid, s);
  if (M <= 4) return launch_correct<F32, 4>(M, bt, grid, s);
  return launch_correct<F32, 8>(M, bt, grid, s);
}

// Tokens per pass: as many as the call has, up to 8, while their staged
// activations fit a block's shared memory (K up to 12288 for 8 tokens, 26624
// for four, 55296 for two or one); beyond that x is gathered from global
// memory.  More passes than three of two tokens each are slower than one of
// eight that gathers (512 x 49152, eight tokens, 13.6 %: 150 and 141 us, with
// 0.3 % 148 and 107); with passes of four, staging is the faster one
// (4096 x 16384, eight tokens: 65 and 77, but 62 and 50 with 0.3 %).
template <bool F32>
cudaError_t launch_correct_idx_mt(int M, const Batch<Prob> &bt, int64_t total, int rows, int Kmax, int num_sms,
                                  cudaStream_t s) {
  const auto fits = [&](int MT) { return idx_smem_bytes(Kmax, MT) <= kIdxMaxSmem; };
  if (M > 4 && fits(8)) return launch_correct_idx<F32, 8, true>(M, bt, total, rows, Kmax, num_sms, s);
  if (M > 2 && fits(4)) return launch_correct_idx<F32, 4, true>(M, bt, total, rows, Kmax, num_sms, s);
  if (M > 1 && M <= 6 && fits(2)) return launch_correct_idx<F32, 2, true>(M, bt, total, rows, Kmax, num_sms, s);
  if (M == 1 && fits(1)) return launch_correct_idx<F32, 1, true>(M, bt, total, rows, Kmax, num_sms, s);
  if (M == 1) return launch_correct_idx<F32, 1, false>(M, bt, total, rows, Kmax, num_sms, s);
  if (M == 2) return launch_correct_idx<F32, 2, false>(M, bt, total, rows, Kmax, num_sms, s);
  if (M <= 4) return launch_correct_idx<F32, 4, false>(M, bt, total, rows, Kmax, num_sms, s);
  return launch_correct_idx<F32, 8, false>(M, bt, total, rows, Kmax, num_sms, s);
}

}  // namespace ew

// The views of every problem (one launch).
cudaError_t launch_ew_views(const EwCall *calls, int count, cudaStream_t s) {
  thread_local ew::Batch<ew::ViewProb> bt;  // large: kept off the stack
  bt.count = count;
  int64_t most = 1;
  for (int i = 0; i < count; ++i) {
    const EwCall &c = calls[i];
    ew::ViewProb &P = bt.prob[i];
    P.mu = reinterpret_cast<const __half *>(c.w->mu);
    P.a0 = reinterpret_cast<const __half *>(c.w->alpha0);
    P.s1v = reinterpret_cast<__half *>(c.s1v);
    P.offv = reinterpret_cast<__half *>(c.offv);
    P.salv = c.salv;
    P.rpv = c.rpv;
    P.N = c.w->N;
    P.K = c.w->K;
    most = std::max<int64_t>(most, (int64_t)P.N * (P.K / kGroup));
  }
  constexpr int64_t per_block = 8 * ew::kViewUnits * ew::kViewThreads;
  const int blocks = (int)std::min<int64_t>((most + per_block - 1) / per_block, 1024);
  return ew::with_batch(bt, [&](const auto &b) {
    return launch_dependent(ew::views_kernel<std::decay_t<decltype(b)>>, dim3(blocks, count), ew::kViewThreads, s, b);
  });
}

// Masks 0..2 of every problem added to its plane-1 result, y written: the
// problems with a correction index through correct_idx_kernel, the others
// through correct_kernel (one launch of each kind present per pass of up
// to 8 tokens).
cudaError_t launch_ew_correct(int M, const EwCall *calls, int count, bool f32, cudaStream_t s) {
  thread_local ew::Batch<ew::Prob> bt;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  bt.count = count;
  for (int pass = 0; pass < 2; ++pass) {
    const bool indexed = pass == 1;
    int most = 0, rows_idx = 0, Kmax = 0;
    int64_t total = 0;
    for (int i = 0; i < count; ++i) {
      const EwCall &c = calls[i];
      ew::Prob &P = bt.prob[i];
      P.mask = c.w->mask;
      P.plane1 = c.w->plane1;
      P.p2rowptr = c.w->p2rowptr;
      P.plane2 = c.w->plane2;
      P.mu = reinterpret_cast<const __half *>(c.w->mu);
      P.a0 = reinterpret_cast<const __half *>(c.w->alpha0);
      P.a1 = reinterpret_cast<const __half *>(c.w->alpha1);
      P.idx_off = c.w->idx_off;
      P.idx = c.w->idx;
      P.x = reinterpret_cast<const __half *>(c.x);
      P.ydense = c.ydense;
      P.y = c.y;
      P.N = c.w->N;
      P.K = c.w->K;
      const bool mine = (c.w->idx_off && c.w->idx) == indexed;
      P.S = ew::warps_per_row(P.N, P.K, sms);
      const int rows = ew::kWarps / P.S;
      P.blocks = mine && !indexed ? (P.N + rows - 1) / rows : 0;
      P.w_begin = total;
      if (mine && indexed) {
        total += (int64_t)P.N * (P.K / kGroup);
        rows_idx = std::min<int64_t>((int64_t)rows_idx + P.N, INT32_MAX / 2);
        Kmax = std::max(Kmax, P.K);
      }
      most = std::max(most, P.blocks);
    }
    if (indexed ? total == 0 : most == 0) continue;
    const cudaError_t e = indexed ? (f32 ? ew::launch_correct_idx_mt<true>(M, bt, total, rows_idx, Kmax, sms, s)
                                         : ew::launch_correct_idx_mt<false>(M, bt, total, rows_idx, Kmax, sms, s))
                                  : (f32 ? ew::launch_correct_mt<true>(M, bt, most, s)
                                         : ew::launch_correct_mt<false>(M, bt, most, s));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace tq
