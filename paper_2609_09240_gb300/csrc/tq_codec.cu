// tq_codec.cu - pack / unpack / salience row-prefix kernels.
//
// The lattice-aware serialization of the paper ("Packing: From Quantization
// to Serialization") stores the discrete supports (trit codes) and their
// parameters instead of fp16 values.  Byte layout (library definition, the
// paper prints none): five trits per byte as a base-3 numeral, digit =
// trit + 1, first trit least significant; a 128-trit group is 26 bytes
// (25 full bytes, then a tail byte with trits 125..127 and pad digits 1);
// plane-1 rows are padded with 0x00 to a multiple of 16 bytes.  Plane 2
// holds only salient groups in (row, group) order.
//
// Every kernel validates what it reads and ORs TQ_DATA_* bits into the
// caller's status word; no kernel traps, and every plane-2 index is checked
// against rowptr[N] before it is used.
#include "tq_common.cuh"
#include "tq_launch.cuh"
#include "tq_sm100.cuh"

namespace tq {

__device__ __forceinline__ int sal_bit(const uint32_t *sal, int W, int n, int g) {
  return (int)((sal[(int64_t)n * W + (g >> 5)] >> (g & 31)) & 1u);
}

// Number of salient groups of row n before group g.
__device__ __forceinline__ int sal_rank(const uint32_t *sal, int W, int n, int g) {
  const uint32_t *row = sal + (int64_t)n * W;
  int r = 0;
  for (int w = 0; w < (g >> 5); ++w) r += __popc(row[w]);
  uint32_t part = row[g >> 5] & ((1u << (g & 31)) - 1u);
  return r + __popc(part);
}

// Set bits of row n at valid group positions, and whether pad bits are set.
__device__ __forceinline__ int row_popc(const uint32_t *sal, int W, int G, int n, bool *pad_bad) {
  const uint32_t *row = sal + (int64_t)n * W;
  int r = 0;
  for (int w = 0; w < W; ++w) {
    uint32_t v = row[w];
    int valid = G - 32 * w;  // valid bits in this word
    if (valid < 32) {
      uint32_t mask = valid > 0 ? ((1u << valid) - 1u) : 0u;
      if (v & ~mask) *pad_bad = true;
      v &= mask;
    }
    r += __popc(v);
  }
  return r;
}

// ---------------------------------------------------------------- rowptr
// One block: each thread sums a contiguous run of rows, then a block scan.
__global__ void __launch_bounds__(1024) rowptr_kernel(int N, int K, const uint32_t *sal,
                                                      int32_t *rowptr, uint32_t *status) {
  const int G = K / kGroup, W = sal_words_of(K);
  const int per = (N + blockDim.x - 1) / blockDim.x;
  const int r0 = threadIdx.x * per;
  const int r1 = min(N, r0 + per);
  grid_dep_launch_next();
  grid_dep_wait();
  bool pad_bad = false;
  int local = 0, cnt[16];  // a thread's rows' counts, up to 16 rows
  if (per <= 16) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      cnt[i] = r0 + i < r1 ? row_popc(sal, W, G, r0 + i, &pad_bad) : 0;
      local += cnt[i];
    }
  } else {
    for (int n = r0; n < r1; ++n) local += row_popc(sal, W, G, n, &pad_bad);
  }
  // inclusive warp scan, then scan of warp totals
  __shared__ int warp_tot[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = local;
  for (int o = 1; o < 32; o <<= 1) {
    int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int nw = blockDim.x >> 5;
    int v = lane < nw ? warp_tot[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    if (lane < nw) warp_tot[lane] = v;  // inclusive over warps
  }
  __syncthreads();
  int base = (wid > 0 ? warp_tot[wid - 1] : 0) + incl - local;
  if (per <= 16) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (r0 + i < r1) rowptr[r0 + i] = base;
      base += cnt[i];
    }
  } else {
    for (int n = r0; n < r1; ++n) {
      rowptr[n] = base;
      bool dummy = false;
      base += row_popc(sal, W, G, n, &dummy);
    }
  }
  if (threadIdx.x == blockDim.x - 1) rowptr[N] = warp_tot[(blockDim.x >> 5) - 1];
  if (pad_bad) atomicOr(status, TQ_DATA_BAD_PAD);
}

// Thread per row: rowptr[0] == 0 and rowptr[n+1] - rowptr[n] == popcount.
__global__ void check_rowptr_kernel(int N, int K, const uint32_t *sal, const int32_t *rowptr,
                                    uint32_t *status) {
  const int G = K / kGroup, W = sal_words_of(K);
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  bool pad_bad = false;
  int c = row_popc(sal, W, G, n, &pad_bad);
  uint32_t st = 0;
  if (pad_bad) st |= TQ_DATA_BAD_PAD;
  if (rowptr[n + 1] - rowptr[n] != c) st |= TQ_DATA_BAD_ROWPTR;
  if (n == 0 && rowptr[0] != 0) st |= TQ_DATA_BAD_ROWPTR;
  if (st) atomicOr(status, st);
}

// ------------------------------------------------------------------- pack
__device__ __forceinline__ uint8_t encode_codes(const int8_t *t, int ntr, uint32_t *st) {
  int v = 0, p = 1;
  for (int i = 0; i < 5; ++i) {
    int d = 1;  // pad digit (trit 0)
    if (i < ntr) {
      int c = t[i];
      if (c < -1 || c > 1) {
        *st |= TQ_DATA_BAD_CODE;
        c = c < -1 ? -1 : 1;
      }
      d = c + 1;
    }
    v += d * p;
    p *= 3;
  }
  return (uint8_t)v;
}

// Thread per plane-1 byte (n, b): blocks stride over rows, threads over a
// row's bytes.
__global__ void pack_kernel(int N, int K, const int8_t *T1, const int8_t *T2, const uint32_t *sal,
                            const int32_t *rowptr, uint8_t *plane1, uint8_t *plane2,
                            uint32_t *status) {
  const int G = K / kGroup, W = sal_words_of(K);
  const int RB = (int)row_bytes_of(K);
  const int32_t nnz = rowptr[N];
  for (int n = blockIdx.x; n < N; n += gridDim.x)
  for (int b = threadIdx.x; b < RB; b += blockDim.x) {
    const int64_t idx = (int64_t)n * RB + b;
    uint32_t st = 0;
    if (b >= G * kGroupBytes) {
      plane1[idx] = 0;
      continue;
    }
    const int g = b / kGroupBytes, pos = b - g * kGroupBytes;
    const int ntr = pos < kFullBytes ? 5 : kTailTrits;
    const int64_t k0 = (int64_t)n * K + (int64_t)g * kGroup + 5 * pos;
    plane1[idx] = encode_codes(T1 + k0, ntr, &st);
    const int s = sal_bit(sal, W, n, g);
    if (T2) {
      if (s) {
        int64_t j = (int64_t)rowptr[n] + sal_rank(sal, W, n, g);
        if (j >= 0 && j < nnz)
          plane2[j * kGroupBytes + pos] = encode_codes(T2 + k0, ntr, &st);
        else
          st |= TQ_DATA_BAD_ROWPTR;
      } else {
        for (int i = 0; i < ntr; ++i)
          if (T2[k0 + i] != 0) st |= TQ_DATA_T2_OUTSIDE;
      }
    } else if (s) {
      st |= TQ_DATA_T2_OUTSIDE;
    }
    if (st) atomicOr(status, st);
  }
}

// ----------------------------------------------------------------- unpack
__device__ __forceinline__ void decode_to(uint8_t v, int ntr, int8_t *t, uint32_t *st) {
  if (v > 242) {
    *st |= TQ_DATA_BAD_BYTE;
    for (int i = 0; i < ntr; ++i) t[i] = 0;
    return;
  }
  int q = v;
  for (int i = 0; i < 5; ++i) {
    int d = q % 3;
    q /= 3;
    if (i < ntr)
      t[i] = (int8_t)(d - 1);
    else if (d != 1)
      *st |= TQ_DATA_BAD_PAD;
  }
}

// Thread per plane-1 byte (n, b): blocks stride over rows, threads over a
// row's bytes.
__global__ void unpack_kernel(int N, int K, const uint8_t *plane1, const uint8_t *plane2,
                              const uint32_t *sal, const int32_t *rowptr, int8_t *T1, int8_t *T2,
                              uint32_t *status) {
  const int G = K / kGroup, W = sal_words_of(K);
  const int RB = (int)row_bytes_of(K);
  const int32_t nnz = rowptr[N];
  for (int n = blockIdx.x; n < N; n += gridDim.x)
  for (int b = threadIdx.x; b < RB; b += blockDim.x) {
    const int64_t idx = (int64_t)n * RB + b;
    uint32_t st = 0;
    const uint8_t v = plane1[idx];
    if (b >= G * kGroupBytes) {
      if (v != 0) atomicOr(status, TQ_DATA_BAD_PAD);
      continue;
    }
    const int g = b / kGroupBytes, pos = b - g * kGroupBytes;
    const int ntr = pos < kFullBytes ? 5 : kTailTrits;
    const int64_t k0 = (int64_t)n * K + (int64_t)g * kGroup + 5 * pos;
    decode_to(v, ntr, T1 + k0, &st);
    if (T2) {
      if (sal_bit(sal, W, n, g)) {
        int64_t j = (int64_t)rowptr[n] + sal_rank(sal, W, n, g);
        if (plane2 && j >= 0 && j < nnz) {
          decode_to(plane2[j * kGroupBytes + pos], ntr, T2 + k0, &st);
        } else {
          st |= TQ_DATA_BAD_ROWPTR;
          for (int i = 0; i < ntr; ++i) T2[k0 + i] = 0;
        }
      } else {
        for (int i = 0; i < ntr; ++i) T2[k0 + i] = 0;
      }
    }
    if (st) atomicOr(status, st);
  }
}

// ----------------------------------------------- warp-staged pack / unpack
// The same bytes and status bits as pack_kernel / unpack_kernel, a warp per
// 32 consecutive groups (of one row or several).  The codes move between
// global and shared memory in 16-byte units (a warp's 4 KB are contiguous),
// each lane encodes or decodes one group in registers, and the packed bytes
// move in 2-byte units, 64 contiguous bytes per access.  Taken when the code
// arrays are 16-byte and the packed planes 2-byte aligned.
// What bounds it: HBM (the codes, read or written once).  A warp has its 8 KB
// of codes under way at once and waits for no other warp; with a CTA per row
// and block barriers between load, encode and store, packing and unpacking a
// 12288 x 4096 projection took 120 us (1.87 TB/s), this takes 58 us (3.87 TB/s;
// pack 33, unpack 30 of them under a profiler, at about 45 % issue).
constexpr int kCodecWarps = 4;
constexpr int kGroupStride = kGroup + 16;  // a group's codes in shared memory (free of bank conflicts)
constexpr int kStageBytesW = 32 * kGroupStride;

// Digits (code + 1) of four codes, bytewise without carries between bytes.
__device__ __forceinline__ uint32_t digits4(uint32_t c) {
  return ((c & 0x7F7F7F7Fu) + 0x01010101u) ^ (c & 0x80808080u);
}
// Bits that are set iff some digit is not 0, 1 or 2.
__device__ __forceinline__ uint32_t not_digits4(uint32_t d) { return (d & 0xFCFCFCFCu) | (d & (d >> 1) & 0x01010101u); }

// The 26 bytes of a group from its 128 codes in shared memory (p), as
// halfwords; a group with an invalid code goes through encode_codes.
__device__ __forceinline__ void encode_group(const unsigned char *p, uint16_t (&h)[13], uint32_t *st) {
  uint32_t d[32], bad = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint4 v = *reinterpret_cast<const uint4 *>(p + 16 * i);
    d[4 * i] = digits4(v.x), d[4 * i + 1] = digits4(v.y), d[4 * i + 2] = digits4(v.z), d[4 * i + 3] = digits4(v.w);
  }
#pragma unroll
  for (int i = 0; i < 32; ++i) bad |= not_digits4(d[i]);
  if (bad) {
#pragma unroll 1
    for (int j = 0; j < 13; ++j) {
      const int8_t *t = reinterpret_cast<const int8_t *>(p) + 10 * j;
      const uint32_t lo = encode_codes(t, 5, st), hi = encode_codes(t + 5, j < 12 ? 5 : kTailTrits, st);
#pragma unroll
      for (int k = 0; k < 13; ++k)  // (no dynamic register index)
        if (k == j) h[k] = (uint16_t)(lo | hi << 8);
    }
    return;
  }
  // byte j: digits 5 j .. 5 j + 4, from the two or three words they lie in
  auto byte = [&](int j) -> uint32_t {
    constexpr uint32_t pw[5] = {1, 3, 9, 27, 81};
    uint32_t v = j < kFullBytes ? 0u : 27u + 81u;  // the tail byte's pad digits are 1
#pragma unroll
    for (int w = 5 * j / 4; w <= (5 * j + 4) / 4 && w < 32; ++w) {
      uint32_t wt = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = 4 * w + k - 5 * j;
        if (i >= 0 && i < 5) wt |= pw[i] << (8 * k);
      }
      v = __dp4a(d[w], wt, v);
    }
    return v;
  };
#pragma unroll
  for (int j = 0; j < 13; ++j) h[j] = (uint16_t)(byte(2 * j) | byte(2 * j + 1) << 8);
}

// A lane's group of a warp's 32: row, group in the row, whether it exists.
struct LaneGroup {
  int n, g;
  bool live;
};
__device__ __forceinline__ LaneGroup lane_group(int64_t q0, int64_t total, int G, int lane) {
  LaneGroup r;
  const int64_t n0 = q0 / G;
  const int e = (int)(q0 - n0 * G) + lane;
  r.n = (int)n0 + e / G;
  r.g = e % G;
  r.live = q0 + lane < total;
  return r;
}
// Halfword u of the warp's packed bytes: lane u / 13's group, its byte
// 2 (u % 13); off: a lane's byte offset in plane 1, or -1 for no group.
// (13 accesses of 64 contiguous bytes.)
template <class F>
__device__ __forceinline__ void for_halfwords(int64_t off, int lane, F f) {
#pragma unroll
  for (int i = 0; i < 13; ++i) {
    const int u = 32 * i + lane, l = u / 13;
    const int64_t o = __shfl_sync(0xffffffffu, off, l);
    f(u, o < 0 ? o : o + 2 * (u - 13 * l));
  }
}
// The check of a row's salience bits and row pointers (check_rowptr_kernel).
__device__ __forceinline__ uint32_t row_status(const uint32_t *sal, const int32_t *rowptr, int W, int G, int n) {
  bool pad_bad = false;
  const int c = row_popc(sal, W, G, n, &pad_bad);
  uint32_t st = pad_bad ? TQ_DATA_BAD_PAD : 0u;
  if (rowptr[n + 1] - rowptr[n] != c || (n == 0 && rowptr[0] != 0)) st |= TQ_DATA_BAD_ROWPTR;
  return st;
}

__global__ void __launch_bounds__(32 * kCodecWarps) pack_warp_kernel(int N, int K, const int8_t *T1, const int8_t *T2,
                                                                   const uint32_t *sal, const int32_t *rowptr,
                                                                   uint8_t *plane1, uint8_t *plane2,
                                                                   uint32_t *status) {
  __shared__ __align__(16) unsigned char stage[kCodecWarps][kStageBytesW];
  const int G = K / kGroup, W = sal_words_of(K), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t RB = row_bytes_of(K), total = (int64_t)N * G;
  const int64_t q0 = ((int64_t)blockIdx.x * kCodecWarps + warp) * 32;
  if (q0 >= total) return;
  unsigned char *sm = stage[warp];
  // chunk 32 i + lane of the warp's codes: group 4 i + lane / 8's 16-byte part lane % 8
  const int64_t chunks = (total - q0) * 8;
  const uint4 *s1 = reinterpret_cast<const uint4 *>(T1 + q0 * kGroup), *s2 = reinterpret_cast<const uint4 *>(T2 + q0 * kGroup);
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  uint4 v1[8], v2[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v1[i] = 32 * i + lane < chunks ? __ldcs(s1 + 32 * i + lane) : zero;
  if (T2) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v2[i] = 32 * i + lane < chunks ? __ldcs(s2 + 32 * i + lane) : zero;
  }
  const LaneGroup L = lane_group(q0, total, G, lane);
  const int64_t off = L.live ? L.n * RB + (int64_t)L.g * kGroupBytes : -1;
  const bool s = L.live && sal_bit(sal, W, L.n, L.g);
  const uint32_t smask = __ballot_sync(0xffffffffu, s);
  uint32_t st = L.live && L.g == 0 ? row_status(sal, rowptr, W, G, L.n) : 0u;
  unsigned char *mine = sm + lane * kGroupStride;
  unsigned char *part = sm + (lane >> 3) * kGroupStride + 16 * (lane & 7);
  uint16_t h[13];
#pragma unroll
  for (int i = 0; i < 8; ++i) *reinterpret_cast<uint4 *>(part + 4 * i * kGroupStride) = v1[i];
  __syncwarp();
  encode_group(mine, h, &st);
  __syncwarp();
  // the bytes go out in order: through shared memory
#pragma unroll
  for (int j = 0; j < 13; ++j) *reinterpret_cast<uint16_t *>(sm + lane * kGroupBytes + 2 * j) = h[j];
  __syncwarp();
  for_halfwords(off, lane, [&](int u, int64_t o) {
    if (o >= 0) *reinterpret_cast<uint16_t *>(plane1 + o) = *reinterpret_cast<const uint16_t *>(sm + 2 * u);
  });
  if (L.live && L.g == G - 1)
    for (int64_t b = off + kGroupBytes; b < (L.n + 1) * RB; b += 2) *reinterpret_cast<uint16_t *>(plane1 + b) = 0;
  if (T2) {
    __syncwarp();
    // second-plane codes outside the salient groups must be zero; the salient
    // groups' go through shared memory
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool sg = (smask >> (4 * i + (lane >> 3))) & 1u;
      if (sg)
        *reinterpret_cast<uint4 *>(part + 4 * i * kGroupStride) = v2[i];
      else if ((v2[i].x | v2[i].y | v2[i].z | v2[i].w) != 0)
        st |= TQ_DATA_T2_OUTSIDE;
    }
    __syncwarp();
    if (s) {
      encode_group(mine, h, &st);
      const int64_t j = (int64_t)rowptr[L.n] + sal_rank(sal, W, L.n, L.g);
      if (j >= 0 && j < rowptr[N]) {
        uint16_t *d = reinterpret_cast<uint16_t *>(plane2 + j * kGroupBytes);
#pragma unroll
        for (int k = 0; k < 13; ++k) d[k] = h[k];
      } else {
        st |= TQ_DATA_BAD_ROWPTR;
      }
    }
  } else if (s) {
    st |= TQ_DATA_T2_OUTSIDE;
  }
  st = __reduce_or_sync(0xffffffffu, st);
  if (st && lane == 0) atomicOr(status, st);
}

// Decode table: a byte's five codes in bytes 0..4, byte 5 nonzero for an
// invalid byte (its codes are zero).
__device__ __forceinline__ uint2 decode_entry(int v) {
  if (v > 242) return make_uint2(0u, 0x100u);
  uint32_t t[5];
#pragma unroll
  for (int i = 0; i < 5; ++i, v /= 3) t[i] = (uint32_t)(v % 3 - 1) & 0xFFu;
  return make_uint2(t[0] | t[1] << 8 | t[2] << 16 | t[3] << 24, t[4]);
}
// A group's 128 codes into shared memory (p) from its 26 bytes (halfwords).
__device__ __forceinline__ void decode_group_codes(const uint16_t (&h)[13], const uint2 *lut, unsigned char *p, uint32_t *st) {
  uint32_t bad = 0, w[32];
  uint2 e = lut[h[0] & 0xFFu];
#pragma unroll
  for (int j = 0; j < 26; ++j) {
    bad |= e.y;
    const uint2 nx = j + 1 < 26 ? lut[(j & 1) ? h[(j + 1) >> 1] & 0xFFu : h[j >> 1] >> 8] : make_uint2(0u, 0u);
    // words whose first code is in byte j: code 4 k = 5 j + i
#pragma unroll
    for (int k = (5 * j + 3) / 4; 4 * k < 5 * j + 5 && k < 32; ++k) {
      const int i = 4 * k - 5 * j;
      const uint32_t tail = __byte_perm(e.y, nx.x, 0x6540);  // code 4, the next byte's codes 0..2
      w[k] = i == 0 ? e.x : i == 4 ? tail : __funnelshift_r(e.x, tail, 8 * i);
    }
    if (j == 25 && !(e.y & 0x100u) && ((e.x >> 24) | (e.y & 0xFFu))) *st |= TQ_DATA_BAD_PAD;
    e = nx;
  }
  if (bad & 0x100u) *st |= TQ_DATA_BAD_BYTE;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<uint4 *>(p + 16 * i) = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
}

__global__ void __launch_bounds__(32 * kCodecWarps) unpack_warp_kernel(int N, int K, const uint8_t *plane1,
                                                                     const uint8_t *plane2, const uint32_t *sal,
                                                                     const int32_t *rowptr, int8_t *T1, int8_t *T2,
                                                                     uint32_t *status) {
  __shared__ __align__(16) unsigned char stage[kCodecWarps][kStageBytesW];
  __shared__ __align__(16) uint2 lut[256];
  const int G = K / kGroup, W = sal_words_of(K), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t RB = row_bytes_of(K), total = (int64_t)N * G;
  const int64_t q0 = ((int64_t)blockIdx.x * kCodecWarps + warp) * 32;
  for (int v = threadIdx.x; v < 256; v += 32 * kCodecWarps) lut[v] = decode_entry(v);
  unsigned char *sm = stage[warp];
  const LaneGroup L = lane_group(q0, total, G, lane);
  const int64_t off = L.live ? L.n * RB + (int64_t)L.g * kGroupBytes : -1;
  uint16_t x[13];
  for_halfwords(off, lane, [&](int u, int64_t o) {
    x[u >> 5] = o >= 0 ? __ldcs(reinterpret_cast<const unsigned short *>(plane1 + o)) : (unsigned short)0;
  });
  const bool s = L.live && sal_bit(sal, W, L.n, L.g);
  const uint32_t smask = __ballot_sync(0xffffffffu, s);
  uint32_t st = L.live && L.g == 0 ? row_status(sal, rowptr, W, G, L.n) : 0u;
  if (L.live && L.g == G - 1)
    for (int64_t b = off + kGroupBytes; b < (L.n + 1) * RB; ++b)
      if (plane1[b] != 0) st |= TQ_DATA_BAD_PAD;
  __syncthreads();  // the table
  if (q0 >= total) return;
#pragma unroll
  for (int i = 0; i < 13; ++i) *reinterpret_cast<uint16_t *>(sm + 2 * (32 * i + lane)) = x[i];
  __syncwarp();
  uint16_t h[13];
#pragma unroll
  for (int j = 0; j < 13; ++j) h[j] = *reinterpret_cast<const uint16_t *>(sm + lane * kGroupBytes + 2 * j);
  __syncwarp();
  unsigned char *mine = sm + lane * kGroupStride;
  const unsigned char *part = sm + (lane >> 3) * kGroupStride + 16 * (lane & 7);
  uint32_t sd = 0;
  decode_group_codes(h, lut, mine, &sd);
  if (L.live) st |= sd;
  __syncwarp();
  const int64_t chunks = (total - q0) * 8;
  uint4 *d1 = reinterpret_cast<uint4 *>(T1 + q0 * kGroup), *d2 = reinterpret_cast<uint4 *>(T2 + q0 * kGroup);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (32 * i + lane < chunks) __stcs(d1 + 32 * i + lane, *reinterpret_cast<const uint4 *>(part + 4 * i * kGroupStride));
  if (T2) {
    // salient groups' records through shared memory, zeros elsewhere
    // (a record per lane; a byte per lane, record after record, took 5 us more)
    if (smask) {
      __syncwarp();
      if (s) {
        const int64_t j = (int64_t)rowptr[L.n] + sal_rank(sal, W, L.n, L.g);
        if (plane2 && j >= 0 && j < rowptr[N]) {
          const uint16_t *r = reinterpret_cast<const uint16_t *>(plane2 + j * kGroupBytes);
#pragma unroll
          for (int k = 0; k < 13; ++k) h[k] = __ldcs(r + k);
          decode_group_codes(h, lut, mine, &st);
        } else {
          st |= TQ_DATA_BAD_ROWPTR;
#pragma unroll
          for (int i = 0; i < 8; ++i) *reinterpret_cast<uint4 *>(mine + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool sg = (smask >> (4 * i + (lane >> 3))) & 1u;
      if (32 * i + lane < chunks)
        __stcs(d2 + 32 * i + lane,
               sg ? *reinterpret_cast<const uint4 *>(part + 4 * i * kGroupStride) : make_uint4(0u, 0u, 0u, 0u));
    }
  }
  st = __reduce_or_sync(0xffffffffu, st);
  if (st && lane == 0) atomicOr(status, st);
}

// ------------------------------------------------------ second-plane index
// One block per group g walks the rows in chunks of blockDim.x, in order;
// a block-wide count (and, for the fill, an exclusive scan of the row bits)
// gives each salient row its place in group g's list.  Group lists start at
// multiples of 16; the entries after a group's last pair, up to the next
// start, are empty.
constexpr int kIdxThreads = 256;

__host__ __device__ __forceinline__ int64_t p2index_capacity(int K, int64_t nnz) {
  return (nnz + 15 * (int64_t)(K / kGroup) + 15) & ~(int64_t)15;
}
__host__ __device__ __forceinline__ int64_t p2index_slot_off(int K) {
  return ((int64_t)(K / kGroup + 1) * 4 + 127) & ~(int64_t)127;
}

// The fill takes rows in chunks: block (g, c) handles group g's rows
// [chunk c, chunk (c + 1)), in rounds of its threads.  A chunk is one round up
// to 16384 rows (four rounds, with their block barriers, took 15 us for
// 4096 x 12288, this 13), and at most 64 chunks are taken, since each
// block counts the group's rows before its own.
static int p2index_chunk(int N) { return kIdxThreads * ((N + 64 * kIdxThreads - 1) / (64 * kIdxThreads)); }

// Salient rows of group g in rows [r0, r1) (the block's threads together;
// every thread gets the total).
__device__ __forceinline__ int p2index_block_count(const uint32_t *sal, int W, int g, int r0, int r1, int *red) {
  int c = 0;
  for (int n = r0 + (int)threadIdx.x; n < r1; n += kIdxThreads) c += sal_bit(sal, W, n, g);
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  int t = 0;
  for (int w = 0; w < kIdxThreads / 32; ++w) t += red[w];
  __syncthreads();
  return t;
}

// Rows of a counting block: one block per group, unless a weight has more
// rows (then the blocks add up, from zero).
constexpr int kIdxCountRows = 16384;

// colptr[g + 1] = salient rows of group g.
__global__ void __launch_bounds__(kIdxThreads) p2index_count_kernel(int N, int K, const uint32_t *sal,
                                                                     int32_t *colptr) {
  __shared__ int red[kIdxThreads / 32];
  const int g = blockIdx.x, r0 = blockIdx.y * kIdxCountRows;
  grid_dep_launch_next();
  grid_dep_wait();
  const int t = p2index_block_count(sal, sal_words_of(K), g, r0, min(N, r0 + kIdxCountRows), red);
  if (threadIdx.x == 0) {
    if (gridDim.y == 1)
      colptr[g + 1] = t;
    else
      atomicAdd(colptr + g + 1, t);
  }
}

__global__ void p2index_zero_kernel(int G, int32_t *colptr) {
  for (int i = threadIdx.x; i <= G; i += blockDim.x) colptr[i] = 0;
}

// colptr[g+1] = colptr[g] + count rounded up to 16, at most the capacity
// (which the counts of a consistent salience map never reach).  One warp.
__global__ void p2index_scan_kernel(int G, int64_t cap, int32_t *colptr) {
  const int lane = threadIdx.x;
  grid_dep_launch_next();
  grid_dep_wait();
  int64_t base = 0;
  for (int g0 = 0; g0 < G; g0 += 32) {
    const int g = g0 + lane;
    int64_t v = g < G ? ((int64_t)colptr[g + 1] + 15) & ~(int64_t)15 : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    v += base;
    if (g < G) colptr[g + 1] = (int32_t)min(v, cap);
    base = __shfl_sync(0xffffffffu, v, 31);
  }
  if (lane == 0) colptr[0] = 0;
}

// One slot: 8 words in the order of logical words 0, 4, 1, 5, 2, 6, 3, 7.
__device__ __forceinline__ void p2index_store_slot(uint8_t *slot, const uint32_t *L) {
  uint4 *d = reinterpret_cast<uint4 *>(slot);
  d[0] = make_uint4(L[0], L[4], L[1], L[5]);
  d[1] = make_uint4(L[2], L[6], L[3], L[7]);
}

__device__ __forceinline__ void p2index_empty_slot(uint8_t *slot) {
  const uint32_t L[8] = {0, 0, 0, 0, 0, 0, 0, 0xffffffffu};
  p2index_store_slot(slot, L);
}

// Entry e of group g: the record j of row n (plane 2 and s2 are 2-byte
// aligned at a record, so the record is read as 13 halves).
__device__ __forceinline__ void p2index_fill_slot(uint8_t *slot, int g, int n, int64_t j, int64_t nnz,
                                                  const uint8_t *plane2, const uint16_t *scale2) {
  if (j < 0 || j >= nnz) {
    p2index_empty_slot(slot);
    return;
  }
  uint32_t L[8] = {0, 0, 0, 0, 0, 0, 0, (uint32_t)n};
  const int h0 = (g % 8) & 1;  // the record starts at logical half h0 (byte o = 2 h0)
  const uint16_t *rec = reinterpret_cast<const uint16_t *>(plane2 + j * kGroupBytes);
#pragma unroll
  for (int i = 0; i < kGroupBytes / 2; ++i) {
    const int h = h0 + i;
    L[h >> 1] |= (uint32_t)rec[i] << (16 * (h & 1));
  }
  const int hs = h0 ? 0 : kGroupBytes / 2;  // s2 in the free half next to the record
  L[hs >> 1] |= (uint32_t)scale2[j] << (16 * (hs & 1));
  p2index_store_slot(slot, L);
}

// Block (g, c) fills the entries of group g's salient rows of chunk c
// (their place: colptr[g] plus the salient rows of the group's earlier
// chunks, counted by the block itself); the group's last chunk empties the
// slots after its last entry.  Block (G, 0) empties the slots from
// colptr[G] to the capacity.
__global__ void __launch_bounds__(kIdxThreads) p2index_fill_kernel(int N, int K, const uint32_t *sal,
                                                                    const int32_t *rowptr, int64_t nnz,
                                                                    const uint8_t *plane2, const uint16_t *scale2,
                                                                    int32_t *index, int chunk) {
  __shared__ int warp_base[kIdxThreads / 32 + 1];
  __shared__ int red[kIdxThreads / 32];
  const int G = K / kGroup, g = blockIdx.x, c = blockIdx.y, W = sal_words_of(K);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  grid_dep_wait();
  uint8_t *slots = reinterpret_cast<uint8_t *>(index) + p2index_slot_off(K);
  if (g == G) {
    if (c != 0) return;
    const int64_t cap = p2index_capacity(K, nnz);
    for (int64_t e = index[G] + threadIdx.x; e < cap; e += kIdxThreads) p2index_empty_slot(slots + 32 * e);
    return;
  }
  const int r0 = c * chunk, r1 = min(N, r0 + chunk);
  if (r0 >= N) return;
  const int64_t lim = index[g + 1];
  int64_t base = index[g] + p2index_block_count(sal, W, g, 0, r0, red);
  for (int n0 = r0; n0 < r1; n0 += kIdxThreads) {
    const int n = n0 + threadIdx.x;
    const bool bit = n < r1 && sal_bit(sal, W, n, g);
    const uint32_t m = __ballot_sync(0xffffffffu, bit);
    if (lane == 0) warp_base[warp] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
      int run = 0;
      for (int w = 0; w < kIdxThreads / 32; ++w) {
        const int cnt = warp_base[w];
        warp_base[w] = run;
        run += cnt;
      }
      warp_base[kIdxThreads / 32] = run;
    }
    __syncthreads();
    if (bit) {
      const int64_t pos = base + warp_base[warp] + __popc(m & ((1u << lane) - 1u));
      if (pos < lim) {  // within the group's entries (the capacity cuts an inconsistent map short)
        const int64_t j = (int64_t)rowptr[n] + sal_rank(sal, W, n, g);
        p2index_fill_slot(slots + 32 * pos, g, n, j, nnz, plane2, scale2);
      }
    }
    base += warp_base[kIdxThreads / 32];
    __syncthreads();
  }
  if (r1 == N)
    for (int64_t e = base + threadIdx.x; e < lim; e += kIdxThreads) p2index_empty_slot(slots + 32 * e);
}

// ------------------------------------------------------------- launchers
static int grid_for(int64_t work, int block) {
  int64_t g = (work + block - 1) / block;
  if (g > 152 * 32) g = 152 * 32;
  return (int)(g < 1 ? 1 : g);
}

// behind_smem: the stream's previous kernel may be one whose CTAs fill shared
// memory.  Beside them this one gets little of the SM's L1 cache, on which its
// strided reads live where a thread has more than 16 rows, so it then waits
// for their end: ternarizing 40000 x 128 took 92 us with an early start and
// takes 66 without (10 % salient 129 and 96).
cudaError_t launch_rowptr(int N, int K, const uint32_t *sal, int32_t *rowptr, uint32_t *status, bool behind_smem,
                          cudaStream_t s) {
  if (behind_smem && N > 16 * 1024) {
    rowptr_kernel<<<1, 1024, 0, s>>>(N, K, sal, rowptr, status);
    return cudaGetLastError();
  }
  return launch_dependent(rowptr_kernel, dim3(1), 1024, s, N, K, sal, rowptr, status);
}

cudaError_t launch_check_rowptr(int N, int K, const uint32_t *sal, const int32_t *rowptr,
                                uint32_t *status, cudaStream_t s) {
  check_rowptr_kernel<<<(N + 255) / 256, 256, 0, s>>>(N, K, sal, rowptr, status);
  return cudaGetLastError();
}

// Whether the warp-staged kernels take these arrays.
static bool warp_codec(int N, int K, const void *T1, const void *T2, const void *plane1, const void *plane2) {
  const int64_t warps = ((int64_t)N * (K / kGroup) + 31) / 32;
  return ((((uintptr_t)T1) | ((uintptr_t)T2)) & 15u) == 0 && ((((uintptr_t)plane1) | ((uintptr_t)plane2)) & 1u) == 0 &&
         (warps + kCodecWarps - 1) / kCodecWarps <= INT32_MAX;
}
static unsigned warp_codec_blocks(int N, int K) {
  return (unsigned)(((int64_t)N * (K / kGroup) + 32 * kCodecWarps - 1) / (32 * kCodecWarps));
}

// Both check the salience map against rowptr as they go (per row; the
// per-byte kernels by a kernel of its own in front).
cudaError_t launch_pack(int N, int K, const int8_t *T1, const int8_t *T2, const uint32_t *sal,
                        const int32_t *rowptr, uint8_t *plane1, uint8_t *plane2, uint32_t *status,
                        cudaStream_t s) {
  if (warp_codec(N, K, T1, T2, plane1, plane2)) {
    pack_warp_kernel<<<warp_codec_blocks(N, K), 32 * kCodecWarps, 0, s>>>(N, K, T1, T2, sal, rowptr, plane1, plane2,
                                                                         status);
    return cudaGetLastError();
  }
  if (cudaError_t e = launch_check_rowptr(N, K, sal, rowptr, status, s)) return e;
  pack_kernel<<<std::min(N, 152 * 16), 256, 0, s>>>(N, K, T1, T2, sal, rowptr, plane1, plane2, status);
  return cudaGetLastError();
}

cudaError_t launch_unpack(int N, int K, const uint8_t *plane1, const uint8_t *plane2,
                          const uint32_t *sal, const int32_t *rowptr, int8_t *T1, int8_t *T2,
                          uint32_t *status, cudaStream_t s) {
  if (warp_codec(N, K, T1, T2, plane1, plane2)) {
    unpack_warp_kernel<<<warp_codec_blocks(N, K), 32 * kCodecWarps, 0, s>>>(N, K, plane1, plane2, sal, rowptr, T1, T2,
                                                                           status);
    return cudaGetLastError();
  }
  if (cudaError_t e = launch_check_rowptr(N, K, sal, rowptr, status, s)) return e;
  unpack_kernel<<<std::min(N, 152 * 16), 256, 0, s>>>(N, K, plane1, plane2, sal, rowptr, T1, T2,
                                                     status);
  return cudaGetLastError();
}

cudaError_t launch_plane2_index(int N, int K, const uint32_t *sal, const int32_t *rowptr, int64_t nnz,
                                const uint8_t *plane2, const uint16_t *scale2, int32_t *index, cudaStream_t s) {
  const int G = K / kGroup, chunk = p2index_chunk(N), C = (N + kIdxCountRows - 1) / kIdxCountRows;
  cudaError_t e;
  if (C > 1) {
    p2index_zero_kernel<<<1, 256, 0, s>>>(G, index);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if ((e = launch_dependent(p2index_count_kernel, dim3(G, C), kIdxThreads, s, N, K, sal, index)) != cudaSuccess) return e;
  if ((e = launch_dependent(p2index_scan_kernel, dim3(1), 32, s, G, p2index_capacity(K, nnz), index)) != cudaSuccess)
    return e;
  return launch_dependent(p2index_fill_kernel, dim3(G + 1, (N + chunk - 1) / chunk), kIdxThreads, s, N, K, sal, rowptr,
                          nnz, plane2, scale2, index, chunk);
}

// ------------------------------------------ element-wise four-mask format
// The paper's representation with four disjoint masks of orders [2, 2, 1, 1]
// ("Model and Representation"), stored as: a 2-bit mask-id plane (element k
// of row n in bits 2 (k mod 16) of word [n][k / 16]); T0 of every element in
// plane 1's group layout (the codec above); per row, the T1 trits of its
// order-2 elements (masks 0 and 1) in increasing k, five per byte, the last
// byte padded with digit 1, row n's bytes from byte rowptr[n].
constexpr int kEwRowWarps = 4;  // rows (warps) per block of the per-row kernels

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Warp per row: plane-2 bytes of the row (ceil(order-2 elements / 5)) into
// rowptr[n + 1]; mask ids above 3 set BAD_CODE.
__global__ void __launch_bounds__(32 * kEwRowWarps) ew_count_kernel(int N, int K, const uint8_t *mask,
                                                                   int32_t *rowptr, uint32_t *status) {
  const int lane = threadIdx.x & 31;
  const int n = blockIdx.x * kEwRowWarps + (threadIdx.x >> 5);
  if (n >= N) return;
  const uint8_t *row = mask + (int64_t)n * K;
  int c = 0;
  uint32_t st = 0;
  for (int k = lane; k < K; k += 32) {
    const uint8_t m = row[k];
    c += m <= 1;
    if (m > 3) st |= TQ_DATA_BAD_CODE;
  }
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) {
    rowptr[n + 1] = (c + 4) / 5;
    if (n == 0) rowptr[0] = 0;
    if (st) atomicOr(status, st);
  }
}

// One block: rowptr[1..N] (bytes per row) into offsets, in place.
__global__ void __launch_bounds__(1024) ew_scan_kernel(int N, int32_t *rowptr) {
  __shared__ int32_t part[1024];
  const int t = threadIdx.x;
  const int r0 = (int)((int64_t)N * t / 1024), r1 = (int)((int64_t)N * (t + 1) / 1024);
  int32_t sum = 0;
  for (int n = r0; n < r1; ++n) sum += rowptr[n + 1];
  part[t] = sum;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int32_t v = t >= o ? part[t - o] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  int32_t run = part[t] - sum;  // exclusive prefix of this thread's rows
  for (int n = r0; n < r1; ++n) {
    run += rowptr[n + 1];
    rowptr[n + 1] = run;
  }
}

// Thread per mask word.
__global__ void ew_mask_pack_kernel(int N, int K, const uint8_t *mask, uint32_t *plane, uint32_t *status) {
  const int64_t total = (int64_t)N * (K / 16);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t *src = mask + i * 16;
    uint32_t w = 0, st = 0;
    for (int j = 0; j < 16; ++j) {
      uint32_t m = src[j];
      if (m > 3) st |= TQ_DATA_BAD_CODE, m = 3;
      w |= m << (2 * j);
    }
    plane[i] = w;
    if (st) atomicOr(status, st);
  }
}

// Thread per plane-1 byte: T0 of every element (the group layout).
__global__ void ew_plane1_pack_kernel(int N, int K, const int8_t *T0, uint8_t *plane1, uint32_t *status) {
  const int G = K / kGroup;
  const int64_t RB = row_bytes_of(K), total = (int64_t)N * RB;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(idx / RB), b = (int)(idx - (int64_t)n * RB);
    if (b >= G * kGroupBytes) {
      plane1[idx] = 0;
      continue;
    }
    uint32_t st = 0;
    const int g = b / kGroupBytes, pos = b - g * kGroupBytes;
    plane1[idx] = encode_codes(T0 + (int64_t)n * K + (int64_t)g * kGroup + 5 * pos, pos < kFullBytes ? 5 : kTailTrits, &st);
    if (st) atomicOr(status, st);
  }
}

// Warp per row: the row's order-2 T1 trits in order, five per byte.  Each
// 32-element chunk ranks its order-2 elements by ballot; their digits join
// the (fewer than 5) left over from earlier chunks in a per-warp ring, whole
// bytes are written, the rest carried on.
__global__ void __launch_bounds__(32 * kEwRowWarps) ew_plane2_pack_kernel(int N, int K, const int8_t *T1,
                                                                         const uint8_t *mask, const int32_t *rowptr,
                                                                         uint8_t *plane2, uint32_t *status) {
  __shared__ uint8_t dig[kEwRowWarps][40];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int n = blockIdx.x * kEwRowWarps + wi;
  if (n >= N) return;
  uint8_t *d = dig[wi];
  const int8_t *t1 = T1 + (int64_t)n * K;
  const uint8_t *mk = mask + (int64_t)n * K;
  const int64_t b0 = rowptr[n], nb = (int64_t)rowptr[n + 1] - rowptr[n];
  int pend = 0;   // digits carried into this chunk
  int64_t out = 0;  // bytes written
  uint32_t st = 0;
  for (int k0 = 0; k0 < K; k0 += 32) {
    const int k = k0 + lane;
    const bool in = k < K;
    const bool o2 = in && mk[k] <= 1;
    int c = in ? t1[k] : 0;
    if (c < -1 || c > 1) st |= TQ_DATA_BAD_CODE, c = c < -1 ? -1 : 1;
    if (in && !o2 && c != 0) st |= TQ_DATA_T2_OUTSIDE;
    const uint32_t bal = __ballot_sync(0xffffffffu, o2);
    if (o2) d[pend + __popc(bal & lanemask_lt())] = (uint8_t)(c + 1);
    __syncwarp();
    const int tot = pend + __popc(bal), full = tot / 5, rem = tot - 5 * full;
    if (lane < full) {
      const uint8_t *q = d + 5 * lane;
      const int v = q[0] + 3 * q[1] + 9 * q[2] + 27 * q[3] + 81 * q[4];
      if (out + lane < nb) plane2[b0 + out + lane] = (uint8_t)v;
    }
    const uint8_t carry = lane < rem ? d[5 * full + lane] : 0;
    __syncwarp();
    if (lane < rem) d[lane] = carry;
    __syncwarp();
    out += full;
    pend = rem;
  }
  if (pend > 0 && lane == 0) {
    int v = 0, p = 1;
    for (int i = 0; i < 5; ++i, p *= 3) v += (i < pend ? d[i] : 1) * p;
    if (out < nb) plane2[b0 + out] = (uint8_t)v;
    ++out;
  }
  if (lane == 0 && out != nb) st |= TQ_DATA_BAD_ROWPTR;
  if (st) atomicOr(status, st);
}

// Thread per mask word: mask ids back.
__global__ void ew_mask_unpack_kernel(int N, int K, const uint32_t *plane, uint8_t *mask) {
  const int64_t total = (int64_t)N * (K / 16);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t w = plane[i];
    for (int j = 0; j < 16; ++j) mask[i * 16 + j] = (uint8_t)((w >> (2 * j)) & 3u);
  }
}

// Thread per plane-1 byte: T0 back (pad bytes must be 0).
__global__ void ew_plane1_unpack_kernel(int N, int K, const uint8_t *plane1, int8_t *T0, uint32_t *status) {
  const int G = K / kGroup;
  const int64_t RB = row_bytes_of(K), total = (int64_t)N * RB;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(idx / RB), b = (int)(idx - (int64_t)n * RB);
    const uint8_t v = plane1[idx];
    if (b >= G * kGroupBytes) {
      if (v != 0) atomicOr(status, TQ_DATA_BAD_PAD);
      continue;
    }
    uint32_t st = 0;
    const int g = b / kGroupBytes, pos = b - g * kGroupBytes;
    decode_to(v, pos < kFullBytes ? 5 : kTailTrits, T0 + (int64_t)n * K + (int64_t)g * kGroup + 5 * pos, &st);
    if (st) atomicOr(status, st);
  }
}

// Warp per row: T1 back from plane 2 (zeros on order-1 elements); bytes
// above 242 and pad digits other than 1 in the row's last byte are flagged.
__global__ void __launch_bounds__(32 * kEwRowWarps) ew_plane2_unpack_kernel(int N, int K, const uint32_t *plane,
                                                                           const int32_t *rowptr,
                                                                           const uint8_t *plane2, int8_t *T1,
                                                                           uint32_t *status) {
  const int lane = threadIdx.x & 31;
  const int n = blockIdx.x * kEwRowWarps + (threadIdx.x >> 5);
  if (n >= N) return;
  const int64_t b0 = rowptr[n], nb = (int64_t)rowptr[n + 1] - rowptr[n];
  const uint32_t *mw = plane + (int64_t)n * (K / 16);
  int base = 0;
  uint32_t st = 0;
  for (int k0 = 0; k0 < K; k0 += 32) {
    const int k = k0 + lane;
    const bool in = k < K;
    const bool o2 = in && ((mw[k >> 4] >> (2 * (k & 15))) & 3u) <= 1;
    const uint32_t bal = __ballot_sync(0xffffffffu, o2);
    int8_t t = 0;
    if (o2) {
      const int r = base + __popc(bal & lanemask_lt());
      if (r / 5 < nb) {
        int v = plane2[b0 + r / 5];
        if (v > 242) st |= TQ_DATA_BAD_BYTE, v = 0;
        for (int i = 0; i < r % 5; ++i) v /= 3;
        t = (int8_t)(v % 3 - 1);
      } else {
        st |= TQ_DATA_BAD_ROWPTR;
      }
    }
    if (in) T1[(int64_t)n * K + k] = t;
    base += __popc(bal);
  }
  if (lane == 0) {
    if ((base + 4) / 5 != nb) st |= TQ_DATA_BAD_ROWPTR;
    if (base % 5 && nb > 0 && (base + 4) / 5 == nb) {
      int v = plane2[b0 + nb - 1];
      if (v <= 242) {
        for (int i = 0; i < 5; ++i, v /= 3)
          if (i >= base % 5 && v % 3 != 1) st |= TQ_DATA_BAD_PAD;
      }
    }
  }
  if (st) atomicOr(status, st);
}

// ----------------------------------------------- element-wise correction index
// Entries of masks 0..2 per row and 2048-element block (uint16
// (k mod 2048) | code << 11, code = 9 q + 3 (T0 + 1) + (T1 + 1)), with int32
// offsets[n nb + b] (nb = ceil(K / 2048)).
constexpr int kIdxBlock = 2048, kIdxShift = 11;

// Warp per row: the count of each block's mask-0..2 elements into
// off[n nb + b + 1] (off[0] = 0); ew_scan_kernel turns them into offsets.
__global__ void __launch_bounds__(32 * kEwRowWarps) ew_index_count_kernel(int N, int K, const uint32_t *plane,
                                                                          int32_t *off) {
  const int lane = threadIdx.x & 31;
  const int n = blockIdx.x * kEwRowWarps + (threadIdx.x >> 5);
  if (n >= N) return;
  const int WK = K / 16, nb = (K + kIdxBlock - 1) / kIdxBlock;
  const uint32_t *mw = plane + (int64_t)n * WK;
  for (int b = 0; b < nb; ++b) {
    int c = 0;
    for (int wi = b * (kIdxBlock / 16) + lane; wi < min(WK, (b + 1) * (kIdxBlock / 16)); wi += 32) {
      const uint32_t m = mw[wi];
      c += __popc(~(m & (m >> 1)) & 0x55555555u);
    }
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) off[(int64_t)n * nb + b + 1] = c;
  }
  if (n == 0 && lane == 0) off[0] = 0;
}

__device__ __forceinline__ int base3_digit(int v, int i) {
  for (int j = 0; j < i; ++j) v /= 3;
  return v % 3;
}

// Warp per row, 32 elements per step (lane = element): each mask-0..2
// element's entry at its rank in the row; T0 from plane 1, T1 from plane 2
// at the element's rank among the row's order-2 elements.  A row whose
// offsets or plane-2 rowptr do not match its mask plane is skipped and
// reported (TQ_DATA_BAD_ROWPTR), so nothing is written outside its range.
__global__ void __launch_bounds__(32 * kEwRowWarps) ew_index_fill_kernel(int N, int K, const uint32_t *plane,
                                                                         const uint8_t *plane1,
                                                                         const int32_t *rowptr,
                                                                         const uint8_t *plane2, const int32_t *off,
                                                                         uint16_t *idx, uint32_t *status) {
  const int lane = threadIdx.x & 31;
  const int n = blockIdx.x * kEwRowWarps + (threadIdx.x >> 5);
  if (n >= N) return;
  const int WK = K / 16, nb = (K + kIdxBlock - 1) / kIdxBlock;
  const uint32_t *mw = plane + (int64_t)n * WK;
  const int64_t e0 = off[(int64_t)n * nb];
  int c3 = 0, c2 = 0;
  for (int wi = lane; wi < WK; wi += 32) {
    const uint32_t m = mw[wi];
    c3 += __popc(~(m & (m >> 1)) & 0x55555555u);
    c2 += __popc(~m & 0xaaaaaaaau);
  }
  for (int o = 16; o; o >>= 1) {
    c3 += __shfl_xor_sync(0xffffffffu, c3, o);
    c2 += __shfl_xor_sync(0xffffffffu, c2, o);
  }
  const int64_t b2 = rowptr[n], nb2 = (int64_t)rowptr[n + 1] - rowptr[n];
  if ((int64_t)off[(int64_t)n * nb + nb] - e0 != c3 || (c2 + 4) / 5 != nb2) {
    if (lane == 0) atomicOr(status, TQ_DATA_BAD_ROWPTR);
    return;
  }
  const uint8_t *p1 = plane1 + (int64_t)n * row_bytes_of(K);
  uint32_t st = 0;
  int run = 0, r2 = 0;
  for (int k0 = 0; k0 < K; k0 += 32) {
    if (k0 % kIdxBlock == 0 && run != (int)(off[(int64_t)n * nb + k0 / kIdxBlock] - e0)) {
      st |= TQ_DATA_BAD_ROWPTR;  // per-block offsets that do not match the mask plane
      break;
    }
    const int k = k0 + lane;
    const uint32_t q = k < K ? (mw[k >> 4] >> (2 * (k & 15))) & 3u : 3u;
    const uint32_t bal3 = __ballot_sync(0xffffffffu, q != 3u), bal2 = __ballot_sync(0xffffffffu, q <= 1u);
    if (q != 3u) {
      const int kg = k % kGroup;
      int v = p1[(int64_t)(k / kGroup) * kGroupBytes + kg / 5];
      if (v > 242) st |= TQ_DATA_BAD_BYTE, v = 242;
      const int d0 = base3_digit(v, kg % 5);
      int d1 = 1;
      if (q <= 1u) {
        const int r = r2 + __popc(bal2 & lanemask_lt());
        int u = plane2[b2 + r / 5];
        if (u > 242) st |= TQ_DATA_BAD_BYTE, u = 242;
        d1 = base3_digit(u, r % 5);
      }
      const uint32_t code = 9u * q + 3u * (uint32_t)d0 + (uint32_t)d1;
      idx[e0 + run + __popc(bal3 & lanemask_lt())] = (uint16_t)((uint32_t)(k % kIdxBlock) | (code << kIdxShift));
    }
    run += __popc(bal3);
    r2 += __popc(bal2);
  }
  for (int o = 16; o; o >>= 1) st |= __shfl_xor_sync(0xffffffffu, st, o);
  if (lane == 0 && st) atomicOr(status, st);
}

cudaError_t launch_ew_index_offsets(int N, int K, const uint32_t *mplane, int32_t *off, cudaStream_t s) {
  const int nb = (K + kIdxBlock - 1) / kIdxBlock;
  ew_index_count_kernel<<<(N + kEwRowWarps - 1) / kEwRowWarps, 32 * kEwRowWarps, 0, s>>>(N, K, mplane, off);
  ew_scan_kernel<<<1, 1024, 0, s>>>(N * nb, off);
  return cudaGetLastError();
}

cudaError_t launch_ew_index_fill(int N, int K, const uint32_t *mplane, const uint8_t *plane1, const int32_t *rowptr,
                                 const uint8_t *plane2, const int32_t *off, uint16_t *idx, uint32_t *status,
                                 cudaStream_t s) {
  ew_index_fill_kernel<<<(N + kEwRowWarps - 1) / kEwRowWarps, 32 * kEwRowWarps, 0, s>>>(N, K, mplane, plane1, rowptr,
                                                                                       plane2, off, idx, status);
  return cudaGetLastError();
}

cudaError_t launch_ew_rowptr(int N, int K, const uint8_t *mask, int32_t *rowptr, uint32_t *status, cudaStream_t s) {
  ew_count_kernel<<<(N + kEwRowWarps - 1) / kEwRowWarps, 32 * kEwRowWarps, 0, s>>>(N, K, mask, rowptr, status);
  ew_scan_kernel<<<1, 1024, 0, s>>>(N, rowptr);
  return cudaGetLastError();
}

cudaError_t launch_ew_pack(int N, int K, const int8_t *T0, const int8_t *T1, const uint8_t *mask,
                           const int32_t *rowptr, uint32_t *mplane, uint8_t *plane1, uint8_t *plane2,
                           uint32_t *status, cudaStream_t s) {
  ew_mask_pack_kernel<<<grid_for((int64_t)N * (K / 16), 256), 256, 0, s>>>(N, K, mask, mplane, status);
  ew_plane1_pack_kernel<<<grid_for((int64_t)N * row_bytes_of(K), 256), 256, 0, s>>>(N, K, T0, plane1, status);
  ew_plane2_pack_kernel<<<(N + kEwRowWarps - 1) / kEwRowWarps, 32 * kEwRowWarps, 0, s>>>(N, K, T1, mask, rowptr,
                                                                                        plane2, status);
  return cudaGetLastError();
}

cudaError_t launch_ew_unpack(int N, int K, const uint32_t *mplane, const uint8_t *plane1, const int32_t *rowptr,
                             const uint8_t *plane2, int8_t *T0, int8_t *T1, uint8_t *mask, uint32_t *status,
                             cudaStream_t s) {
  ew_mask_unpack_kernel<<<grid_for((int64_t)N * (K / 16), 256), 256, 0, s>>>(N, K, mplane, mask);
  ew_plane1_unpack_kernel<<<grid_for((int64_t)N * row_bytes_of(K), 256), 256, 0, s>>>(N, K, plane1, T0, status);
  ew_plane2_unpack_kernel<<<(N + kEwRowWarps - 1) / kEwRowWarps, 32 * kEwRowWarps, 0, s>>>(N, K, mplane, rowptr,
                                                                                          plane2, T1, status);
  return cudaGetLastError();
}

}  // namespace tq
