// pipe_expand_weights: residual expansion of a weight matrix (Sec. 3.1, Eq. 2-3 and the masked
// form), with the per-channel symmetric quantizer of Eq. 1.
//
// Most layers: one pass over W that quantizes every row K times in registers, one block that decides which order keeps
// which group, one copy of the kept rows' codes to their orders (expand_chain_kernel and behind it).
// Masks over single weights, the L2 score and row lengths that path does not take, per order: [group select, orders >= 2]
// -> one fused pass over the kept rows that (order 1: finds the row maximum,) divides, rounds, packs both code layouts,
// updates the residual with one FMA per element and leaves the next order's row absmax behind: streaming passes,
// 128-bit loads, warp-shuffle reductions, one block per row.
#include <cstring>
#include <mutex>

#include "pipe_common.cuh"

namespace pipe {

constexpr int kRowThreads = 256;

__device__ __forceinline__ uint32_t warp_max_u32(uint32_t v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}

// Max over the block of an unsigned value; result valid in every thread.
__device__ __forceinline__ uint32_t block_max_u32(uint32_t v) {
  __shared__ uint32_t part[32];
  __shared__ uint32_t total;
  v = warp_max_u32(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) part[warp] = v;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < (blockDim.x + 31) / 32 ? part[lane] : 0u;
    w = warp_max_u32(w);
    if (lane == 0) total = w;
  }
  __syncthreads();
  const uint32_t r = total;
  __syncthreads();
  return r;
}

// |v| as an ordered unsigned key: for finite floats the order of the keys is the order of the
// magnitudes, and every Inf/NaN maps to a key >= 0x7f800000.
__device__ __forceinline__ uint32_t abs_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// score[j] = max over the g rows of group j of a[] ; one thread per group.
__global__ void group_score_kernel(const float* __restrict__ a, int G, int g, float* __restrict__ score) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= G) return;
  float m = 0.f;
  for (int u = 0; u < g; ++u) m = fmaxf(m, a[static_cast<int64_t>(j) * g + u]);
  score[j] = m;
}

// keep[j] = 1 iff fewer than n_keep groups precede j in the order (score descending, index
// ascending).  Scores are non-negative finite floats, so the comparison is exact and the
// result does not depend on any reduction order.
template <typename S>
__global__ void group_rank_kernel(const S* __restrict__ score, int G, int n_keep, int32_t* __restrict__ keep) {
  // one warp per group: its lanes share the G comparisons (a count, so the order of the additions does not matter)
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (j >= G) return;
  const S sj = score[j];
  int rank = 0;
  for (int t = lane; t < G; t += 32) {
    const S si = score[t];
    rank += (si > sj) || (si == sj && t < j);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, d);
  if (lane == 0) keep[j] = rank < n_keep ? 1 : 0;
}

// Second score of the structured mask (PIPE_SCORE_L2): the squared Euclidean norm of the group's residual rows in
// binary64, with the order of the additions fixed as include/pipe.h states it so that the kept lists can be compared
// bit for bit: one warp per row, lane l sums the squares of the elements l, l + 32, ... in ascending order (a square
// of a binary32 value is exact in binary64), then the 32 partial sums are added as a tree with offsets 16, 8, 4, 2, 1.
__global__ void __launch_bounds__(256) row_sumsq_kernel(const float* __restrict__ r, int64_t ld, int O, int I, double* __restrict__ rowsq) {
  const int o = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (o >= O) return;
  const float* row = r + static_cast<int64_t>(o) * ld;
  double s = 0.0;
  for (int i = lane; i < I; i += 32) {
    const double v = static_cast<double>(row[i]);
    s = __dadd_rn(s, __dmul_rn(v, v));
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s = __dadd_rn(s, __shfl_down_sync(0xffffffffu, s, off));
  if (lane == 0) rowsq[o] = s;
}

// score[j] = sum over the group's rows, ascending, of rowsq; one thread per group.
__global__ void group_score_l2_kernel(const double* __restrict__ rowsq, int G, int g, double* __restrict__ score) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= G) return;
  double s = 0.0;
  for (int u = 0; u < g; ++u) s = __dadd_rn(s, rowsq[static_cast<int64_t>(j) * g + u]);
  score[j] = s;
}

// Unstructured mask (pipe_layer_desc::keep_elems): per row, the magnitude key of the n-th largest entry of the
// residual and the index up to which entries EQUAL to it are kept (ties go to the lower index).  One block per row:
// a radix select over the four bytes of the key, then a bisection on the index among the ties.  An entry i of the
// row is kept iff key_i > thr, or key_i == thr and i <= tie_cut.
__global__ void __launch_bounds__(256) row_topn_kernel(const float* __restrict__ r, int64_t ld, int I, int n,
                                                       uint32_t* __restrict__ thr_out, int32_t* __restrict__ cut_out) {
  __shared__ int hist[256];
  __shared__ uint32_t sh_prefix;
  __shared__ int sh_remaining, sh_count;
  const float* row = r + static_cast<int64_t>(blockIdx.x) * ld;
  uint32_t prefix = 0, mask = 0;
  int remaining = n;
  for (int shift = 24; shift >= 0; shift -= 8) {
    hist[threadIdx.x] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < I; i += blockDim.x) {
      const uint32_t k = abs_key(row[i]);
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 0xffu], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int b = 255, rem = remaining;
      while (b > 0 && hist[b] < rem) rem -= hist[b--];   // the bin that holds the rem-th largest of the candidates
      sh_prefix = prefix | (static_cast<uint32_t>(b) << shift);
      sh_remaining = rem;
    }
    __syncthreads();
    prefix = sh_prefix;
    remaining = sh_remaining;
    mask |= 0xffu << shift;
    __syncthreads();
  }
  // `remaining` of the entries equal to prefix are kept: the smallest index c such that #{i <= c : key_i == prefix} = remaining
  int lo = 0, hi = I - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (threadIdx.x == 0) sh_count = 0;
    __syncthreads();
    int c = 0;
    for (int i = threadIdx.x; i <= mid; i += blockDim.x) c += abs_key(row[i]) == prefix;
    if (c) atomicAdd(&sh_count, c);
    __syncthreads();
    const int total = sh_count;
    __syncthreads();
    if (total >= remaining) hi = mid;
    else lo = mid + 1;
  }
  if (threadIdx.x == 0) {
    thr_out[blockIdx.x] = prefix;
    cut_out[blockIdx.x] = lo;
  }
}

// Exclusive prefix sum of keep[] -> cum[0..G], and the ascending list of kept groups.
// keep == nullptr means "all groups kept".  Single block of 1024 threads.
__global__ void __launch_bounds__(1024) group_compact_kernel(const int32_t* __restrict__ keep, int G,
                                                             int32_t* __restrict__ cum, int32_t* __restrict__ kept) {
  __shared__ int32_t chunk_sum[1024];
  const int per = (G + blockDim.x - 1) / blockDim.x;
  const int b = threadIdx.x * per, e = min(G, b + per);
  int32_t s = 0;
  for (int j = b; j < e; ++j) s += keep ? keep[j] : 1;
  chunk_sum[threadIdx.x] = s;
  __syncthreads();
  // inclusive Hillis-Steele scan over the chunk sums
  for (int d = 1; d < blockDim.x; d <<= 1) {
    int32_t v = threadIdx.x >= d ? chunk_sum[threadIdx.x - d] : 0;
    __syncthreads();
    chunk_sum[threadIdx.x] += v;
    __syncthreads();
  }
  int32_t run = threadIdx.x == 0 ? 0 : chunk_sum[threadIdx.x - 1];
  for (int j = b; j < e; ++j) {
    cum[j] = run;
    if (!keep || keep[j]) kept[run++] = j;
  }
  if (threadIdx.x == blockDim.x - 1) cum[G] = chunk_sum[blockDim.x - 1];
}

// Group selection of one order in ONE block, for layers of up to kFusedGroups groups: scores, ranks and
// the compacted list stay in shared memory (three tiny launches less per sparse order).  Same rule and
// same exact comparisons as the three kernels above.
constexpr int kFusedGroups = 512;   // one group per thread; a power of two (the sorting network's size)
__global__ void __launch_bounds__(kFusedGroups) group_select_kernel(const float* __restrict__ a, int G, int g, int n_keep,
                                                            int32_t* __restrict__ cum, int32_t* __restrict__ kept) {
  // Rank = position in the order (score descending, index ascending), found by sorting the keys
  // (score bits, ~index) in descending order: scores are non-negative floats, whose order is the order of their bit
  // patterns, so the keys are distinct integers and the sorted order is unique (a bitonic network of 45 rounds over
  // the 512 slots; slots beyond G hold the smallest key and end up last).
  __shared__ unsigned long long key[kFusedGroups];
  __shared__ int32_t flag[kFusedGroups];
  __shared__ int32_t chunk_sum[kFusedGroups];
  const int tid = threadIdx.x;
  {
    unsigned long long kv = 0ull;
    if (tid < G) {
      // the group's row maxima: independent loads (four at a time where the rows allow vector loads)
      const float* rows = a + static_cast<int64_t>(tid) * g;
      float m0 = 0.f, m1 = 0.f, m2 = 0.f, m3 = 0.f;
      int u = 0;
      if ((g & 3) == 0 && (reinterpret_cast<uintptr_t>(rows) & 15) == 0) {
#pragma unroll 4
        for (; u < g; u += 4) {
          const float4 v = *reinterpret_cast<const float4*>(rows + u);
          m0 = fmaxf(m0, v.x);
          m1 = fmaxf(m1, v.y);
          m2 = fmaxf(m2, v.z);
          m3 = fmaxf(m3, v.w);
        }
      }
#pragma unroll 4
      for (; u < g; ++u) m0 = fmaxf(m0, rows[u]);
      const float m = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
      kv = (static_cast<unsigned long long>(__float_as_uint(m)) << 32) | (0xffffffffu - static_cast<uint32_t>(tid));
    }
    key[tid] = kv;
  }
  __syncthreads();
  for (int k = 2; k <= kFusedGroups; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      const int other = tid ^ j;
      if (other > tid) {
        const unsigned long long x = key[tid], y = key[other];
        const bool descending = (tid & k) == 0;
        if (descending ? x < y : x > y) {
          key[tid] = y;
          key[other] = x;
        }
      }
      __syncthreads();
    }
  }
  if (tid < G) flag[0xffffffffu - static_cast<uint32_t>(key[tid])] = tid < n_keep ? 1 : 0;
  __syncthreads();
  const int per = (G + blockDim.x - 1) / blockDim.x;
  const int b = threadIdx.x * per, e = min(G, b + per);
  int32_t sum = 0;
  for (int j = b; j < e; ++j) sum += flag[j];
  chunk_sum[threadIdx.x] = sum;
  __syncthreads();
  for (int d = 1; d < blockDim.x; d <<= 1) {
    int32_t v = threadIdx.x >= d ? chunk_sum[threadIdx.x - d] : 0;
    __syncthreads();
    chunk_sum[threadIdx.x] += v;
    __syncthreads();
  }
  int32_t run = threadIdx.x == 0 ? 0 : chunk_sum[threadIdx.x - 1];
  for (int j = b; j < e; ++j) {
    cum[j] = run;
    if (flag[j]) kept[run++] = j;
  }
  if (threadIdx.x == blockDim.x - 1) cum[G] = chunk_sum[blockDim.x - 1];
}

// Pack 16 codes (each already in [-qmax, qmax]) into the canonical and the kernel layout.
// canonical: field e at bit e*b of the stream; kernel: see include/pipe.h.
template <int BITS>
__device__ __forceinline__ void pack16(const int (&q)[16], uint32_t (&canon)[4], uint32_t (&kern)[4]) {
  if (BITS == 8) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      uint32_t v = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) v |= (static_cast<uint32_t>(q[4 * w + e]) & 0xffu) << (8 * e);
      canon[w] = v;
      kern[w] = v;
    }
  } else if (BITS == 4) {
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      uint32_t c = 0, k = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t f = static_cast<uint32_t>(q[8 * w + e]) & 0xfu;
        c |= f << (4 * e);
        const int h = e >> 2, j = e & 3;  // code 4h+j -> nibble 2j+h
        k |= f << (4 * (2 * j + h));
      }
      canon[w] = c;
      kern[w] = k;
    }
  } else {
    uint32_t c = 0, k = 0;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const uint32_t f = static_cast<uint32_t>(q[e]) & 0x3u;
      c |= f << (2 * e);
      const int h = e >> 2, j = e & 3;  // code 4h+j -> bits 8j+2h
      k |= f << (8 * j + 2 * h);
    }
    canon[0] = c;
    kern[0] = k;
  }
}

struct QuantizeRowsArgs {
  const float* src;      // residual entering this order ([O, ld_src])
  int64_t ld_src;
  float* dst;            // residual leaving this order ([O, ld_dst]) or nullptr (last order)
  int64_t ld_dst;
  float* a;              // [O] row absmax: read (this order's), overwritten (next order's) if dst
  int first;             // order 1: the row maximum is not in a[] yet, the block finds it itself
  int* status;
  const int32_t* kept;   // [rows/g] ascending kept groups
  uint8_t* codes;        // canonical [rows, canon_row_bytes]
  uint8_t* kcodes;       // streaming layout [ceil(I/128), rows, 128*BITS/8]
  uint8_t* wcodes;       // int8 copy in the tensor-core operand layout [ceil(I/128), rows, 128] or nullptr (see pipe.h)
  int rows;              // compacted rows of this order
  float* scales;         // [rows]
  int I, g, qmax;
  int canon_row_bytes, kernel_row_bytes;
  const uint32_t* mask_thr;   // unstructured mask of this order, per ORIGINAL row (nullptr: every entry is kept):
  const int32_t* mask_cut;    // an entry is kept iff its magnitude key > thr, or == thr and its index <= cut
};

// One block per compacted row: Eq. 1 on the residual, then the residual update of Eq. 3.
template <int BITS>
__global__ void __launch_bounds__(kRowThreads, 5) quantize_rows_kernel(const QuantizeRowsArgs p) {
  const int n = blockIdx.x;
  const int o = p.kept[n / p.g] * p.g + n % p.g;
  const float* src = p.src + static_cast<int64_t>(o) * p.ld_src;
  float* dst = p.dst ? p.dst + static_cast<int64_t>(o) * p.ld_dst : nullptr;
  const float fq = static_cast<float>(p.qmax);
  float amax;
  if (p.first) {
    // order 1 (Eq. 1 on W itself): one more pass over the row, which the second pass then finds in cache
    uint32_t mk = 0;
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
      const int n4 = p.I >> 2;
      const float4* r4 = reinterpret_cast<const float4*>(src);
      for (int i = threadIdx.x; i < n4; i += blockDim.x) {
        const float4 v = r4[i];
        mk = max(max(mk, abs_key(v.x)), max(abs_key(v.y), max(abs_key(v.z), abs_key(v.w))));
      }
      for (int i = (n4 << 2) + threadIdx.x; i < p.I; i += blockDim.x) mk = max(mk, abs_key(src[i]));
    } else {
      for (int i = threadIdx.x; i < p.I; i += blockDim.x) mk = max(mk, abs_key(src[i]));
    }
    mk = block_max_u32(mk);
    if (threadIdx.x == 0 && mk >= 0x7f800000u) raise_status(p.status, PIPE_ERR_NONFINITE);
    amax = __uint_as_float(mk);
  } else {
    amax = p.a[o];
  }
  const float s = __fdiv_rn(amax, fq);
  const bool masked = p.mask_thr != nullptr;
  const uint32_t mthr = masked ? p.mask_thr[o] : 0u;
  const int mcut = masked ? p.mask_cut[o] : 0;
  __syncthreads();  // every thread has read a[o] before thread 0 overwrites it at the end
  if (threadIdx.x == 0) p.scales[n] = s;
  uint8_t* crow = p.codes + static_cast<int64_t>(n) * p.canon_row_bytes;
  constexpr int kStepBytes = 128 * BITS / 8;  // packed bytes of one row in one 128-code reduction block
  constexpr int kChunkBytes = 16 * BITS / 8;  // bytes of 16 packed codes
  constexpr int kWords = kChunkBytes / 4;
  const int I = p.I;
  const int I_pad = p.kernel_row_bytes * 8 / BITS;
  const bool src_vec = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  const bool dst_vec = dst && (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
  const bool canon_vec = (reinterpret_cast<uintptr_t>(crow) & 3) == 0;
  uint32_t m = 0;
  constexpr int CPW = 32 / BITS;   // codes per packed 32-bit word
  constexpr int LPW = CPW / 4;     // lanes that share one word when a lane holds 4 consecutive codes
  const bool lanewise = (I % CPW == 0) && src_vec && (!dst || dst_vec) && canon_vec && (p.canon_row_bytes % 4 == 0);
  if (lanewise) {
    // Lane-contiguous form: per trip a warp covers 512 consecutive elements, lane L holding the four quads at
    // offsets w * 128 + 4 L (w = 0..3), so every load and store instruction of the warp touches one contiguous
    // run.  A packed word then takes its fields from LPW neighbouring lanes; each lane shifts its four codes
    // to their places in both layouts and the lanes OR their parts together.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int h = lane & (LPW - 1);
    for (int base = warp * 512; base < I_pad; base += nwarps * 512) {
      float4 v[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int e0 = base + w * 128 + lane * 4;
        v[w] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e0 < I) v[w] = *reinterpret_cast<const float4*>(src + e0);   // plain load: src may alias dst
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int e0 = base + w * 128 + lane * 4;
        float x[4] = {v[w].x, v[w].y, v[w].z, v[w].w};
        uint32_t f4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float c = 0.f;
          bool take = s != 0.f;
          if (masked) {
            const uint32_t key = abs_key(x[j]);
            take = take && (key > mthr || (key == mthr && e0 + j <= mcut));
          }
          if (take) {
            c = rintf(__fdiv_rn(x[j], s));         // round half to even
            c = fminf(fmaxf(c, -fq), fq);
            x[j] = __fmaf_rn(-s, c, x[j]);         // exact new residual, rounded once
          }
          m = max(m, abs_key(x[j]));
          f4[j] = static_cast<uint32_t>(static_cast<int>(c));
        }
        if (dst && e0 < I) *reinterpret_cast<float4*>(dst + e0) = make_float4(x[0], x[1], x[2], x[3]);
        // The four codes as the four bytes of a word, then both packed layouts from that word with masks and shifts
        // on all four fields at once.  Canonical: field e at bit e * b of the stream (this lane's four fields are
        // e = 4 h + j); streaming layout: field 4 h + j at bit 8 j + b h (see include/pipe.h).
        const uint32_t wv = __byte_perm(__byte_perm(f4[0], f4[1], 0x0040), __byte_perm(f4[2], f4[3], 0x0040), 0x5410);
        uint32_t cc, ck;
        if (BITS == 8) {
          cc = ck = wv;
        } else if (BITS == 4) {
          const uint32_t t = wv & 0x0F0F0F0Fu;
          const uint32_t u = (t | (t >> 4)) & 0x00FF00FFu;
          cc = ((u | (u >> 8)) & 0xFFFFu) << (16 * h);
          ck = t << (4 * h);
        } else {
          const uint32_t t = wv & 0x03030303u;
          const uint32_t u = (t | (t >> 6)) & 0x000F000Fu;
          cc = ((u | (u >> 12)) & 0xFFu) << (8 * h);
          ck = t << (2 * h);
        }
#pragma unroll
        for (int d = 1; d < LPW; d <<= 1) {
          cc |= __shfl_xor_sync(0xffffffffu, cc, d);
          ck |= __shfl_xor_sync(0xffffffffu, ck, d);
        }
        if (p.wcodes && e0 < I_pad) {
          // the lane's four codes are four bytes of piece (e0 & 127) / 16 of the row's block, which is stored as piece
          // ((e0 & 127) / 16) ^ (n & 7)
          uint8_t* wdst = p.wcodes + (static_cast<int64_t>(e0 >> 7) * p.rows + n) * 128 + (((((e0 & 127) >> 4) ^ (n & 7)) << 4) | (e0 & 15));
          *reinterpret_cast<uint32_t*>(wdst) = wv;
        }
        if (h == 0 && e0 < I_pad) {
          uint8_t* kdst = p.kcodes + (static_cast<int64_t>(e0 >> 7) * p.rows + n) * kStepBytes + (e0 & 127) * BITS / 8;
          *reinterpret_cast<uint32_t*>(kdst) = ck;
          if (e0 < I) *reinterpret_cast<uint32_t*>(crow + e0 * BITS / 8) = cc;
        }
      }
    }
  } else
  for (int i0 = threadIdx.x * 16; i0 < I_pad; i0 += blockDim.x * 16) {
    float v[16];
    const bool full = i0 + 16 <= I;
    if (full && src_vec) {
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const float4 t = reinterpret_cast<const float4*>(src + i0)[w];  // plain load: src may alias dst
        v[4 * w] = t.x; v[4 * w + 1] = t.y; v[4 * w + 2] = t.z; v[4 * w + 3] = t.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = (i0 + e < I) ? src[i0 + e] : 0.f;
    }
    int q[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      float c = 0.f;
      const uint32_t key = abs_key(v[e]);
      if (s != 0.f && (!masked || key > mthr || (key == mthr && i0 + e <= mcut))) {
        c = rintf(__fdiv_rn(v[e], s));           // round half to even
        c = fminf(fmaxf(c, -fq), fq);
        v[e] = __fmaf_rn(-s, c, v[e]);           // exact new residual, rounded once
      }
      q[e] = static_cast<int>(c);
      m = max(m, abs_key(v[e]));
    }
    if (dst) {
      if (full && dst_vec) {
#pragma unroll
        for (int w = 0; w < 4; ++w)
          reinterpret_cast<float4*>(dst + i0)[w] = make_float4(v[4 * w], v[4 * w + 1], v[4 * w + 2], v[4 * w + 3]);
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (i0 + e < I) dst[i0 + e] = v[e];
      }
    }
    uint32_t canon[4], kern[4];
    pack16<BITS>(q, canon, kern);
    if (p.wcodes) {
      uint32_t wv[4];
#pragma unroll
      for (int w = 0; w < 4; ++w)
        wv[w] = (static_cast<uint32_t>(q[4 * w]) & 0xffu) | ((static_cast<uint32_t>(q[4 * w + 1]) & 0xffu) << 8) |
                ((static_cast<uint32_t>(q[4 * w + 2]) & 0xffu) << 16) | (static_cast<uint32_t>(q[4 * w + 3]) << 24);
      uint8_t* wdst = p.wcodes + (static_cast<int64_t>(i0 >> 7) * p.rows + n) * 128 + ((((i0 & 127) >> 4) ^ (n & 7)) << 4);
      *reinterpret_cast<uint4*>(wdst) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
    }
    const int byte0 = i0 * BITS / 8;
    // streaming layout: reduction-block major, [i0 / 128][row][128 codes]; padded, always whole words
    uint8_t* kdst = p.kcodes + (static_cast<int64_t>(i0 >> 7) * p.rows + n) * kStepBytes + (i0 & 127) * BITS / 8;
#pragma unroll
    for (int w = 0; w < kWords; ++w) reinterpret_cast<uint32_t*>(kdst)[w] = kern[w];
    if (i0 < I) {
      if (full && canon_vec) {
#pragma unroll
        for (int w = 0; w < kWords; ++w) reinterpret_cast<uint32_t*>(crow + byte0)[w] = canon[w];
      } else {
        const int nbytes = min(kChunkBytes, p.canon_row_bytes - byte0);
        for (int bb = 0; bb < nbytes; ++bb) crow[byte0 + bb] = static_cast<uint8_t>(canon[bb >> 2] >> (8 * (bb & 3)));
      }
    }
  }
  if (dst) {
    m = block_max_u32(m);
    if (threadIdx.x == 0) p.a[o] = __uint_as_float(m);
  }
}

// Channel-block table of one cluster of orders (see pipe.h): the groups are walked from 0 and a block is closed
// when the next group would take its stacked rows beyond PIPE_BLOCK_ROWS or its channels beyond PIPE_BLOCK_CHANNELS.
// One thread block per cluster: all threads gather the rows every group stacks (kept orders of the cluster only),
// thread 0 then cuts the blocks.
constexpr int kTableSets = 2 * (PIPE_MAX_ORDERS + 1);   // channel-block tables, then decode-unit tables
struct BlockTableArgs {
  const int32_t* cum[kTableSets][8];   // prefix counts of the cluster's orders
  int nk[kTableSets];
  int32_t* out[kTableSets];
  int cap[kTableSets];
  int limit[kTableSets];   // rows a block of the cluster may stack
  int G, g;
};

constexpr int kTableChunk = 2048;
constexpr int kTableThreads = 256;

// One thread block per table.  The groups are taken in chunks: all threads gather the rows every group of the chunk
// stacks (kept orders of the cluster only) and form their running sums; the first warp then cuts the blocks.  The
// greedy rule "close the block when the next group would take it beyond the limit" needs, for a block that starts at
// group b, the first group whose running sum from b exceeds the limit (or that would be the block's max_groups + 1-th):
// the sums are non-decreasing, so the lanes test 32 candidates at a time and the first hit is the cut.
__device__ __forceinline__ void cut_table(const BlockTableArgs& a, const int m) {
  __shared__ int pre_s[kTableChunk];            // inclusive running sum of the chunk's rows
  __shared__ int part_s[kTableThreads];
  int32_t* out = a.out[m];
  if (!out) return;
  int cur_rows = 0, cur_groups = 0, n = 0;      // (warp 0: the same in every lane)
  const int max_groups = PIPE_BLOCK_CHANNELS / a.g > 0 ? PIPE_BLOCK_CHANNELS / a.g : 1;
  const int lane = threadIdx.x & 31;
  constexpr int kPer = kTableChunk / kTableThreads;
  for (int base = 0; base < a.G; base += kTableChunk) {
    const int cnt = min(kTableChunk, a.G - base);
    // rows of this thread's kPer consecutive groups, then a scan of the threads' totals
    int r[kPer];
    int tot = 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int j = threadIdx.x * kPer + u;
      int v = 0;
      if (j < cnt)
        for (int q = 0; q < a.nk[m]; ++q) v += (a.cum[m][q][base + j + 1] - a.cum[m][q][base + j]) * a.g;
      tot += v;
      r[u] = tot;
    }
    part_s[threadIdx.x] = tot;
    __syncthreads();
    for (int d = 1; d < kTableThreads; d <<= 1) {
      const int v = threadIdx.x >= d ? part_s[threadIdx.x - d] : 0;
      __syncthreads();
      part_s[threadIdx.x] += v;
      __syncthreads();
    }
    const int before = threadIdx.x == 0 ? 0 : part_s[threadIdx.x - 1];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int j = threadIdx.x * kPer + u;
      if (j < cnt) pre_s[j] = before + r[u];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      if (base == 0 && lane == 0) out[1] = 0;
      int pos = 0, s0 = 0;   // next group of the chunk to place; running sum before it
      while (pos < cnt) {
        for (int off = 0;; off += 32) {
          const int c = pos + off + lane;
          const bool valid = c < cnt;
          const int rsum = valid ? pre_s[c] - s0 : 0;   // rows of the groups pos .. c
          const int ng = cur_groups + off + lane;       // groups of the block before c
          const bool cut = valid && ng > 0 && (cur_rows + rsum > a.limit[m] || ng + 1 > max_groups);
          const unsigned hit = __ballot_sync(0xffffffffu, cut);
          if (hit) {
            const int f = off + __ffs(hit) - 1;         // group pos + f opens the next block
            if (lane == 0 && n < a.cap[m]) out[2 + n] = base + pos + f;   // (the capacity bound holds by construction; never write past it)
            ++n;
            cur_rows = 0;
            cur_groups = 0;
            pos += f;
            s0 = pos > 0 ? pre_s[pos - 1] : 0;
            break;
          }
          if (pos + off + 32 >= cnt) {                  // the rest of the chunk joins the block under construction
            cur_rows += pre_s[cnt - 1] - s0;
            cur_groups += cnt - pos;
            pos = cnt;
            break;
          }
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (n < a.cap[m]) out[2 + n] = a.G;
    ++n;
    out[0] = n <= a.cap[m] ? n : 0;
  }
}

__global__ void __launch_bounds__(kTableThreads) block_table_kernel(const __grid_constant__ BlockTableArgs a) {
  grid_wait();
  grid_release();
  cut_table(a, blockIdx.x);
}

// Block records (layout in pipe.h): one thread block per (block of a table, table).
struct BlockRecordArgs {
  const int32_t* cum[PIPE_MAX_ORDERS + 1][8];   // prefix counts of the cluster's orders
  const float* scales[PIPE_MAX_ORDERS + 1][8];  // their row scales
  int nk[PIPE_MAX_ORDERS + 1];
  const int32_t* tbl[PIPE_MAX_ORDERS + 1];      // the channel-block table (n, b_0 .. b_n)
  uint8_t* out[PIPE_MAX_ORDERS + 1];
  int cap[PIPE_MAX_ORDERS + 1];
  int g;
  int* status;
};

__global__ void block_record_kernel(const __grid_constant__ BlockRecordArgs a) {
  grid_wait();
  grid_release();
  const int m = blockIdx.y, cb = blockIdx.x;
  if (!a.out[m]) return;
  const int n_blocks = a.tbl[m][0];
  if (n_blocks > a.cap[m]) {   // cannot happen (the capacity is a bound on the cut); never write past it
    if (cb == 0 && threadIdx.x == 0) raise_status(a.status, PIPE_ERR_WORKSPACE);
    return;
  }
  if (cb >= n_blocks) return;
  __shared__ int rowbase_s[9], start_s[8];
  const int j0 = a.tbl[m][1 + cb], j1 = a.tbl[m][2 + cb];
  const int nk = a.nk[m];
  if (threadIdx.x == 0) {
    int rb = 0;
    for (int q = 0; q < 8; ++q) {
      rowbase_s[q] = rb;
      start_s[q] = 0;
      if (q < nk) {
        const int lo = a.cum[m][q][j0], hi = a.cum[m][q][j1];
        start_s[q] = lo * a.g;
        rb += (hi - lo) * a.g;
      }
    }
    rowbase_s[8] = rb;
  }
  __syncthreads();
  uint8_t* rec = a.out[m] + static_cast<size_t>(cb) * kRecBytes;
  int32_t* hdr = reinterpret_cast<int32_t*>(rec);
  int16_t* colmap = reinterpret_cast<int16_t*>(rec + kRecColmapOff);
  float* scale = reinterpret_cast<float*>(rec + kRecScaleOff);
  const int c0 = j0 * a.g, c1 = j1 * a.g, n_total = rowbase_s[8];
  for (int i = threadIdx.x; i < kRecHeaderInts; i += blockDim.x) {
    int v = 0;
    if (i == 0) v = c0;
    else if (i == 1) v = c1;
    else if (i == 2) v = nk;
    else if (i == 3) v = n_total;
    else if (i >= kRecRowbase && i < kRecRowbase + 8) v = rowbase_s[i - kRecRowbase];
    else if (i >= kRecStart && i < kRecStart + 8) v = start_s[i - kRecStart];
    hdr[i] = v;
  }
  const int nch = (c1 - c0) >> 3;
  for (int e = threadIdx.x; e < kRecColmapEntries; e += blockDim.x) {
    const int cc = e >> 3, q = e & 7;
    int col = -1;
    if (q < nk && cc < nch) {
      const int c = c0 + 8 * cc;
      const int j = c / a.g;
      const int lo = a.cum[m][q][j], hi = a.cum[m][q][j + 1];
      if (hi > lo) col = rowbase_s[q] + lo * a.g + c % a.g - start_s[q];
    }
    colmap[e] = static_cast<int16_t>(col);
  }
  for (int r = threadIdx.x; r < PIPE_BLOCK_ROWS; r += blockDim.x) {
    float v = 0.f;
    if (r < n_total) {
      int q = 0;
      while (q + 1 < nk && r >= rowbase_s[q + 1]) ++q;
      v = a.scales[m][q][start_s[q] + (r - rowbase_s[q])];
    }
    scale[r] = v;
  }
}

// ------------------------------------------------------------------------------------------------
// The expansion with ONE pass over the weights.
//
// How often a row has been quantized decides its residual: the residual entering a row's (j+1)-th quantization, its
// "level" j, does not depend on WHICH orders kept the row.  So a row's scales and codes of all K levels come from one
// pass with the row in registers (expand_chain_kernel); which order uses which level is known as soon as the group
// maxima of every level are (select_orders_kernel, one block, walks the orders); and a third kernel copies the kept
// rows' packed codes from level storage to their orders (place_orders_kernel).
// Against one pass per order this neither writes nor re-reads the fp32 residual (8 bytes an element and order) and
// pays with codes of levels that no order uses (b / 8 bytes each, and their arithmetic): 4096 x 11008 and back, int4,
// K = 4, gamma = 0.5: 600 -> 222 us; 8192 x 8192 ternary, K = 8, gamma = 0.25 (8 levels computed, 2.75 used on
// average): 464 -> 200 us.  The level storage takes the place of the residual in the workspace.
// Layers this does not take (chain_fits) run one pass per order: the unstructured mask and the L2 score need the
// residual itself, rows beyond 16384 do not fit a block's registers, rows that are not whole 16-code chunks, and large
// layers that use few of many levels.
struct ChainOut {
  uint8_t* codes;
  uint8_t* kcodes;
  uint8_t* wcodes;
  float* scales;
};
struct ChainArgs {
  const float* W;
  int64_t ldw;
  ChainOut out[PIPE_MAX_ORDERS];   // levels below `direct` go straight to the order of that number
  int direct;                      // 1, or K when every order keeps every row
  uint8_t* temp;                   // packed codes (streaming field order, row-major) of the levels from `direct` on
  int temp_pitch;
  float* lvl_scale;                // [K][O]
  uint32_t* lvl_max;               // [K][G] largest magnitude bits of the group's rows entering a level
  int O, I, I_pad, g, G, K, qmax;
  int canon_row_bytes;
  int* status;
};

// Both packed layouts of 16 codes given as the four bytes of four words.
template <int BITS>
__device__ __forceinline__ void pack_bytes(const uint32_t (&wv)[4], uint32_t (&kern)[4]) {
  if (BITS == 8) {
#pragma unroll
    for (int w = 0; w < 4; ++w) kern[w] = wv[w];
  } else if (BITS == 4) {
#pragma unroll
    for (int w = 0; w < 2; ++w) kern[w] = (wv[2 * w] & 0x0F0F0F0Fu) | ((wv[2 * w + 1] << 4) & 0xF0F0F0F0u);
  } else {
    kern[0] = (wv[0] & 0x03030303u) | ((wv[1] & 0x03030303u) << 2) | ((wv[2] & 0x03030303u) << 4) | ((wv[3] & 0x03030303u) << 6);
  }
}
// A word of the canonical layout from the same codes' word of the streaming layout (see include/pipe.h).
template <int BITS>
__device__ __forceinline__ uint32_t canon_of_kern(uint32_t k) {
  if (BITS == 8) return k;
  uint32_t c = 0;
  if (BITS == 4) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t t = (k >> (4 * h)) & 0x0F0F0F0Fu;
      const uint32_t u = (t | (t >> 4)) & 0x00FF00FFu;
      c |= ((u | (u >> 8)) & 0xFFFFu) << (16 * h);
    }
  } else {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const uint32_t t = (k >> (2 * h)) & 0x03030303u;
      const uint32_t u = (t | (t >> 6)) & 0x000F000Fu;
      c |= ((u | (u >> 12)) & 0xFFu) << (8 * h);
    }
  }
  return c;
}
// The int8 codes (four per word) of field h of a streaming-layout word, sign extended byte by byte.
template <int BITS>
__device__ __forceinline__ uint32_t bytes_of_kern(uint32_t k, int h) {
  if (BITS == 8) return k;
  if (BITS == 4) {
    const uint32_t t = (k >> (4 * h)) & 0x0F0F0F0Fu;
    return t | ((t & 0x08080808u) * 0x1Eu);
  }
  const uint32_t t = (k >> (2 * h)) & 0x03030303u;
  return t | ((t & 0x02020202u) * 0x7Eu);
}

// The estimate of one level (see expand_chain_kernel): the reciprocal of its step, and the residual magnitude from which a
// code has to be divided for.  A step of zero quantizes nothing: with rcp = 0 every code is 0 and the residual stays.
__device__ __forceinline__ void level_estimate(float s, float near_half, float& rcp, float& limit) {
  const bool fast = quant_step_is_fast(s);
  rcp = 0.f;
  if (fast) asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(s));
  limit = fast ? s * near_half : s == 0.f ? __uint_as_float(0x7f800000u) : -1.f;
}
__device__ __forceinline__ float code_by_division(float x, float s, float fq) {
  float c = 0.f;
  if (s != 0.f) c = fminf(fmaxf(rintf(__fdiv_rn(x, s)), -fq), fq);
  return c;
}
static __device__ __noinline__ uint32_t codes4_by_division(float x0, float x1, float x2, float x3, float s, float fq) {
  const float q[4] = {code_by_division(x0, s, fq), code_by_division(x1, s, fq), code_by_division(x2, s, fq), code_by_division(x3, s, fq)};
  uint32_t b = 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) b |= (static_cast<uint32_t>(static_cast<int>(q[e])) & 0xffu) << (8 * e);
  return b;
}
// Four elements through all levels up to j (out of line: a few chunks in a thousand): residual after level j and its codes
// as the bytes of a word.  lvl_s: the scales of the levels below j.  Divides only where the estimate cannot decide, like the
// levels themselves: weights on a coarse grid (an integer model's) put many quotients on a boundary, at several levels.
static __device__ __noinline__ void replay_quad(const float4* src, const float* lvl_s, int j, float s, float fq, float near_half, float4* resid, uint32_t* codes) {
  const float4 v = src ? __ldg(src) : make_float4(0.f, 0.f, 0.f, 0.f);
  float x[4] = {v.x, v.y, v.z, v.w}, q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int l = 0; l <= j; ++l) {
    const float sl = l < j ? lvl_s[l] : s;
    float rcp, limit, x1[4];
    level_estimate(sl, near_half, rcp, limit);
    float m = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      q[e] = __fsub_rn(__fmaf_rn(x[e], rcp, 12582912.f), 12582912.f);
      x1[e] = __fmaf_rn(-sl, q[e], x[e]);
      m = fmaxf(m, fabsf(x1[e]));
    }
    if (m >= limit) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        q[e] = code_by_division(x[e], sl, fq);
        x1[e] = __fmaf_rn(-sl, q[e], x[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = x1[e];
  }
  *resid = make_float4(x[0], x[1], x[2], x[3]);
  uint32_t b = 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) b |= (static_cast<uint32_t>(static_cast<int>(q[e])) & 0xffu) << (8 * e);
  *codes = b;
}

constexpr int kChainMaxI = 16384;

// One block per row, PER chunks of 16 consecutive elements per thread.  Bound by its instructions, so a level costs an
// element three packed operations (two elements each) beside half a maximum and the packing: r * (1 / s) + 1.5 * 2^23 (the
// fused addition rounds to nearest even), the code as a float, the residual.  What DEFINES the code is the IEEE
// quotient; it and the estimate can differ only next to a rounding boundary, where |residual| is within
// s * |t| * 2^-22 of s / 2: so the maximum that the next level needs anyway tells whether a chunk has to be replayed from
// the weights, and the old residual need not be kept (the reciprocal is off by 2^-23, the quotient's own rounding by 2^-24, relative; |t| <= qmax because |x| <= amax,
// which is also why no clamp is needed while s has a usable reciprocal).
// The packing is arithmetic too: sum_e (code_e + 2^(b-1)) 2^(b e) over the codes of 16 bits of a packed word, on top of
// 1.5 * 2^23, is exact in binary32 and stands in the low 16 bits of its pattern; the offsets are the fields' sign bits, which
// an exclusive or takes away.  A pair holds the elements i and i + 2 of a quad, so that its halves lead to the low and to the
// high half of the same word.  (9.1 instructions per element and level in all for int4, 7.3 for 2 bits, issue slots 72 % busy, against 11 with scalar
// operations and byte permutations: 11008 x 4096 int4 K = 4 73 -> 66 us, 8192 x 8192 ternary K = 8 184 -> 155.)
// Ordinary weights replay a few chunks in a thousand.  Weights on a coarse grid put quotients on a boundary all over, at
// every level; a block that had to replay in an eighth of its threads therefore keeps, from the next level on, the old
// residual of a quad until its maximum is known, and divides the quad alone.
template <int BITS, int PER, int MAXT, int MINB>   // PER: 16-code chunks per thread
__global__ void __launch_bounds__(MAXT, MINB) expand_chain_kernel(const __grid_constant__ ChainArgs p) {
  __shared__ uint32_t part[2][32];
  __shared__ float lvl_s[PIPE_MAX_ORDERS];
  const int o = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const float fq = static_cast<float>(p.qmax);
  constexpr float kMagic = 12582912.f;
  constexpr int kWords = BITS / 2;            // packed words of 16 codes
  constexpr int kStepBytes = 128 * BITS / 8;
  constexpr uint32_t kSigns = BITS == 8 ? 0x80808080u : (BITS == 4 ? 0x88888888u : 0xAAAAAAAAu);   // sign bits of a word's fields
  // |residual| / s from which a chunk is divided: 1/2 - (qmax 2^-22 + 2^-23)
  const float near_half = 0.5f - (fq * 2.384185791015625e-07f + 1.1920928955078125e-07f);
  f32x2 r[PER][8];   // pair 2 w + i: elements 4 w + i and 4 w + i + 2
  float mf = 0.f;
#pragma unroll
  for (int c = 0; c < PER; ++c) {
    const int e0 = (tid + c * blockDim.x) * 16;
    if (e0 < p.I) {
      const float4* src = reinterpret_cast<const float4*>(p.W + static_cast<int64_t>(o) * p.ldw + e0);
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const float4 v = __ldg(src + w);
        r[c][2 * w] = pack_f2(v.x, v.z);
        r[c][2 * w + 1] = pack_f2(v.y, v.w);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) r[c][i] = 0;
    }
  }
#pragma unroll
  for (int c = 0; c < PER; ++c)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float lo, hi;
      unpack_f2(r[c][i], lo, hi);
      mf = max3_abs_nan(mf, lo, hi);
    }
  uint32_t mk = __float_as_uint(mf);
  // (the weights were complete when the launch before this one, which zeroes the level maxima, started)
  grid_wait();
  grid_release();
  uint8_t* temp_row = p.temp + static_cast<int64_t>(o) * p.temp_pitch;   // this row in the level being written
  const int64_t temp_step = static_cast<int64_t>(p.O) * p.temp_pitch;
  bool careful = false;
  int replays = 0;
#pragma unroll 1
  for (int j = 0; j < p.K; ++j) {
    // largest magnitude entering this level (one barrier per level: the partial maxima alternate between two rows)
    mk = __reduce_max_sync(0xffffffffu, mk);
    if (lane == 0) part[j & 1][warp] = mk;
    // (a block that had to replay in an eighth of its threads keeps to the careful form from here on)
    careful = __syncthreads_count(replays) * 8 > blockDim.x || careful;
    replays = 0;
    mk = __reduce_max_sync(0xffffffffu, lane < nwarps ? part[j & 1][lane] : 0u);
    const float s = BITS == 2 ? __uint_as_float(mk) : __fdiv_rn(__uint_as_float(mk), fq);   // (2 bits: qmax = 1)
    const bool direct = j < p.direct;
    if (tid == 0) {
      lvl_s[j] = s;   // (read at later levels, behind their barriers)
      if (j == 0 && mk >= 0x7f800000u) raise_status(p.status, PIPE_ERR_NONFINITE);
      (direct ? p.out[j].scales : p.lvl_scale + static_cast<int64_t>(j) * p.O)[o] = s;
      if (j > 0 && p.direct == 1) atomicMax(p.lvl_max + static_cast<int64_t>(j) * p.G + o / p.g, mk);
    }
    float rcp, limit;
    level_estimate(s, near_half, rcp, limit);
    const f32x2 rcp2 = both_f2(rcp), neg_s2 = both_f2(-s), magic2 = both_f2(kMagic), neg_magic2 = both_f2(-kMagic);
    constexpr float kBias = kMagic + static_cast<float>(kSigns & 0xffffu);
    mk = 0;
#pragma unroll
    for (int c = 0; c < PER; ++c) {
      const int chunk = tid + c * blockDim.x, e0 = chunk * 16;
      uint32_t kern[4];
      float m = 0.f;
      if (careful) {
        uint32_t wv[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          float x[4], u[4], x1[4];
          unpack_f2(r[c][2 * w], x[0], x[2]);
          unpack_f2(r[c][2 * w + 1], x[1], x[3]);
          float m4 = 0.f;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            u[e] = __fmaf_rn(x[e], rcp, kMagic);
            x1[e] = __fmaf_rn(-s, __fsub_rn(u[e], kMagic), x[e]);
            m4 = fmaxf(m4, fabsf(x1[e]));
          }
          wv[w] = pack4_low_bytes(u[0], u[1], u[2], u[3]);
          if (m4 >= limit) {
            wv[w] = codes4_by_division(x[0], x[1], x[2], x[3], s, fq);
            m4 = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              x1[e] = __fmaf_rn(-s, static_cast<float>(static_cast<int8_t>(wv[w] >> (8 * e))), x[e]);
              m4 = fmaxf(m4, fabsf(x1[e]));
            }
          }
          r[c][2 * w] = pack_f2(x1[0], x1[2]);
          r[c][2 * w + 1] = pack_f2(x1[1], x1[3]);
          m = fmaxf(m, m4);
        }
        pack_bytes<BITS>(wv, kern);
      } else {
        constexpr int kQuads = 8 / BITS;   // quads whose codes share a packed word
        float m1 = 0.f;
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
          f32x2 acc = both_f2(kBias);
#pragma unroll
          for (int h = 0; h < kQuads; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              f32x2& x = r[c][2 * (k * kQuads + h) + i];
              const f32x2 q = add_f2(fma_f2(x, rcp2, magic2), neg_magic2);
              x = fma_f2(neg_s2, q, x);   // exact new residual, rounded once
              acc = h + i == 0 ? add_f2(q, acc) : fma_f2(q, both_f2(static_cast<float>(1u << (8 * i + BITS * h))), acc);
              float lo, hi;
              unpack_f2(x, lo, hi);
              (i ? m1 : m) = max3_abs(i ? m1 : m, lo, hi);
            }
          float lo, hi;
          unpack_f2(acc, lo, hi);
          kern[k] = __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x5410) ^ kSigns;
        }
        m = fmaxf(m, m1);
      }
      if (!careful && m >= limit) {
        replays = 1;
        // (the old residual is overwritten: the chunk goes through all levels again)
        m = 0.f;
        uint32_t wv[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          float4 v;
          replay_quad(e0 < p.I ? reinterpret_cast<const float4*>(p.W + static_cast<int64_t>(o) * p.ldw + e0) + w : nullptr, lvl_s, j, s, fq, near_half, &v, &wv[w]);
          r[c][2 * w] = pack_f2(v.x, v.z);
          r[c][2 * w + 1] = pack_f2(v.y, v.w);
          m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
        }
        pack_bytes<BITS>(wv, kern);
      }
      mk = max(mk, __float_as_uint(m));
      auto store = [](uint8_t* dst, const uint32_t (&w)[4]) {
        if constexpr (kWords == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        else if constexpr (kWords == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
        else *reinterpret_cast<uint32_t*>(dst) = w[0];
      };
      if (!direct) {
        if (e0 < p.I) store(temp_row + chunk * (2 * BITS), kern);
      } else {
        const ChainOut& out = p.out[j];
        if (e0 < p.I_pad) {
          store(out.kcodes + (static_cast<int64_t>(e0 >> 7) * p.O + o) * kStepBytes + (e0 & 127) * BITS / 8, kern);
          if (out.wcodes) {
            uint32_t wv[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) wv[w] = bytes_of_kern<BITS>(kern[w * BITS / 8], w % (8 / BITS));
            *reinterpret_cast<uint4*>(out.wcodes + (static_cast<int64_t>(e0 >> 7) * p.O + o) * 128 + ((((e0 & 127) >> 4) ^ (o & 7)) << 4)) =
                make_uint4(wv[0], wv[1], wv[2], wv[3]);
          }
        }
        if (e0 < p.I) {
          uint32_t canon[4];
#pragma unroll
          for (int w = 0; w < 4; ++w) canon[w] = w < kWords ? canon_of_kern<BITS>(kern[w]) : 0u;
          store(out.codes + static_cast<int64_t>(o) * p.canon_row_bytes + chunk * (2 * BITS), canon);
        }
      }
    }
    if (!direct) temp_row += temp_step;
  }
}

// Which order keeps which group at which level, all orders in one block: per order the n_keep groups of largest score
// (the maximum at the group's present level; ties to the lower index, as everywhere; non-negative floats order like
// their bits).  The n_keep-th largest score is found by counting the keys at and above three probes that quarter the interval
// which holds it, until a probe has exactly n_keep (the usual end, after about log4 of the number of groups) or one value is
// left.  A step of that search is one barrier, and so is the compaction, for which a thread holds neighbouring groups.
constexpr int kSelThreads = 1024;
constexpr int kSelPer = 8;
constexpr int kSelMaxGroups = kSelThreads * kSelPer;
struct SelectArgs {
  const uint32_t* lvl_max;   // [K][G]
  int32_t* lvl_of;           // [K][n_keep]: level of every kept slot of an order (order 1 is dense: level 0)
  int32_t* cum[PIPE_MAX_ORDERS];
  int32_t* kept[PIPE_MAX_ORDERS];
  int G, K, n_keep;
};

template <int PER>   // groups per thread: few for few groups, an order's time is its instructions one after the other
__global__ void __launch_bounds__(kSelThreads) select_orders_kernel(const __grid_constant__ SelectArgs p) {
  __shared__ uint32_t part_lo[32], part_hi[32], part_n[2][2][32], part_c[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int per = (p.G + blockDim.x - 1) / blockDim.x, j0 = tid * per;   // this thread's groups: j0 .. j0 + per - 1
  grid_wait();
  grid_release();
  // key: score at the group's present level, plus one (0: no group); next: at the level behind it, asked for ahead of use
  uint32_t lvl[PER], key[PER], next[PER];
  auto score = [&](int c, uint32_t l) -> uint32_t {
    return c < per && j0 + c < p.G && l < static_cast<uint32_t>(p.K) ? __ldcg(p.lvl_max + static_cast<int64_t>(l) * p.G + j0 + c) + 1u : 0u;
  };
#pragma unroll
  for (int c = 0; c < PER; ++c) {
    lvl[c] = 1;
    key[c] = score(c, 1);
  }
  int round = 0;
  for (int k = 1; k < p.K; ++k) {
    uint32_t lo = 0xffffffffu, hi = 0;
#pragma unroll
    for (int c = 0; c < PER; ++c) {
      next[c] = score(c, lvl[c] + 1);
      if (key[c] != 0) {
        lo = min(lo, key[c]);
        hi = max(hi, key[c]);
      }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      part_lo[warp] = lo;
      part_hi[warp] = hi;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lane < nwarps ? part_lo[lane] : 0xffffffffu);
    hi = __reduce_max_sync(0xffffffffu, lane < nwarps ? part_hi[lane] : 0u);
    // more than n_keep keys are >= lo (every group has a key: it has been taken k - 1 times at most), `above` < n_keep are > hi
    int above = 0;
    int ties = p.G;            // how many of the keys equal to the threshold are kept, lowest index first
    uint32_t thr = lo;
    while (true) {
      if (lo == hi) {
        thr = lo;
        ties = p.n_keep - above;
        break;
      }
      const uint32_t q = (hi - lo) >> 2;
      const uint32_t m[3] = {lo + q + 1, lo + 2 * q + 1, lo + 3 * q + 1};   // in (lo, hi]
      uint32_t n01 = 0, n2 = 0;
#pragma unroll
      for (int c = 0; c < PER; ++c) {
        n01 += (key[c] >= m[0] ? 1u : 0u) + (key[c] >= m[1] ? 0x10000u : 0u);
        n2 += key[c] >= m[2] ? 1u : 0u;
      }
      n01 = __reduce_add_sync(0xffffffffu, n01);
      n2 = __reduce_add_sync(0xffffffffu, n2);
      if (lane == 0) {
        part_n[round & 1][0][warp] = n01;
        part_n[round & 1][1][warp] = n2;
      }
      __syncthreads();
      n01 = __reduce_add_sync(0xffffffffu, lane < nwarps ? part_n[round & 1][0][lane] : 0u);
      n2 = __reduce_add_sync(0xffffffffu, lane < nwarps ? part_n[round & 1][1][lane] : 0u);
      ++round;
      const int n[3] = {static_cast<int>(n01 & 0xffffu), static_cast<int>(n01 >> 16), static_cast<int>(n2)};
      if (n[0] == p.n_keep || n[1] == p.n_keep || n[2] == p.n_keep) {
        thr = n[2] == p.n_keep ? m[2] : (n[1] == p.n_keep ? m[1] : m[0]);
        break;
      }
      if (n[2] > p.n_keep) {
        lo = m[2];
      } else if (n[1] > p.n_keep) {
        lo = m[1];
        hi = m[2] - 1;
        above = n[2];
      } else if (n[0] > p.n_keep) {
        lo = m[0];
        hi = m[1] - 1;
        above = n[1];
      } else {
        hi = m[0] - 1;
        above = n[0];
      }
    }
    uint32_t mine = 0;   // keys above the threshold << 16, keys at it
#pragma unroll
    for (int c = 0; c < PER; ++c) mine += (key[c] > thr ? 0x10000u : 0u) + (key[c] == thr ? 1u : 0u);
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
    }
    if (lane == 31) part_c[warp] = incl;
    __syncthreads();
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? part_c[lane] : 0u) + incl - mine;
    int gt = static_cast<int>(before >> 16), eq = static_cast<int>(before & 0xffffu);
#pragma unroll
    for (int c = 0; c < PER; ++c) {
      const int j = j0 + c;
      if (c >= per || j >= p.G) continue;
      const int pos = gt + min(eq, ties);
      const bool over = key[c] > thr, at = key[c] == thr;
      p.cum[k][j] = pos;
      if (over || (at && eq < ties)) {
        p.kept[k][pos] = j;
        p.lvl_of[static_cast<int64_t>(k) * p.n_keep + pos] = static_cast<int>(lvl[c]);
        ++lvl[c];
        key[c] = next[c];
      }
      gt += over;
      eq += at;
    }
    if (tid == 0) p.cum[k][p.G] = p.n_keep;
  }
}

// The kept rows' codes from level storage to their orders (both layouts, and the int8 copy where the layer keeps one),
// one block per (order, kept group); the first blocks cut the channel-block and decode-unit tables meanwhile, whose
// serial walk would otherwise stand alone at the end of the expansion (18 us on 4096 -> 11008).
// UW: words a thread moves at a time, 4 where rows are whole 16-byte pieces, else the words of 16 codes.
struct PlaceArgs {
  ChainOut out[PIPE_MAX_ORDERS];
  const int32_t* kept[PIPE_MAX_ORDERS];
  const int32_t* lvl_of;
  const float* lvl_scale;
  const uint8_t* temp;
  int temp_pitch;
  int O, g, n_keep, rows;          // rows: kept rows of a sparse order
  int canon_row_bytes, kblocks, tables;
  BlockTableArgs tab;
};

template <int BITS, int UW>
__global__ void __launch_bounds__(kTableThreads) place_orders_kernel(const __grid_constant__ PlaceArgs p) {
  grid_wait();
  grid_release();
  if (blockIdx.x < static_cast<unsigned>(p.tables)) {
    cut_table(p.tab, blockIdx.x);
    return;
  }
  const int b = blockIdx.x - p.tables;
  const int k = 1 + b / p.n_keep, slot = b % p.n_keep;
  const int j = p.kept[k][slot], lvl = p.lvl_of[static_cast<int64_t>(k) * p.n_keep + slot];
  const ChainOut& out = p.out[k];
  const int n0 = slot * p.g, o0 = j * p.g;
  const uint8_t* src = p.temp + (static_cast<int64_t>(lvl - 1) * p.O + o0) * p.temp_pitch;
  for (int u = threadIdx.x; u < p.g; u += kTableThreads) out.scales[n0 + u] = p.lvl_scale[static_cast<int64_t>(lvl) * p.O + o0 + u];
  constexpr int kStepBytes = 128 * BITS / 8;
  constexpr int UB = 4 * UW;                    // bytes of a piece
  constexpr int kPieces = kStepBytes / UB;      // pieces of a row in one reduction block
  const int per = p.g * kPieces;                // pieces of the group in one reduction block
  const int tid = threadIdx.x;
  const int kpar = per <= kTableThreads ? kTableThreads / per : 1;
  const int kb0 = per <= kTableThreads ? tid / per : 0;
  if (kb0 >= kpar) return;
  for (int q = per <= kTableThreads ? tid % per : tid; q < per; q += kTableThreads) {
    const int u = q / kPieces, piece = q % kPieces, n = n0 + u;
    const uint8_t* row = src + static_cast<int64_t>(u) * p.temp_pitch + piece * UB;
    uint8_t* crow = out.codes + static_cast<int64_t>(n) * p.canon_row_bytes + piece * UB;
    uint8_t* krow = out.kcodes + static_cast<int64_t>(n) * kStepBytes + piece * UB;
    const int64_t kstep = static_cast<int64_t>(p.rows) * kStepBytes;
#pragma unroll 4
    for (int kb = kb0; kb < p.kblocks; kb += kpar) {
      const int byte0 = kb * kStepBytes + piece * UB;
      const bool in_row = byte0 < p.canon_row_bytes;
      uint32_t w[UW];
#pragma unroll
      for (int i = 0; i < UW; ++i) w[i] = 0u;
      if (in_row) {
        if constexpr (UW == 4) {
          const uint4 v = __ldg(reinterpret_cast<const uint4*>(row + kb * kStepBytes));
          w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
        } else if constexpr (UW == 2) {
          const uint2 v = __ldg(reinterpret_cast<const uint2*>(row + kb * kStepBytes));
          w[0] = v.x, w[1] = v.y;
        } else {
          w[0] = __ldg(reinterpret_cast<const uint32_t*>(row + kb * kStepBytes));
        }
      }
      uint32_t c[UW];
#pragma unroll
      for (int i = 0; i < UW; ++i) c[i] = canon_of_kern<BITS>(w[i]);
      uint8_t* kd = krow + kb * kstep;
      uint8_t* cd = crow + kb * kStepBytes;
      if constexpr (UW == 4) {
        *reinterpret_cast<uint4*>(kd) = make_uint4(w[0], w[1], w[2], w[3]);
        if (in_row) *reinterpret_cast<uint4*>(cd) = make_uint4(c[0], c[1], c[2], c[3]);
      } else if constexpr (UW == 2) {
        *reinterpret_cast<uint2*>(kd) = make_uint2(w[0], w[1]);
        if (in_row) *reinterpret_cast<uint2*>(cd) = make_uint2(c[0], c[1]);
      } else {
        *reinterpret_cast<uint32_t*>(kd) = w[0];
        if (in_row) *reinterpret_cast<uint32_t*>(cd) = c[0];
      }
      if (out.wcodes) {
        // 16 codes are one 16-byte piece of the operand layout, at its place in the swizzled row
        constexpr int kPer16 = BITS / 2;          // words of 16 codes
        uint8_t* wrow = out.wcodes + (static_cast<int64_t>(kb) * p.rows + n) * 128;
#pragma unroll
        for (int i = 0; i < UW / kPer16; ++i) {
          uint32_t v[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) v[h] = bytes_of_kern<BITS>(w[i * kPer16 + h * BITS / 8], h % (8 / BITS));
          const int p16 = piece * (UW / kPer16) + i;
          *reinterpret_cast<uint4*>(wrow + ((p16 ^ (n & 7)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]);
        }
      }
    }
  }
}

// Header, the trivial kept lists (order 1; every order where all groups are kept) and zeroed level maxima.
struct ChainInitArgs {
  uint32_t* hdr;
  pipe_layer_desc desc;
  int32_t* cum[PIPE_MAX_ORDERS];
  int32_t* kept[PIPE_MAX_ORDERS];
  int lists, G;
  uint32_t* lvl_max;
  int64_t n_max;
};

__device__ __forceinline__ void write_header(uint32_t* hdr, const pipe_layer_desc& d) {
  {
    hdr[0] = kBlobMagic;
    hdr[1] = 1;  // format version
    int32_t* o = reinterpret_cast<int32_t*>(hdr + 2);
    o[0] = d.out_features; o[1] = d.in_features; o[2] = d.weight_bits; o[3] = d.num_orders;
    o[4] = d.group_size; o[5] = d.keep_groups; o[6] = d.num_branches;
    for (int m = 0; m < PIPE_MAX_ORDERS; ++m) o[7 + m] = d.branch_orders[m];
  }
}
__global__ void write_header_kernel(uint32_t* hdr, pipe_layer_desc d) {
  if (threadIdx.x == 0) write_header(hdr, d);
}

__global__ void __launch_bounds__(256) chain_init_kernel(const __grid_constant__ ChainInitArgs p) {
  grid_wait();
  grid_release();
  const int64_t i0 = blockIdx.x * 256ll + threadIdx.x, step = gridDim.x * 256ll;
  if (i0 == 0) write_header(p.hdr, p.desc);
  for (int64_t i = i0; i < p.n_max; i += step) p.lvl_max[i] = 0u;
  for (int k = 0; k < p.lists; ++k)
    for (int64_t j = i0; j <= p.G; j += step) {
      p.cum[k][j] = static_cast<int32_t>(j);
      if (j < p.G) p.kept[k][j] = static_cast<int32_t>(j);
    }
}

// The chain's level storage inside the expansion workspace; false: the layer runs one pass per order.
struct ChainPlan {
  uint64_t temp, lvl_scale, lvl_max, lvl_of;   // byte offsets
  int temp_pitch;
};
static bool chain_fits(const LayerInfo& L, const float* W, int64_t ldw, ChainPlan* c) {
  if (L.keep_elems > 0 || L.score_mode != PIPE_SCORE_MAXABS) return false;
  if (L.I % 16 != 0 || round_up(L.I, kKernelKAlign) > kChainMaxI || L.G > kSelMaxGroups) return false;
  if ((reinterpret_cast<uintptr_t>(W) & 15) || ldw % 4 != 0) return false;
  const int levels = L.n_keep == L.G ? 0 : L.K - 1;   // levels that need storage
  // Many levels of which few are used (high orders that keep little of a large layer): a level costs 0.4 ps an element whether
  // a row uses it or not, an order 1.5 ps an element of its kept rows (and 2000 elements' worth a row) and 10 us of
  // selection, the first one 0.6 ps more for its maximum.  Measured, orders against chain, ternary: K = 16 16384 x 16384
  // gamma = 0.01 897 / 1831 us, 0.1 1430 / 1874, 0.2 2025 / 1934; 28672 x 4096 0.05 721 / 736, 0.1 901 / 755; 8192 x 8192
  // 0.01 426 / 478, 0.1 574 / 501; K = 8 16384 x 16384 0.01 692 / 817, 0.1 947 / 829, 8192 x 8192 0.01 295 / 233.
  const double n = static_cast<double>(L.O) * L.I;
  if (levels && 0.4 * L.K * n > 0.6 * n + 1.5 * L.lay.total_rows * (L.I + 2000.0) + 1e7 * (L.K - 1)) return false;
  c->temp_pitch = round_up(L.lay.canon_row_bytes, 16);
  uint64_t off = 0;
  c->temp = off;
  off += round_up<uint64_t>(static_cast<uint64_t>(levels) * L.O * c->temp_pitch, 256);
  c->lvl_scale = off;
  if (levels) off += round_up<uint64_t>(static_cast<uint64_t>(L.K) * L.O * 4, 256);
  c->lvl_max = off;
  if (levels) off += round_up<uint64_t>(static_cast<uint64_t>(L.K) * L.G * 4, 256);
  c->lvl_of = off;
  if (levels) off += round_up<uint64_t>(static_cast<uint64_t>(L.K) * L.n_keep * 4, 256);
  return off <= L.lay.expand_ws_bytes;   // (more than 32 bits of codes per element beyond order 1 does not fit)
}

}  // namespace pipe

using namespace pipe;

// In a stream capture a mark would not do: a launch on ANOTHER stream that has joined behind the expansion gets an edge of the same
// kind as one behind it on its own stream, programmatic, where outside of captures an event stands for full completion.  The
// expansion's last kernel releases its dependents early, so it is followed by an empty node, and what comes behind it has an ordinary edge.
// captured: the stream is in a capture.
static pipe_status close_in_capture(cudaStream_t s, bool* captured) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  cudaGraph_t graph = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t n = 0;
  cudaError_t e = cudaStreamGetCaptureInfo(s, &status, nullptr, &graph, &deps, &n);
  if (e != cudaSuccess || status != cudaStreamCaptureStatusActive) return cuda_ok(e);
  *captured = true;
  cudaGraphNode_t end = nullptr;
  e = cudaGraphAddEmptyNode(&end, graph, deps, n);
  if (e == cudaSuccess) e = cudaStreamUpdateCaptureDependencies(s, &end, 1, cudaStreamSetCaptureDependencies);
  return cuda_ok(e);
}

extern "C" pipe_status pipe_expand_weights(const pipe_layer_desc* desc, const float* d_W, int64_t ldw, void* d_blob,
                                           size_t blob_bytes, void* d_ws, size_t ws_bytes, void* stream) {
  LayerInfo L;
  pipe_status st = resolve_layer(desc, &L);
  if (st != PIPE_OK) return st;
  if (!d_W || !d_blob || !d_ws) return PIPE_ERR_INVALID_ARG;
  if (ldw < L.I) return PIPE_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(d_W) & 3) || (reinterpret_cast<uintptr_t>(d_blob) & (PIPE_BLOB_ALIGN - 1)) ||
      (reinterpret_cast<uintptr_t>(d_ws) & 255))
    return PIPE_ERR_ALIGNMENT;
  if (blob_bytes < L.lay.blob_bytes || ws_bytes < L.lay.expand_ws_bytes) return PIPE_ERR_WORKSPACE;
  int* status = device_status_word();
  if (!status) return PIPE_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  uint8_t* ws = static_cast<uint8_t*>(d_ws);
  const int64_t I4 = round_up(L.I, 4);
  float* resid = reinterpret_cast<float*>(ws);
  uint64_t off = round_up<uint64_t>(static_cast<uint64_t>(L.O) * I4 * 4, 256);
  float* a = reinterpret_cast<float*>(ws + off);
  off += round_up<uint64_t>(static_cast<uint64_t>(L.O) * 4, 256);
  float* score = reinterpret_cast<float*>(ws + off);          // G doubles for the L2 score, G floats otherwise
  double* score64 = reinterpret_cast<double*>(ws + off);
  off += round_up<uint64_t>(static_cast<uint64_t>(L.G) * 8, 256);
  int32_t* keep = reinterpret_cast<int32_t*>(ws + off);
  off += round_up<uint64_t>(static_cast<uint64_t>(L.G) * 4, 256);
  double* rowsq = nullptr;
  if (L.score_mode == PIPE_SCORE_L2) {
    rowsq = reinterpret_cast<double*>(ws + off);
    off += round_up<uint64_t>(static_cast<uint64_t>(L.O) * 8, 256);
  }
  uint32_t* mask_thr = nullptr;
  int32_t* mask_cut = nullptr;
  if (L.keep_elems > 0) {
    mask_thr = reinterpret_cast<uint32_t*>(ws + off);
    off += round_up<uint64_t>(static_cast<uint64_t>(L.O) * 4, 256);
    mask_cut = reinterpret_cast<int32_t*>(ws + off);
    off += round_up<uint64_t>(static_cast<uint64_t>(L.O) * 4, 256);
  }
  uint8_t* blob = static_cast<uint8_t*>(d_blob);

  // channel-block tables (entries 0 .. M) and decode-unit tables (entries M + 1 .. 2 M + 1: the same cut with the
  // layout's row limits), one thread block per table
  BlockTableArgs t;
  std::memset(&t, 0, sizeof(t));
  t.G = L.G;
  t.g = L.g;
  bool any = false, any_blk = false;
  for (int m = 0; m <= L.M; ++m) {
    const int k0 = (m < L.M) ? L.branch_begin[m] : 0, k1 = (m < L.M) ? L.branch_begin[m + 1] : L.K;
    if (L.lay.blk_off[m] != 0) {
      t.nk[m] = k1 - k0;
      for (int q = 0; q < k1 - k0; ++q) t.cum[m][q] = reinterpret_cast<const int32_t*>(blob + L.lay.cum_off[k0 + q]);
      t.out[m] = reinterpret_cast<int32_t*>(blob + L.lay.blk_off[m]);
      t.cap[m] = L.lay.blk_cap[m];
      // even blocks: the fewest blocks that could hold the cluster's rows, their mean size plus one group of slack
      int64_t R = 0;
      for (int k = k0; k < k1; ++k) R += L.lay.rows[k];
      t.limit[m] = block_row_limit(R, L.O, k1 - k0, L.g);
      any = any_blk = true;
    }
    if (L.lay.dec_off[m] != 0) {
      const int e = L.M + 1 + m;
      t.nk[e] = k1 - k0;
      for (int q = 0; q < k1 - k0; ++q) t.cum[e][q] = reinterpret_cast<const int32_t*>(blob + L.lay.cum_off[k0 + q]);
      t.out[e] = reinterpret_cast<int32_t*>(blob + L.lay.dec_off[m]);
      t.cap[e] = L.G;
      t.limit[e] = L.lay.dec_limit[m];
      any = true;
    }
  }
  const int tables = any ? 2 * (L.M + 1) : 0;

  ChainPlan plan;
  if (chain_fits(L, d_W, ldw, &plan)) {
    const bool dense = L.K == 1 || L.n_keep == L.G;
    ChainInitArgs ini;
    std::memset(&ini, 0, sizeof(ini));
    ChainArgs ch;
    std::memset(&ch, 0, sizeof(ch));
    SelectArgs sel;
    std::memset(&sel, 0, sizeof(sel));
    PlaceArgs pl;
    std::memset(&pl, 0, sizeof(pl));
    for (int k = 0; k < L.K; ++k) {
      ini.cum[k] = sel.cum[k] = reinterpret_cast<int32_t*>(blob + L.lay.cum_off[k]);
      ini.kept[k] = sel.kept[k] = reinterpret_cast<int32_t*>(blob + L.lay.kept_off[k]);
      pl.kept[k] = sel.kept[k];
      ChainOut& out = ch.out[k];
      out.codes = blob + L.lay.codes_off[k];
      out.kcodes = blob + L.lay.kcodes_off[k];
      out.wcodes = L.lay.wcodes_off[k] ? blob + L.lay.wcodes_off[k] : nullptr;
      out.scales = reinterpret_cast<float*>(blob + L.lay.scales_off[k]);
      pl.out[k] = out;
    }
    ini.hdr = reinterpret_cast<uint32_t*>(blob);
    ini.desc = *desc;
    ini.lists = dense ? L.K : 1;
    ini.G = L.G;
    ini.lvl_max = reinterpret_cast<uint32_t*>(ws + plan.lvl_max);
    ini.n_max = dense ? 0 : static_cast<int64_t>(L.K) * L.G;
    const int64_t init_n = ini.n_max > L.G + 1 ? ini.n_max : L.G + 1;
    const int64_t init_grid = ceil_div<int64_t>(init_n, 256);
    launch_overlapped(chain_init_kernel, dim3(static_cast<int>(init_grid < 64 ? init_grid : 64)), 256, 1, true, s, ini);
    ch.W = d_W;
    ch.ldw = ldw;
    ch.direct = dense ? L.K : 1;
    ch.temp = ws + plan.temp;
    ch.temp_pitch = plan.temp_pitch;
    ch.lvl_scale = reinterpret_cast<float*>(ws + plan.lvl_scale);
    ch.lvl_max = ini.lvl_max;
    ch.O = L.O; ch.I = L.I; ch.I_pad = round_up(L.I, kKernelKAlign); ch.g = L.g; ch.G = L.G; ch.K = L.K; ch.qmax = L.qmax;
    ch.canon_row_bytes = L.lay.canon_row_bytes;
    ch.status = status;
    // Two chunks per thread at 64 registers, or three at 80 where rows beyond 8192 elements leave an SM two or three blocks
    // and three chunks make it one more, to hide the blocks' barriers behind each other.  Whole expansions of 4096 rows,
    // int4 K = 4 / ternary K = 8 / int8 K = 2, two against three chunks: 8448 120 / 176 / 90 against 116 / 163 / 85 us,
    // 9216 126 / 178 / 92 against 120 / 165 / 87, 11008 157 / 210 / 114 against 144 / 196 / 102, 12288 161 / 220 / 121
    // against 149 / 200 / 108; as many blocks either way: 10240 131 / 181 / 98 against 134 / 189 / 98; shorter rows: 7168
    // 100 / 143 against 104 / 151, 8192 113 / 154 against 116 / 162.
    const int threads2 = round_up(ceil_div(ch.I_pad / 16, 2), 32), threads3 = round_up(ceil_div(ch.I_pad / 16, 3), 32);
    const bool long_rows = ch.I_pad > 8192 && ch.I_pad <= 12288 && 65536 / (threads3 * 80) > 65536 / (threads2 * 64);
    const int threads = long_rows ? threads3 : threads2;
#define PIPE_CHAIN(B)                                                                       \
  if (long_rows) launch_overlapped(expand_chain_kernel<B, 3, 256, 3>, dim3(L.O), threads, 1, true, s, ch);   \
  else launch_overlapped(expand_chain_kernel<B, 2, 512, 2>, dim3(L.O), threads, 1, true, s, ch);
    if (L.bits == 8) { PIPE_CHAIN(8) } else if (L.bits == 4) { PIPE_CHAIN(4) } else { PIPE_CHAIN(2) }
#undef PIPE_CHAIN
    count_launch(2);
    if (!dense) {
      sel.lvl_max = ini.lvl_max;
      sel.lvl_of = reinterpret_cast<int32_t*>(ws + plan.lvl_of);
      sel.G = L.G; sel.K = L.K; sel.n_keep = L.n_keep;
      // (two groups per thread up to 1024 of them, four up to 2048, eight beyond: seven orders of 512 groups 18 us, 24 with eight
      // groups per thread always)
      const int sel_per = L.G <= 1024 ? 2 : (L.G <= 2048 ? 4 : kSelPer);
      const int sel_threads = round_up(ceil_div(L.G, sel_per), 32);
      if (sel_per == 2) launch_overlapped(select_orders_kernel<2>, dim3(1), sel_threads, 1, true, s, sel);
      else if (sel_per == 4) launch_overlapped(select_orders_kernel<4>, dim3(1), sel_threads, 1, true, s, sel);
      else launch_overlapped(select_orders_kernel<kSelPer>, dim3(1), sel_threads, 1, true, s, sel);
      pl.lvl_of = sel.lvl_of;
      pl.lvl_scale = ch.lvl_scale;
      pl.temp = ch.temp;
      pl.temp_pitch = plan.temp_pitch;
      pl.O = L.O; pl.g = L.g; pl.n_keep = L.n_keep; pl.rows = L.n_keep * L.g;
      pl.canon_row_bytes = L.lay.canon_row_bytes;
      pl.kblocks = ceil_div(L.I, kKernelKAlign);
      pl.tables = tables;
      pl.tab = t;
      const int grid = tables + (L.K - 1) * L.n_keep;
      const bool whole = L.lay.canon_row_bytes % 16 == 0;
      if (L.bits == 8) launch_overlapped(place_orders_kernel<8, 4>, dim3(grid), kTableThreads, 1, true, s, pl);
      else if (L.bits == 4 && whole) launch_overlapped(place_orders_kernel<4, 4>, dim3(grid), kTableThreads, 1, true, s, pl);
      else if (L.bits == 4) launch_overlapped(place_orders_kernel<4, 2>, dim3(grid), kTableThreads, 1, true, s, pl);
      else if (whole) launch_overlapped(place_orders_kernel<2, 4>, dim3(grid), kTableThreads, 1, true, s, pl);
      else launch_overlapped(place_orders_kernel<2, 1>, dim3(grid), kTableThreads, 1, true, s, pl);
      count_launch(2);
    } else if (tables) {
      launch_overlapped(block_table_kernel, dim3(tables), kTableThreads, 1, true, s, t);
      count_launch(1);
    }
  } else {
    write_header_kernel<<<1, 32, 0, s>>>(reinterpret_cast<uint32_t*>(blob), *desc);
    count_launch(1);
    for (int k = 0; k < L.K; ++k) {
      int32_t* kept = reinterpret_cast<int32_t*>(blob + L.lay.kept_off[k]);
      int32_t* cum = reinterpret_cast<int32_t*>(blob + L.lay.cum_off[k]);
      const bool dense = (k == 0) || (L.n_keep == L.G);
      if (!dense && L.G <= kFusedGroups && L.score_mode == PIPE_SCORE_MAXABS) {
        group_select_kernel<<<1, kFusedGroups, 0, s>>>(a, L.G, L.g, L.n_keep, cum, kept);
        count_launch(1);
      } else {
        if (!dense && L.score_mode == PIPE_SCORE_L2) {
          // (a sparse order is never the first, so the current residual is in the workspace)
          row_sumsq_kernel<<<ceil_div(L.O, 8), 256, 0, s>>>(resid, I4, L.O, L.I, rowsq);
          group_score_l2_kernel<<<ceil_div(L.G, 256), 256, 0, s>>>(rowsq, L.G, L.g, score64);
          group_rank_kernel<double><<<ceil_div(L.G, 8), 256, 0, s>>>(score64, L.G, L.n_keep, keep);
          count_launch(3);
        } else if (!dense) {
          group_score_kernel<<<ceil_div(L.G, 256), 256, 0, s>>>(a, L.G, L.g, score);
          group_rank_kernel<float><<<ceil_div(L.G, 8), 256, 0, s>>>(score, L.G, L.n_keep, keep);
          count_launch(2);
        }
        group_compact_kernel<<<1, 1024, 0, s>>>(dense ? nullptr : keep, L.G, cum, kept);
        count_launch(1);
      }
      QuantizeRowsArgs q;
      q.src = (k == 0) ? d_W : resid;
      q.ld_src = (k == 0) ? ldw : I4;
      q.dst = (k + 1 < L.K) ? resid : nullptr;
      q.ld_dst = I4;
      q.a = a;
      q.first = (k == 0) ? 1 : 0;
      q.status = status;
      q.kept = kept;
      q.codes = blob + L.lay.codes_off[k];
      q.kcodes = blob + L.lay.kcodes_off[k];
      q.wcodes = L.lay.wcodes_off[k] ? blob + L.lay.wcodes_off[k] : nullptr;
      q.scales = reinterpret_cast<float*>(blob + L.lay.scales_off[k]);
      q.I = L.I; q.g = L.g; q.qmax = L.qmax;
      q.canon_row_bytes = L.lay.canon_row_bytes;
      q.kernel_row_bytes = L.lay.kernel_row_bytes;
      q.rows = L.lay.rows[k];
      q.mask_thr = nullptr;
      q.mask_cut = nullptr;
      if (L.keep_elems > 0 && k > 0) {
        row_topn_kernel<<<L.O, 256, 0, s>>>(resid, I4, L.I, L.keep_elems, mask_thr, mask_cut);
        count_launch(1);
        q.mask_thr = mask_thr;
        q.mask_cut = mask_cut;
      }
      const int rows = L.lay.rows[k];
      if (L.bits == 8) quantize_rows_kernel<8><<<rows, kRowThreads, 0, s>>>(q);
      else if (L.bits == 4) quantize_rows_kernel<4><<<rows, kRowThreads, 0, s>>>(q);
      else quantize_rows_kernel<2><<<rows, kRowThreads, 0, s>>>(q);
      count_launch(1);
    }
    if (tables) {
      block_table_kernel<<<tables, kTableThreads, 0, s>>>(t);
      count_launch(1);
    }
  }
  if (any_blk) {
    // the records of the blocks just cut
    BlockRecordArgs r;
    std::memset(&r, 0, sizeof(r));
    r.g = L.g;
    r.status = status;
    int max_cap = 0;
    for (int m = 0; m <= L.M; ++m) {
      if (L.lay.rec_off[m] == 0) continue;
      const int k0 = (m < L.M) ? L.branch_begin[m] : 0, k1 = (m < L.M) ? L.branch_begin[m + 1] : L.K;
      r.nk[m] = k1 - k0;
      for (int q = 0; q < k1 - k0; ++q) {
        r.cum[m][q] = reinterpret_cast<const int32_t*>(blob + L.lay.cum_off[k0 + q]);
        r.scales[m][q] = reinterpret_cast<const float*>(blob + L.lay.scales_off[k0 + q]);
      }
      r.tbl[m] = reinterpret_cast<const int32_t*>(blob + L.lay.blk_off[m]);
      r.out[m] = blob + L.lay.rec_off[m];
      r.cap[m] = L.lay.rec_cap[m];
      max_cap = max_cap > r.cap[m] ? max_cap : r.cap[m];
    }
    if (max_cap > 0) {
      launch_overlapped(block_record_kernel, dim3(max_cap, L.M + 1), 256, 1, true, s, r);
      count_launch(1);
    }
  }
  st = launch_status();
  bool captured = false;
  const pipe_status closed = close_in_capture(s, &captured);
  if (!captured) mark_expansion(s);   // a forward call that follows on this stream must not read the blob ahead of its dependency wait
  return st == PIPE_OK ? closed : st;
}

// ------------------------------------------------------------------------------------------------
// pipe_expand_weights_static: the same expansion for callers that cannot allocate device memory.
// Its workspace is the fixed array below, which is part of the library image: every GPU that
// loads the library holds PIPE_STATIC_SCRATCH_BYTES for it until the process exits.
namespace {

static __device__ __align__(256) unsigned char g_expand_scratch[PIPE_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_addr[kMaxDevices] = {nullptr};

// Device address of the array on the current device.  In host code the name g_expand_scratch is
// only a handle for the runtime, not an address a kernel could use; the address has to be asked
// for, once per device, while that device is current.
pipe_status static_scratch(void** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return PIPE_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_expand_scratch) != cudaSuccess || !p) return PIPE_ERR_CUDA;
    g_scratch_addr[dev] = p;
  }
  *out = g_scratch_addr[dev];
  return PIPE_OK;
}

}  // namespace

extern "C" pipe_status pipe_expand_weights_static(const pipe_layer_desc* desc, const float* d_W, int64_t ldw,
                                                  void* d_blob, size_t blob_bytes, void* stream) {
  LayerInfo L;
  pipe_status st = resolve_layer(desc, &L);
  if (st != PIPE_OK) return st;
  // the layer's workspace (fp32 residual + per-row and per-group arrays) must fit the fixed array
  if (L.lay.expand_ws_bytes > static_cast<uint64_t>(PIPE_STATIC_SCRATCH_BYTES)) return PIPE_ERR_WORKSPACE;
  void* scratch = nullptr;
  st = static_scratch(&scratch);
  if (st != PIPE_OK) return st;
  // Nothing in the workspace has to start at zero: levels and their maxima, or the residual, the row maxima, the group
  // scores and the keep flags, are all written by this call before it reads them, so what an earlier call left behind is
  // simply overwritten.
  return pipe_expand_weights(desc, d_W, ldw, d_blob, blob_bytes, scratch, PIPE_STATIC_SCRATCH_BYTES, stream);
}
