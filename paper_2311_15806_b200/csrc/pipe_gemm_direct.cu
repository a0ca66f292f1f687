// Small-token kernel of the expanded layer (Appendix B, Eq. 9; Sec. 3.2 for the branches): up to 16 tokens.
//
// With a handful of tokens the layer is bound by reading the packed weight codes from HBM once, so little stands between that
// stream and the registers that consume it.  A CTA owns a contiguous range of output channels of one branch; in every
// order of the branch that is a contiguous run of compacted rows, cut into groups of 8 rows.  Two groups -- of whatever
// orders, as long as they meet the same input -- are the 16 rows of a warp-level integer MMA (mma.sync m16n8k32: weights as
// the 16-row operand, tokens as the 8-column operand), so a branch of one dense and one half-empty order costs its 1.5
// orders and nothing is padded but the last pair.  A warp takes up to three pairs and every KS-th stage of the reduction axis
// (a reduction block of 128 codes, two of them with 2-bit codes) and brings its operands into a ring of its own with
// asynchronous copies of 16 bytes per lane: a lane reads back the weights that it copied itself, and no other warp is waited for.
// (Bulk copies cost an SM 50 to 60 ns each whatever their size: 57 MB in pieces of 512 bytes take 43 us, of 1.5 KB 14 to 19.)
// The warps of a CTA are dealt to its sets of pairs by their size, and the CTAs to the branches by their bytes.  At the end the
// warps add their exact int32 sums in shared memory and the fixed-order fp32 epilogue runs once per output.
#include <mutex>

#include "pipe_common.cuh"

namespace pipe {

namespace sd {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
// (one CTA per SM, with the next launch's beside it, leaves half of the warps and of the bytes in flight: 4096 -> 11008 -> 4096,
// int4, K = 4, M = 2, T = 1 and 13 with quantization 57 and 73 us, two 39 and 46)
constexpr int kCtasPerSm = 2;
constexpr int kPairs = 3;        // most pairs of row groups per warp
constexpr int kMaxDepth = 6;     // most stages of a warp's ring
constexpr int kMaxOrd = 8;       // orders per branch (of all predictors in a summed launch)

struct Params {
  ForwardArgs f;
  const uint8_t* kbase;             // lowest address of the streaming sections (16-byte aligned)
  uint32_t koff[PIPE_MAX_ORDERS];   // (kcodes of order k - kbase) / 16
  int kblocks;                      // reduction blocks of 128 codes
  int nstages;                      // stages of the reduction axis: a block, or two with 2-bit codes
  int depth, stage_bytes;           // ring of a warp
  int shift;                        // 8 - b
  int slabs;                        // O / 8
  int cta0[PIPE_MAX_ORDERS + 1];    // first CTA of every branch, then the total
  int nkmax;                        // most orders any branch has
  int set_pairs;                    // most pairs of a set: kPairs, or fewer where the ring would be too shallow
  int own_max, pairs_max;           // most slabs (of 8 channels) / pairs of row groups any CTA can have
  uint32_t split_mask;              // SUMMED: bit k marks the order (k > 0) that opens the next predictor
  int8_t input[PIPE_MAX_ORDERS];    // SUMMED: the predictor whose input an order meets
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
// 16 bytes from global to shared memory, past L1; the second form brings `real` of them and zeros.
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16_part(uint32_t dst, const void* src, int real) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(real) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All but the newest n groups of this lane (n < kMaxDepth) have landed.
__device__ __forceinline__ void copy_wait(int n) {
  switch (n) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
  }
}
__device__ __forceinline__ uint4 lds128(const uint8_t* p) { return *reinterpret_cast<const uint4*>(p); }

__device__ __forceinline__ void mma_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The CTA's rows: order ko has `rows` of them from compacted row `row0` on, which are the 8-row groups g0 .. of the CTA's pool.
// Groups of one input are consecutive; the next input's start at an even number, so no pair mixes inputs.
struct Rows {
  int row0[kMaxOrd], rows[kMaxOrd], g0[kMaxOrd];
};

// One warp's work: N pairs from pair0 on, the stages ki, ki + ks, ... of the reduction axis.  before_x, after_x: what the warp has
// to do once between its first weight copies and its first activation copies (the dependency wait) and behind those.
template <int BITS, int NT, int N, bool ZP, class BeforeX, class AfterX>
__device__ __forceinline__ void run_pairs(const Params& p, const Rows& rows, uint8_t* ring, int* sums, int k0, int nk, int pair0, int in, int ki, int ks,
                                          BeforeX before_x, AfterX after_x) {
  constexpr int KB = BITS == 2 ? 2 : 1;             // reduction blocks of a stage
  constexpr int SUB = BITS == 8 ? 2 : 1;            // 16-byte chunks per lane, group and stage
  constexpr int XCH = 8 / BITS;                     // 16-byte activation chunks per weight chunk and token
  constexpr int kRow16 = BITS;                      // 16-byte chunks of a row in one reduction block
  constexpr uint32_t kGroupBytes = 512 * SUB;       // of a group in a stage
  constexpr uint32_t kXOff = 2 * N * kGroupBytes;
  const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const int T = static_cast<int>(p.f.T);
  // ---- where the groups lie: lane l < 2 N looks up group 2 pair0 + l
  uint32_t off = 0, str = 0;
  bool here = false;
  if (lane < 2 * N) {
    const int gi = 2 * pair0 + lane;
    for (int ko = 0; ko < nk; ++ko) {
      const int r = 8 * (gi - rows.g0[ko]);
      if (r >= 0 && r < rows.rows[ko]) {
        off = p.koff[k0 + ko] + static_cast<uint32_t>(rows.row0[ko] + r) * kRow16;
        str = static_cast<uint32_t>(p.f.order[k0 + ko].rows) * kRow16;
        here = true;
      }
    }
  }
  const uint32_t present = __ballot_sync(0xffffffffu, here);
  // this lane's chunk of a group's rows of one block, in 16-byte units (2 bits: lanes 2, 3 of a quad take the second block;
  // 8 bits: and the chunk four further on)
  const uint32_t place = BITS == 4 ? lane : (BITS == 8 ? gid * 8 + tig : gid * 2 + (tig & 1));
  uint32_t offs[2 * N], strs[2 * N];
#pragma unroll
  for (int h = 0; h < 2 * N; ++h) {
    offs[h] = __shfl_sync(0xffffffffu, off, h) + place;
    strs[h] = __shfl_sync(0xffffffffu, str, h);
  }
  const uint32_t stage0 = smem_u32(ring), depth = static_cast<uint32_t>(p.depth), x_bytes = static_cast<uint32_t>(T) * 128u;
  const int mine = ki < p.nstages ? (p.nstages - ki + ks - 1) / ks : 0;   // stages of this warp
  auto issue_w = [&](int i, uint32_t slot) {
    const int kb = (ki + i * ks) * KB + (BITS == 2 ? tig >> 1 : 0);
    const uint32_t dst = stage0 + slot * p.stage_bytes + lane * 16;
    if (BITS == 2 && kb >= p.kblocks) return;   // (the second block of the last stage may lie beyond the axis)
#pragma unroll
    for (int h = 0; h < 2 * N; ++h)
      if ((present >> h) & 1u) {
        const uint8_t* src = p.kbase + (static_cast<uint64_t>(offs[h] + static_cast<uint32_t>(kb) * strs[h]) << 4);
#pragma unroll
        for (int sub = 0; sub < SUB; ++sub) copy16(dst + h * kGroupBytes + sub * 512, src + 64 * sub);
      }
  };
  // activations: eight lanes bring a row's 128 bytes of a block
  const int8_t* x_src = p.f.branch[in].xq + static_cast<int64_t>(lane >> 3) * p.f.ldxq + 16 * (lane & 7);
  auto issue_x = [&](int i, uint32_t slot) {
    const uint32_t dst = stage0 + slot * p.stage_bytes + kXOff + lane * 16;
#pragma unroll
    for (int b = 0; b < KB; ++b) {
      const int kb = (ki + i * ks) * KB + b, left = p.f.I - (kb * 128 + 16 * (lane & 7));
      if (KB == 2 && kb >= p.kblocks) break;
      const int8_t* src = x_src + static_cast<int64_t>(kb) * 128;
      for (int t = lane >> 3; t < T; t += 4, src += 4 * p.f.ldxq) {
        const uint32_t d = dst + b * x_bytes + (t - (lane >> 3)) * 128;
        if (left >= 16) copy16(d, src);
        else copy16_part(d, left > 0 ? src : p.f.branch[in].xq, left > 0 ? left : 0);
      }
    }
  };
  for (uint32_t i = 0; i < depth; ++i) {
    if (static_cast<int>(i) < mine) issue_w(i, i);
    copy_commit();
  }
  before_x();
  for (uint32_t i = 0; i < depth; ++i) {
    if (static_cast<int>(i) < mine) issue_x(i, i);
    copy_commit();
  }
  after_x();
  int acc[N][NT][4];
#pragma unroll
  for (int u = 0; u < N; ++u)
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[u][t][e] = 0;
  uint32_t slot = 0;
  for (int i = 0; i < mine; ++i) {
    copy_wait(p.depth - 1);
    __syncwarp();   // (the activations of the stage are other lanes' copies)
    const uint8_t* st = ring + slot * p.stage_bytes;
    const int kb = (ki + i * ks) * KB;
#pragma unroll
    for (int sub = 0; sub < SUB; ++sub) {
      const int kbs = BITS == 2 ? tig >> 1 : 0;
      // (a second block beyond the axis holds stale bytes: such lanes contribute zero weights)
      const bool live = BITS != 2 || kb + kbs < p.kblocks;
      uint4 w[2 * N];
#pragma unroll
      for (int h = 0; h < 2 * N; ++h) {
        w[h] = make_uint4(0, 0, 0, 0);
        if (live && ((present >> h) & 1u)) w[h] = lds128(st + h * kGroupBytes + sub * 512 + lane * 16);
      }
      const int byte = BITS == 8 ? (tig + 4 * sub) * 16 : (BITS == 4 ? tig * 32 : (tig & 1) * 64);   // of its 128 in the block
#pragma unroll
      for (int v = 0; v < XCH; ++v) {
        uint4 x[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          x[t] = make_uint4(0, 0, 0, 0);
          if (gid + 8 * t < T) x[t] = lds128(st + kXOff + kbs * x_bytes + (gid + 8 * t) * 128 + byte + 16 * v);
          // (asymmetric activations: the last token column is fed ones, its sums are the row sums of the codes)
          if (ZP && t == NT - 1 && gid == 7) x[t] = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
        }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int mm = 2 * v + m;
#pragma unroll
          for (int u = 0; u < N; ++u) {
            uint32_t a0, a1, b0, b1;
            mma_frag<BITS>(w[2 * u], mm, a0, a1);
            mma_frag<BITS>(w[2 * u + 1], mm, b0, b1);
#pragma unroll
            for (int t = 0; t < NT; ++t) mma_s8(acc[u][t], a0, b0, a1, b1, m ? x[t].z : x[t].x, m ? x[t].w : x[t].y);
          }
        }
      }
    }
    __syncwarp();   // every lane has read the stage
    if (i + p.depth < mine) {
      issue_w(i + p.depth, slot);
      issue_x(i + p.depth, slot);
    }
    copy_commit();
    slot = slot + 1 == depth ? 0u : slot + 1;
  }
  copy_wait(0);
#pragma unroll
  for (int u = 0; u < N; ++u)
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) atomicAdd(sums + (((pair0 + u) * NT + t) * 4 + e) * 32 + lane, acc[u][t][e]);
}

// SUMMED: a summed ensemble in one launch (every predictor's chain starts from zero, the bias closes the first one, the chains
// are added in ascending predictor order), whether the predictors share their input or not.
// ZP: asymmetric activations, sum_i (c - z) q = sum_i c q - z sum_i q.
// (Two CTAs per SM leave a thread 128 registers.  Five of the 24 forms spill some: 2 bits with two token tiles, 12 to 24 bytes stored, and the
// plain 8-bit one with one tile, 16.)
template <int BITS, int NT, bool SUMMED, bool ZP>
__global__ void __launch_bounds__(kThreads, 2) direct_forward_kernel(const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ Rows rows;
  __shared__ float sx_s[PIPE_MAX_ORDERS];
  __shared__ int zp_s[PIPE_MAX_ORDERS];
  uint8_t* ring_gen = smem_raw + (((smem_u32(smem_raw) + 127u) & ~127u) - smem_u32(smem_raw));
  int* sums = reinterpret_cast<int*>(ring_gen + kWarps * p.depth * p.stage_bytes);   // [pairs_max][NT][4][32]
  int* loc = sums + p.pairs_max * NT * 128;                            // [own_max][nkmax]: group of the pool, or -1
  float* bias_s = reinterpret_cast<float*>(loc + p.own_max * p.nkmax); // [own_max][8]
  float* scale = bias_s + p.own_max * 8;                               // [own_max][nkmax][8]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // Everything that belongs to the layer -- row lists, scales, the first weights -- is read ahead of the wait for the launch before:
  // the layer is complete when a CTA starts (a launch directly behind an expansion is an ordinary one, see launch_direct).  This
  // launch's dependents start at once: the launch before was complete, or past this same point, when this CTA started, so no
  // expansion queued earlier is still running beside them.
  grid_release();
  int b = 0;
  if (!SUMMED)
    while (b + 1 < p.f.num_branches && static_cast<int>(blockIdx.x) >= p.cta0[b + 1]) ++b;
  const BranchArgs& br = p.f.branch[b];
  const int k0 = br.k_begin, nk = br.k_end - br.k_begin;
  const int ctas = p.cta0[b + 1] - p.cta0[b], ci = static_cast<int>(blockIdx.x) - p.cta0[b];
  const int base = p.slabs / ctas, rem = p.slabs % ctas;
  const int s0 = ci * base + min(ci, rem), own = base + (ci < rem ? 1 : 0);   // this CTA's slabs of 8 channels
  auto input_of = [&](int ko) { return SUMMED ? static_cast<int>(p.input[ko]) : b; };
  uint8_t* ring = ring_gen + warp * p.depth * p.stage_bytes;

  if (warp == 0) {
    if (lane < nk) {
      const int32_t* cum = p.f.order[k0 + lane].cum;
      const int r0 = rows_before(cum, s0 * 8, p.f.O, p.f.g);
      rows.row0[lane] = r0;
      rows.rows[lane] = rows_before(cum, (s0 + own) * 8, p.f.O, p.f.g) - r0;
    }
    __syncwarp();
    if (lane == 0) {
      int g = 0;
      for (int ko = 0; ko < nk; ++ko) {
        if (ko > 0 && input_of(ko) != input_of(ko - 1)) g = (g + 1) & ~1;
        rows.g0[ko] = g;
        g += rows.rows[ko] >> 3;
      }
    }
  } else {
    for (int e = tid - 32; e < p.pairs_max * NT * 128; e += kThreads - 32) sums[e] = 0;
  }
  __syncthreads();
  // ---- sets of up to set_pairs pairs of one input, evenly cut: set number s -> first pair, pairs, input (0 pairs: no such set)
  auto find_set = [&](int s, int& pair0, int& n, int& in) {
    n = 0;
    for (int ko = 0; ko < nk;) {
      in = input_of(ko);
      const int first = rows.g0[ko];
      int end = first;
      for (; ko < nk && input_of(ko) == in; ++ko) end = rows.g0[ko] + (rows.rows[ko] >> 3);
      const int pairs = (end - first + 1) >> 1, sets = (pairs + p.set_pairs - 1) / p.set_pairs;
      if (s < sets) {
        const int small = pairs / sets, more = pairs % sets;
        n = small + (s < more ? 1 : 0);
        pair0 = (first >> 1) + s * small + min(s, more);
        return;
      }
      s -= sets;
    }
  };
  int pair0 = 0, n = 0, in = 0;
  find_set(lane, pair0, n, in);
  const int nsets = __popc(__ballot_sync(0xffffffffu, n > 0));   // (32: that many or more)
  int set = warp, ki = 0, ks = 1;
  if (nsets <= kWarps) {
    // the warps left over go, one by one, to the set with most pairs per warp
    int cnt = n > 0 ? 1 : 0;
    for (int i = nsets; i < kWarps; ++i) {
      const uint32_t load = cnt ? static_cast<uint32_t>(n) * 840u / static_cast<uint32_t>(cnt) : 0u;
      const uint32_t top = __reduce_max_sync(0xffffffffu, load);
      if (lane == __ffs(__ballot_sync(0xffffffffu, load == top)) - 1) ++cnt;
    }
    int before = 0;
    for (int s = 0; s < nsets; ++s) {
      const int c = __shfl_sync(0xffffffffu, cnt, s);
      if (warp >= before && warp < before + c) {
        set = s;
        ki = warp - before;
        ks = c;
      }
      before += c;
    }
  }
  // ---- what every thread does once: the dependency wait behind its first weight copies, the tables of the epilogue behind its
  // first activation copies
  bool waited = false, made = false;
  auto wait_once = [&]() {
    if (!waited) grid_wait();
    waited = true;
  };
  auto tables_once = [&]() {
    if (made) return;
    made = true;
    if (tid < PIPE_MAX_ORDERS && (SUMMED ? tid < p.f.num_branches : tid == b)) {
      sx_s[tid] = __ldcg(p.f.branch[tid].sx);
      if (ZP) zp_s[tid] = p.f.branch[tid].zp ? __ldcg(p.f.branch[tid].zp) : 0;
    }
    for (int e = tid; e < own * 8; e += kThreads) bias_s[e] = p.f.bias && br.add_bias ? __ldcg(p.f.bias + s0 * 8 + e) : 0.f;
    for (int e = tid; e < own * nk; e += kThreads) {
      const int li = e / nk, ko = e % nk;
      const int c0 = (s0 + li) * 8, j = c0 / p.f.g;
      const int32_t* cum = p.f.order[k0 + ko].cum;
      const int lo = __ldg(cum + j), hi = __ldg(cum + j + 1);
      const int row = lo * p.f.g + c0 % p.f.g;
      loc[e] = hi > lo ? rows.g0[ko] + ((row - rows.row0[ko]) >> 3) : -1;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), c = a;
      if (hi > lo) {   // (the section is 256-byte aligned, the row a multiple of 8)
        const float4* src = reinterpret_cast<const float4*>(p.f.order[k0 + ko].scales + row);
        a = __ldg(src);
        c = __ldg(src + 1);
      }
      float* dst = scale + 8 * e;
      dst[0] = a.x, dst[1] = a.y, dst[2] = a.z, dst[3] = a.w, dst[4] = c.x, dst[5] = c.y, dst[6] = c.z, dst[7] = c.w;
    }
  };
  for (;; set += kWarps) {
    find_set(set, pair0, n, in);
    if (n == 0) break;
    if (n == 1) run_pairs<BITS, NT, 1, ZP>(p, rows, ring, sums, k0, nk, pair0, in, ki, ks, wait_once, tables_once);
    else if (n == 2) run_pairs<BITS, NT, 2, ZP>(p, rows, ring, sums, k0, nk, pair0, in, ki, ks, wait_once, tables_once);
    else run_pairs<BITS, NT, kPairs, ZP>(p, rows, ring, sums, k0, nk, pair0, in, ki, ks, wait_once, tables_once);
    if (nsets <= kWarps) break;
  }
  wait_once();     // (a warp without a set)
  tables_once();
  __syncthreads();

  // ---- fixed-order epilogue, one output per thread at a time, neighbouring threads on neighbouring channels
  const int nch = own * 8, items = nch * static_cast<int>(p.f.T);
  const bool bias = p.f.bias && br.add_bias;
  const float os = p.f.q8_out ? __ldcg(br.out_scale) : 0.f;
  if (p.f.q8_out && tid == 0 && !(os >= 0.f && os < __uint_as_float(0x7f800000u))) raise_status(p.f.status, PIPE_ERR_INVALID_ARG);
  for (int it = tid; it < items; it += kThreads) {
    const int tok = it / nch, ch = it - tok * nch, li = ch >> 3, r = ch & 7;
    const float bv = bias_s[ch];
    float y = 0.f, ysum = 0.f;
    bool first_chain = true;
    auto close_chain = [&]() {
      if (first_chain) ysum = bias ? __fadd_rn(y, bv) : y;
      else ysum = __fadd_rn(ysum, y);
      first_chain = false;
      y = 0.f;
    };
    // accumulator registers 0, 1 of lane 4 r + q hold the tokens 2 q, 2 q + 1 of a pair's first group, 2, 3 of its second
    const int* cell0 = sums + (tok >> 3) * 128 + (tok & 1) * 32 + r * 4 + ((tok & 7) >> 1);
    for (int ko = 0; ko < nk; ++ko) {
      if (SUMMED && ((p.split_mask >> ko) & 1u)) close_chain();
      const int gi = loc[li * nk + ko];
      if (gi < 0) continue;
      const int m = input_of(ko);
      int a = cell0[(gi >> 1) * NT * 128 + (gi & 1) * 64] >> p.shift;   // exact: the sum carries a factor 2^shift
      // (the row's sum of codes: the last token column, i.e. the second column of lane 4 r + 3 of the last token tile)
      if (ZP) a -= zp_s[m] * (sums[((gi >> 1) * NT + NT - 1) * 128 + (gi & 1) * 64 + 32 + r * 4 + 3] >> p.shift);
      y = __fmaf_rn(__int2float_rn(a), __fmul_rn(scale[(li * nk + ko) * 8 + r], sx_s[m]), y);
      if (p.f.partials) {
        const int row = rows.row0[ko] + (gi - rows.g0[ko]) * 8 + r;
        p.f.partials[static_cast<int64_t>(tok) * p.f.total_rows + p.f.order[k0 + ko].row_off + row] = a;
      }
    }
    float v = y;
    if (SUMMED) {
      close_chain();
      v = ysum;
    } else if (bias) {
      v = __fadd_rn(v, bv);
    }
    const int c = s0 * 8 + ch;
    if (p.f.q8_out) {
      // inner layer of a branch: sigma, then the next layer's input quantizer (Sec. 3.2)
      br.yq[static_cast<int64_t>(tok) * p.f.ldyq + c] = static_cast<int8_t>(quant_lane_exact(apply_activation(v, p.f.relu), os));
      continue;
    }
    float* dst = br.y + static_cast<int64_t>(tok) * p.f.ldy + c;
    if (br.accumulate) v = __fadd_rn(__ldcg(dst), v);
    *dst = v;
  }
}

using Kernel = void (*)(const Params);

static Kernel pick_kernel(int bits, int nt, bool summed, bool zp) {
#define PIPE_SD_PICK(B)                                                                                               \
  if (nt == 1)                                                                                                        \
    return summed ? (zp ? direct_forward_kernel<B, 1, true, true> : direct_forward_kernel<B, 1, true, false>)         \
                  : (zp ? direct_forward_kernel<B, 1, false, true> : direct_forward_kernel<B, 1, false, false>);      \
  return summed ? (zp ? direct_forward_kernel<B, 2, true, true> : direct_forward_kernel<B, 2, true, false>)           \
                : (zp ? direct_forward_kernel<B, 2, false, true> : direct_forward_kernel<B, 2, false, false>);
  if (bits == 8) { PIPE_SD_PICK(8) }
  if (bits == 4) { PIPE_SD_PICK(4) }
  PIPE_SD_PICK(2)
#undef PIPE_SD_PICK
}

// SM count, and the largest dynamic shared memory every instantiation may be launched with (set once per device).
struct DeviceSetup {
  int sms = 0, smem_max = 0, smem_half = 0;   // dynamic shared memory of a CTA alone on its SM, and of one of two
  bool ok = false;
};
static const DeviceSetup& device_setup() {
  constexpr int kMaxDevices = 64;
  static DeviceSetup setups[kMaxDevices];
  static std::once_flag once[kMaxDevices];
  static const DeviceSetup bad;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return bad;
  std::call_once(once[dev], [dev] {
    DeviceSetup& d = setups[dev];
    int optin = 0, sm = 0, reserved = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return;
    if (cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) return;
    if (cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess) return;
    if (cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return;
    constexpr int kStatic = 1024;   // (the kernel's static shared memory is below this)
    d.smem_max = optin - kStatic;
    d.smem_half = sm / 2 - reserved - kStatic;
    for (int bits = 2; bits <= 8; bits *= 2)
      for (int i = 0; i < 8; ++i)
        if (cudaFuncSetAttribute(pick_kernel(bits, 1 + (i & 1), (i & 2) != 0, (i & 4) != 0), cudaFuncAttributeMaxDynamicSharedMemorySize, d.smem_max) != cudaSuccess)
          return;
    d.ok = true;
  });
  return setups[dev];
}

}  // namespace sd

// summed: a.branch[0 .. num_branches) are the predictors of a summed ensemble, whose orders run as one cluster.
// (queue = false: only say whether the kernel takes the call; any: also what the streaming kernel is ahead on, see the two rules below)
static pipe_status launch_direct(const ForwardArgs& a, cudaStream_t stream, bool summed, bool any, bool queue = true) {
  using namespace sd;
  const bool zp = has_zero_point(a);   // (its row sums take the place of a token)
  if (a.T > (zp ? 15 : 16) || a.g % 8 != 0 || a.O % 8 != 0 || (zp && a.q8_out) || a.conv_on) return PIPE_ERR_UNSUPPORTED;
  if (a.ldxq % 16 != 0) return PIPE_ERR_UNSUPPORTED;
  for (int m = 0; m < a.num_branches; ++m)
    if (reinterpret_cast<uintptr_t>(a.branch[m].xq) & 15) return PIPE_ERR_UNSUPPORTED;
  const DeviceSetup& ds = device_setup();
  if (!ds.ok) return PIPE_ERR_CUDA;
  Params p;
  p.f = a;
  p.split_mask = 0;
  int units = a.num_branches, inputs = 1;
  if (summed) {
    const int first = a.branch[0].k_begin;
    for (int m = 0; m < a.num_branches; ++m) {
      if (m > 0 && (a.branch[m].k_begin != a.branch[m - 1].k_end || a.branch[m].y != a.branch[0].y)) return PIPE_ERR_UNSUPPORTED;
      if (a.branch[m].k_end - first > kMaxOrd) return PIPE_ERR_UNSUPPORTED;
      if (m > 0) p.split_mask |= 1u << (a.branch[m].k_begin - first);
      // (predictors on the first one's input share its pairs)
      const bool same = a.branch[m].xq == a.branch[0].xq && a.branch[m].sx == a.branch[0].sx && a.branch[m].zp == a.branch[0].zp;
      for (int k = a.branch[m].k_begin; k < a.branch[m].k_end; ++k) p.input[k - first] = static_cast<int8_t>(same ? 0 : m);
    }
    inputs = a.num_branches;   // (a bound on the changes of input along the orders)
    p.f.branch[0].k_end = a.branch[a.num_branches - 1].k_end;
    p.f.branch[0].accumulate = 0;
    units = 1;
  }
  int k_lo = PIPE_MAX_ORDERS, k_hi = 0;
  p.nkmax = 0;
  for (int m = 0; m < units; ++m) {
    const int nk = p.f.branch[m].k_end - p.f.branch[m].k_begin;
    p.nkmax = nk > p.nkmax ? nk : p.nkmax;
    k_lo = p.f.branch[m].k_begin < k_lo ? p.f.branch[m].k_begin : k_lo;
    k_hi = p.f.branch[m].k_end > k_hi ? p.f.branch[m].k_end : k_hi;
  }
  if (p.nkmax > kMaxOrd) return PIPE_ERR_UNSUPPORTED;
  p.kblocks = ceil_div(a.I, 128);
  p.nstages = a.bits == 2 ? ceil_div(p.kblocks, 2) : p.kblocks;
  p.shift = 8 - a.bits;
  p.slabs = a.O / 8;
  p.kbase = a.order[k_lo].kcodes;
  for (int k = k_lo; k < k_hi; ++k) p.kbase = a.order[k].kcodes < p.kbase ? a.order[k].kcodes : p.kbase;
  int64_t rows[PIPE_MAX_ORDERS] = {}, total = 0;
  for (int m = 0; m < units; ++m) {
    for (int k = p.f.branch[m].k_begin; k < p.f.branch[m].k_end; ++k) rows[m] += a.order[k].rows;
    total += rows[m];
  }
  for (int k = k_lo; k < k_hi; ++k) {
    const uint64_t d = static_cast<uint64_t>(a.order[k].kcodes - p.kbase);
    if ((d & 15) || ((d + static_cast<uint64_t>(a.order[k].rows) * a.kernel_row_bytes) >> 4) >= 0xffffffffull) return PIPE_ERR_UNSUPPORTED;
    p.koff[k] = static_cast<uint32_t>(d >> 4);
  }
  // CTAs to the branches by their rows.  Layers that leave a CTA little (below two pair-stages per warp) get half of them: fewer
  // warps without a stage, fewer set-ups (3072 x 768, M = 2 6.6 us with two CTAs per SM).
  const int ctas = total / 16 * p.nstages < static_cast<int64_t>(2 * kWarps * kCtasPerSm) * ds.sms ? ds.sms : kCtasPerSm * ds.sms;
  if (units > ctas) return PIPE_ERR_UNSUPPORTED;
  int share[PIPE_MAX_ORDERS], used = 0;
  for (int m = 0; m < units; ++m) {
    const int64_t n = static_cast<int64_t>(ctas) * rows[m] / total;
    share[m] = static_cast<int>(n < 1 ? 1 : (n > p.slabs ? p.slabs : n));
    used += share[m];
  }
  for (; used < ctas; ++used) {   // (what the divisions left over: to the branch with most rows per CTA)
    int best = -1;
    for (int m = 0; m < units; ++m)
      if (share[m] < p.slabs && (best < 0 || rows[m] * share[best] > rows[best] * share[m])) best = m;
    if (best < 0) break;
    ++share[best];
  }
  p.cta0[0] = 0;
  p.own_max = 0;
  for (int m = 0; m < units; ++m) {
    p.cta0[m + 1] = p.cta0[m] + share[m];
    const int own = ceil_div(p.slabs, share[m]);
    p.own_max = own > p.own_max ? own : p.own_max;
  }
  p.pairs_max = (p.own_max * p.nkmax + inputs + 1) / 2;
  const int nt = a.T <= (zp ? 7 : 8) ? 1 : 2;
  // The warps' rings: as deep as half of an SM's shared memory allows, with sets of two pairs where three would leave less than
  // two stages (8 bits from 8 tokens on, 2 bits from 13), then of one.  A CTA that takes more than half of an SM makes the grid two
  // rounds (4096 x 4096 int8 K = 2, T = 8 10 -> 18 us): the whole of an SM only where even that does not fit, whose tables are those of
  // 100 thousand channels and more.
  const int64_t tables = 128 + static_cast<int64_t>(p.pairs_max) * nt * 512 + static_cast<int64_t>(p.own_max) * (p.nkmax * 36 + 32);
  int64_t depth = 0;
  for (p.set_pairs = kPairs; p.set_pairs > 0; --p.set_pairs) {
    p.stage_bytes = 2 * p.set_pairs * (a.bits == 8 ? 1024 : 512) + (a.bits == 2 ? 2 : 1) * static_cast<int>(a.T) * 128;
    depth = (ds.smem_half - tables) / (kWarps * p.stage_bytes);
    if (depth >= 2 || depth >= p.nstages) break;
  }
  const bool two_rounds = p.set_pairs == 0;
  if (two_rounds) {
    p.set_pairs = 1;
    depth = (ds.smem_max - tables) / (kWarps * p.stage_bytes);
  }
  if (depth > kMaxDepth) depth = kMaxDepth;
  if (depth > p.nstages) depth = p.nstages;
  if (depth < 1) return PIPE_ERR_UNSUPPORTED;
  // Two rounds cost by the rows, the weight-streaming kernel by the slabs and the positions of their order pairs, half empty or not.
  // So they pay on one token tile where a branch has more than four orders (eight positions) and at most three rows per output channel
  // (us, streaming / here: 128256 x 2048 int4 K = 8, 2.75 rows, T = 1 and 8 200 / 154 and 200 / 180; 128256 x 2048 int8 K = 5, two rows, T = 8
  // 183 / 139; 128256 x 1024 int4 K = 6, 3.5 rows, T = 1 104 / 120; four orders and fewer: 200000 x 1024 K = 4, T = 1 90 / 129, 128256 x 2048
  // K = 4 M = 2, T = 8 94 / 169, K = 6 M = 2 152 / 225; two token tiles: 128256 x 4096 K = 4, T = 16 217 / 338, 98304 x 2048 K = 8 169 / 223).
  // 2 bits: 65536 x 2048 K = 8, T = 8 75 / 85, M = 2 74 / 90.
  if (two_rounds && !any && (nt > 1 || a.bits == 2 || p.nkmax <= 4 || total > 3 * static_cast<int64_t>(a.O) * units)) return PIPE_ERR_UNSUPPORTED;
  // 2 bits, two token tiles, sets of one pair: a stage's activations, 256 codes of every token, are more than twice its weights, and every set
  // brings them; the streaming kernel brings them once per CTA (8192 x 8192 K = 8 M = 4, T = 16 58 / 82 us, 8192 x 4096 M = 2 28 / 44,
  // 11008 x 2048 23 / 28; kept rows a quarter: 19.4 / 18.6).  Sets of two pairs: T = 13 58 / 45, 8192 x 4096 28.4 / 25.4, 4096 x 4096 K = 4,
  // T = 16 11.2 / 9.9, 11008 x 4096 K = 3 20.8 / 16.0, 4096 x 11008 K = 6 M = 2 22.6 / 23.6.  One token tile, one pair: 65536 x 2048 K = 8, T = 6
  // 75 / 52.
  if (a.bits == 2 && nt > 1 && p.set_pairs < 2 && !any) return PIPE_ERR_UNSUPPORTED;
  p.depth = static_cast<int>(depth);
  if (!queue) return PIPE_OK;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = a.blob_settled ? 1 : 0;   // (not where the blob may be under construction)
  cfg.gridDim = dim3(p.cta0[units], 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(tables + depth * kWarps * p.stage_bytes);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, pick_kernel(a.bits, nt, summed, zp), p) != cudaSuccess) return PIPE_ERR_CUDA;
  count_launch(1);
  return launch_status();
}

pipe_status forward_direct(const ForwardArgs& a, cudaStream_t stream, bool any) {
  if (a.T == 0) return PIPE_OK;
  const bool sum_mode = a.num_branches > 1 && a.branch[1].accumulate;
  if (!sum_mode) return launch_direct(a, stream, false, any);
  // one launch for predictors that share their input, or two predictors of at most two orders each on inputs of their own; declined,
  // it is for the weight-streaming kernel, which also takes them together
  bool together = true;
  for (int m = 1; m < a.num_branches; ++m)
    together = together && a.branch[m].xq == a.branch[0].xq && a.branch[m].sx == a.branch[0].sx && a.branch[m].zp == a.branch[0].zp;
  together = together || (a.num_branches == 2 && a.branch[0].k_end - a.branch[0].k_begin <= 2 && a.branch[1].k_end - a.branch[1].k_begin <= 2);
  // Predictors of more orders than one launch takes are one launch each: the streaming kernel takes no more of them together either, and
  // its launches are the slower ones (shared input, cold weights, us, streaming / here: 4096 x 4096 int4 K = 12, M = 6, T = 1, 8, 16
  // 55.5 / 47.6, 56.9 / 48.4, 66.8 / 51.7; 2048 x 2048 int8 K = 10, M = 3 27.3 / 12.8, 28.1 / 13.3, 26.3 / 14.7).
  together = together && a.branch[a.num_branches - 1].k_end - a.branch[0].k_begin <= sd::kMaxOrd;
  if (together) return launch_direct(a, stream, true, any);
  return launch_each_predictor(a, [&](const ForwardArgs& one, bool queue) { return launch_direct(one, stream, false, any, queue); });
}

}  // namespace pipe
