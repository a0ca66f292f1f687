// pipe_quantize_act / pipe_quantize_act_ex: per-tensor quantization of the layer input (Appendix B, Eq. 9: the layer
// consumes Q(x) and one scale lambda_x; Sec. 4.3 for the narrow and asymmetric forms).
//
// Tensors of kTinyQuads to kSmallQuads quads: ONE launch of one cluster, which keeps the tensor in registers, exchanges
// its maxima through distributed shared memory and writes the codes.  Others: (1) a range pass whose clusters each leave
// their maxima in the workspace (no atomics, so nothing has to be zeroed first), (2) a pass that reads those, divides /
// rounds half to even / clamps and stores.  The launches use programmatic stream serialization: their blocks stand ready when
// the launch before ends (but for the range pass of a large tensor, see quantize_impl).  The second pass walks the tensor from
// its END, where the first pass stopped: what is still in the 126 MB L2 is then read from there before it is evicted.  The last
// launch of either form lets ITS dependents start at once: a forward call that follows sets itself up (and, where it is allowed
// to, fetches weights) beside it and waits for it before touching the codes.  (The first launch of either form releases only
// behind its own wait, so whatever stands before the quantization on the stream -- an expansion, say -- is complete when such
// a forward call starts.)
// Measured against zeroing + range pass + quantize pass as three plain launches (graphs of 20 calls, inputs beyond L2 where
// large; asymmetric in brackets): 4096 elements 8.3 -> 2.5 us (8.4 -> 2.7), 65 thousand 8.3 -> 3.7 (9.2 -> 4.5), a million
// 8.4 -> 6.3 (13.2 -> 6.5), 17 million 35.5 -> 28.5 (56.6 -> 29.3), 67 million 115 -> 96 (145 -> 98).  The one-launch form ends
// where one cluster's SMs take longer to read the tensor than a second launch costs (131 thousand elements; at 262 thousand
// 7.2 against 6.0 in one run).
#include "pipe_common.cuh"

namespace pipe {

constexpr int kQThreads = 256;        // quantize pass
constexpr int kRangeThreads = 1024;   // range pass: 18 clusters of 8 such CTAs fill 144 of the 148 SMs, and three words
constexpr int kRangeClusters = 18;    // per cluster fit the 256-byte workspace
constexpr int kClusterCtas = 8;
constexpr int kFlatUnroll = 4;
constexpr int64_t kKeepQuads = (80ll << 20) / 16;   // tail of a large tensor that the range pass leaves in L2
constexpr int kSmallPer = 4;          // quads per thread of the one-launch form
constexpr int64_t kTinyQuads = kClusterCtas * 32;   // below: not a warp of quads for every CTA; two launches, as for any
                                                    // tensor the one-launch form does not take
constexpr int64_t kSmallQuads = static_cast<int64_t>(kClusterCtas) * 1024 * kSmallPer;

__device__ __forceinline__ uint32_t q_abs_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// What a pass collects: the largest magnitude key (non-finite check, symmetric scale) and, for the asymmetric
// quantizer, the bits of max(x, 0) and of max(-x, 0): non-negative floats, whose order is the order of their bits.
template <bool EX>
struct Range {
  uint32_t v[EX ? 3 : 1] = {};
  __device__ __forceinline__ void add(float x) {
    v[0] = max(v[0], q_abs_key(x));
    if constexpr (EX) {
      v[1] = __float_as_uint(fmaxf(__uint_as_float(v[1]), x));    // (from +0 on, never NaN)
      v[2] = __float_as_uint(fmaxf(__uint_as_float(v[2]), -x));
    }
  }
  __device__ __forceinline__ void add4(const float4& f) { add(f.x), add(f.y), add(f.z), add(f.w); }
};
template <bool EX>
constexpr int kRangeWords = EX ? 3 : 1;

__device__ __forceinline__ uint32_t q_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void q_store_remote(uint32_t* local, uint32_t rank, uint32_t v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(local))), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void q_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Maxima of the cluster, in every thread of the CTAs of rank below `readers` (the others read nothing of meaning).  The
// caller has already met the cluster once: a CTA that has not started must not be written to.
template <bool EX>
__device__ __forceinline__ void cluster_max(Range<EX>& r, int readers) {
  constexpr int W = kRangeWords<EX>;
  __shared__ uint32_t part[W][32];
  __shared__ uint32_t all[W][kClusterCtas];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, r.v[w] & 0x7fffffffu);   // (a maximum of -0 is 0)
    if (lane == 0) part[w][warp] = m;
  }
  __syncthreads();
  const uint32_t rank = q_cluster_rank();
  if (warp == 0) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t m = __reduce_max_sync(0xffffffffu, lane < nwarps ? part[w][lane] : 0u);
      if (lane < readers) q_store_remote(&all[w][rank], lane, m);
    }
  }
  __syncwarp();
  q_cluster_sync();
#pragma unroll
  for (int w = 0; w < W; ++w) {
    uint32_t m = 0;
#pragma unroll
    for (int c = 0; c < kClusterCtas; ++c) m = max(m, all[w][c]);
    r.v[w] = m;
  }
}

struct QuantArgs {
  const float* x;
  int8_t* xq;
  int64_t T, ldx, ldxq;
  int I;
  int chunks_per_row;   // ceil(I / 16)
  int64_t total_chunks;
  int64_t quads;        // FLAT: T * I / 4
  int vec_in, vec_out;  // rows are 16-byte aligned on the input / output side
  uint32_t* ws;         // [kRangeClusters][words]
  const float* static_scale;
  const float* static_range;
  float* sx;
  int32_t* zp;
  int act_bits, asym;
  int* status;
  int overlap;          // the range pass overlaps its neighbours' ends
};

// The quantizer of a call: scale, and for the forms of Sec. 4.3 zero point and code range.
template <bool EX>
struct Quantizer {
  float s, r, z, cmin = -127.f, cmax = 127.f;
  bool fast;
  // (report: the thread that writes the scale and raises errors)
  __device__ __forceinline__ Quantizer(const QuantArgs& p, const Range<EX>& range, bool report) {
    const uint32_t mbits = range.v[0];
    const float inf = __uint_as_float(0x7f800000u);
    bool bad_arg = false;
    z = 0.f;
    if constexpr (!EX) {
      s = p.static_scale ? *p.static_scale : __fdiv_rn(__uint_as_float(mbits), 127.f);
      bad_arg = p.static_scale && !(s >= 0.f && s < inf);
    } else {
      const float half = static_cast<float>(1 << (p.act_bits - 1));
      if (!p.asym) {
        const float qx = half - 1.f;
        s = p.static_scale ? *p.static_scale : __fdiv_rn(__uint_as_float(mbits), qx);
        bad_arg = p.static_scale && !(s >= 0.f && s < inf);
        cmin = -qx;
        cmax = qx;
      } else {
        float lo = -__uint_as_float(range.v[2]), hi = __uint_as_float(range.v[1]);
        if (p.static_range) {
          lo = p.static_range[0];
          hi = p.static_range[1];
          bad_arg = !(lo <= 0.f && hi >= 0.f && lo > -inf && hi < inf);
        }
        s = __fdiv_rn(__fsub_rn(hi, lo), 2.f * half - 1.f);
        cmin = -half;
        cmax = half - 1.f;
        if (s != 0.f) z = fminf(fmaxf(rintf(__fsub_rn(-half, __fdiv_rn(lo, s))), cmin), cmax);
      }
      if (bad_arg) s = 0.f, z = 0.f;
    }
    if (report) {
      *p.sx = s;
      if constexpr (EX) *p.zp = static_cast<int32_t>(z);
      if (mbits >= 0x7f800000u) raise_status(p.status, PIPE_ERR_NONFINITE);
      if (bad_arg) raise_status(p.status, PIPE_ERR_INVALID_ARG);
    }
    fast = quant_step_is_fast(s);
    r = fast ? __frcp_rn(s) : 0.f;
  }
  // clamp(rne(v / s) + z) as a byte.
  __device__ __forceinline__ uint32_t lane_exact(float v) const {
    float q = z;
    if (s != 0.f) q = fminf(fmaxf(__fadd_rn(rintf(__fdiv_rn(v, s)), z), cmin), cmax);
    return static_cast<uint32_t>(static_cast<int>(q)) & 0xffu;
  }
  // Four codes.  The quotient is estimated as t = v * rn(1 / s), off by less than |t| * 2^-21 (at most 2^-13 inside the
  // code range), clamped -- the limits less z are integers, so clamping before the rounding is the same -- and rounded by
  // an addition (code_magic); a quad with an estimate that close to a rounding boundary is divided.  The pass is bound by
  // its instructions once the loads hit the L2: eight per element against over twenty with a compare, a divide under
  // a predicate and a conversion for each.
  __device__ __forceinline__ uint32_t quad(const float4& f) const {
    const float v[4] = {f.x, f.y, f.z, f.w};
    const float lo = EX ? cmin - z : -127.f, hi = EX ? cmax - z : 127.f;
    float u[4];
    float edge = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) u[e] = code_magic(fminf(fmaxf(__fmul_rn(v[e], r), lo), hi), 0.f, edge);
    if (!fast || edge >= 0.5f - 1.220703125e-04f)
      return lane_exact(v[0]) | (lane_exact(v[1]) << 8) | (lane_exact(v[2]) << 16) | (lane_exact(v[3]) << 24);
    if constexpr (EX) {
#pragma unroll
      for (int e = 0; e < 4; ++e) u[e] = __fadd_rn(u[e], z);   // (exact: integers in a binade of spacing one)
    }
    return pack4_low_bytes(u[0], u[1], u[2], u[3]);
  }
};

__device__ __forceinline__ void load16(const QuantArgs& p, int64_t c, float (&v)[16], int64_t& t, int& i0) {
  t = c / p.chunks_per_row;
  i0 = static_cast<int>(c - t * p.chunks_per_row) * 16;
  const float* row = p.x + t * p.ldx;
  if (p.vec_in && i0 + 16 <= p.I) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float4 f = __ldcg(reinterpret_cast<const float4*>(row + i0) + w);
      v[4 * w] = f.x; v[4 * w + 1] = f.y; v[4 * w + 2] = f.z; v[4 * w + 3] = f.w;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = (i0 + e < p.I) ? row[i0 + e] : 0.f;
  }
}

// Range pass.  FLAT: the tensor is one array of quads (ldx == ldxq == I, I a multiple of 4, 16-byte aligned input): a warp
// reads 512 contiguous bytes per instruction, four of them in flight per thread.
template <bool EX, bool FLAT>
__global__ void __launch_bounds__(kRangeThreads) act_range_kernel(const __grid_constant__ QuantArgs p) {
  grid_wait();
  if (p.overlap) grid_release();
  q_cluster_sync();   // every CTA of the cluster runs before another one writes its shared memory
  Range<EX> range;
  const int64_t first = blockIdx.x * static_cast<int64_t>(kRangeThreads) + threadIdx.x;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kRangeThreads;
  if constexpr (FLAT) {
    const float4* x = reinterpret_cast<const float4*>(p.x);
    int64_t i = first;
    // (what lies further from the end than the L2 keeps is read as evict-first, so that the end stays)
    for (; i + (kFlatUnroll - 1) * stride < p.quads - kKeepQuads; i += kFlatUnroll * stride) {
      float4 f[kFlatUnroll];
#pragma unroll
      for (int u = 0; u < kFlatUnroll; ++u) f[u] = __ldcs(x + i + u * stride);
#pragma unroll
      for (int u = 0; u < kFlatUnroll; ++u) range.add4(f[u]);
    }
    for (; i + (kFlatUnroll - 1) * stride < p.quads; i += kFlatUnroll * stride) {
      float4 f[kFlatUnroll];
#pragma unroll
      for (int u = 0; u < kFlatUnroll; ++u) f[u] = __ldcg(x + i + u * stride);
#pragma unroll
      for (int u = 0; u < kFlatUnroll; ++u) range.add4(f[u]);
    }
    for (; i < p.quads; i += stride) range.add4(__ldcg(x + i));
  } else {
    for (int64_t c = first; c < p.total_chunks; c += stride) {
      float v[16];
      int64_t t;
      int i0;
      load16(p, c, v, t, i0);
#pragma unroll
      for (int e = 0; e < 16; ++e) range.add(v[e]);
    }
  }
  cluster_max<EX>(range, 1);
  if (q_cluster_rank() == 0 && threadIdx.x == 0) {
    const int cluster = blockIdx.x / kClusterCtas;
#pragma unroll
    for (int w = 0; w < kRangeWords<EX>; ++w) p.ws[cluster * kRangeWords<EX> + w] = range.v[w];
  }
}

// Quantize pass: lambda_x and the codes.
template <bool EX, bool FLAT>
__global__ void __launch_bounds__(kQThreads) act_quantize_kernel(const __grid_constant__ QuantArgs p, int clusters) {
  grid_release();
  grid_wait();
  Range<EX> range;
  {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 0; w < kRangeWords<EX>; ++w)
      range.v[w] = __reduce_max_sync(0xffffffffu, lane < clusters ? p.ws[lane * kRangeWords<EX> + w] : 0u);
  }
  const Quantizer<EX> qz(p, range, blockIdx.x == 0 && threadIdx.x == 0);
  const int64_t first = blockIdx.x * static_cast<int64_t>(kQThreads) + threadIdx.x;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kQThreads;
  if constexpr (FLAT) {
    const float4* x = reinterpret_cast<const float4*>(p.x) + (p.quads - 1);   // from the last quad down
    uint32_t* xq = reinterpret_cast<uint32_t*>(p.xq) + (p.quads - 1);
    int64_t i = first;
    for (; i + (kFlatUnroll - 1) * stride < p.quads; i += kFlatUnroll * stride) {
      float4 f[kFlatUnroll];
#pragma unroll
      for (int u = 0; u < kFlatUnroll; ++u) f[u] = __ldcs(x - (i + u * stride));
#pragma unroll
      for (int u = 0; u < kFlatUnroll; ++u) xq[-(i + u * stride)] = qz.quad(f[u]);
    }
    for (; i < p.quads; i += stride) xq[-i] = qz.quad(__ldcg(x - i));
  } else {
    for (int64_t c = first; c < p.total_chunks; c += stride) {
      float v[16];
      int64_t t;
      int i0;
      load16(p, c, v, t, i0);
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = qz.quad(make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]));
      int8_t* orow = p.xq + t * p.ldxq;
      if (p.vec_out && i0 + 16 <= p.I) {
        *reinterpret_cast<uint4*>(orow + i0) = make_uint4(w[0], w[1], w[2], w[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (i0 + e < p.I) orow[i0 + e] = static_cast<int8_t>(w[e >> 2] >> (8 * (e & 3)));
      }
    }
  }
}

// Both passes in one launch of one cluster (FLAT tensors of at most PER quads per thread).
template <bool EX, int PER>
__global__ void __launch_bounds__(1024) act_small_kernel(const __grid_constant__ QuantArgs p) {
  grid_wait();
  grid_release();
  const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = kClusterCtas * blockDim.x;
  const int quads = static_cast<int>(p.quads);
  const float4* x = reinterpret_cast<const float4*>(p.x);
  float4 f[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) f[u] = first + u * stride < quads ? __ldcg(x + first + u * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
  q_cluster_sync();   // every CTA of the cluster runs before another one writes its shared memory
  Range<EX> range;
#pragma unroll
  for (int u = 0; u < PER; ++u) range.add4(f[u]);
  cluster_max<EX>(range, kClusterCtas);
  const Quantizer<EX> qz(p, range, blockIdx.x == 0 && threadIdx.x == 0);
#pragma unroll
  for (int u = 0; u < PER; ++u)
    if (first + u * stride < quads) reinterpret_cast<uint32_t*>(p.xq)[first + u * stride] = qz.quad(f[u]);
}

__global__ void act_empty_kernel(const float* static_scale, float* sx_out, int32_t* zp_out) {
  if (threadIdx.x == 0) {
    *sx_out = static_scale ? *static_scale : 0.f;
    if (zp_out) *zp_out = 0;
  }
}

template <typename... P, typename... A>
static pipe_status launch_q(void (*k)(P...), int grid, int block, bool cluster, bool overlap, cudaStream_t s, A... args) {
  if (launch_overlapped(k, dim3(grid, 1, 1), block, cluster ? kClusterCtas : 1, overlap, s, args...) != cudaSuccess) return PIPE_ERR_CUDA;
  count_launch(1);
  return PIPE_OK;
}

template <bool EX>
static pipe_status quantize_impl(QuantArgs p, cudaStream_t s) {
  p.status = device_status_word();
  if (!p.status) return PIPE_ERR_CUDA;
  if (p.T == 0) {
    act_empty_kernel<<<1, 32, 0, s>>>(p.static_scale, p.sx, EX ? p.zp : nullptr);
    count_launch(1);
    return launch_status();
  }
  p.chunks_per_row = ceil_div(p.I, 16);
  p.total_chunks = p.T * p.chunks_per_row;
  p.vec_in = ((reinterpret_cast<uintptr_t>(p.x) & 15) == 0) && (p.ldx % 4 == 0);
  p.vec_out = ((reinterpret_cast<uintptr_t>(p.xq) & 15) == 0) && (p.ldxq % 16 == 0);
  const bool flat = (p.T == 1 || (p.ldx == p.I && p.ldxq == p.I)) && p.I % 4 == 0 && (reinterpret_cast<uintptr_t>(p.x) & 15) == 0 &&
                    (reinterpret_cast<uintptr_t>(p.xq) & 3) == 0;
  p.quads = p.T * (p.I / 4);
  pipe_status st;
  if (flat && p.quads >= kTinyQuads && p.quads <= kSmallQuads) {
    const int per_cta = static_cast<int>(ceil_div<int64_t>(p.quads, kClusterCtas));
    const int per = per_cta <= 1024 ? 1 : kSmallPer;
    const int threads = round_up(ceil_div(per_cta, per), 32);
    if (per == 1) st = launch_q(act_small_kernel<EX, 1>, kClusterCtas, threads, true, true, s, p);
    else st = launch_q(act_small_kernel<EX, kSmallPer>, kClusterCtas, threads, true, true, s, p);
    return st == PIPE_OK ? launch_status() : st;
  }
  int sms = 148, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t items = flat ? ceil_div<int64_t>(p.quads, kFlatUnroll) : p.total_chunks;
  const int64_t want_c = ceil_div<int64_t>(items, kRangeThreads * kClusterCtas);
  const int clusters = static_cast<int>(want_c < kRangeClusters ? want_c : kRangeClusters);
  const int64_t want = ceil_div<int64_t>(items, kQThreads);
  const int grid = static_cast<int>(want < static_cast<int64_t>(sms) * 8 ? want : static_cast<int64_t>(sms) * 8);
  // The range pass of a tensor that fills the chip starts only when the launch before has ended, and releases nobody ahead of
  // its end: brought in while that one still holds some SMs, its clusters crowd onto the first free ones (67 million elements,
  // back to back: 49 us on an empty chip, 91 that way, 60 with one CTA to an SM).
  p.overlap = clusters < kRangeClusters;
  // (with a static scale the first pass still serves the non-finite check of the input)
  st = flat ? launch_q(act_range_kernel<EX, true>, clusters * kClusterCtas, kRangeThreads, true, p.overlap != 0, s, p)
            : launch_q(act_range_kernel<EX, false>, clusters * kClusterCtas, kRangeThreads, true, p.overlap != 0, s, p);
  if (st != PIPE_OK) return st;
  st = flat ? launch_q(act_quantize_kernel<EX, true>, grid, kQThreads, false, true, s, p, clusters)
            : launch_q(act_quantize_kernel<EX, false>, grid, kQThreads, false, true, s, p, clusters);
  return st == PIPE_OK ? launch_status() : st;
}

}  // namespace pipe

using namespace pipe;

extern "C" pipe_status pipe_quantize_act(const float* d_x, int64_t T, int32_t I, int64_t ldx, const float* d_static_scale,
                                         int8_t* d_xq, int64_t ldxq, float* d_sx, void* d_ws, size_t ws_bytes,
                                         void* stream) {
  if (T < 0 || I <= 0) return PIPE_ERR_INVALID_ARG;
  if (!d_sx || !d_ws) return PIPE_ERR_INVALID_ARG;
  if (T > 0 && (!d_x || !d_xq)) return PIPE_ERR_INVALID_ARG;
  if (ldx < I || ldxq < I) return PIPE_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(d_x) & 3) || (reinterpret_cast<uintptr_t>(d_ws) & 255) ||
      (reinterpret_cast<uintptr_t>(d_sx) & 3))
    return PIPE_ERR_ALIGNMENT;
  if (ws_bytes < 256) return PIPE_ERR_WORKSPACE;
  QuantArgs p = {};
  p.x = d_x; p.xq = d_xq; p.T = T; p.ldx = ldx; p.ldxq = ldxq; p.I = I;
  p.ws = static_cast<uint32_t*>(d_ws);
  p.static_scale = d_static_scale;
  p.sx = d_sx;
  const pipe_status st = quantize_impl<false>(p, static_cast<cudaStream_t>(stream));
  // (this call's kernels now stand between an expansion and what follows)
  if (st == PIPE_OK) take_expansion_mark(static_cast<cudaStream_t>(stream));
  return st;
}

extern "C" pipe_status pipe_quantize_act_ex(const float* d_x, int64_t T, int32_t I, int64_t ldx, int32_t act_bits,
                                            int32_t asymmetric, const float* d_static_scale, const float* d_static_range,
                                            int8_t* d_xq, int64_t ldxq, float* d_sx, int32_t* d_zp, void* d_ws,
                                            size_t ws_bytes, void* stream) {
  if (T < 0 || I <= 0) return PIPE_ERR_INVALID_ARG;
  if (!(act_bits == 8 || act_bits == 6 || act_bits == 4)) return PIPE_ERR_INVALID_ARG;
  if (!d_sx || !d_zp || !d_ws) return PIPE_ERR_INVALID_ARG;
  if (T > 0 && (!d_x || !d_xq)) return PIPE_ERR_INVALID_ARG;
  if (ldx < I || ldxq < I) return PIPE_ERR_INVALID_ARG;
  if (asymmetric ? d_static_scale != nullptr : d_static_range != nullptr) return PIPE_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(d_x) & 3) || (reinterpret_cast<uintptr_t>(d_ws) & 255) || (reinterpret_cast<uintptr_t>(d_sx) & 3) ||
      (reinterpret_cast<uintptr_t>(d_zp) & 3) || (reinterpret_cast<uintptr_t>(d_static_scale) & 3) ||
      (reinterpret_cast<uintptr_t>(d_static_range) & 3))
    return PIPE_ERR_ALIGNMENT;
  if (ws_bytes < 256) return PIPE_ERR_WORKSPACE;
  QuantArgs p = {};
  p.x = d_x; p.xq = d_xq; p.T = T; p.ldx = ldx; p.ldxq = ldxq; p.I = I;
  p.ws = static_cast<uint32_t*>(d_ws);
  p.static_scale = d_static_scale;
  p.static_range = d_static_range;
  p.sx = d_sx;
  p.zp = d_zp;
  p.act_bits = act_bits;
  p.asym = asymmetric ? 1 : 0;
  const pipe_status st = quantize_impl<true>(p, static_cast<cudaStream_t>(stream));
  // (kernels follow: they stand between an expansion and what comes next on the stream)
  if (st == PIPE_OK) take_expansion_mark(static_cast<cudaStream_t>(stream));
  return st;
}

// ------------------------------------------------------------------------------------------------
// Explicit lowering of a quantized NHWC tensor to the rows of the convolution's GEMM, for the geometries the implicit
// convolution does not take (channel counts that are not multiples of 128: a network's first layer, narrow layers).
namespace pipe {

struct LowerArgs {
  const int8_t* x;
  int8_t* rows;
  int64_t ld_rows, total;   // total = T * kh * kw * ceil(C / 16) pieces of up to 16 channels
  int N, H, W, C, kh, kw, ph, pw, sh, sw, Ho, Wo, cpieces;
  int vec;                  // 16-byte loads and stores are possible (C % 16 == 0, aligned pointers and pitch)
};

__global__ void __launch_bounds__(256) lower_conv_input_kernel(const __grid_constant__ LowerArgs a) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < a.total; i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int piece = static_cast<int>(i % a.cpieces);
    int64_t r = i / a.cpieces;
    const int tap = static_cast<int>(r % (a.kh * a.kw));
    const int64_t t = r / (a.kh * a.kw);
    const int wo = static_cast<int>(t % a.Wo);
    const int ho = static_cast<int>((t / a.Wo) % a.Ho);
    const int n = static_cast<int>(t / (static_cast<int64_t>(a.Wo) * a.Ho));
    const int h = a.sh * ho + tap / a.kw - a.ph, w = a.sw * wo + tap % a.kw - a.pw;
    const bool in = h >= 0 && h < a.H && w >= 0 && w < a.W;
    const int c0 = piece * 16, nc = min(16, a.C - c0);
    int8_t* dst = a.rows + t * a.ld_rows + static_cast<int64_t>(tap) * a.C + c0;
    const int8_t* src = a.x + ((static_cast<int64_t>(n) * a.H + h) * a.W + w) * a.C + c0;
    if (a.vec) {
      *reinterpret_cast<uint4*>(dst) = in ? __ldg(reinterpret_cast<const uint4*>(src)) : make_uint4(0, 0, 0, 0);
    } else {
      for (int c = 0; c < nc; ++c) dst[c] = in ? __ldg(src + c) : static_cast<int8_t>(0);
    }
  }
}

}  // namespace pipe

extern "C" pipe_status pipe_lower_conv_input(const pipe_conv_geom* geom, const int8_t* d_xq, int8_t* d_rows, int64_t ld_rows,
                                             void* stream) {
  if (!geom || !d_xq || !d_rows) return PIPE_ERR_INVALID_ARG;
  if (geom->batch < 1 || geom->height < 1 || geom->width < 1 || geom->channels < 1 || geom->kernel_h < 1 || geom->kernel_w < 1 ||
      geom->stride_h < 0 || geom->stride_w < 0 || geom->pad_h < 0 || geom->pad_w < 0)
    return PIPE_ERR_INVALID_ARG;
  const int sh = geom->stride_h > 0 ? geom->stride_h : 1, sw = geom->stride_w > 0 ? geom->stride_w : 1;
  if (geom->pad_h >= geom->kernel_h || geom->pad_w >= geom->kernel_w) return PIPE_ERR_SHAPE;
  if (geom->height + 2 * geom->pad_h < geom->kernel_h || geom->width + 2 * geom->pad_w < geom->kernel_w) return PIPE_ERR_SHAPE;
  const int64_t I = static_cast<int64_t>(geom->kernel_h) * geom->kernel_w * geom->channels;
  if (I > INT32_MAX || ld_rows < I) return PIPE_ERR_INVALID_ARG;
  LowerArgs a;
  a.x = d_xq; a.rows = d_rows; a.ld_rows = ld_rows;
  a.N = geom->batch; a.H = geom->height; a.W = geom->width; a.C = geom->channels;
  a.kh = geom->kernel_h; a.kw = geom->kernel_w; a.ph = geom->pad_h; a.pw = geom->pad_w; a.sh = sh; a.sw = sw;
  a.Ho = (a.H + 2 * a.ph - a.kh) / sh + 1;
  a.Wo = (a.W + 2 * a.pw - a.kw) / sw + 1;
  a.cpieces = ceil_div(a.C, 16);
  a.total = static_cast<int64_t>(a.N) * a.Ho * a.Wo * a.kh * a.kw * a.cpieces;
  a.vec = (a.C % 16 == 0 && ld_rows % 16 == 0 && !(reinterpret_cast<uintptr_t>(d_xq) & 15) && !(reinterpret_cast<uintptr_t>(d_rows) & 15)) ? 1 : 0;
  int sms = 148, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = ceil_div<int64_t>(a.total, 256);
  const int grid = static_cast<int>(want < static_cast<int64_t>(sms) * 16 ? want : static_cast<int64_t>(sms) * 16);
  lower_conv_input_kernel<<<grid > 0 ? grid : 1, 256, 0, static_cast<cudaStream_t>(stream)>>>(a);
  count_launch(1);
  const pipe_status st = launch_status();
  if (st == PIPE_OK) take_expansion_mark(static_cast<cudaStream_t>(stream));
  return st;
}
