// Device and host helpers shared by the tcgen05 kernels of libpipe (one-SM kernel, SM-pair kernel, decode
// kernel, diagnostics): mbarrier operations with bounded waits, TMA tensor loads, the shared-memory matrix
// descriptor and the instruction descriptor of tcgen05.mma kind::i8, accumulator loads, the conversion-free
// re-quantization of the fused inner-layer epilogue, and tensor-map encoding through the runtime's
// driver-entry-point query.  The descriptor encodings, the 128-byte swizzle and the tensor-map call are fixed by
// the hardware interface.
#pragma once

#include <cuda.h>

#include <mutex>

#include "pipe_common.cuh"

namespace pipe {
namespace tcc {

constexpr long long kWaitLimitCycles = 4000000000ll;  // about 2 s per wait at the maximum SM clock

// Position in a ring of `depth` slots: slot index and phase parity, advanced without divisions.
struct RingPos {
  uint32_t slot, phase;
  __device__ __forceinline__ void advance(uint32_t by, uint32_t depth) {  // by <= depth
    slot += by;
    if (slot >= depth) {
      slot -= depth;
      phase ^= 1u;
    }
  }
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// For barriers that the other CTA of a pair signals: the wait acquires at cluster scope.
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait.  Returns false when the CTA is aborting (this wait or another one expired).
// The bound is counted in SM cycles; the abort flag and the clock are looked at only every few
// polls so that a barrier that completes soon is seen with little delay.
// SLEEP_NS > 0: a wait that is expected to last long (an epilogue warp waiting for a whole tile's MMAs) backs off
// between polls, so that its polling does not take shared-memory and issue slots from the warps that feed the MMAs.
template <bool CLUSTER = false, int SLEEP_NS = 0>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          long long limit = kWaitLimitCycles) {
  if (CLUSTER ? mbar_try_cluster(bar, parity) : mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 16; ++i) {
      if (CLUSTER ? mbar_try_cluster(bar, parity) : mbar_try(bar, parity)) return true;
      if (SLEEP_NS > 0) __nanosleep(SLEEP_NS);
    }
    if (*abort_flag) return false;
    if (clock64() - t0 > limit) {
      *abort_flag = 1;
      raise_status(status, PIPE_ERR_TIMEOUT);
      return false;
    }
  }
}

// After the last issue: wait (bounded) until the copies of the last `depth` ring slots have landed,
// so that no copy is still writing into this CTA's shared memory when it exits.
__device__ __forceinline__ void drain_ring(uint32_t full0, uint32_t issued, int depth, long long limit = kWaitLimitCycles) {
  for (uint32_t j = (issued > static_cast<uint32_t>(depth) ? issued - depth : 0); j < issued; ++j) {
    const int s = j % depth;
    const uint32_t ph = (j / depth) & 1;
    const long long t0 = clock64();
    while (!mbar_try(full0 + 8u * s, ph) && clock64() - t0 < limit) {
    }
  }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

// Four-dimensional tile of an NHWC tensor (coordinates innermost first: channel, x, y, image);
// coordinates outside the tensor read zeros, which is the convolution's padding.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor of a K-major int8 tile whose rows are 128 bytes, stored as
// 8-row atoms of 1024 bytes with the 128-byte swizzle (the layout TMA writes with SWIZZLE_128B).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);  // start address
  d |= static_cast<uint64_t>(1) << 16;                 // leading byte offset (unused for swizzled K-major)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;         // stride byte offset: next 8-row atom
  d |= static_cast<uint64_t>(1) << 46;                 // descriptor version of this architecture
  d |= static_cast<uint64_t>(2) << 61;                 // 128-byte swizzle
  return d;
}

// Instruction descriptor: D = int32, A and B = signed int8, both K-major, M = m (128, or 256 over an SM pair), N = n.
__device__ __forceinline__ uint32_t idesc_i8(int m, int n) {
  return (2u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(m >> 4) << 24);
}

__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate ? 1u : 0u)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}

// The codes clamp(rne(sigma(v) / s)) of the fused inner-layer epilogue, eight at a time, without a conversion
// instruction, a division or a full-precision exp / erf on the common path.  An estimate t of sigma(v) / s, clamped to
// +-127 (a t beyond 127 has a true quotient above 126.9, whose code is 127), is added to 1.5 * 2^23, where the spacing
// of binary32 is one, so the addition itself rounds to the nearest integer, ties to even, and leaves the code in the
// low byte of the sum.  `edge` collects the largest |t - code| + (bound on the error of t): at 0.5 or more an estimate
// lies so close to a rounding boundary that what DEFINES the code -- apply_activation in binary32, then the IEEE
// quotient -- may round the other way, and codes4_exact evaluates the definition.  The codes are therefore the same
// bits as with the definition everywhere.
// Why: the drain is bound by its instructions.  With expf / erff and a division per output the SiLU and GeLU drains
// took longer than the MMAs they should hide behind.  Measured before -> after (K = 4, M = 2, T = 4096): 4096 -> 11008
// with SiLU 596 -> 342 us (fp32 output: 302), 768 -> 3072 with GeLU 175 -> 84 us (fp32 output: 57), and with ReLU, which
// gains from the fallback being out of line, 86 -> 69 us.
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// sigma(v) r for kinds 2 to 4 of apply_activation, estimated, and `err`: a bound on its distance from the quotient that
// defines the code (2^-21 of it for the product with r = rn(1 / s) in place of that quotient).
//   SiLU v q and sigmoid q, q = 1 / (1 + 2^(-v log2 e)), on the approximate exponential and reciprocal: the rounded
//     argument of the exponential contributes |v| 1.5 * 2^-24, the exponential 2^-22, the reciprocal, the other
//     roundings and the reference's own less than 2^-21 together, as fractions of the estimate.  (Beyond v = -86 the
//     exponential overflows and the estimate is 0 where sigma is below 1e-35: no usable step, all above 1e-30, makes that
//     a code other than 0.)
//   GeLU v / 2 + |v| / 2 erf(|v| / sqrt 2) with erf by formula 7.1.26 of Abramowitz and Stegun (absolute error 1.5e-7):
//     2^-20 of |v| r.  (Written so that no maximum is needed: the drain's busiest pipe is the one that does the maxima and
//     byte permutations.)
// Over every binary32 v in +-80 the largest distance measured (r = 1) is 0.47 (SiLU), 0.26 (GeLU), 0.47 (sigmoid) of err.
// Scaled by r inside the estimate and without the maximum: 768 -> 3072 GeLU 78 -> 76 us, SiLU 74 -> 71, ReLU 64 -> 60.
// (err: a number whose magnitude is the bound.)  Two at a time on the packed arithmetic, whose halves round like the scalar
// operations; what has no packed form -- the approximate functions, an absolute value inside a multiplication -- is done twice.
template <int KIND>
__device__ __forceinline__ f32x2 smooth_estimate2(f32x2 v, float r, f32x2& err) {
  float v0, v1;
  unpack_f2(v, v0, v1);
  if constexpr (KIND == 3) {
    const f32x2 hv = mul_f2(v, both_f2(__fmul_rn(0.5f, r)));
    const f32x2 t = pack_f2(rcp_approx(__fmaf_rn(0.23164189f, fabsf(v0), 1.f)), rcp_approx(__fmaf_rn(0.23164189f, fabsf(v1), 1.f)));   // 0.3275911 / sqrt 2
    float a0, a1;
    unpack_f2(mul_f2(mul_f2(v, v), both_f2(-0.72134752f)), a0, a1);
    const f32x2 e = pack_f2(ex2_approx(a0), ex2_approx(a1));                // exp(-v^2 / 2)
    f32x2 h = fma_f2(t, both_f2(-1.061405429f), both_f2(1.453152027f));     // (minus the polynomial)
    h = fma_f2(t, h, both_f2(-1.421413741f));
    h = fma_f2(t, h, both_f2(0.284496736f));
    h = fma_f2(t, h, both_f2(-0.254829592f));
    const f32x2 erf_v = fma_f2(mul_f2(t, h), e, both_f2(1.f));
    err = mul_f2(hv, both_f2(2.86102294921875e-06f));                       // |v| r (2^-20 + 2^-21)
    float h0, h1, f0, f1;
    unpack_f2(hv, h0, h1);
    unpack_f2(erf_v, f0, f1);
    return pack_f2(__fmaf_rn(fabsf(h0), f0, h0), __fmaf_rn(fabsf(h1), f1, h1));
  } else {
    float a0, a1;
    unpack_f2(mul_f2(v, both_f2(-1.44269504f)), a0, a1);
    f32x2 q = add_f2(both_f2(1.f), pack_f2(ex2_approx(a0), ex2_approx(a1)));
    unpack_f2(q, a0, a1);
    q = pack_f2(rcp_approx(a0), rcp_approx(a1));
    const f32x2 t = mul_f2(KIND == 2 ? mul_f2(v, q) : q, both_f2(r));
    // |t| (|v| 2^-23 + 1.5 * 2^-20, + 2^-21)
    err = mul_f2(t, pack_f2(__fmaf_rn(fabsf(v0), 1.1920928955078125e-07f, 1.9073486328125e-06f),
                            __fmaf_rn(fabsf(v1), 1.1920928955078125e-07f, 1.9073486328125e-06f)));
    return t;
  }
}

// Four codes by the definition (out of line: the drain's loop is sensitive to its instruction footprint).
static __device__ __noinline__ uint32_t codes4_exact(float a, float b, float c, float d, int kind, float s) {
  return quant_lane_exact(apply_activation(a, kind), s) | (quant_lane_exact(apply_activation(b, kind), s) << 8) |
         (quant_lane_exact(apply_activation(c, kind), s) << 16) | (quant_lane_exact(apply_activation(d, kind), s) << 24);
}

// Two estimates clamped to [lo, 127] and rounded by an addition (see code_magic): the codes stand in the low bytes of u0, u1.
// RELATIVE: err is a factor, the bound its product with the clamped estimate.
template <bool RELATIVE>
__device__ __forceinline__ void code_magic2(f32x2 t, f32x2 err, float lo, float& u0, float& u1, float& edge) {
  float t0, t1, d0, d1, e0, e1;
  unpack_f2(t, t0, t1);
  t = pack_f2(fminf(fmaxf(t0, lo), 127.f), fminf(fmaxf(t1, lo), 127.f));
  if (RELATIVE) err = mul_f2(t, err);
  const f32x2 u = add_f2(t, both_f2(12582912.f));
  unpack_f2(sub_f2(t, sub_f2(u, both_f2(12582912.f))), d0, d1);
  unpack_f2(err, e0, e1);
  edge = max3(edge, __fadd_rn(fabsf(d0), fabsf(e0)), __fadd_rn(fabsf(d1), fabsf(e1)));
  unpack_f2(u, u0, u1);
}

template <int KIND>
__device__ __forceinline__ void smooth_codes8(const f32x2 (&y)[4], float r, float (&uu)[8], float& edge) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    f32x2 err;
    const f32x2 t = smooth_estimate2<KIND>(y[e], r, err);
    code_magic2<false>(t, err, -127.f, uu[2 * e], uu[2 * e + 1], edge);
  }
}

// kind: the activation; s: the output step; r = rn(1 / s), usable when `fast`.
__device__ __forceinline__ void q8_codes8(const f32x2 (&y)[4], int kind, float s, float r, bool fast, uint32_t& w0, uint32_t& w1) {
  float uu[8];
  float edge = fast ? 0.f : 1.f;
  if (kind < 2) {
    const float lo = kind == 1 ? 0.f : -127.f;   // ReLU: max(v, 0) r = max(v r, 0)
#pragma unroll
    for (int e = 0; e < 4; ++e) code_magic2<true>(mul_f2(y[e], both_f2(r)), both_f2(4.76837158203125e-07f), lo, uu[2 * e], uu[2 * e + 1], edge);
  } else if (kind == 2) {
    smooth_codes8<2>(y, r, uu, edge);
  } else if (kind == 3) {
    smooth_codes8<3>(y, r, uu, edge);
  } else {
    smooth_codes8<4>(y, r, uu, edge);
  }
  w0 = pack4_low_bytes(uu[0], uu[1], uu[2], uu[3]);
  w1 = pack4_low_bytes(uu[4], uu[5], uu[6], uu[7]);
  if (edge >= 0.5f) {   // an estimate too close to a rounding boundary to decide (or the step has no usable reciprocal)
    float v[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) unpack_f2(y[e], v[2 * e], v[2 * e + 1]);
    w0 = codes4_exact(v[0], v[1], v[2], v[3], kind, s);
    w1 = codes4_exact(v[4], v[5], v[6], v[7], kind, s);
  }
}

// ---------------------------------------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeFn encode_fn() {
  static std::once_flag once;
  static EncodeFn fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  });
  return fn;
}

inline bool make_map_2d(CUtensorMap* map, const void* base, uint64_t inner_bytes, uint64_t rows, uint64_t pitch_bytes,
                        uint32_t box_inner, uint32_t box_rows, CUtensorMapSwizzle swz) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {inner_bytes, rows};
  const cuuint64_t strides[1] = {pitch_bytes};
  const cuuint32_t box[2] = {box_inner, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// NHWC int8 tensor as a 4-D map; one box = 128 channels x 8 x 8 pixels of one image (64 rows of 128 bytes).
inline bool make_map_nhwc(CUtensorMap* map, const void* base, int N, int H, int W, int C, int sh, int sw) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(W), static_cast<cuuint64_t>(H),
                              static_cast<cuuint64_t>(N)};
  const cuuint64_t strides[3] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(W) * C,
                                 static_cast<cuuint64_t>(H) * W * C};
  // 8 x 8 pixels at the convolution's stride: the box spans 8 * stride positions and the copy takes every
  // stride-th of them
  const cuuint32_t box[4] = {128, static_cast<cuuint32_t>(8 * sw), static_cast<cuuint32_t>(8 * sh), 1};
  const cuuint32_t estr[4] = {1, static_cast<cuuint32_t>(sw), static_cast<cuuint32_t>(sh), 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 output [rows, channels] with a row pitch: one box = 16 channels x 32 rows (64-byte rows, 64-byte swizzle).
inline bool make_map_out_2d(CUtensorMap* map, const float* base, uint64_t channels, uint64_t rows, uint64_t pitch_elems) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {channels, rows};
  const cuuint64_t strides[1] = {pitch_elems * 4};
  const cuuint32_t box[2] = {16, 32};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 output of a convolution, pixels in NHW order with a pixel pitch: one box = 16 channels x 8 pixels x 4 image
// rows of one image (half of an 8 x 8 patch); what hangs over the right or lower edge of the image is not written.
inline bool make_map_out_nhwc(CUtensorMap* map, const float* base, int N, int Ho, int Wo, uint64_t channels, uint64_t pitch_elems) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {channels, static_cast<cuuint64_t>(Wo), static_cast<cuuint64_t>(Ho), static_cast<cuuint64_t>(N)};
  const cuuint64_t strides[3] = {pitch_elems * 4, pitch_elems * 4 * Wo, pitch_elems * 4 * Wo * Ho};
  const cuuint32_t box[4] = {16, 8, 4, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tcc
}  // namespace pipe
