// Per-unit quantiser: normalised spectral vectors (fp32) -> the stored unit
// format the forward reads (codes, fp16 scale and zero per group).
//
// BitsMoE quantises every spectral unit p (a column of P, length I) with its
// own bit-width b in {0,1,2,3,4,6,8,16} (appendix "Piecewise Reconstruction
// Error for Bit Allocation"), one scale per group of `group` elements along
// the unit (group 128 in the paper's experiments):
//   b = 2, 3, 4  symmetric uniform Q_b (Eq. app_scalar_quantization_uk) with
//                the MSE-optimal scale (Eq. app_low_bit_opt_scale), searched
//                over `grid` fp16 candidates s_c = fp16(rho 2^(2-b) c / grid)
//   b = 6, 8     Q_b with s = rho / q_max, rho = ||p||_inf (Eqs.
//                app_high_bit_rho_eta, app_uk_scale)
//   b = 1        sign quantiser s_1 sign(p), s_1 = mean |p|, sign(0) = +1
//                (Eq. app_one_bit_quantization)
//   b = 0        evicted (Eq. app_zero_bit_vector); b = 16: fp16 values
// Stored as code = q + 2^(b-1), zero = 2^(b-1) (sign: code [p >= 0], zero
// 1/2, scale 2 s_1), so that p_hat = scale (code - zero).
//
// Arithmetic: fp32 with every operation rounded once (no contraction in the
// error sums), the quotient p / s as p times the correctly rounded fp32
// reciprocal of s, error sums over the group's elements in order, the least
// error winning with ties to the smaller candidate index, so the result is a
// deterministic function of the inputs.
//
// Work decomposition: one warp per (unit, group), the group's elements staged in shared
// memory.  The scale search first scores every ST-th candidate (one or two a lane); the
// others are scored only where a lower bound on their error does not exceed the least
// one found.  The bound: the codes of a scale are the nearest ones, so with the codes q'
// of s', ||x - s q(s)|| <= ||x - s q'|| <= ||x - s' q'|| + |s - s'| ||q'||, and ||q'|| <=
// ||q(s_lo)|| for every s' >= s_lo (the levels shrink as the scale grows); taken from the
// scored neighbours on both sides, with 1e-4 of each term for rounding (the sums' and
// near ties': below 2e-5).  What is left is scored in full, in the same steps, so the
// least error and its index are those of a search over all.  One lexicographic (error,
// index) warp reduction picks the scale.  The search is ALU-bound: the fp32 input is
// read once and the codes written once.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "device.cuh"
#include "internal.h"

namespace {

constexpr int kQWarps = 8;
constexpr int kQThreads = kQWarps * 32;
constexpr int kQMaxGroup = 256;
constexpr float kRne = 12582912.f;   // 1.5 * 2^23: t + kRne - kRne rounds |t| <= 2^22 to nearest even

struct QArgs {
  const float* p;
  const uint8_t* bits;
  int64_t items;   // U * ng
  int I, group, ng, grid;
  uint16_t* codes;
  uint16_t* scale;
  uint16_t* zero;
  int* status;
};

__device__ __forceinline__ float f16_round(float x) { return __half2float(__float2half_rn(x)); }
__device__ __forceinline__ uint32_t f16_bits(float x) { return (uint32_t)__half_as_ushort(__float2half_rn(x)); }
__device__ __forceinline__ bool bits_supported(int b) {
  return b == 0 || b == 1 || b == 2 || b == 3 || b == 4 || b == 6 || b == 8 || b == 16;
}
// a scale that is positive and finite in fp16
__device__ __forceinline__ bool usable(float s) { return s > 0.f && s <= 65504.f; }
// clamp(round(v * r), qmin, qmax): clamping first gives the same level (the bounds are integers)
__device__ __forceinline__ float level(float v, float r, float qmin, float qmax) {
  const float t = fminf(fmaxf(__fmul_rn(v, r), qmin), qmax);
  return __fsub_rn(__fadd_rn(t, kRne), kRne);
}
// candidate c (1-based) of the scale search
__device__ __forceinline__ float candidate(float top, int c, int grid) {
  return f16_round(__fdiv_rn(__fmul_rn(top, (float)c), (float)grid));
}

// Scores of K candidates (scale sc, reciprocal rc) of a lane over the group, and with NORM the squared norm of
// their codes.  Two elements at a time in packed fp32 (every operation rounded as the scalar one: 5.5 issue
// slots an element and candidate instead of 8, the two clamps on the other pipe); the squares are added one by
// one, in order.
template <int K, bool NORM>
__device__ __forceinline__ void score(const float* v, int g, const float (&sc)[K], const float (&rc)[K], float (&e)[K],
                                      float (&nn)[K], float qmin, float qmax) {
  using u64 = unsigned long long;
  auto pack = [](float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
  };
  auto unpack = [](u64 r, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); };
  const u64 up = pack(kRne, kRne), down = pack(-kRne, -kRne);
  u64 s2[K], r2[K], n2[K];
#pragma unroll
  for (int m = 0; m < K; ++m) {
    s2[m] = pack(-sc[m], -sc[m]);
    r2[m] = pack(rc[m], rc[m]);
    n2[m] = 0ull;
  }
#pragma unroll 4
  for (int i = 0; i < g; i += 4) {
    const ulonglong2 x4 = *reinterpret_cast<const ulonglong2*>(v + i);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const u64 x = h ? x4.y : x4.x;
#pragma unroll
      for (int m = 0; m < K; ++m) {
        u64 t, q, d;
        float a, b;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(x), "l"(r2[m]));
        unpack(t, a, b);
        a = fminf(fmaxf(a, qmin), qmax);
        b = fminf(fmaxf(b, qmin), qmax);
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(q) : "l"(pack(a, b)), "l"(up));
        asm("add.rn.f32x2 %0, %0, %1;" : "+l"(q) : "l"(down));
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(s2[m]), "l"(q), "l"(x));   // sc * q is exact (11 x 4 bits)
        asm("mul.rn.f32x2 %0, %0, %0;" : "+l"(d));
        if constexpr (NORM) asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(n2[m]) : "l"(q));
        unpack(d, a, b);
        e[m] = __fadd_rn(__fadd_rn(e[m], a), b);
      }
    }
  }
  if constexpr (NORM) {
#pragma unroll
    for (int m = 0; m < K; ++m) {
      float a, b;
      unpack(n2[m], a, b);
      nn[m] = a + b;
    }
  }
}

// (error, index) of the better of two, the smaller index on ties.
__device__ __forceinline__ void better(float& be, int& bc, float e, int c) {
  if (e < be || (e == be && c < bc)) {
    be = e;
    bc = c;
  }
}
__device__ __forceinline__ void warp_better(float& be, int& bc) {
#pragma unroll
  for (int o = 16; o; o >>= 1) better(be, bc, __shfl_xor_sync(0xFFFFFFFFu, be, o), __shfl_xor_sync(0xFFFFFFFFu, bc, o));
}

// One warp's scored candidates and the list of those left to score.
template <int NC>
struct SearchMem {
  // candidates a lane scores first: strides of 4, 8, 8 and 16 from 128 candidates on, below it all of them.  16384 units
  // of 768, us with this and with the other K: 64 candidates 193 / 224, 128 233 / 310, 256 300 / 327, 512 435 / 414
  // (the one stride that is not the faster), 1024 613 / 654.
  static constexpr int K = NC == 1 || NC == 4 || NC == 8 ? 1 : 2;
  static constexpr int ST = NC / K;                      // their stride
  float s[32 * K], err[32 * K], norm[32 * K];            // scale, ||x - s q|| and ||q||
  uint16_t list[ST > 1 ? 32 * NC : 1];
};

// Scores the candidates c[k] (0: none).
template <int K, bool NORM>
__device__ __forceinline__ void score_candidates(const float* v, int g, float top, int grid, const int (&c)[K], float qmin,
                                                 float qmax, float (&sc)[K], float (&e)[K], float (&nn)[K]) {
  float rc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {   // a skipped candidate starts (and stays) at +inf error
    const float s = c[k] ? candidate(top, c[k], grid) : 0.f;
    const bool ok = usable(s);
    sc[k] = ok ? s : 1.f;
    rc[k] = __frcp_rn(sc[k]);
    e[k] = ok ? 0.f : __int_as_float(0x7F800000);
  }
  score<K, NORM>(v, g, sc, rc, e, nn, qmin, qmax);
}

// Scale search of one group for b in {2, 3, 4}: 32 NC candidates.
template <int NC>
__device__ float search_scale(const float* v, int g, float rho, int b, int grid, int lane, SearchMem<NC>& sm) {
  constexpr int K = SearchMem<NC>::K, ST = SearchMem<NC>::ST;
  const float qmax = (float)((1 << (b - 1)) - 1), qmin = -(float)(1 << (b - 1));
  const float top = __fmul_rn(rho, b == 2 ? 1.f : (b == 3 ? 0.5f : 0.25f));
  const float kInf = __int_as_float(0x7F800000);
  float be = kInf;
  int bc = 0x7FFFFFFF;
  const float cap = sqrtf((float)g) * -qmin;   // ||q|| of any codes
  {
    int c[K];
    float sc[K], e[K], nn[K];
#pragma unroll
    for (int k = 0; k < K; ++k) c[k] = (lane + 32 * k + 1) * ST;
    score_candidates<K, (ST > 1)>(v, g, top, grid, c, qmin, qmax, sc, e, nn);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      better(be, bc, e[k], c[k]);
      if constexpr (ST > 1) {   // no bound from a skipped candidate or an overflowed sum
        const bool ok = e[k] < kInf;
        sm.s[lane + 32 * k] = candidate(top, c[k], grid);
        sm.err[lane + 32 * k] = ok ? sqrtf(e[k]) * 0.9999f : 0.f;
        sm.norm[lane + 32 * k] = ok ? sqrtf(nn[k]) * 1.0001f : cap;
      }
    }
    warp_better(be, bc);
  }
  if constexpr (ST > 1) {
    __syncwarp();
    const float lim = sqrtf(be) * 1.0001f;
    int cnt = 0;
#pragma unroll 1
    for (int m = 0; m < NC; ++m) {
      const int c = lane + 1 + 32 * m, hi = c / ST, lo = hi - 1;   // scored neighbours: (lo + 1) ST < c < (hi + 1) ST
      const float s = candidate(top, c, grid);
      bool keep = c % ST != 0 && usable(s);
      if (keep) {
        const float nq = lo >= 0 ? sm.norm[lo] : cap;
        if (sm.err[hi] - (sm.s[hi] - s) * nq > lim) keep = false;
        if (lo >= 0 && sm.err[lo] - (s - sm.s[lo]) * nq > lim) keep = false;
      }
      const unsigned mk = __ballot_sync(0xFFFFFFFFu, keep);
      if (keep) sm.list[cnt + __popc(mk & ((1u << lane) - 1u))] = (uint16_t)c;
      cnt += __popc(mk);
    }
    __syncwarp();
    int i = 0;
    for (; cnt - i > 32; i += 64) {
      const int c[2] = {(int)sm.list[i + lane], i + 32 + lane < cnt ? (int)sm.list[i + 32 + lane] : 0};
      float sc[2], e[2], nn[2];
      score_candidates<2, false>(v, g, top, grid, c, qmin, qmax, sc, e, nn);
      better(be, bc, e[0], c[0]);
      if (c[1]) better(be, bc, e[1], c[1]);
    }
    if (i < cnt) {
      const int c[1] = {i + lane < cnt ? (int)sm.list[i + lane] : 0};
      float sc[1], e[1], nn[1];
      score_candidates<1, false>(v, g, top, grid, c, qmin, qmax, sc, e, nn);
      if (c[0]) better(be, bc, e[0], c[0]);
    }
    warp_better(be, bc);
    __syncwarp();   // the next group's search writes the lists
  }
  return be < kInf ? candidate(top, bc, grid) : 0.f;
}

template <int NC>
__global__ void __launch_bounds__(kQThreads) k_quantize(QArgs a) {
  __shared__ __align__(16) float sv[kQWarps][kQMaxGroup];
  __shared__ SearchMem<NC> found[kQWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* v = sv[w];
  const int g = a.group;
  for (int64_t it = (int64_t)blockIdx.x * kQWarps + w; it < a.items; it += (int64_t)gridDim.x * kQWarps) {
    const int64_t u = it / a.ng;
    const int gi = (int)(it - u * a.ng);
    const int b = __ldg(a.bits + u);
    const size_t base = (size_t)u * a.I + (size_t)gi * g;
    uint32_t* dst = reinterpret_cast<uint32_t*>(a.codes + base);   // two codes a word
    float mx = 0.f;
    __syncwarp();   // the previous item's reads of v are done
    for (int i = lane; i < g / 4; i += 32) {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(a.p + base) + i);
      reinterpret_cast<float4*>(v)[i] = x;
      mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
    }
    const float rho = warp_max(mx);
    __syncwarp();
    float s = 0.f, zp = 0.f;
    if (b == 0 || !bits_supported(b)) {
      for (int i = lane; i < g / 2; i += 32) dst[i] = 0u;
      if (b != 0 && lane == 0 && a.status) atomicCAS(a.status, 0, BITSMOE_ERR_UNSUPPORTED_BITS);
    } else if (b == 16) {
      for (int i = lane; i < g / 2; i += 32) dst[i] = f16_bits(v[2 * i]) | (f16_bits(v[2 * i + 1]) << 16);
    } else if (b == 1) {
      // s_1 = mean |p| over the group, summed in element order
      float acc = 0.f;
      if (lane == 0) {
#pragma unroll 8
        for (int i = 0; i < g; ++i) acc = __fadd_rn(acc, fabsf(v[i]));
      }
      acc = __shfl_sync(0xFFFFFFFFu, acc, 0);
      s = f16_round(__fmul_rn(2.f, __fdiv_rn(acc, (float)g)));
      zp = 0.5f;
      for (int i = lane; i < g / 2; i += 32)
        dst[i] = (v[2 * i] >= 0.f ? 1u : 0u) | ((v[2 * i + 1] >= 0.f ? 1u : 0u) << 16);
    } else {
      const float half = (float)(1 << (b - 1));
      if (b <= 4) {
        s = search_scale<NC>(v, g, rho, b, a.grid, lane, found[w]);
      } else {
        s = f16_round(__fdiv_rn(rho, half - 1.f));
        if (!usable(s)) s = 0.f;
      }
      zp = half;
      const float r = s > 0.f ? __frcp_rn(s) : 0.f;
      const float qmax = half - 1.f, qmin = -half;
      for (int i = lane; i < g / 2; i += 32) {
        const float q0 = s > 0.f ? level(v[2 * i], r, qmin, qmax) : 0.f;
        const float q1 = s > 0.f ? level(v[2 * i + 1], r, qmin, qmax) : 0.f;
        dst[i] = (uint32_t)(int)(q0 + half) | ((uint32_t)(int)(q1 + half) << 16);
      }
    }
    if (lane == 0) {
      const size_t o = (size_t)u * a.ng + gi;
      a.scale[o] = (uint16_t)f16_bits(s);
      a.zero[o] = (uint16_t)f16_bits(zp);
    }
  }
}

template <int NC>
cudaError_t launch_q(const QArgs& a, cudaStream_t st) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_quantize<NC>, kQThreads, 0);
  if (e != cudaSuccess) return e;
  const int64_t need = (a.items + kQWarps - 1) / kQWarps;
  const int64_t full = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
  const int blocks = (int)(need < full ? need : full);
  k_quantize<NC><<<blocks, kQThreads, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

extern "C" int bitsmoe_quantize_units(const float* p, const uint8_t* bits, int64_t U, int I, int group, int grid,
                                      uint16_t* codes, uint16_t* scale, uint16_t* zero, int* status,
                                      void* stream) {
  if (U < 0 || I < 1) return BITSMOE_ERR_INVALID_ARG;
  if (!bmoe::group_ok(group) || I % group) return BITSMOE_ERR_SHAPE;
  if (grid != 32 && grid != 64 && grid != 128 && grid != 256 && grid != 512 && grid != 1024)
    return BITSMOE_ERR_INVALID_ARG;
  if (U == 0) return BITSMOE_OK;
  if (!p || !bits || !codes || !scale || !zero) return BITSMOE_ERR_INVALID_ARG;
  if ((uintptr_t)p % 16 || (uintptr_t)codes % 16 || (uintptr_t)scale % 2 || (uintptr_t)zero % 2 ||
      (uintptr_t)status % 4)
    return BITSMOE_ERR_ALIGNMENT;
  QArgs a{p, bits, U * (int64_t)(I / group), I, group, I / group, grid, codes, scale, zero, status};
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  switch (grid) {
    case 32: e = launch_q<1>(a, st); break;
    case 64: e = launch_q<2>(a, st); break;
    case 128: e = launch_q<4>(a, st); break;
    case 256: e = launch_q<8>(a, st); break;
    case 512: e = launch_q<16>(a, st); break;
    default: e = launch_q<32>(a, st); break;
  }
  return e == cudaSuccess ? BITSMOE_OK : bmoe::record_cuda_error((int)e);
}
