// Expert factors of calls with several tokens, on the warp-level tensor-core
// instruction (mma.sync m16n8k16, f16 operands, fp32 accumulators):
//
//   gate/up[t][h][i] = sum_j p_hat_{h,e}[i, j] alpha_{h,e,j} z_h[t][j]          (h = gate, up)
//   h_t[i]           = SiLU(gate[t][i]) up[t][i]
//   s[t][j']        += g_{t,e} alpha_{dn,e,j'} sum_i p_hat_{dn,e}[i, j'] h_t[i]
//   p_hat[i, j]      = scale_{j,g(i)} (q_ij - zero_{j,g(i)})                     (group g along i)
//
// A code c, written as the bit pattern of an fp16 number, is the subnormal
// c 2^-24 (exact below 2048), so two codes that a 32-bit word holds 16 bits apart
// become one A register by a shift and a mask: no conversion, no byte permute and
// no shared-memory round trip (a tcgen05 operand has to be written to shared memory
// or TMEM first).  The activation side (gate/up: scale alpha z; down: h) is an
// fp16 pair hi + lo of about 22 bits, scaled by a power of two per token; both
// halves accumulate into the same fp32 accumulator, and zero points enter as
// per-token corrections in fp32.
//
// Why mma.sync: with few tokens an expert the codes, not the products, are the
// work.  On GB300 an m16n8k16 takes 2 SM clocks (128 codes a clock against 8
// tokens) while a tcgen05.mma of M = 128 and N <= 64 takes about 95 clocks an
// instruction (21 codes a clock), and the codes then have to be written to shared
// memory; the decode itself runs at about 60 codes a clock and SM.
//
// A K-step is 16 consecutive unit slots (gate/up) or rows (down).  Lane (g, t) =
// (lane / 4, lane % 4) of a warp holds the products' K indices 4 t .. 4 t + 3: word
// w of a packed stream holds those four codes at bits 8 m + b k (m = 0 .. 3), so the
// registers are ((w >> b k) & mask) for m = 0, 2 and ((w >> b k + 8) & mask) for m = 1, 3.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "device.cuh"

namespace {

constexpr int kStagePiece = 4096;   // bytes of down codes a warp stages at a time

// Token tiles of the call, and their share of a kernel's work: active expert a has cnt[a] tokens from
// pair_list[pst[a]], in tiles of NT.  Tile tt of expert a owns M_a consecutive units of the kernel's flat
// unit order, M_a = (ub[a + 1] - ub[a]) / tiles; a unit weighs tile_weight of its tile's tokens, and wb is
// the prefix of the weights.  A block takes the units between two equal cuts of the total weight.
struct MTiles {
  int* e;
  int* cnt;
  int* pst;
  int* ub;    // [na + 1]
  int* wb;    // [na + 1]
  int* row;   // first row of the expert's tokens, experts padded to 8 rows
  int na;
};
__host__ __device__ inline uint32_t mtiles_bytes(int A_max) { return ((6u * (uint32_t)A_max + 2u) * 4u + 15u) & ~15u; }

__device__ MTiles mtiles_at(uint8_t* sm, int A_max) {
  MTiles t;
  t.e = reinterpret_cast<int*>(sm);
  t.cnt = t.e + A_max;
  t.pst = t.cnt + A_max;
  t.ub = t.pst + A_max;
  t.wb = t.ub + A_max + 1;
  t.row = t.wb + A_max + 1;
  t.na = 0;
  return t;
}
// Relative time of a tile of nt tokens (measured: the decode of the codes is shared by a tile's groups of
// 8 tokens, the operand and the products are not).
__device__ __forceinline__ int tile_weight(int nt) { return 1 + 3 * ((nt + 7) >> 3); }

// Whole block; the routing is published.  per_tile(e): units of a token tile of expert e.
template <class F>
__device__ void mtiles_build(const Fwd& p, int A_max, int NT, MTiles& t, F per_tile) {
  const int tid = threadIdx.x, lane = tid & 31;
  t.na = min(p.active[0], A_max);
  for (int a = tid; a < t.na; a += (int)blockDim.x) {
    const int e = p.active[1 + a], c = p.expert_count[e];
    t.e[a] = e;
    t.cnt[a] = c;
    t.pst[a] = p.expert_start[e];
    const int m = per_tile(e), f = c / NT, r = c - f * NT;
    t.ub[a] = (f + (r > 0)) * m;
    t.wb[a] = (f * tile_weight(NT) + (r > 0 ? tile_weight(r) : 0)) * m;
  }
  __syncthreads();
  if (tid < 32) {   // exclusive prefixes
    int ru = 0, rw = 0, rr = 0;
    for (int a0 = 0; a0 < t.na; a0 += 32) {
      const int a = a0 + lane;
      const int u = a < t.na ? t.ub[a] : 0, w = a < t.na ? t.wb[a] : 0;
      const int r8 = a < t.na ? (t.cnt[a] + 7) & ~7 : 0;
      int ui = u, wi = w, ri = r8;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v1 = __shfl_up_sync(0xFFFFFFFFu, ui, o), v2 = __shfl_up_sync(0xFFFFFFFFu, wi, o);
        const int v3 = __shfl_up_sync(0xFFFFFFFFu, ri, o);
        if (lane >= o) {
          ui += v1;
          wi += v2;
          ri += v3;
        }
      }
      if (a < t.na) {
        t.ub[a] = ru + ui - u;
        t.wb[a] = rw + wi - w;
        t.row[a] = rr + ri - r8;
      }
      ru += __shfl_sync(0xFFFFFFFFu, ui, 31);
      rw += __shfl_sync(0xFFFFFFFFu, wi, 31);
      rr += __shfl_sync(0xFFFFFFFFu, ri, 31);
    }
    if (lane == 0) {
      t.ub[t.na] = ru;
      t.wb[t.na] = rw;
    }
  }
  __syncthreads();
}

// The largest index i < n with base[i] <= v.
__device__ __forceinline__ int find_le(const int* base, int n, int v) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int m = (lo + hi) >> 1;
    if (base[m] <= v) lo = m;
    else hi = m;
  }
  return lo;
}
// First unit of block b of nb.
__device__ int cut_unit(const MTiles& t, int NT, int b, int nb) {
  const int W = t.wb[t.na], x = (int)((long long)W * b / nb);
  if (b >= nb || x >= W) return t.ub[t.na];
  const int a = find_le(t.wb, t.na, x);   // the last expert that starts at or before: one with units
  const int c = t.cnt[a], f = c / NT, tiles = f + (c > f * NT), m = (t.ub[a + 1] - t.ub[a]) / tiles;
  const int wf = tile_weight(NT), full = f * m * wf;
  int r = x - t.wb[a];
  if (r < full) return t.ub[a] + (r + wf - 1) / wf;
  r -= full;
  const int wp = tile_weight(c - f * NT);
  return t.ub[a] + f * m + (r + wp - 1) / wp;
}

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 ld4s(const uint8_t* p) { return *reinterpret_cast<const uint4*>(p); }

// fp32 pair (a, b) -> fp16 pair hi (truncated to 11 significant bits) and lo (the rest, rounded)
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const float ha = __uint_as_float(__float_as_uint(a) & 0xFFFFE000u);
  const float hb = __uint_as_float(__float_as_uint(b) & 0xFFFFE000u);
  const __half2 h2 = __floats2half2_rn(ha, hb);
  const __half2 l2 = __floats2half2_rn(a - ha, b - hb);
  hi = *reinterpret_cast<const uint32_t*>(&h2);
  lo = *reinterpret_cast<const uint32_t*>(&l2);
}

// 2^S with m 2^S in [2^13, 2^14) (1 for m = 0 or not finite), |S| <= 100.
__device__ __forceinline__ float scale_pow2(float m) {
  if (!(m > 0.f) || !(m < 3.0e38f)) return 1.f;
  int ex;
  frexpf(m, &ex);
  return ldexpf(1.f, max(-100, min(100, 14 - ex)));
}

// Bit position of a B-bit code in its fp16 element: the code times 2^kPos stays below 2048, where the bit
// pattern is linear.  As high as it fits: the tensor core aligns a product by its operands' exponents, so
// with the code in the lowest bits the sum kept only about 16 bits of each product (measured: gate/up off
// by 9e-6 of their norm against 4e-7).
template <int B>
__host__ __device__ constexpr int code_pos() { return B <= 3 ? 8 : B == 4 ? 7 : B == 6 ? 5 : 3; }

// The two A registers of one row (or unit) word: codes m = 0, 2 (lo) and m = 1, 3 (hi) of field k = sh / B.
// The left shift is a multiplication (it runs beside the ALU's shifts and masks).
template <int B>
__device__ __forceinline__ void a_regs(uint32_t w, int sh, uint32_t mul, uint32_t& lo, uint32_t& hi) {
  constexpr uint32_t M = ((1u << B) - 1u) * 0x00010001u << code_pos<B>();
  lo = (w * mul) & M;
  hi = (w >> (sh + 8 - code_pos<B>())) & M;
}
// The same of a code in two planes: PB low bits in w at field shift sh, HB high bits in h at field shift hs.
template <int PB, int HB>
__device__ __forceinline__ void a_regs2(uint32_t w, int sh, uint32_t mul, uint32_t h, int hs, uint32_t& lo, uint32_t& hi) {
  constexpr int P = code_pos<PB + HB>();
  constexpr uint32_t M = ((1u << PB) - 1u) * 0x00010001u << P, MH = ((1u << HB) - 1u) * 0x00010001u << (P + PB);
  lo = ((w * mul) & M) | (__funnelshift_l(h, h, P + PB - hs) & MH);
  hi = ((w >> (sh + 8 - P)) & M) | (__funnelshift_l(h, h, (P + PB - 8 - hs) & 31) & MH);
}

// ---------------------------------------------------------------------------
// Gate/up operand of calls past the decode batch
// ---------------------------------------------------------------------------
// az[h][row][slot]: alpha z 2^S of every (projection, routed token), in the order in which a warp of the
// gate/up kernel reads it: a token tile of `rows` rows (a multiple of 8) holds [slot / 4][row][4], so that a
// K-step of 8 tokens is one 16-byte load a lane (four full lines a warp).  Gathered in the kernel itself, z
// costs four 4-byte loads from as many sectors for each of a tile's row blocks (1024 tokens of the
// Qwen3-shaped layer: gate/up 988 us).
constexpr int kZgThreads = 256;
constexpr int kZgQuads = 128;   // slot quads of a work item (8 tokens each)

__global__ void __launch_bounds__(kZgThreads) k_zgather(Fwd p, MArgs x) {
  extern __shared__ __align__(128) uint8_t msm[];
  __shared__ int s_ok;
  const int tid = threadIdx.x, kNT = 8 * x.ntm;
  MTiles tb = mtiles_at(msm, x.A_max);
  pdl_trigger();
  if (tid == 0) s_ok = wait_flag(p.route_flag);
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
    pdl_wait();
    return;
  }
  mtiles_build(p, x.A_max, 8, tb, [](int) { return 1; });
  const int ng = tb.ub[tb.na], nch = (x.nsp / 4 + kZgQuads - 1) / kZgQuads;
  pdl_wait();   // z and max |z| come from the projection
  const int tk = tid & 7, q0 = tid >> 3;
  for (int w = blockIdx.x; w < ng * 2 * nch; w += gridDim.x) {
    const int gi = w % ng, hc = w / ng, h = hc & 1, ch = hc >> 1;
    const int a = find_le(tb.ub, tb.na, gi), e = tb.e[a], n8 = gi - tb.ub[a];
    const ExpertDesc& xd = p.desc[h * p.E + e];
    const int nq = __ldg(&xd.nslots) >> 2;
    const int* un = reinterpret_cast<const int*>(p.img + __ldg(&xd.unit_off));
    const float* al = reinterpret_cast<const float*>(p.img + __ldg(&xd.alpha_off));
    const int tt = n8 / x.ntm, rows = min(kNT, ((tb.cnt[a] - tt * kNT) + 7) & ~7);
    const bool live = 8 * n8 + tk < tb.cnt[a];
    const int tok = live ? p.pair_list[tb.pst[a] + 8 * n8 + tk] / p.k : 0;
    const float bs = live ? scale_pow2(__ldg(x.msa + h * p.E + e) * __uint_as_float(__ldcg(p.zmax + h * p.T + tok))) : 0.f;
    const float* z = p.z + ((size_t)h * p.T + tok) * p.n_pad;
    float* dst = x.az + ((size_t)h * x.rt + tb.row[a] + tt * kNT) * x.nsp + (size_t)((n8 - tt * x.ntm) * 8 + tk) * 4;
#pragma unroll
    for (int i = 0; i < kZgQuads / (kZgThreads / 8); ++i) {
      const int q = ch * kZgQuads + q0 + i * (kZgThreads / 8);
      if (q < nq) {
        const int4 u = __ldg(reinterpret_cast<const int4*>(un) + q);
        const float4 av = __ldg(reinterpret_cast<const float4*>(al) + q);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (live) v = make_float4(av.x * z[u.x] * bs, av.y * z[u.y] * bs, av.z * z[u.z] * bs, av.w * z[u.w] * bs);
        *reinterpret_cast<float4*>(dst + (size_t)q * rows * 4) = v;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Gate/up
// ---------------------------------------------------------------------------
// Units in (token tile, projection, group of R row blocks, segment) order.  A block takes a contiguous run
// of units; inside it, warp w has row block w % R of the group and part w / R of each run of segments, so
// that the warps of a block read the same operand (L1).  A warp streams its segments' codes and slot
// metadata through its own two-stage ring (two bulk copies a segment) and adds its partial rows into
// gate/up.  The operand is az (AZ), or for the decode batch (at most 8 tokens, no extra launch) gathered
// from z stored token-fastest, where a unit's 8 tokens are one sector.
struct GCur {
  int pos;               // unit at which the current (tile, projection, row group) run starts (>= hi: the end)
  int end;               // its end (inside the block's units)
  int a, tt, h, rb;      // expert index and token tile, projection, row block
  int sg, sg1;           // segment, end of the warp's part
  int first;
};

// 32 rows (from byte row16 of a chunk) of K-step ks of a bucket: A registers of rows 4 g .. 4 g + 3.
template <int B>
__device__ __forceinline__ void rl_a(const uint8_t* code, int ks, int ntl, int row16, int t, uint32_t (&lo)[4],
                                     uint32_t (&hi)[4]) {
  if (B == 3) {
    const uint8_t* c = code + (ks >> 1) * (3 * kChunkBytes) + row16;
    const uint4 w = ld4s(c + (ks & 1) * kChunkBytes), h = ld4s(c + 2 * kChunkBytes);
    const int sh = 2 * t, hs = t + 4 * (ks & 1);
    const uint32_t mul = 1u << (code_pos<3>() - sh);
    a_regs2<2, 1>(w.x, sh, mul, h.x, hs, lo[0], hi[0]);
    a_regs2<2, 1>(w.y, sh, mul, h.y, hs, lo[1], hi[1]);
    a_regs2<2, 1>(w.z, sh, mul, h.z, hs, lo[2], hi[2]);
    a_regs2<2, 1>(w.w, sh, mul, h.w, hs, lo[3], hi[3]);
  } else if (B == 6) {
    const uint8_t* c = code + min(ks, ntl - 1) * (3 * kChunkBytes) + row16;
    const uint4 w = ld4s(c + (t >> 1) * kChunkBytes), h = ld4s(c + 2 * kChunkBytes);
    const int sh = 4 * (t & 1), hs = 2 * t;
    const uint32_t mul = 1u << (code_pos<6>() - sh);
    a_regs2<4, 2>(w.x, sh, mul, h.x, hs, lo[0], hi[0]);
    a_regs2<4, 2>(w.y, sh, mul, h.y, hs, lo[1], hi[1]);
    a_regs2<4, 2>(w.z, sh, mul, h.z, hs, lo[2], hi[2]);
    a_regs2<4, 2>(w.w, sh, mul, h.w, hs, lo[3], hi[3]);
  } else {
    const int tile = B == 1 ? ks >> 1 : min(B == 2 ? ks : B == 4 ? 2 * ks + (t >> 1) : 4 * ks + t, ntl - 1);
    const int sh = B == 1 ? t + 4 * (ks & 1) : B == 2 ? 2 * t : B == 4 ? 4 * (t & 1) : 0;
    const uint32_t mul = 1u << (code_pos<B>() - sh);
    const uint4 w = ld4s(code + tile * kChunkBytes + row16);
    a_regs<B>(w.x, sh, mul, lo[0], hi[0]);
    a_regs<B>(w.y, sh, mul, lo[1], hi[1]);
    a_regs<B>(w.z, sh, mul, lo[2], hi[2]);
    a_regs<B>(w.w, sh, mul, lo[3], hi[3]);
  }
}

// What a lane reads its operand from (run of one token tile and projection).
template <int NTM>
struct GOp {
  const float* az;          // AZ: the tile's az, at this lane's token row
  int rows4;                //     floats between slot quads
  const float* zt[NTM];     // else: z column of this lane's token (unit-major)
  int zstride;              //     floats between units
  float bs[NTM];            //     2^S of this lane's token
};

// A warp's K-steps: KP an iteration; NT groups of 8 tokens; the next iteration's operand is loaded while
// this one is computed, across the buckets of a segment (AZ: across the run's segments too).
template <int NT, int KP, int NTM, bool AZ>
__device__ __forceinline__ void gu_load(const GOp<NTM>& o, const int* su, int slot, int limit, float4 (&zn)[KP][NT]) {
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    const int s = min(slot + 16 * k, limit);
    if (AZ) {
      const float* q = o.az + (s >> 2) * o.rows4;
#pragma unroll
      for (int n = 0; n < NT; ++n) zn[k][n] = *reinterpret_cast<const float4*>(q + 32 * n);
    } else {
      const int4 u = *reinterpret_cast<const int4*>(su + s);
#pragma unroll
      for (int n = 0; n < NT; ++n)
        zn[k][n] = make_float4(__ldcg(o.zt[n] + u.x * o.zstride), __ldcg(o.zt[n] + u.y * o.zstride),
                               __ldcg(o.zt[n] + u.z * o.zstride), __ldcg(o.zt[n] + u.w * o.zstride));
    }
  }
}

// A bucket's run of tiles; s0: its first slot (in the segment, AZ: in the projection), limit: the last slot
// quad that may be loaded ahead, sa / ssz at its first slot (ssz rows `zs` words apart), G scale groups
// inside the 128 rows.
template <int B, int NT, int KP, int NTM, int G, bool AZ>
__device__ __forceinline__ void gu_bucket(const uint8_t* code, int ntl, const GOp<NTM>& o, const int* su, int s0, int limit,
                                          const float* sa, const uint32_t* ssz, int zs, int lane, float4 (&zn)[KP][NT],
                                          float (&acc)[8][NTM][4], float (&cs)[G][NTM]) {
  constexpr float fB = 1.f / (float)(1 << (code_pos<B>() - 3));   // the code's position, taken back in B
  const int g = lane >> 2, t = lane & 3;
  const int nsl = ntl * rl_units(B), nks = (nsl + 15) >> 4;
  float ce[G][NT];   // zero-point corrections
#pragma unroll
  for (int gl = 0; gl < G; ++gl)
#pragma unroll
    for (int n = 0; n < NT; ++n) ce[gl][n] = 0.f;
#pragma unroll 1
  for (int ks = 0; ks < nks; ks += KP) {
    float4 zc[KP][NT];
#pragma unroll
    for (int k = 0; k < KP; ++k)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        zc[k][n] = zn[k][n];
        if (!AZ) {
          zc[k][n].x *= o.bs[n];
          zc[k][n].y *= o.bs[n];
          zc[k][n].z *= o.bs[n];
          zc[k][n].w *= o.bs[n];
        }
      }
    gu_load<NT, KP, NTM, AZ>(o, su, s0 + (ks + KP < nks ? 16 * (ks + KP) : nsl) + 4 * t, limit, zn);
#pragma unroll
    for (int gl = 0; gl < G; ++gl) {
      uint32_t bh[KP][NT][2], bl[KP][NT][2];
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        const int sl = 16 * (ks + k) + 4 * t, slc = min(sl, nsl - 4);
        uint4 sz = *reinterpret_cast<const uint4*>(ssz + gl * zs + slc);
        const float f = sl < nsl ? fB : 0.f;   // past the bucket: the codes read are another slot's
        float w0 = f16lo(sz.x) * f, w1 = f16lo(sz.y) * f, w2 = f16lo(sz.z) * f, w3 = f16lo(sz.w) * f;
        if (!AZ) {
          const float4 al = *reinterpret_cast<const float4*>(sa + slc);
          w0 *= al.x;
          w1 *= al.y;
          w2 *= al.z;
          w3 *= al.w;
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const float v0 = w0 * zc[k][n].x, v1 = w1 * zc[k][n].y, v2 = w2 * zc[k][n].z, v3 = w3 * zc[k][n].w;
          ce[gl][n] = fmaf(f16hi(sz.x), v0, fmaf(f16hi(sz.y), v1, fmaf(f16hi(sz.z), v2, fmaf(f16hi(sz.w), v3, ce[gl][n]))));
          split_pair(v0, v2, bh[k][n][0], bl[k][n][0]);
          split_pair(v1, v3, bh[k][n][1], bl[k][n][1]);
        }
      }
#pragma unroll
      for (int jj = 0; jj < 4 / G; ++jj) {
        const int j = gl * (4 / G) + jj;
#pragma unroll
        for (int k = 0; k < KP; ++k) {
          uint32_t lo[4], hi[4];
          rl_a<B>(code, ks + k, ntl, 16 * (8 * j + g), t, lo, hi);
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            mma_16816(acc[2 * j][n], lo[0], lo[1], hi[0], hi[1], bl[k][n][0], bl[k][n][1]);
            mma_16816(acc[2 * j + 1][n], lo[2], lo[3], hi[2], hi[3], bl[k][n][0], bl[k][n][1]);
          }
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            mma_16816(acc[2 * j][n], lo[0], lo[1], hi[0], hi[1], bh[k][n][0], bh[k][n][1]);
            mma_16816(acc[2 * j + 1][n], lo[2], lo[3], hi[2], hi[3], bh[k][n][0], bh[k][n][1]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int gl = 0; gl < G; ++gl)
#pragma unroll
    for (int n = 0; n < NT; ++n) cs[gl][n] = fmaf(ce[gl][n], 1.f / fB, cs[gl][n]);
}

template <int NT, int KP, int NTM, int G, bool AZ>
__device__ __forceinline__ void gu_segment(const CStage& r, const uint8_t* st, const GOp<NTM>& o, int limit, int lane,
                                           bool first, float4 (&zn)[KP][NTM], float (&acc)[8][NTM][4], float (&cs)[G][NTM]) {
  const int zs = (int)(r.mb >> 2);
  const int* su = reinterpret_cast<const int*>(st + r.bytes);                       // !AZ only
  const float* sa = reinterpret_cast<const float*>(su + zs);                        // !AZ only
  const uint32_t* sz = reinterpret_cast<const uint32_t*>(st + r.bytes + (AZ ? 0u : 2u * r.mb));
  int s0 = AZ ? (int)r.slot0 : 0;
  const int lim = AZ ? limit : zs - 4;
  float4 z[KP][NT];
#pragma unroll
  for (int k = 0; k < KP; ++k)
#pragma unroll
    for (int n = 0; n < NT; ++n) z[k][n] = zn[k][n];
  if (!AZ || first) gu_load<NT, KP, NTM, AZ>(o, su, s0 + 4 * (lane & 3), lim, z);
  for (int q = 0; q < r.nr; ++q) {
    const int b = r.bits[q], ntl = r.ntl[q];
    switch (b) {
      case 1: gu_bucket<1, NT, KP, NTM, G, AZ>(st, ntl, o, su, s0, lim, sa, sz, zs, lane, z, acc, cs); break;
      case 2: gu_bucket<2, NT, KP, NTM, G, AZ>(st, ntl, o, su, s0, lim, sa, sz, zs, lane, z, acc, cs); break;
      case 3: gu_bucket<3, NT, KP, NTM, G, AZ>(st, ntl, o, su, s0, lim, sa, sz, zs, lane, z, acc, cs); break;
      case 4: gu_bucket<4, NT, KP, NTM, G, AZ>(st, ntl, o, su, s0, lim, sa, sz, zs, lane, z, acc, cs); break;
      case 6: gu_bucket<6, NT, KP, NTM, G, AZ>(st, ntl, o, su, s0, lim, sa, sz, zs, lane, z, acc, cs); break;
      default: gu_bucket<8, NT, KP, NTM, G, AZ>(st, ntl, o, su, s0, lim, sa, sz, zs, lane, z, acc, cs); break;
    }
    st += (uint32_t)ntl * rl_chunks(b) * kChunkBytes;
    const int ns = ntl * rl_units(b);
    s0 += ns;
    sa += ns;
    sz += ns;
  }
#pragma unroll
  for (int k = 0; k < KP; ++k)
#pragma unroll
    for (int n = 0; n < NT; ++n) zn[k][n] = z[k][n];
}

constexpr int kMW = 12;   // warps of a block

template <int NTM, int G, bool AZ>
__global__ void __launch_bounds__(kMW * 32, 1) k_gu_mma(Fwd p, MArgs x) {
  constexpr int kNT = 8 * NTM, KP = NTM == 1 ? 2 : 1;
  const int kW = (int)blockDim.x >> 5;   // as many warps as their rings fit in shared memory
  extern __shared__ __align__(128) uint8_t msm[];
  __shared__ uint64_t bars[kMW][2];
  __shared__ CStage recs[kMW][2];
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  uint8_t* ring = msm + (size_t)wid * 2 * x.gu_stage;
  MTiles tb = mtiles_at(msm + (size_t)kW * 2 * x.gu_stage, x.A_max);

  pdl_trigger();
  if (lane == 0) {
    mbar_init(&bars[wid][0]);
    mbar_init(&bars[wid][1]);
  }
  if (tid == 0) s_ok = wait_flag(p.route_flag);
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
    pdl_wait();
    return;
  }
  const int R = x.gu_r, KH = kW / R, nrg = (p.NRB + R - 1) / R, M = 2 * nrg * p.nseg;
  mtiles_build(p, x.A_max, kNT, tb, [&](int) { return M; });
  const int lo = cut_unit(tb, kNT, (int)blockIdx.x, (int)gridDim.x);
  const int hi = cut_unit(tb, kNT, (int)blockIdx.x + 1, (int)gridDim.x);
  const int wr = wid % R, wk = wid / R;   // row block of the group, part of the run (wk == KH: no work)

  // the warp's part of the run that starts at c.pos, skipping runs that have none for it
  auto first_of = [&](GCur& c) {
    for (; c.pos < hi; c.pos = c.end) {
      const int tau = c.pos / M;
      int i = c.pos - tau * M;
      c.h = i >= nrg * p.nseg;
      i -= c.h * nrg * p.nseg;
      const int rg = i / p.nseg, s0 = i - rg * p.nseg;
      c.end = min(hi, c.pos + p.nseg - s0);
      c.rb = rg * R + wr;
      if (wk >= KH || c.rb >= p.NRB) continue;
      const int len = c.end - c.pos;
      c.sg = s0 + len * wk / KH;
      c.sg1 = s0 + len * (wk + 1) / KH;
      if (c.sg == c.sg1) continue;
      c.a = find_le(tb.ub, tb.na, c.pos);
      c.tt = (c.pos - tb.ub[c.a]) / M;
      c.first = 1;
      return;
    }
  };
  auto advance = [&](GCur& c) {
    c.first = 0;
    if (++c.sg < c.sg1) return;
    c.pos = c.end;
    first_of(c);
  };
  // word `lane` of the cursor's staging record
  auto record = [&](const GCur& c) -> uint32_t {
    if (c.pos >= hi || lane >= (int)(sizeof(CStage) / 4)) return 0u;
    return __ldg(reinterpret_cast<const uint32_t*>(x.cst + ((size_t)c.h * p.E + tb.e[c.a]) * p.nseg + c.sg) + lane);
  };
  auto issue = [&](int s, const GCur& c, uint32_t rw) {
    if (lane < (int)(sizeof(CStage) / 4)) reinterpret_cast<uint32_t*>(&recs[wid][s])[lane] = rw;
    const uint64_t code0 = (uint64_t)__shfl_sync(0xFFFFFFFFu, rw, 0) | ((uint64_t)__shfl_sync(0xFFFFFFFFu, rw, 1) << 32);
    const uint32_t rbs = __shfl_sync(0xFFFFFFFFu, rw, 8), bytes = __shfl_sync(0xFFFFFFFFu, rw, 10);
    const uint32_t mb = __shfl_sync(0xFFFFFFFFu, rw, 11), meta0 = __shfl_sync(0xFFFFFFFFu, rw, 18);
    if (lane == 0) {
      uint64_t* bar = &bars[wid][s];
      uint8_t* dst = ring + (size_t)s * x.gu_stage;
      // the record's metadata of a row block: unit indices, alphas (not needed beside az), scale/zero rows
      const uint32_t skip = AZ ? 2u * mb : 0u, mt = bytes ? (2u + G) * mb - skip : 0u;
      fence_proxy_async();   // the stage was last read by the generic proxy
      mbar_expect_tx(bar, bytes + mt);
      if (bytes) {
        bulk_g2s(dst, p.img + code0 + (uint64_t)c.rb * rbs, bytes, bar);
        bulk_g2s(dst + bytes, x.meta + meta0 + (size_t)c.rb * (2u + G) * mb + skip, mt, bar);
      }
    }
  };

  GCur c;
  c.pos = lo;
  first_of(c);
  uint32_t rn = 0;
  GCur n = c;
  if (c.pos < hi) {
    issue(0, c, record(c));
    advance(n);
    rn = record(n);
  }
  pdl_wait();   // z and max |z| come from the projection
  bool ok = true;
  float acc[8][NTM][4];
  float cs[G][NTM];
  GOp<NTM> o;
  float4 zn[KP][NTM];
  float inv[NTM];   // 2^-S of this lane's token
  int ntk = 0, limit = 0;
  bool need = false;   // the run's first operand is still to be loaded
  for (int i = 0; c.pos < hi; ++i) {
    __syncwarp();   // the other stage has been read by every lane
    if (n.pos < hi) issue((i + 1) & 1, n, rn);
    GCur n2 = n;
    if (n.pos < hi) advance(n2);
    rn = record(n2);
    if (c.first) {   // the run's tokens, their operand and its powers of two
      const int e = tb.e[c.a];
      ntk = min(kNT, tb.cnt[c.a] - c.tt * kNT);
      const float ms = __ldg(x.msa + c.h * p.E + e);
      if (AZ) {
        o.rows4 = 4 * min(kNT, (ntk + 7) & ~7);
        o.az = x.az + ((size_t)c.h * x.rt + tb.row[c.a] + c.tt * kNT) * x.nsp + 4 * g;
        limit = max(0, __ldg(&p.desc[c.h * p.E + e].nslots) - 4);
      }
      o.zstride = p.T;
      need = true;
#pragma unroll
      for (int q = 0; q < NTM; ++q) {
        const int tok = p.pair_list[tb.pst[c.a] + c.tt * kNT + min(8 * q + g, ntk - 1)] / p.k;
        o.zt[q] = p.z + (size_t)c.h * p.n_pad * p.T + tok;
        o.bs[q] = scale_pow2(ms * __uint_as_float(__ldcg(p.zmax + c.h * p.T + tok)));
        inv[q] = 1.f / o.bs[q];
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
          for (int w = 0; w < 4; ++w) acc[m][q][w] = 0.f;
#pragma unroll
        for (int gl = 0; gl < G; ++gl) cs[gl][q] = 0.f;
      }
    }
    ok &= mbar_wait(&bars[wid][i & 1], (uint32_t)(i >> 1) & 1u);
    __syncwarp();
    const CStage& r = recs[wid][i & 1];
    const uint8_t* st = ring + (size_t)(i & 1) * x.gu_stage;
    if (r.nr > 0) {
      if (NTM == 1 || ntk <= 8) gu_segment<1, KP, NTM, G, AZ>(r, st, o, limit, lane, need, zn, acc, cs);
      else gu_segment<NTM, KP, NTM, G, AZ>(r, st, o, limit, lane, need, zn, acc, cs);
      need = false;
    }
    if (c.sg + 1 == c.sg1) {   // the part's end: its partial rows into gate/up
#pragma unroll
      for (int q = 0; q < NTM; ++q) {
        if (8 * q >= ntk) break;
        float co[G];
#pragma unroll
        for (int gl = 0; gl < G; ++gl) {   // the token's correction, summed over the K lanes
          float v = cs[gl][q];
          v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
          v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
          co[gl] = v;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int col = 2 * t + u;
          const float iv = __shfl_sync(0xFFFFFFFFu, inv[q], 4 * col), f24 = 2097152.f * iv;   // 2^(24 - 3 - S)
          float cc[G];
#pragma unroll
          for (int gl = 0; gl < G; ++gl) cc[gl] = __shfl_sync(0xFFFFFFFFu, co[gl], 4 * col) * iv;
          if (8 * q + col < ntk) {
            const int pr = p.pair_list[tb.pst[c.a] + c.tt * kNT + 8 * q + col];
            float* gp = p.gu + ((size_t)pr * 2 + c.h) * p.I_pad + c.rb * kRows + 4 * g;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float k0 = cc[j * G / 4];
              red_add_v4(gp + 32 * j, fmaf(acc[2 * j][q][u], f24, -k0), fmaf(acc[2 * j][q][u + 2], f24, -k0),
                         fmaf(acc[2 * j + 1][q][u], f24, -k0), fmaf(acc[2 * j + 1][q][u + 2], f24, -k0));
            }
          }
        }
      }
    }
    c = n;
    n = n2;
  }
  if (!ok && lane == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
}

// ---------------------------------------------------------------------------
// Down
// ---------------------------------------------------------------------------
// Unit-lane tiles (32 units): a warp item = (token tile, run of row blocks, unit tile).  The items of a
// block are consecutive; for each (token tile, run) among them the block forms h = SiLU(gate) up once, as
// B fragments in shared memory, and its warps take the unit tiles, whose codes they stream in pieces of
// at most kStagePiece bytes through their own two-stage ring.
struct DCur {
  int pos, end;          // segment of the block's range: [pos, end) of the flat items, one (tile, run)
  int tau, a, tt, rc;    // its token tile (expert a's tile tt) and run of row blocks
  int tile0;             // unit tile of item `pos`
  int tile, rb, nrb;     // the warp's unit tile, row block and row blocks of the piece
  int seq;               // unit tiles the warp has started (parity of the metadata slot)
};

// K-step ks (16 rows) of a row block: A registers of unit `u16 / 16` of the tile
template <int B>
__device__ __forceinline__ void ul_a(const uint8_t* code, int ks, int u16, int t, uint32_t& lo, uint32_t& hi) {
  auto word = [&](int chunk, int w) {
    return *reinterpret_cast<const uint32_t*>(code + chunk * kChunkBytes + u16 + 4 * w);
  };
  const int sh = B == 1 ? t + 4 * (ks & 1) : B == 2 || B == 3 ? 2 * t : B == 8 ? 0 : 4 * (t & 1);
  const uint32_t mul = 1u << (code_pos<B>() - sh);
  if (B == 1) a_regs<1>(word(0, ks >> 1), sh, mul, lo, hi);
  else if (B == 2) a_regs<2>(word(ks >> 2, ks & 3), sh, mul, lo, hi);
  else if (B == 4) a_regs<4>(word(ks >> 1, 2 * (ks & 1) + (t >> 1)), sh, mul, lo, hi);
  else if (B == 8) a_regs<8>(word(ks, t), sh, mul, lo, hi);
  else if (B == 3) a_regs2<2, 1>(word(ks >> 2, ks & 3), sh, mul, word(2, ks >> 1), t + 4 * (ks & 1), lo, hi);
  else a_regs2<4, 2>(word(ks >> 1, 2 * (ks & 1) + (t >> 1)), sh, mul, word(4 + (ks >> 2), ks & 3), 2 * t, lo, hi);
}

// One row block of a tile: out += scale (P 2^(24 - S) - zero sum(h)) per group
template <int B, int NT, int NTM, int G>
__device__ __forceinline__ void dn_rb(const uint8_t* code, const uint4* hf, int hstride, const float4* hz, int zstride,
                                      const uint32_t* sz, int lane, float (&out)[2][NTM][4]) {
  constexpr float fP = 1.f / (float)(1 << code_pos<B>());   // the codes' position
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int gl = 0; gl < G; ++gl) {
    float P[2][NT][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int w = 0; w < 4; ++w) P[m][n][w] = 0.f;
#pragma unroll
    for (int k = 0; k < 8 / G; ++k) {
      const int ks = gl * (8 / G) + k;
      uint32_t lo[4], hi[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) ul_a<B>(code, ks, 16 * (g + 8 * u), t, lo[u], hi[u]);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const uint4 b = hf[n * hstride + ks * 32 + lane];
        mma_16816(P[0][n], lo[0], lo[1], hi[0], hi[1], b.x, b.y);
        mma_16816(P[1][n], lo[2], lo[3], hi[2], hi[3], b.x, b.y);
        mma_16816(P[0][n], lo[0], lo[1], hi[0], hi[1], b.z, b.w);
        mma_16816(P[1][n], lo[2], lo[3], hi[2], hi[3], b.z, b.w);
      }
    }
    float sc[4], zp[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t w = sz[gl * 32 + g + 8 * u];
      sc[u] = f16lo(w);
      zp[u] = f16hi(w);
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      float4 z = hz[gl * zstride + n * 4 + t];   // tokens 2 t and 2 t + 1: (sum, 2^(24 - S)) each
      z.y *= fP;
      z.w *= fP;
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        out[m][n][0] = fmaf(sc[2 * m], fmaf(P[m][n][0], z.y, -zp[2 * m] * z.x), out[m][n][0]);
        out[m][n][1] = fmaf(sc[2 * m], fmaf(P[m][n][1], z.w, -zp[2 * m] * z.z), out[m][n][1]);
        out[m][n][2] = fmaf(sc[2 * m + 1], fmaf(P[m][n][2], z.y, -zp[2 * m + 1] * z.x), out[m][n][2]);
        out[m][n][3] = fmaf(sc[2 * m + 1], fmaf(P[m][n][3], z.w, -zp[2 * m + 1] * z.z), out[m][n][3]);
      }
    }
  }
}

template <int NT, int NTM, int G>
__device__ __forceinline__ void dn_piece(int b, int nrb, const uint8_t* code, const uint4* hf, int hstride,
                                         const float4* hz, int zstride, const uint32_t* sz, int rb, int group, int lane,
                                         float (&out)[2][NTM][4]) {
  // sz: the tile's scale/zero rows from the run's first group on; rb: the piece's first row block in the run
#pragma unroll 1
  for (int r = 0; r < nrb; ++r) {
    const uint8_t* cb = code + (size_t)r * b * kChunkBytes;
    const uint4* hb = hf + (rb + r) * 8 * 32;
    const float4* zb = hz + (rb + r) * G * zstride;
    const uint32_t* sb = sz + (G > 1 ? (rb + r) * G : (rb + r) * kRows / group) * 32;
    switch (b) {
      case 1: dn_rb<1, NT, NTM, G>(cb, hb, hstride, zb, zstride, sb, lane, out); break;
      case 2: dn_rb<2, NT, NTM, G>(cb, hb, hstride, zb, zstride, sb, lane, out); break;
      case 3: dn_rb<3, NT, NTM, G>(cb, hb, hstride, zb, zstride, sb, lane, out); break;
      case 4: dn_rb<4, NT, NTM, G>(cb, hb, hstride, zb, zstride, sb, lane, out); break;
      case 6: dn_rb<6, NT, NTM, G>(cb, hb, hstride, zb, zstride, sb, lane, out); break;
      default: dn_rb<8, NT, NTM, G>(cb, hb, hstride, zb, zstride, sb, lane, out); break;
    }
  }
}

// Shared-memory plan of k_dn_mma.
struct DPlan {
  uint32_t ring, meta, hf, hz, tabs, total;
};
__host__ __device__ inline DPlan d_plan(int ntm, int G, int warps, const MArgs& x) {
  DPlan s;
  uint32_t o = 0;
  s.ring = o;
  o += (uint32_t)warps * 2u * kStagePiece;
  s.meta = o;
  o += (uint32_t)warps * 2u * x.dn_meta;
  s.hf = o;
  o += (uint32_t)ntm * x.dn_rc * 8u * 32u * 16u;
  s.hz = o;
  o += (uint32_t)x.dn_rc * G * ntm * 8u * 8u;
  s.tabs = o;
  o += mtiles_bytes(x.A_max);
  s.total = (o + 15u) & ~15u;
  return s;
}

template <int NTM, int G>
__global__ void __launch_bounds__(kMW * 32, 1) k_dn_mma(Fwd p, MArgs x) {
  constexpr int kW = kMW, kNT = 8 * NTM;
  extern __shared__ __align__(128) uint8_t msm[];
  __shared__ uint64_t bars[kW][2];
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  const DPlan L = d_plan(NTM, G, kW, x);
  uint8_t* ring = msm + L.ring + (size_t)wid * 2 * kStagePiece;
  uint8_t* meta = msm + L.meta + (size_t)wid * 2 * x.dn_meta;
  uint4* hf = reinterpret_cast<uint4*>(msm + L.hf);       // [NTM][dn_rc][8 K-steps][32 lanes]
  float2* hz = reinterpret_cast<float2*>(msm + L.hz);     // [dn_rc][G][kNT] (sum of h, 2^(24 - S))
  MTiles tb = mtiles_at(msm + L.tabs, x.A_max);
  const int RC = x.dn_rc, nrc = (p.NRB + RC - 1) / RC;
  const ExpertDesc* dd = p.desc + 2 * p.E;

  pdl_trigger();
  if (lane == 0) {
    mbar_init(&bars[wid][0]);
    mbar_init(&bars[wid][1]);
  }
  if (tid == 0) s_ok = wait_flag(p.route_flag);
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
    pdl_wait();
    return;
  }
  mtiles_build(p, x.A_max, kNT, tb, [&](int e) { return nrc * __ldg(&dd[e].ntiles); });
  const int lo = cut_unit(tb, kNT, (int)blockIdx.x, (int)gridDim.x);
  const int hi = cut_unit(tb, kNT, (int)blockIdx.x + 1, (int)gridDim.x);

  // the segment that starts at flat item c.pos (< hi)
  auto seg_at = [&](DCur& c) {
    c.a = find_le(tb.ub, tb.na, c.pos);   // the last expert that starts at or before: one with items
    const int nt = (tb.ub[c.a + 1] - tb.ub[c.a]) / (((tb.cnt[c.a] + kNT - 1) / kNT) * nrc);
    const int q = c.pos - tb.ub[c.a], tr = q / nt;
    c.tile0 = q - tr * nt;
    c.tt = tr / nrc;
    c.rc = tr - c.tt * nrc;
    c.end = min(hi, c.pos + nt - c.tile0);
  };
  auto piece_len = [&](int bits, int left) { return min(left, bits <= 1 ? 8 : bits <= 2 ? 4 : bits <= 4 ? 2 : 1); };
  // the warp's first unit tile at or after the segment, skipping segments without one
  auto first_tile = [&](DCur& c) {
    for (;;) {
      if (c.pos >= hi) return;
      seg_at(c);
      c.tile = c.tile0 + wid;
      c.rb = 0;
      if (c.tile < c.tile0 + (c.end - c.pos)) return;
      c.pos = c.end;
    }
  };
  // words of the unit tile's staging record (12 words: lane l holds word l)
  auto record = [&](const DCur& c) -> uint32_t {
    if (c.pos >= hi || lane >= (int)(sizeof(DStage) / 4)) return 0u;
    return __ldg(reinterpret_cast<const uint32_t*>(x.dst + (size_t)tb.e[c.a] * p.ul_max_tiles + c.tile) + lane);
  };
  auto run_nrb = [&](const DCur& c) { return min(RC, p.NRB - c.rc * RC); };
  auto issue = [&](int s, DCur& c, uint32_t rw) {
    const uint64_t code = (uint64_t)__shfl_sync(0xFFFFFFFFu, rw, 0) | ((uint64_t)__shfl_sync(0xFFFFFFFFu, rw, 1) << 32);
    const uint32_t bits = __shfl_sync(0xFFFFFFFFu, rw, 9), mt = __shfl_sync(0xFFFFFFFFu, rw, 10);
    c.nrb = piece_len((int)bits, run_nrb(c) - c.rb);
    if (lane == 0) {
      uint64_t* bar = &bars[wid][s];
      const uint32_t bytes = (uint32_t)c.nrb * bits * kChunkBytes;
      fence_proxy_async();   // the stage was last read by the generic proxy
      uint32_t tx = bytes, szb = 0;
      if (c.rb == 0) {   // the tile's units, alphas and its scale/zero rows of this run
        const int g0 = c.rc * RC * kRows / p.group, g1 = min(p.NG, ((c.rc * RC + run_nrb(c)) * kRows + p.group - 1) / p.group);
        szb = (uint32_t)(g1 - g0) * 128u;
        tx += 256u + szb;
        mbar_expect_tx(bar, tx);
        uint8_t* md = meta + (size_t)(c.seq & 1) * x.dn_meta;
        bulk_g2s(md, x.meta + mt, 256u, bar);
        bulk_g2s(md + 256, x.meta + mt + 256u + (uint32_t)g0 * 128u, szb, bar);
      } else {
        mbar_expect_tx(bar, tx);
      }
      bulk_g2s(ring + (size_t)s * kStagePiece, p.img + code + (uint64_t)(c.rc * RC + c.rb) * bits * kChunkBytes, bytes, bar);
    }
  };
  auto advance = [&](DCur& c) {   // the next piece
    c.rb += c.nrb;
    if (c.rb < run_nrb(c)) return;
    c.rb = 0;
    c.tile += kW;
    ++c.seq;
    if (c.tile < c.tile0 + (c.end - c.pos)) return;
    c.pos = c.end;
    first_tile(c);
  };

  DCur n;   // the piece being staged
  n.pos = lo;
  n.seq = 0;
  n.nrb = 0;
  first_tile(n);
  uint32_t rn = record(n), rnn = 0;
  int i = 0;        // pieces consumed
  DCur c = n;       // the piece being consumed
  uint32_t rcw = rn;
  if (n.pos < hi) {
    issue(0, n, rn);
    c = n;
    advance(n);
    rn = record(n);
  }
  pdl_wait();   // gate/up come from the previous kernel
  bool ok = true;
  DCur sgm;
  for (sgm.pos = lo; sgm.pos < hi; sgm.pos = sgm.end) {
    seg_at(sgm);
    __syncthreads();   // the previous segment's h has been read
    const int nrb = run_nrb(sgm), ntk = min(kNT, tb.cnt[sgm.a] - sgm.tt * kNT);
    const int pst = tb.pst[sgm.a] + sgm.tt * kNT;
    const int ntc = (ntk + 7) & ~7;
    for (int w = wid; w < ntc * nrb; w += kW) {   // a warp per (token, row block): 4 rows a lane
      const int tk = w / nrb, rb = w - tk * nrb;
      float4 h4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (tk < ntk) {
        const int pr = p.pair_list[pst + tk];
        const float* gp = p.gu + (size_t)pr * 2 * p.I_pad + (sgm.rc * RC + rb) * kRows + 4 * lane;
        const float4 gv = __ldcg(reinterpret_cast<const float4*>(gp));
        const float4 uv = __ldcg(reinterpret_cast<const float4*>(gp + p.I_pad));
        h4.x = gv.x / (1.f + __expf(-gv.x)) * uv.x;
        h4.y = gv.y / (1.f + __expf(-gv.y)) * uv.y;
        h4.z = gv.z / (1.f + __expf(-gv.z)) * uv.z;
        h4.w = gv.w / (1.f + __expf(-gv.w)) * uv.w;
      }
      const float am = warp_max(fmaxf(fmaxf(fabsf(h4.x), fabsf(h4.y)), fmaxf(fabsf(h4.z), fabsf(h4.w))));
      float sum = (h4.x + h4.y) + (h4.z + h4.w);
#pragma unroll
      for (int o = 16 / G; o; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
      const float sc = scale_pow2(am);
      uint4 v;
      split_pair(h4.x * sc, h4.z * sc, v.x, v.z);
      split_pair(h4.y * sc, h4.w * sc, v.y, v.w);
      hf[((size_t)(tk >> 3) * RC + rb) * 256 + (lane >> 2) * 32 + (tk & 7) * 4 + (lane & 3)] = v;
      if ((lane & (32 / G - 1)) == 0) hz[((size_t)rb * G + lane / (32 / G)) * kNT + tk] = make_float2(sum, 16777216.f / sc);
    }
    __syncthreads();
    // this warp's unit tiles of the segment
    const int tend = sgm.tile0 + (sgm.end - sgm.pos);
    for (int tile = sgm.tile0 + wid; tile < tend; tile += kW) {
      float out[2][NTM][4];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int q = 0; q < NTM; ++q)
#pragma unroll
          for (int w = 0; w < 4; ++w) out[m][q][w] = 0.f;
      const int bits = (int)__shfl_sync(0xFFFFFFFFu, rcw, 9);
      const uint8_t* md = meta + (size_t)(c.seq & 1) * x.dn_meta;
      for (int rb = 0; rb < nrb; ++i) {
        __syncwarp();   // the other stage has been read by every lane
        const int np = c.nrb;
        const DCur nc = n;
        rnn = rn;
        if (n.pos < hi) {
          issue((i + 1) & 1, n, rn);
          c = n;
          advance(n);
          rn = record(n);
        } else {
          c = nc;
        }
        ok &= mbar_wait(&bars[wid][i & 1], (uint32_t)(i >> 1) & 1u);
        __syncwarp();
        const uint8_t* code = ring + (size_t)(i & 1) * kStagePiece;
        const uint32_t* szp = reinterpret_cast<const uint32_t*>(md + 256);
        const float4* hz4 = reinterpret_cast<const float4*>(hz);
        if (NTM == 1 || ntk <= 8)
          dn_piece<1, NTM, G>(bits, np, code, hf, RC * 256, hz4, kNT / 2, szp, rb, p.group, lane, out);
        else
          dn_piece<NTM, NTM, G>(bits, np, code, hf, RC * 256, hz4, kNT / 2, szp, rb, p.group, lane, out);
        rb += np;
        rcw = rnn;
      }
      // s += g alpha out
      const int* un = reinterpret_cast<const int*>(md);
      const float* al = reinterpret_cast<const float*>(md + 128);
#pragma unroll
      for (int q = 0; q < NTM; ++q) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int tk = 8 * q + 2 * t + u;
          if (tk >= ntk) continue;
          const int pr = p.pair_list[pst + tk];
          const float pw = p.pair_weight[pr];
          float* sp = p.s + (size_t)(pr / p.k) * p.n_pad;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float a = al[g + 8 * v];
            if (a != 0.f) atomicAdd(sp + un[g + 8 * v], pw * a * out[v >> 1][q][u + 2 * (v & 1)]);
          }
        }
      }
      __syncwarp();   // the tile's metadata slot may be refilled
    }
  }
  if (!ok && lane == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
}

}  // namespace

namespace bmoe {

// Largest staged gate/up segment of a layer: codes, unit indices, alphas and G scale/zero rows.
uint32_t mma_gu_stage(const std::vector<CStage>& cst, int G, bool az) {
  uint32_t m = 0;
  for (const CStage& r : cst)
    if (r.bytes) m = std::max(m, r.bytes + ((az ? 0u : 2u) + (uint32_t)G) * r.mb);
  return (m + 127u) & ~127u;
}

constexpr uint32_t kMaxSmem = 222u * 1024u;   // dynamic shared memory of a block (static parts beside it)

static uint32_t gu_smem(const MArgs& x, int warps) { return (uint32_t)warps * 2u * x.gu_stage + mtiles_bytes(x.A_max); }
// Warps of a gate/up block: as many as kMW whose rings fit, 0 when not even four do.
static int gu_warps(const MArgs& x) {
  int w = kMW;
  while (w >= 4 && gu_smem(x, w) > kMaxSmem) --w;
  return w >= 4 ? w : 0;
}

// Row blocks a gate/up block works on at once: the split warps = R x parts with the fewest idle warps
// (the larger R where equal: its warps share the operand's reads).
static int gu_rows(int NRB, int warps) {
  int best = 1;
  double bu = 0;
  for (int R = std::min(NRB, warps); R >= 1; --R) {
    const double u = (double)NRB / ((NRB + R - 1) / R * R) * (R * (warps / R)) / warps;
    if (u > bu + 1e-9) {
      bu = u;
      best = R;
    }
  }
  return best;
}

uint64_t mma_az_floats(const ImageHeader& hd, int T, int k, int* rt, int* nsp) {
  const int P = T * k, A = std::min(hd.E, P);
  *rt = (int)align_up((uint64_t)P + 7 * (uint64_t)A, 8);
  *nsp = (int)align_up((uint64_t)hd.n + 7 * 32, 4);   // units and the padding of seven buckets (< 32 slots each)
  return 2ull * (uint64_t)*rt * (uint64_t)*nsp;
}

bool mma_args(const ImageHeader& hd, int T, int k, bool az, uint32_t gu_stage, MArgs* x) {
  std::memset(x, 0, sizeof(*x));
  const int G = std::max(1, kRows / hd.group);
  x->ntm = T <= 16 ? 1 : 2;
  x->A_max = std::min(hd.E, T * k);
  x->use_az = az;
  mma_az_floats(hd, T, k, &x->rt, &x->nsp);
  x->gu_stage = gu_stage;
  const int gw = gu_stage > 0 ? gu_warps(*x) : 0;
  if (gw <= 0) return false;
  x->gu_r = gu_rows(hd.NRB, gw);
  const int need = std::max(1, hd.group / kRows);   // whole groups a run of row blocks
  x->dn_rc = std::max(need, std::min(hd.NRB, 8) / need * need);
  x->dn_meta = 256u + 128u * (uint32_t)(x->dn_rc * kRows / hd.group);
  return d_plan(x->ntm, G, kMW, *x).total <= kMaxSmem;
}

template <class K>
static cudaError_t mm_launch(K kernel, int grid, int threads, uint32_t smem, const Fwd& p, const MArgs& x, cudaStream_t st,
                             bool pdl, uint32_t* done) {
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (smem > *done) {
      const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      *done = smem;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, p, x);
}

template <int NTM, int G>
static cudaError_t mm_pair(bool down, const Fwd& p, const MArgs& x, int sms, cudaStream_t st, bool pdl) {
  static uint32_t done[3] = {0, 0, 0};
  if (down) return mm_launch(k_dn_mma<NTM, G>, sms, kMW * 32, d_plan(NTM, G, kMW, x).total, p, x, st, pdl, &done[0]);
  const int w = gu_warps(x);
  if constexpr (NTM == 1) {
    if (!x.use_az) return mm_launch(k_gu_mma<1, G, false>, sms, w * 32, gu_smem(x, w), p, x, st, pdl, &done[1]);
  }
  return mm_launch(k_gu_mma<NTM, G, true>, sms, w * 32, gu_smem(x, w), p, x, st, pdl, &done[2]);
}

cudaError_t launch_expert_mma(bool down, const Fwd& p, const MArgs& x, int sms, cudaStream_t st, bool pdl) {
  const int G = std::max(1, kRows / p.group);
  if (!down && x.use_az) {
    static uint32_t done = 0;
    const cudaError_t e = mm_launch(k_zgather, 4 * sms, kZgThreads, mtiles_bytes(x.A_max), p, x, st, pdl, &done);
    if (e != cudaSuccess) return e;
  }
  if (x.ntm == 2)
    return G == 1 ? mm_pair<2, 1>(down, p, x, sms, st, pdl)
                  : G == 2 ? mm_pair<2, 2>(down, p, x, sms, st, pdl) : mm_pair<2, 4>(down, p, x, sms, st, pdl);
  return G == 1 ? mm_pair<1, 1>(down, p, x, sms, st, pdl)
                : G == 2 ? mm_pair<1, 2>(down, p, x, sms, st, pdl) : mm_pair<1, 4>(down, p, x, sms, st, pdl);
}

}  // namespace bmoe
