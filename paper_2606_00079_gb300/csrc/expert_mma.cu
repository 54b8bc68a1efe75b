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
#include <numeric>

#include "device.cuh"
#include "tc.cuh"

namespace {

constexpr int kCW = kMmaWarps;      // consumer warps of both kernels
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
  int na;
};
__host__ __device__ inline uint32_t mtiles_bytes(int A_max) { return ((5u * (uint32_t)A_max + 2u) * 4u + 15u) & ~15u; }

__device__ MTiles mtiles_at(uint8_t* sm, int A_max) {
  MTiles t;
  t.e = reinterpret_cast<int*>(sm);
  t.cnt = t.e + A_max;
  t.pst = t.cnt + A_max;
  t.ub = t.pst + A_max;
  t.wb = t.ub + A_max + 1;
  t.na = 0;
  return t;
}
// Relative time of a tile of nt tokens (measured: the decode of the codes is shared by a tile's groups of
// 8 tokens, the operand and the products are not).
__device__ __forceinline__ int tile_weight(int nt) { return 1 + ((nt + 7) >> 3); }

// Whole block; the routing is published.  per_tile(e): units of a token tile of expert e.  An expert, a count or a
// list outside the call's (another call on the same workspace, or a workspace that was not zero-filled) gets no
// units, and the status word says so.  (An early return instead cost the down kernel spills.)
template <class F>
__device__ void mtiles_build(const Fwd& p, int A_max, int lose, int NT, MTiles& t, F per_tile) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int na = p.active[0];
  bool bad = na < 0 || na > A_max;
  t.na = bad ? 0 : na;
  for (int a = tid; a < t.na; a += (int)blockDim.x) {
    const int e = p.active[1 + a];
    // Read side by side, at a place that is there whatever e is (one after the other's check: 8 tokens 60.9 us
    // against 60.5; without a branch 60.1, but 1024 tokens 719 against 711).
    const int es = (int)min((unsigned)e, (unsigned)p.E - 1u);
    const int c = p.expert_count[es] + (lose & 2) * p.T, start = p.expert_start[es], m = per_tile(es);
    if (e != es || (unsigned)(c - 1) >= (unsigned)p.T || (unsigned)start > (unsigned)(p.P - c)) {
      bad = true;
      t.ub[a] = t.wb[a] = t.cnt[a] = 0;
      continue;
    }
    t.e[a] = e;
    t.cnt[a] = c;
    t.pst[a] = start;
    const int f = c / NT, r = c - f * NT;
    t.ub[a] = (f + (r > 0)) * m;
    t.wb[a] = (f * tile_weight(NT) + (r > 0 ? tile_weight(r) : 0)) * m;
  }
  if (bad) atomicCAS(p.status, 0, BITSMOE_ERR_WORKSPACE_STATE);
  __syncthreads();
  if (tid < 32) {   // exclusive prefixes
    int ru = 0, rw = 0;
    for (int a0 = 0; a0 < t.na; a0 += 32) {
      const int a = a0 + lane;
      const int u = a < t.na ? t.ub[a] : 0, w = a < t.na ? t.wb[a] : 0;
      int ui = u, wi = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v1 = __shfl_up_sync(0xFFFFFFFFu, ui, o), v2 = __shfl_up_sync(0xFFFFFFFFu, wi, o);
        if (lane >= o) {
          ui += v1;
          wi += v2;
        }
      }
      if (a < t.na) {
        t.ub[a] = ru + ui - u;
        t.wb[a] = rw + wi - w;
      }
      ru += __shfl_sync(0xFFFFFFFFu, ui, 31);
      rw += __shfl_sync(0xFFFFFFFFu, wi, 31);
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
  const int W = t.wb[t.na], wq = W / nb;
  const int x = wq * b + (W - wq * nb) * b / nb;   // W b / nb in 32 bits
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

// Packed fp32 pairs (each operation rounded as the scalar one; one issue slot for two: the gate/up kernel's
// operands so, 386 -> 368 us at 1024 tokens).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// split_pair of (v0, v2) and (v1, v3), given (v0, v1) and (v2, v3)
__device__ __forceinline__ void split_quad(uint64_t v01, uint64_t v23, uint32_t (&hi)[2], uint32_t (&lo)[2]) {
  const uint64_t kMask = 0xFFFFE000FFFFE000ull, minus = pack2(-1.f, -1.f);
  const uint64_t h01 = v01 & kMask, h23 = v23 & kMask;
  const uint64_t r01 = fma2(h01, minus, v01), r23 = fma2(h23, minus, v23);
  float a, b, c, d;
  auto half2 = [](float x, float y) {
    const __half2 h = __floats2half2_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&h);
  };
  unpack2(h01, a, b);
  unpack2(h23, c, d);
  hi[0] = half2(a, c);
  hi[1] = half2(b, d);
  unpack2(r01, a, b);
  unpack2(r23, c, d);
  lo[0] = half2(a, c);
  lo[1] = half2(b, d);
}

// 2^S with m 2^S in [2^13, 2^14) (1 for m = 0 or not finite), LO <= S <= 126: below 2^-112 the operand shrinks towards
// 1, which an fp16 pair still holds, above 2^(14 - LO) it grows up to fp16's largest.
template <int LO>
__device__ __forceinline__ float scale_pow2(float m) {
  if (!(m > 0.f) || !(m < 3.0e38f)) return 1.f;
  int ex;
  frexpf(m, &ex);
  return ldexpf(1.f, max(LO, min(126, 14 - ex)));
}
constexpr int kGuLo = -106;         // gate/up undo 2^(S - 21) in one factor
constexpr int kDnLo = -114;         // down in two: 2^(12 - S) with h's sums, 2^12 with the gate weight (exact, and
constexpr float kDnPart = 4096.f;   // whatever q h sums to stays inside fp32 where its product with the scale does)

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
// Gate/up
// ---------------------------------------------------------------------------
// Units in (token tile, projection, group of R row blocks, segment) order, the segments of a run taken with a
// stride: they hold equal bytes, so a segment of 1-bit units has four times the slots (and work) of one of
// 4-bit units, and a stride spreads them over the blocks and groups (in order, the blocks of the 8-token call
// ended between 21 and 33 us).  A block takes a contiguous run of units.  Its 12 consumer warps form KH groups of R: the warps of a group work on the same segment, one
// row block each, and the groups take parts of each run of segments.  4 / KH helper warps a group fill its
// two-stage ring: bulk copies of the R row blocks' codes and scale/zero rows, and the operand alpha z 2^S of
// the segment's slots, gathered from z once for the group (the consumers, at three warps a scheduler, cannot
// hide a global load: gathering in them, or reading a gathered copy from memory, left long-scoreboard stalls
// of 3 issue slots an instruction).  The consumers decode, multiply and add their partial rows into gate/up.
constexpr int kHW = 4;                       // helper warps of both kernels
constexpr int kMmThreads = (kCW + kHW) * 32;
constexpr int kMaxKH = 4;
static_assert(kCW <= 16, "a stage's copies are issued by 16 lanes each for the codes and the scale/zero rows");

struct GCur {
  int pos;               // unit at which the current (tile, projection, row group) run starts (>= hi: the end)
  int end;               // its end (inside the block's units)
  int a, tt, h, rg;      // expert index and token tile, projection, group of row blocks
  int i, i1;             // index of the segment in the run's order, end of the block's part of the run
  int first;
};

// A stage's description for the consumers.
struct GInfo {
  CStage rec;
  int flags;             // 1 first of the run, 2 last, 4 end of the block's work
  int h, rg, ntk, run;   // projection, group of row blocks, tokens of the tile, parity of the run
  int pad_[3];
};
struct GRun {            // rows of a run's token tile
  int pair[16];
  float inv[16];         // 2^-S
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
    const uint8_t* c = code + ks * (3 * kChunkBytes) + row16;
    const uint4 w = ld4s(c + (t >> 1) * kChunkBytes), h = ld4s(c + 2 * kChunkBytes);
    const int sh = 4 * (t & 1), hs = 2 * t;
    const uint32_t mul = 1u << (code_pos<6>() - sh);
    a_regs2<4, 2>(w.x, sh, mul, h.x, hs, lo[0], hi[0]);
    a_regs2<4, 2>(w.y, sh, mul, h.y, hs, lo[1], hi[1]);
    a_regs2<4, 2>(w.z, sh, mul, h.z, hs, lo[2], hi[2]);
    a_regs2<4, 2>(w.w, sh, mul, h.w, hs, lo[3], hi[3]);
  } else {
    const int tile = B == 1 ? ks >> 1 : B == 2 ? ks : min(B == 4 ? 2 * ks + (t >> 1) : 4 * ks + t, ntl - 1);
    const int sh = B == 1 ? t + 4 * (ks & 1) : B == 2 ? 2 * t : B == 4 ? 4 * (t & 1) : 0;
    const uint32_t mul = 1u << (code_pos<B>() - sh);
    const uint4 w = ld4s(code + tile * kChunkBytes + row16);
    a_regs<B>(w.x, sh, mul, lo[0], hi[0]);
    a_regs<B>(w.y, sh, mul, lo[1], hi[1]);
    a_regs<B>(w.z, sh, mul, lo[2], hi[2]);
    a_regs<B>(w.w, sh, mul, lo[3], hi[3]);
  }
}

// Operand rows in shared memory: [slot quad][8 NTM rows][4 slots] fp32, the quads kQS bytes apart (32 bytes
// of padding: the four K lanes of a warp then read different banks).
template <int NTM>
__host__ __device__ constexpr int az_quad() { return 128 * NTM + 32; }

// A bucket's run of tiles: NT groups of 8 tokens, G scale groups inside the 128 rows; az: the operand of the
// bucket's first slot at this lane's row, ssz: its scale/zero word (rows `zs` words apart).
template <int B, int NT, int NTM, int G>
__device__ __forceinline__ void gu_bucket(const uint8_t* code, int ntl, const uint8_t* az, const uint32_t* ssz, int zs,
                                          int lane, float (&acc)[8][NTM][4], float (&cs)[G][NTM]) {
  constexpr float fB = 1.f / (float)(1 << (code_pos<B>() - 3));   // the code's position, taken back in B
  constexpr int kQS = az_quad<NTM>(), JP = G <= 2 ? 2 : 1;
  const int g = lane >> 2, t = lane & 3;
  const int nsl = ntl * rl_units(B), nks = (nsl + 15) >> 4;
  float ce[G][NT];   // zero-point corrections
#pragma unroll
  for (int gl = 0; gl < G; ++gl)
#pragma unroll
    for (int n = 0; n < NT; ++n) ce[gl][n] = 0.f;
#pragma unroll 1
  for (int ks = 0; ks < nks; ++ks) {
    const int sl = 16 * ks + 4 * t, slc = min(sl, nsl - 4);
    const float f = sl < nsl ? fB : 0.f;   // past the bucket: the codes read are another slot's
    const uint64_t f2 = pack2(f, f);
    ulonglong2 zc[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) zc[n] = *reinterpret_cast<const ulonglong2*>(az + (slc >> 2) * kQS + 128 * n);
#pragma unroll
    for (int gl = 0; gl < G; ++gl) {
      uint32_t bh[NT][2], bl[NT][2];
      const uint4 sz = *reinterpret_cast<const uint4*>(ssz + gl * zs + slc);
      const uint64_t w01 = mul2(pack2(f16lo(sz.x), f16lo(sz.y)), f2), w23 = mul2(pack2(f16lo(sz.z), f16lo(sz.w)), f2);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const uint64_t v01 = mul2(w01, zc[n].x), v23 = mul2(w23, zc[n].y);
        float v0, v1, v2, v3;
        unpack2(v01, v0, v1);
        unpack2(v23, v2, v3);
        ce[gl][n] = fmaf(f16hi(sz.x), v0, fmaf(f16hi(sz.y), v1, fmaf(f16hi(sz.z), v2, fmaf(f16hi(sz.w), v3, ce[gl][n]))));
        split_quad(v01, v23, bh[n], bl[n]);
      }
#pragma unroll
      for (int jj = 0; jj < 4 / G; jj += JP) {
        uint32_t lo[JP][4], hi[JP][4];
#pragma unroll
        for (int q = 0; q < JP; ++q) rl_a<B>(code, ks, ntl, 16 * (8 * (gl * (4 / G) + jj + q) + g), t, lo[q], hi[q]);
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int q = 0; q < JP; ++q) {
            const int j = gl * (4 / G) + jj + q;
            mma_16816(acc[2 * j][n], lo[q][0], lo[q][1], hi[q][0], hi[q][1], bl[n][0], bl[n][1]);
            mma_16816(acc[2 * j + 1][n], lo[q][2], lo[q][3], hi[q][2], hi[q][3], bl[n][0], bl[n][1]);
          }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int q = 0; q < JP; ++q) {
            const int j = gl * (4 / G) + jj + q;
            mma_16816(acc[2 * j][n], lo[q][0], lo[q][1], hi[q][0], hi[q][1], bh[n][0], bh[n][1]);
            mma_16816(acc[2 * j + 1][n], lo[q][2], lo[q][3], hi[q][2], hi[q][3], bh[n][0], bh[n][1]);
          }
      }
    }
  }
#pragma unroll
  for (int gl = 0; gl < G; ++gl)
#pragma unroll
    for (int n = 0; n < NT; ++n) cs[gl][n] = fmaf(ce[gl][n], 1.f / fB, cs[gl][n]);
}

// A staged segment: st = the warp's codes, sz its scale/zero rows, az the group's operand at this lane's row.
template <int NT, int NTM, int G>
__device__ __forceinline__ void gu_segment(const CStage& r, const uint8_t* st, const uint32_t* sz, const uint8_t* az,
                                           int lane, float (&acc)[8][NTM][4], float (&cs)[G][NTM]) {
  const int zs = (int)(r.mb >> 2), nr = r.nr;
  for (int q = 0; q < nr; ++q) {
    const int b = r.bits[q], ntl = r.ntl[q];
    switch (b) {
      case 1: gu_bucket<1, NT, NTM, G>(st, ntl, az, sz, zs, lane, acc, cs); break;
      case 2: gu_bucket<2, NT, NTM, G>(st, ntl, az, sz, zs, lane, acc, cs); break;
      case 3: gu_bucket<3, NT, NTM, G>(st, ntl, az, sz, zs, lane, acc, cs); break;
      case 4: gu_bucket<4, NT, NTM, G>(st, ntl, az, sz, zs, lane, acc, cs); break;
      case 6: gu_bucket<6, NT, NTM, G>(st, ntl, az, sz, zs, lane, acc, cs); break;
      default: gu_bucket<8, NT, NTM, G>(st, ntl, az, sz, zs, lane, acc, cs); break;
    }
    st += (uint32_t)ntl * rl_chunks(b) * kChunkBytes;
    const int ns = ntl * rl_units(b);
    az += (ns >> 2) * az_quad<NTM>();
    sz += ns;
  }
}

template <int NTM, int G>
__global__ void __launch_bounds__(kMmThreads, 1) k_gu_mma(Fwd p, MArgs x) {
  constexpr int kNT = 8 * NTM, kQS = az_quad<NTM>();
  extern __shared__ __align__(128) uint8_t msm[];
  __shared__ uint64_t full[kMaxKH][2], empty[kMaxKH][2];
  __shared__ __align__(16) GInfo infos[kMaxKH][2];
  __shared__ GRun runs[kMaxKH][2];
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int R = x.gu_r, KH = x.gu_kh, HG = kHW / KH;
  MTiles tb = mtiles_at(msm + (size_t)KH * 2 * x.gu_stage, x.A_max);

  pdl_trigger();
  if (tid == 0) {
    for (int q = 0; q < KH; ++q)
      for (int s = 0; s < 2; ++s) {
        mbar_init_n(&full[q][s], 1 + HG);   // the copies' expectation, and each helper's part of the operand
        mbar_init_n(&empty[q][s], R);
      }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_ok = wait_flag(p.route_flag);
  }
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
    pdl_wait();
    return;
  }
  const int nrg = (p.NRB + R - 1) / R, M = 2 * nrg * p.nseg;
  mtiles_build(p, x.A_max, x.lose, kNT, tb, [&](int) { return M; });
  bool ok = true;

  if (wid >= kCW) {
    // ---- helpers
    const int hw = wid - kCW, gr = hw / HG, sub = hw - gr * HG;
    if (gr >= KH) {
      pdl_wait();
      return;
    }
    const int lo = cut_unit(tb, kNT, (int)blockIdx.x, (int)gridDim.x);
    const int hi = cut_unit(tb, kNT, (int)blockIdx.x + 1, (int)gridDim.x);
    uint8_t* ring = msm + (size_t)gr * 2 * x.gu_stage;
    // the group's part of the run that starts at c.pos, skipping runs that have none for it
    auto first_of = [&](GCur& c) {
      for (; c.pos < hi; c.pos = c.end) {
        const int tau = c.pos / M;
        int i = c.pos - tau * M;
        c.h = i >= nrg * p.nseg;
        i -= c.h * nrg * p.nseg;
        c.rg = i / p.nseg;
        const int s0 = i - c.rg * p.nseg;
        c.end = min(hi, c.pos + p.nseg - s0);
        c.i = s0 + (gr + tau + c.h) % KH;   // every KH-th segment; which group starts changes from run to run
        c.i1 = s0 + c.end - c.pos;
        if (c.i >= c.i1) continue;
        c.a = find_le(tb.ub, tb.na, c.pos);
        c.tt = (c.pos - tb.ub[c.a]) / M;
        c.first = 1;
        return;
      }
    };
    auto advance = [&](GCur& c) {
      c.first = 0;
      if ((c.i += KH) < c.i1) return;
      c.pos = c.end;
      first_of(c);
    };
    // word `lane` of the cursor's staging record
    auto record = [&](const GCur& c) -> uint32_t {
      if (c.pos >= hi || lane >= (int)(sizeof(CStage) / 4)) return 0u;
      return __ldg(reinterpret_cast<const uint32_t*>(x.cst + ((size_t)c.h * p.E + tb.e[c.a]) * p.nseg + c.i * x.seg_stride % p.nseg) + lane);
    };
    auto pair_of = [&](const GCur& c) {   // lane < 16: the pair of the tile's row `lane`
      const int ntk = min(kNT, tb.cnt[c.a] - c.tt * kNT);
      return p.pair_list[tb.pst[c.a] + c.tt * kNT + min(lane & 15, ntk - 1)];
    };
    // Pipeline, so that no latency but the copies' own follows the release of a stage: the records are loaded
    // two stages ahead, the units and alphas of a stage's first 128 slots one stage ahead, and their z (the
    // first kRB rows) before the wait for the stage.
    constexpr int kRB = 4 * NTM;
    GCur c, n;
    c.pos = lo;
    first_of(c);
    n = c;
    uint32_t rw = record(c), rwn = 0;
    int pr = 0, prn = 0;
    if (c.pos < hi) {
      pr = pair_of(c);
      advance(n);
      rwn = record(n);
      prn = n.pos < hi && n.first ? pair_of(n) : pr;
    }
    auto units = [&](uint32_t r, int q, int4& u, float4& al) {   // slot quad q of the segment of record r
      const uint32_t mb = __shfl_sync(0xFFFFFFFFu, r, 11), m0 = __shfl_sync(0xFFFFFFFFu, r, 18);
      u = make_int4(0, 0, 0, 0);
      al = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q < (int)(mb >> 4)) {
        u = __ldg(reinterpret_cast<const int4*>(x.meta + m0) + q);
        al = __ldg(reinterpret_cast<const float4*>(x.meta + m0 + mb) + q);
      }
    };
    int4 uc, un;
    float4 ac, an;
    units(rw, lane, uc, ac);
    int tok = 0, run = 0;
    float bs = 1.f;
    int i = 0;
    for (;; ++i) {
      const int s = i & 1;
      GInfo& f = infos[gr][s];
      if (c.pos >= hi) {
        if (i >= 2) ok &= mbar_wait(&empty[gr][s], (uint32_t)((i >> 1) - 1) & 1u, x.spin);
        if (!__all_sync(0xFFFFFFFFu, ok)) break;
        if (lane == 0) {
          if (sub == 0) {
            f.flags = 4;
            mbar_arrive(&full[gr][s]);
          }
          mbar_arrive(&full[gr][s]);
        }
        if (i == 0) pdl_wait();
        break;
      }
      const int ntk = min(kNT, tb.cnt[c.a] - c.tt * kNT);
      const int r0 = ntk * sub / HG, r1 = ntk * (sub + 1) / HG;   // this helper's rows
      const uint32_t bytes = __shfl_sync(0xFFFFFFFFu, rw, 10), mb = __shfl_sync(0xFFFFFFFFu, rw, 11), zb = G * mb;
      const int nq = (int)(mb >> 4);
      uint8_t* st = ring + (size_t)s * x.gu_stage;
      uint8_t* az = st + (size_t)R * (bytes + zb);
      const float* zh = p.z + (size_t)c.h * p.T * p.n_pad;
      auto copies = [&]() {   // the description, and lane r < R: codes, lane 16 + r: scale/zero rows of row block r
        const uint64_t code0 =
            (uint64_t)__shfl_sync(0xFFFFFFFFu, rw, 0) | ((uint64_t)__shfl_sync(0xFFFFFFFFu, rw, 1) << 32);
        const uint32_t rbs = __shfl_sync(0xFFFFFFFFu, rw, 8), meta0 = __shfl_sync(0xFFFFFFFFu, rw, 18);
        if (lane < (int)(sizeof(CStage) / 4)) reinterpret_cast<uint32_t*>(&f.rec)[lane] = rw;
        const int nrb = min(R, p.NRB - c.rg * R);
        if (lane == 0) {
          f.flags = (c.first ? 1 : 0) | (c.i + KH >= c.i1 ? 2 : 0);
          f.h = c.h;
          f.rg = c.rg;
          f.ntk = ntk;
          f.run = run & 1;
          mbar_expect_tx(&full[gr][s], (uint32_t)nrb * (bytes + zb));
        }
        __syncwarp();
        const int r = lane & 15, rb = c.rg * R + r;
        if (r < nrb && bytes) {
          fence_proxy_async();   // the stage was last read by the generic proxy
          if (lane < 16) bulk_g2s(st + (size_t)r * bytes, p.img + code0 + (uint64_t)rb * rbs, bytes, &full[gr][s]);
          else bulk_g2s(st + (size_t)R * bytes + (size_t)r * zb, x.meta + meta0 + (size_t)rb * (2u + G) * mb + 2u * mb, zb,
                        &full[gr][s]);
        }
      };
      if (i == 0) {   // the first stage's copies before the wait for the projection
        if (sub == 0) copies();
        pdl_wait();   // z and max |z|
      }
      if (c.first) {
        tok = pr / p.k;
        bs = scale_pow2<kGuLo>(__ldg(x.msa + c.h * p.E + tb.e[c.a]) * __uint_as_float(__ldcg(p.zmax + c.h * p.T + tok)));
      }
      float4 v[kRB];
      auto gather = [&](int r, const int4& u, bool live) {   // rows r .. r + kRB - 1 of one slot quad
#pragma unroll
        for (int w = 0; w < kRB; ++w) {
          const float* z = zh + (size_t)__shfl_sync(0xFFFFFFFFu, tok, max(0, min(r + w, r1 - 1))) * p.n_pad;
          if (live && r + w < r1) v[w] = make_float4(z[u.x], z[u.y], z[u.z], z[u.w]);
        }
      };
      auto put = [&](int r, int q, const float4& al) {
#pragma unroll
        for (int w = 0; w < kRB; ++w) {
          const float b = __shfl_sync(0xFFFFFFFFu, bs, max(0, min(r + w, r1 - 1)));
          if (q < nq && r + w < r1)
            *reinterpret_cast<float4*>(az + (size_t)q * kQS + (r + w) * 16) =
                make_float4(al.x * v[w].x * b, al.y * v[w].y * b, al.z * v[w].z * b, al.w * v[w].w * b);
        }
      };
      gather(r0, uc, lane < nq);
      units(rwn, lane, un, an);   // of the next stage
      GCur n2 = n;
      if (n.pos < hi) advance(n2);
      const uint32_t rwn2 = record(n2);
      const int prn2 = n2.pos < hi && n2.first ? pair_of(n2) : prn;
      if (i >= 2) ok &= mbar_wait(&empty[gr][s], (uint32_t)((i >> 1) - 1) & 1u, x.spin);
      if (!__all_sync(0xFFFFFFFFu, ok)) break;
      if (i > 0 && sub == 0) copies();
      if (c.first && sub == 0 && lane < 16) {
        runs[gr][run & 1].pair[lane] = pr;
        runs[gr][run & 1].inv[lane] = 1.f / bs;
      }
      put(r0, lane, ac);
      for (int r = r0 + kRB; r < r1; r += kRB) {
        gather(r, uc, lane < nq);
        put(r, lane, ac);
      }
      for (int q = 32; q < nq; q += 32) {   // more than 128 slots
        int4 u;
        float4 al;
        units(rw, q + lane, u, al);
        for (int r = r0; r < r1; r += kRB) {
          gather(r, u, q + lane < nq);
          put(r, q + lane, al);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[gr][s]);
      run += c.i + KH >= c.i1;
      c = n;
      n = n2;
      rw = rwn;
      rwn = rwn2;
      pr = prn;
      prn = prn2;
      uc = un;
      ac = an;
    }
    // No block leaves with copies in flight, whichever wait ran out: those of the last stage, and after a wait that
    // ran out here those of the stage before it (otherwise it was consumed, and its slot holds the end mark).
    if (sub == 0)
      for (int j = max(0, __all_sync(0xFFFFFFFFu, ok) ? i - 1 : i - 2); j < i; ++j)
        mbar_wait(&full[gr][j & 1], (uint32_t)(j >> 1) & 1u);
  } else {
    // ---- consumers
    pdl_wait();   // gate/up are cleared by the projection
    const int gr = wid / R, wr = wid - gr * R, g = lane >> 2, t = lane & 3;
    if (gr < KH) {
      const uint8_t* ring = msm + (size_t)gr * 2 * x.gu_stage;
      float acc[8][NTM][4];
      float cs[G][NTM];
      for (int i = 0;; ++i) {
        const int s = i & 1;
        ok &= mbar_wait(&full[gr][s], (uint32_t)(i >> 1) & 1u, x.spin);
        if (!__all_sync(0xFFFFFFFFu, ok)) break;   // a wait ran out: nothing of the stage can be used
        const GInfo& f = infos[gr][s];
        const int flags = f.flags;
        if (flags & 4) break;
        if (flags & 1) {
#pragma unroll
          for (int q = 0; q < NTM; ++q) {
#pragma unroll
            for (int m = 0; m < 8; ++m)
#pragma unroll
              for (int w = 0; w < 4; ++w) acc[m][q][w] = 0.f;
#pragma unroll
            for (int gl = 0; gl < G; ++gl) cs[gl][q] = 0.f;
          }
        }
        const int rb = f.rg * R + wr, ntk = f.ntk;
        if (rb < p.NRB) {
          const uint32_t bytes = f.rec.bytes, zb = G * f.rec.mb;
          const uint8_t* st = ring + (size_t)s * x.gu_stage;
          const uint32_t* sz = reinterpret_cast<const uint32_t*>(st + (size_t)R * bytes + (size_t)wr * zb);
          const uint8_t* az = st + (size_t)R * (bytes + zb) + g * 16;
          if (NTM == 1 || ntk <= 8) gu_segment<1, NTM, G>(f.rec, st + (size_t)wr * bytes, sz, az, lane, acc, cs);
          else gu_segment<NTM, NTM, G>(f.rec, st + (size_t)wr * bytes, sz, az, lane, acc, cs);
          if (flags & 2) {   // the part's end: its partial rows into gate/up
            const GRun& rr = runs[gr][f.run];
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
                const float iv = rr.inv[8 * q + col], f24 = 2097152.f * iv;   // 2^(24 - 3 - S)
                float cc[G];
#pragma unroll
                for (int gl = 0; gl < G; ++gl) cc[gl] = __shfl_sync(0xFFFFFFFFu, co[gl], 4 * col) * iv;
                if (8 * q + col < ntk) {
                  float* gp = p.gu + ((size_t)rr.pair[8 * q + col] * 2 + f.h) * p.I_pad + rb * kRows + 4 * g;
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
        }
        __syncwarp();
        if (lane == 0 && !(i == 0 && (x.lose & 1) && blockIdx.x == 0)) mbar_arrive(&empty[gr][s]);
      }
    }
  }
  if (!ok && lane == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
}

// ---------------------------------------------------------------------------
// Down
// ---------------------------------------------------------------------------
// Unit-lane tiles (32 units): an item = (token tile, run of row blocks, unit tile); a segment = the items of
// one (token tile, run).  A block takes consecutive items and its consumer warps every kCW-th of them,
// whatever their segment; they stream their tiles' codes in pieces of at most kStagePiece bytes through their
// own rings of three stages (with two, a piece's copy took longer than the work on the other: 254 us at
// 1024 tokens with the tensor pipe 34% busy).  Four helper warps form h = SiLU(gate) up of each segment, as B fragments in one of
// two shared-memory slots, while the consumers work on the segment before (formed by all warps between two
// block barriers, h took 3.6 us of latency a segment, and a block whose 12 items lay in two segments ran twice
// as long: the 8-token call's blocks ended between 44 and 55 us).
struct DCur {
  int p;                 // flat item (>= hi: the end)
  int pos, end;          // its segment: items [pos, end) of the block's range
  int ord;               // the segment's number in the block
  int a, tt, rc;         // expert index, token tile, run of row blocks
  int tile0;             // unit tile of item `pos`
  int rb;                // row block of the run
  int ms;                // the tile's metadata slot
};

// The packed words of four K-steps (64 rows, half hf of a row block) of one unit (its 16-byte chunks at
// `ln`, 512 bytes apart) that this lane needs, and from them the A registers of K-step 4 hf + k.
template <int B>
struct UlWords {
  uint32_t w[4];   // word of K-step k
  uint32_t h[4];   // 3 and 6 bits: its high-plane word
};
template <int B>
__device__ __forceinline__ void ul_load(const uint8_t* ln, int hf, int t, UlWords<B>& u) {
  auto word = [&](int chunk, int w) { return *reinterpret_cast<const uint32_t*>(ln + chunk * kChunkBytes + 4 * w); };
  if (B == 1) {          // a word = 32 rows: two K-steps
    const uint2 v = *reinterpret_cast<const uint2*>(ln + 8 * hf);
    u.w[0] = u.w[1] = v.x;
    u.w[2] = u.w[3] = v.y;
  } else if (B == 2 || B == 3) {   // a word = a K-step
    const uint4 v = *reinterpret_cast<const uint4*>(ln + hf * kChunkBytes);
    u.w[0] = v.x;
    u.w[1] = v.y;
    u.w[2] = v.z;
    u.w[3] = v.w;
    if (B == 3) {
      const uint2 x = *reinterpret_cast<const uint2*>(ln + 2 * kChunkBytes + 8 * hf);
      u.h[0] = u.h[1] = x.x;
      u.h[2] = u.h[3] = x.y;
    }
  } else if (B == 4 || B == 6) {   // a word = 8 rows: lanes t < 2 the first of a K-step's two words
#pragma unroll
    for (int k = 0; k < 4; ++k) u.w[k] = word(2 * hf + (k >> 1), 2 * (k & 1) + (t >> 1));
    if (B == 6) {
      const uint4 x = *reinterpret_cast<const uint4*>(ln + (4 + hf) * kChunkBytes);
      u.h[0] = x.x;
      u.h[1] = x.y;
      u.h[2] = x.z;
      u.h[3] = x.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) u.w[k] = word(4 * hf + k, t);
  }
}
template <int B>
__device__ __forceinline__ void ul_a(const UlWords<B>& u, int k, int t, uint32_t& lo, uint32_t& hi) {
  const int sh = B == 1 ? t + 4 * (k & 1) : B == 2 || B == 3 ? 2 * t : B == 8 ? 0 : 4 * (t & 1);
  const uint32_t mul = 1u << (code_pos<B>() - sh);
  if (B == 3) a_regs2<2, 1>(u.w[k], sh, mul, u.h[k], t + 4 * (k & 1), lo, hi);
  else if (B == 6) a_regs2<4, 2>(u.w[k], sh, mul, u.h[k], 2 * t, lo, hi);
  else a_regs<B>(u.w[k], sh, mul, lo, hi);
}

// One row block of a tile: out += scale (P 2^(24 - S) - zero sum(h)) / 2^12 per group.  The hi and lo products of a
// K-step go into the same accumulators, all hi ones first (apart, they took 16 registers more and spilled: 283 us
// at 1024 tokens against 272; 258 with nothing spilled).
template <int B, int NT, int NTM, int G>
__device__ __forceinline__ void dn_rb(const uint8_t* code, const uint4* hf, int hstride, const float4* hz, int zstride,
                                      const uint32_t* sz, int lane, float (&out)[2][NTM][4]) {
  constexpr float fP = 1.f / (float)(1 << code_pos<B>());   // the codes' position
  constexpr int KS = 8 / G;                                  // K-steps of a group
  const int g = lane >> 2, t = lane & 3;
  float P[2][NT][4];
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    UlWords<B> w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ul_load<B>(code + 16 * (g + 8 * u), half, t, w[u]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int ks = 4 * half + k, gl = ks / KS;
      if (ks % KS == 0) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int q = 0; q < 4; ++q) P[m][n][q] = 0.f;
      }
      uint32_t lo[4], hi[4], bl[NT][2];
#pragma unroll
      for (int u = 0; u < 4; ++u) ul_a<B>(w[u], k, t, lo[u], hi[u]);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const uint4 b = hf[n * hstride + ks * 32 + lane];
        bl[n][0] = b.z;
        bl[n][1] = b.w;
        mma_16816(P[0][n], lo[0], lo[1], hi[0], hi[1], b.x, b.y);
        mma_16816(P[1][n], lo[2], lo[3], hi[2], hi[3], b.x, b.y);
      }
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        mma_16816(P[0][n], lo[0], lo[1], hi[0], hi[1], bl[n][0], bl[n][1]);
        mma_16816(P[1][n], lo[2], lo[3], hi[2], hi[3], bl[n][0], bl[n][1]);
      }
      if (ks % KS == KS - 1) {
        float sc[4], zp[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t v = sz[gl * 32 + g + 8 * u];
          sc[u] = f16lo(v);
          zp[u] = f16hi(v);
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          float4 z = hz[gl * zstride + n * 4 + t];   // tokens 2 t and 2 t + 1: (sum, 2^(24 - S)) / 2^12 each
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

constexpr int kDnStages = 3;   // most stages of a consumer's ring

// Rows of a segment's token tile.
struct DRow {
  int off;      // token * n_pad
  float pw;     // gate weight times 2^12
};

// Shared-memory plan of k_dn_mma.
struct DPlan {
  uint32_t ring, meta, hf, hz, rows, tabs, total;
  uint32_t hfs, hzs;   // bytes of an h slot: fragments, sums
};
__host__ __device__ inline DPlan d_plan(int ntm, int G, const MArgs& x) {
  DPlan s;
  uint32_t o = 0;
  s.ring = o;
  o += (uint32_t)(kCW * x.dn_st) * kStagePiece;
  s.meta = o;
  o += (uint32_t)(kCW * x.dn_st) * x.dn_meta;
  s.hfs = (uint32_t)ntm * x.dn_rc * 8u * 32u * 16u;
  s.hf = o;
  o += 2u * s.hfs;
  s.hzs = (uint32_t)x.dn_rc * G * ntm * 8u * 8u;
  s.hz = o;
  o += 2u * s.hzs;
  s.rows = o;
  o += 2u * 16u * (uint32_t)sizeof(DRow);
  s.tabs = o;
  o += mtiles_bytes(x.A_max);
  s.total = (o + 15u) & ~15u;
  return s;
}

// Registers of the down kernel's consumer and helper warps: 3 x 128 x 144 + 128 x 80 = 65536, what the block is launched
// with (512 x 128).
__device__ __forceinline__ void regs_consumer() { asm volatile("setmaxnreg.inc.sync.aligned.u32 144;"); }
__device__ __forceinline__ void regs_helper() { asm volatile("setmaxnreg.dec.sync.aligned.u32 80;"); }

template <int NTM, int G>
__global__ void __launch_bounds__(kMmThreads, 1) k_dn_mma(Fwd p, MArgs x) {
  constexpr int kNT = 8 * NTM;
  extern __shared__ __align__(128) uint8_t msm[];
  __shared__ uint64_t bars[kCW][kDnStages], hfull[2], hempty[2];
  __shared__ int tbits[kCW][kDnStages];
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  const DPlan L = d_plan(NTM, G, x);
  MTiles tb = mtiles_at(msm + L.tabs, x.A_max);
  const int RC = x.dn_rc, nrc = (p.NRB + RC - 1) / RC;
  const ExpertDesc* dd = p.desc + 2 * p.E;

  pdl_trigger();
  if (tid == 0) {
    for (int w = 0; w < kCW; ++w)
      for (int s = 0; s < kDnStages; ++s) mbar_init_n(&bars[w][s], 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init_n(&hfull[s], kHW);
      mbar_init_n(&hempty[s], kCW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_ok = wait_flag(p.route_flag);
  }
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
    pdl_wait();
    return;
  }
  mtiles_build(p, x.A_max, x.lose, kNT, tb, [&](int e) { return nrc * __ldg(&dd[e].ntiles); });
  const int lo = cut_unit(tb, kNT, (int)blockIdx.x, (int)gridDim.x);
  const int hi = cut_unit(tb, kNT, (int)blockIdx.x + 1, (int)gridDim.x);
  bool ok = true;

  // the segment that starts at item c.pos (< hi)
  auto seg_at = [&](DCur& c) {
    c.a = find_le(tb.ub, tb.na, c.pos);   // the last expert that starts at or before: one with items
    const int nt = (tb.ub[c.a + 1] - tb.ub[c.a]) / (((tb.cnt[c.a] + kNT - 1) / kNT) * nrc);
    const int q = c.pos - tb.ub[c.a], tr = q / nt;
    c.tile0 = q - tr * nt;
    c.tt = tr / nrc;
    c.rc = tr - c.tt * nrc;
    c.end = min(hi, c.pos + nt - c.tile0);
  };
  auto run_nrb = [&](const DCur& c) { return min(RC, p.NRB - c.rc * RC); };

  if (wid >= kCW) {
    // ---- helpers: h of one segment after the other
    regs_helper();
    pdl_wait();   // gate/up come from the previous kernel
    const int hw = wid - kCW;
    DCur c;
    c.pos = lo;
    for (int k = 0; c.pos < hi; ++k, c.pos = c.end) {
      seg_at(c);
      const int s = k & 1, nrb = run_nrb(c), ntk = min(kNT, tb.cnt[c.a] - c.tt * kNT), rb0 = c.rc * RC;
      const int pr = p.pair_list[tb.pst[c.a] + c.tt * kNT + min(lane & 15, ntk - 1)];
      const float pw = hw == 0 ? p.pair_weight[pr] : 0.f;
      if (k >= 2) ok &= mbar_wait(&hempty[s], (uint32_t)((k >> 1) - 1) & 1u, x.spin);
      if (!__all_sync(0xFFFFFFFFu, ok)) break;
      uint4* hf = reinterpret_cast<uint4*>(msm + L.hf + s * L.hfs);     // [NTM][RC][8 K-steps][32 lanes]
      float2* hz = reinterpret_cast<float2*>(msm + L.hz + s * L.hzs);   // [RC][G][kNT] (sum of h, 2^(24 - S)) / 2^12
      if (hw == 0 && lane < 16) {
        DRow r;
        r.off = pr / p.k * p.n_pad;
        r.pw = pw * kDnPart;
        reinterpret_cast<DRow*>(msm + L.rows)[s * 16 + lane] = r;
      }
      // a warp per (token, row block), 4 rows a lane; four at a time (rows past the tile's tokens are left
      // as they are: their columns of the products are not read)
      constexpr int kB = 4;
      for (int w0 = hw; w0 < ntk * nrb; w0 += kB * kHW) {
        float4 gv[kB], uv[kB];
#pragma unroll
        for (int q = 0; q < kB; ++q) {
          const int w = min(w0 + q * kHW, ntk * nrb - 1), tk = w / nrb, rb = w - tk * nrb;
          const float* gp = p.gu + (size_t)__shfl_sync(0xFFFFFFFFu, pr, tk) * 2 * p.I_pad + (rb0 + rb) * kRows + 4 * lane;
          gv[q] = __ldcg(reinterpret_cast<const float4*>(gp));
          uv[q] = __ldcg(reinterpret_cast<const float4*>(gp + p.I_pad));
        }
#pragma unroll
        for (int q = 0; q < kB; ++q) {
          const int w = w0 + q * kHW;
          if (w >= ntk * nrb) break;
          const int tk = w / nrb, rb = w - tk * nrb;
          float4 h4;
          h4.x = gv[q].x / (1.f + __expf(-gv[q].x)) * uv[q].x;
          h4.y = gv[q].y / (1.f + __expf(-gv[q].y)) * uv[q].y;
          h4.z = gv[q].z / (1.f + __expf(-gv[q].z)) * uv[q].z;
          h4.w = gv[q].w / (1.f + __expf(-gv[q].w)) * uv[q].w;
          const float am = warp_max(fmaxf(fmaxf(fabsf(h4.x), fabsf(h4.y)), fmaxf(fabsf(h4.z), fabsf(h4.w))));
          float sum = (h4.x + h4.y) + (h4.z + h4.w);
#pragma unroll
          for (int o = 16 / G; o; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
          const float sc = scale_pow2<kDnLo>(am);
          uint4 v;
          split_pair(h4.x * sc, h4.z * sc, v.x, v.z);
          split_pair(h4.y * sc, h4.w * sc, v.y, v.w);
          hf[((size_t)(tk >> 3) * RC + rb) * 256 + (lane >> 2) * 32 + (tk & 7) * 4 + (lane & 3)] = v;
          if ((lane & (32 / G - 1)) == 0)
            hz[((size_t)rb * G + lane / (32 / G)) * kNT + tk] = make_float2(sum / kDnPart, (16777216.f / kDnPart) / sc);
        }
      }
      __syncwarp();
      if (lane == 0 && !(k == 0 && (x.lose & 1) && blockIdx.x == 0)) mbar_arrive(&hfull[s]);
    }
  } else {
    // ---- consumers
    regs_consumer();
    const int S = x.dn_st;
    uint8_t* ring = msm + L.ring + (size_t)wid * S * kStagePiece;
    uint8_t* meta = msm + L.meta + (size_t)wid * S * x.dn_meta;
    auto piece_len = [&](int bits, int left) { return min(left, bits <= 1 ? 8 : bits <= 2 ? 4 : bits <= 4 ? 2 : 1); };
    auto walk = [&](DCur& c) {   // to the segment of item c.p (the block's end: past its last segment)
      while (c.pos < hi && c.p >= c.end) {
        c.pos = c.end;
        ++c.ord;
        if (c.pos < hi) seg_at(c);
      }
    };
    // word `lane` of the unit tile's staging record
    auto record = [&](const DCur& c) -> uint32_t {
      if (c.p >= hi || lane >= (int)(sizeof(DStage) / 4)) return 0u;
      return __ldg(reinterpret_cast<const uint32_t*>(x.dst + (size_t)tb.e[c.a] * p.ul_max_tiles + c.tile0 + c.p - c.pos) +
                   lane);
    };
    auto advance = [&](DCur& c, int nrb) {   // past a piece of nrb row blocks; true: to another tile
      c.rb += nrb;
      if (c.rb < run_nrb(c)) return false;
      c.rb = 0;
      c.p += kCW;
      if (++c.ms == S) c.ms = 0;
      walk(c);
      return true;
    };

    DCur n;   // the piece to be staged next, S - 1 ahead of the one consumed
    n.p = lo + wid;
    n.pos = lo;
    n.ord = n.ms = n.rb = 0;
    if (lo < hi) seg_at(n);
    walk(n);
    DCur c = n;
    uint32_t rn = record(n);
    int ps = 0;   // its stage
    auto issue = [&]() {
      if (n.p >= hi) return;
      const uint64_t code = (uint64_t)__shfl_sync(0xFFFFFFFFu, rn, 0) | ((uint64_t)__shfl_sync(0xFFFFFFFFu, rn, 1) << 32);
      const uint32_t bits = __shfl_sync(0xFFFFFFFFu, rn, 9), mt = __shfl_sync(0xFFFFFFFFu, rn, 10);
      const int nrb = piece_len((int)bits, run_nrb(n) - n.rb);
      if (lane == 0) {
        uint64_t* bar = &bars[wid][ps];
        const uint32_t bytes = (uint32_t)nrb * bits * kChunkBytes;
        fence_proxy_async();   // the stage was last read by the generic proxy
        if (n.rb == 0) {   // the tile's units, alphas and its scale/zero rows of this run
          const int g0 = n.rc * RC * kRows / p.group;
          const int g1 = min(p.NG, ((n.rc * RC + run_nrb(n)) * kRows + p.group - 1) / p.group);
          const uint32_t szb = (uint32_t)(g1 - g0) * 128u;
          mbar_expect_tx(bar, bytes + 256u + szb);
          uint8_t* md = meta + (size_t)n.ms * x.dn_meta;
          tbits[wid][n.ms] = (int)bits;
          bulk_g2s(md, x.meta + mt, 256u, bar);
          bulk_g2s(md + 256, x.meta + mt + 256u + (uint32_t)g0 * 128u, szb, bar);
        } else {
          mbar_expect_tx(bar, bytes);
        }
        bulk_g2s(ring + (size_t)ps * kStagePiece, p.img + code + (uint64_t)(n.rc * RC + n.rb) * bits * kChunkBytes, bytes,
                 bar);
      }
      if (++ps == S) ps = 0;
      if (advance(n, nrb)) rn = record(n);
    };
    for (int k = 0; k < S - 1; ++k) issue();
    pdl_wait();   // s is cleared, and h's inputs are written, by earlier kernels
    int held = -1;   // the segment whose h the warp holds
    auto hold = [&](int ord) {
      while (held < ord) {
        if (held >= 0) {
          __syncwarp();
          if (lane == 0) mbar_arrive(&hempty[held & 1]);
        }
        ++held;
        ok &= mbar_wait(&hfull[held & 1], (uint32_t)(held >> 1) & 1u, x.spin);
        if (!__all_sync(0xFFFFFFFFu, ok)) return;
      }
    };
    int cs = 0;
    uint32_t cph = 0;   // stage and phase of the piece being consumed
    while (c.p < hi) {   // a unit tile
      hold(c.ord);
      bool live = __all_sync(0xFFFFFFFFu, ok);   // a wait that ran out ends the warp's work
      if (!live) break;
      const int hs = held & 1, nrb = run_nrb(c), ntk = min(kNT, tb.cnt[c.a] - c.tt * kNT);
      const uint4* hf = reinterpret_cast<const uint4*>(msm + L.hf + hs * L.hfs);
      const float4* hz4 = reinterpret_cast<const float4*>(msm + L.hz + hs * L.hzs);
      float out[2][NTM][4];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int q = 0; q < NTM; ++q)
#pragma unroll
          for (int w = 0; w < 4; ++w) out[m][q][w] = 0.f;
      const uint8_t* md = meta + (size_t)c.ms * x.dn_meta;
      int bits = 0;
      for (int rb = 0; rb < nrb;) {
        __syncwarp();   // the stage before has been read by every lane
        issue();
        ok &= mbar_wait(&bars[wid][cs], cph, x.spin);
        live = __all_sync(0xFFFFFFFFu, ok);
        if (!live) break;
        if (rb == 0) bits = tbits[wid][c.ms];
        const int np = piece_len(bits, nrb - rb);
        const uint8_t* code = ring + (size_t)cs * kStagePiece;
        const uint32_t* szp = reinterpret_cast<const uint32_t*>(md + 256);
        if (NTM == 1 || ntk <= 8)
          dn_piece<1, NTM, G>(bits, np, code, hf, RC * 256, hz4, kNT / 2, szp, rb, p.group, lane, out);
        else
          dn_piece<NTM, NTM, G>(bits, np, code, hf, RC * 256, hz4, kNT / 2, szp, rb, p.group, lane, out);
        rb += np;
        if (++cs == S) {
          cs = 0;
          cph ^= 1u;
        }
      }
      if (!live) {   // the piece waited for is in flight too
        mbar_wait(&bars[wid][cs], cph);
        if (++cs == S) {
          cs = 0;
          cph ^= 1u;
        }
        break;
      }
      // s += g alpha out
      const int* un = reinterpret_cast<const int*>(md);
      const float* al = reinterpret_cast<const float*>(md + 128);
      const DRow* rows = reinterpret_cast<const DRow*>(msm + L.rows) + hs * 16;
#pragma unroll
      for (int q = 0; q < NTM; ++q) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int tk = 8 * q + 2 * t + u;
          if (tk >= ntk) continue;
          const DRow r = rows[tk];
          float* sp = p.s + r.off;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float a = al[g + 8 * v];
            if (a != 0.f) atomicAdd(sp + un[g + 8 * v], r.pw * a * out[v >> 1][q][u + 2 * (v & 1)]);
          }
        }
      }
      __syncwarp();   // the tile's metadata slot may be refilled
      advance(c, nrb);
    }
    // No block leaves with copies in flight: after a wait that ran out, the pieces requested and not waited for
    // (fewer than S).
    while (cs != ps) {
      mbar_wait(&bars[wid][cs], cph);
      if (++cs == S) {
        cs = 0;
        cph ^= 1u;
      }
    }
    // the segments that are left (the cursor has walked to the block's end: ord = their number)
    if (__all_sync(0xFFFFFFFFu, ok) && c.ord > 0) hold(c.ord - 1);
  }
  if (!ok && lane == 0) atomicCAS(p.status, 0, BITSMOE_ERR_TIMEOUT);
}

}  // namespace

namespace bmoe {

// Largest staged segment of a gate/up group of R row blocks: codes and G scale/zero rows of each, and the
// operand of ntm groups of 8 tokens.
uint32_t mma_gu_stage(const std::vector<CStage>& cst, int G, int ntm, int R) {
  uint32_t m = 0;
  for (const CStage& r : cst)
    if (r.bytes)
      m = std::max(m, (uint32_t)R * (r.bytes + (uint32_t)G * r.mb) +
                          (r.mb / 16u) * (uint32_t)(ntm == 1 ? az_quad<1>() : az_quad<2>()));
  return (m + 127u) & ~127u;
}

constexpr uint32_t kMaxSmem = 224u * 1024u;   // dynamic shared memory of a block (static parts beside it)

static uint32_t gu_smem(const MArgs& x) { return (uint32_t)x.gu_kh * 2u * x.gu_stage + mtiles_bytes(x.A_max); }

// The split of the consumer warps into KH groups of R row blocks: the fewest idle warps among the splits
// whose rings fit (the larger R where equal: its warps share the gathered operand).
static bool gu_split(int NRB, const uint32_t* stages, MArgs* x) {
  double bu = 0;
  for (int R = std::min(NRB, kCW); R >= 1; --R) {
    MArgs c = *x;
    c.gu_r = R;
    c.gu_kh = std::min(kMaxKH, kCW / R);
    c.gu_stage = stages[R];
    while (c.gu_kh > 1 && gu_smem(c) > kMaxSmem) --c.gu_kh;
    if (!c.gu_stage || gu_smem(c) > kMaxSmem) continue;
    const double u = (double)NRB / ((NRB + R - 1) / R * R) * (R * c.gu_kh) / kCW;
    if (u > bu + 1e-9) {
      bu = u;
      *x = c;
    }
  }
  return bu > 0;
}

bool mma_args(const ImageHeader& hd, int T, int k, const uint32_t (&stages)[2][kCW + 1], MArgs* x) {
  std::memset(x, 0, sizeof(*x));
  const int G = std::max(1, kRows / hd.group);
  x->ntm = T <= 16 ? 1 : 2;
  x->A_max = std::min(hd.E, T * k);
  if (!gu_split(hd.NRB, stages[x->ntm - 1], x)) return false;
  x->seg_stride = std::max(1, (int)(0.382 * hd.nseg + 0.5));
  while (std::gcd(x->seg_stride, hd.nseg) != 1) ++x->seg_stride;
  // A down run: whole groups; at most 4 row blocks, so that the two h slots leave room for three stages a
  // consumer and that a block's 12 consumers have several items each (one of 13 items of a whole expert's rows,
  // 8 us each, doubled the 8-token call's time); up to 8 past 256 tokens, where the additions into s, one
  // sector each, weigh more (1024 tokens: 334 us with runs of 3, 262 us with 6).  Whole calls on both sides of the
  // lines, us with 3 and 2 runs of at most 4 row blocks and with one run of up to 8 (Qwen3-shaped layer, uneven
  // experts, 6 row blocks): 9 tokens 68 / 70 / 71, 16 77 / 80 / 83, 17 85 / 87 / 92, 48 115 / 118 / 129, 192
  // 226 / 222 / 228, 256 281 / 275 / 275, 257 289 / 283 / 280, 400 396 / 392 / 375, 1024 879 / 875 / 808; even
  // experts, 64 tokens 158 / 154 / 156, 256 271 / 265 / 263, 512 441 / 431 / 412.
  const int need = std::max(1, hd.group / kRows), most = T > 256 ? 8 : 4;
  const int runs = std::max((hd.NRB + most - 1) / most, T <= 16 ? 3 : T <= 256 ? 2 : 1), rows = (hd.NRB + runs - 1) / runs;
  const int rc0 = std::max(need, (rows + need - 1) / need * need);
  for (int pass = 0; pass < 2; ++pass)
    for (x->dn_rc = rc0; x->dn_rc >= need; x->dn_rc -= need) {
      x->dn_meta = 256u + 128u * (uint32_t)(x->dn_rc * kRows / hd.group);
      for (x->dn_st = kDnStages; x->dn_st >= (pass || T > 256 ? 2 : 3); --x->dn_st)
        if (d_plan(x->ntm, G, *x).total <= kMaxSmem) return true;
    }
  return false;
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
  static uint32_t done[2] = {0, 0};
  if (down) return mm_launch(k_dn_mma<NTM, G>, sms, kMmThreads, d_plan(NTM, G, x).total, p, x, st, pdl, &done[0]);
  return mm_launch(k_gu_mma<NTM, G>, sms, kMmThreads, gu_smem(x), p, x, st, pdl, &done[1]);
}

cudaError_t launch_expert_mma(bool down, const Fwd& p, const MArgs& x, int sms, cudaStream_t st, bool pdl) {
  const int G = std::max(1, kRows / p.group);
  if (x.ntm == 2)
    return G == 1 ? mm_pair<2, 1>(down, p, x, sms, st, pdl)
                  : G == 2 ? mm_pair<2, 2>(down, p, x, sms, st, pdl) : mm_pair<2, 4>(down, p, x, sms, st, pdl);
  return G == 1 ? mm_pair<1, 1>(down, p, x, sms, st, pdl)
                : G == 2 ? mm_pair<1, 2>(down, p, x, sms, st, pdl) : mm_pair<1, 4>(down, p, x, sms, st, pdl);
}

}  // namespace bmoe
