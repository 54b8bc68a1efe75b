// Per-projection bit allocation: which bit-width every spectral unit gets.
//
// BitsMoE chooses b_u in {0,1,2,3,4,6,8,16} for the units of one projection
// type by the ILP of Eq. ilp_piecewise_eps: minimise sum_u C_u(b_u) subject to
// sum_u b_u <= B_h, with C_u(b) = alpha_u^2 beta_u^gamma E_u(b) (Eq.
// app_component_loss_final) and the piecewise distortion of Eq.
// piecewise_expected_eps (eta 2^(-2b) for b >= 6 with eta = d rho^2 / 3,
// kappa_b for 2..4, sin^2 theta = 1 - ||p||_1^2 / d for 1 bit, 1 for 0 bits).
// The paper hands the ILP to a commercial solver; here it is solved by the
// Lagrangian relaxation of the multiple-choice knapsack plus a greedy fill:
//
//   k_alloc_cost   one warp per 32 units, eight rows streamed side by side:
//                  rho = max |p| and ||p||_1 (an exact fixed-point sum, so the
//                  order of the lanes does not matter)
//                  per unit, then each lane builds its unit's costs and the
//                  lower convex hull of (b, C(b)) from b = 0 (ties to the
//                  smaller b, efficiencies capped so they never increase); an
//                  increment's key is (bits of its efficiency) << 32 | ~u
//   radix select   four passes over the 16-bit digits of the keys: a histogram
//                  of the increments' bit counts by digit, then the digit where
//                  the bits taken so far would pass B_h (k_alloc_scan); after the
//                  last pass the cut K* is the key of the first increment group
//                  that does not fit.  The cost kernel counts the first digit
//                  itself; k_alloc_compact collects the keys of the cut digit's
//                  bucket (and counts their second digit), so that the last two
//                  passes (k_alloc_hist) see a short list, or all keys again
//                  where the bucket is larger than the list
//   k_alloc_final  every unit takes its increments with key > K* (the
//                  Lagrangian solution) and exposes its next one; per block and
//                  bit count the largest exposed key
//   k_fill         while a next increment fits the bits left, the one with the
//                  largest key is taken (one block, from the per-block maxima;
//                  only the block of the unit taken is looked through again)
//
// Everything is fp32 with each operation rounded once, in the same steps as
// the allocation oracle, so the bit-widths are a deterministic function of
// the inputs.  The cost kernel streams the units once (HBM-bound); the rest
// works on 64 bytes per unit of workspace.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"

namespace {

constexpr int kAW = 8;                 // warps per block of the cost kernel
constexpr int kBW = 16;                // ... and of its bulk-copy form
constexpr int kNB = 8;                 // bit-width options
constexpr int kNS = 7;                 // at most 7 hull increments
constexpr int kDigits = 65536;
constexpr int kScanBlocks = 32;        // blocks of the digit scan, 2048 digits each
constexpr int kList = 65536;           // entries of the compacted bucket
constexpr int kFinalBlocks = 512;      // blocks of the final pass (rows of the fill's table)
constexpr int kMaxDb = 16;             // largest bit count of an increment
__constant__ int c_bits[kNB] = {0, 1, 2, 3, 4, 6, 8, 16};

struct AllocState {
  unsigned long long prefix;   // key bits decided by the radix passes
  unsigned long long above;    // bits of the increments above the current bucket (all taken)
  unsigned long long kstar;    // the cut: increments with key > kstar are taken (0: all)
  unsigned long long used;     // bits after the cut
  unsigned long long wtot[kScanBlocks];   // digit scan: bits of each block's digits
  int all_fit;                 // every increment fits: nothing to select
  unsigned int done;           // digit scan: blocks finished
  unsigned int nlist;          // keys of the first digit's cut bucket (the list holds them when <= kList)
};

struct AllocWs {
  AllocState* st;
  unsigned long long* hist;    // [2][kDigits]: a pass counts in one while its scan clears the other
  unsigned long long* keys;    // [kNS][U], 0 = none
  uint8_t* reach;              // [kNS][U] option index reached by each increment
  uint8_t* taken;              // [U]
  unsigned long long* nkey;    // [U] next increment's key (0 = none)
  uint8_t* ndb;                // [U] its bits
  unsigned long long* lkey;    // [kList] the cut bucket's keys
  uint8_t* ldb;                // [kList] their bits
  unsigned long long* best;    // [kFinalBlocks][kMaxDb + 1] largest next key of a block's units by its bits
  int64_t U;
};

constexpr int kParts = 10;
size_t ws_layout(int64_t U, size_t* off) {
  size_t o = 0;
  auto put = [&](int i, size_t bytes) {
    off[i] = o;
    o = (o + bytes + 255) / 256 * 256;
  };
  put(0, sizeof(AllocState));
  put(1, (size_t)2 * kDigits * 8);
  put(2, (size_t)U * kNS * 8);
  put(3, (size_t)U * kNS);
  put(4, (size_t)U);
  put(5, (size_t)U * 8);
  put(6, (size_t)U);
  put(7, (size_t)kList * 8);
  put(8, (size_t)kList);
  put(9, (size_t)kFinalBlocks * (kMaxDb + 1) * 8);
  return o;
}

__device__ __forceinline__ float weight(float a, float b, float gamma) {
  float bg;
  if (gamma == 0.f) bg = 1.f;
  else if (gamma == 0.5f) bg = __fsqrt_rn(b);
  else if (gamma == 1.f) bg = b;
  else bg = powf(b, gamma);
  return __fmul_rn(__fmul_rn(a, a), bg);
}

// Costs and hull of one unit (one lane): increment s at keys[32 s], reach[32 s].
__device__ void unit_hull(float rho, long long l1fix, int d, float w, float k2, float k3, float k4, uint32_t u,
                          unsigned long long* keys, uint8_t* reach) {
  const float l1 = __fmul_rn(__ll2float_rn(l1fix), 9.094947017729282e-13f);   // 2^-40
  const float sin2 = __fsub_rn(1.f, __fdiv_rn(__fmul_rn(l1, l1), (float)d));
  const float eta = __fdiv_rn(__fmul_rn(__fmul_rn(rho, rho), (float)d), 3.f);
  float C[kNB];
  C[0] = w;                                  // w * 1
  C[1] = __fmul_rn(w, sin2);
  C[2] = __fmul_rn(w, k2);
  C[3] = __fmul_rn(w, k3);
  C[4] = __fmul_rn(w, k4);
  C[5] = __fmul_rn(w, __fmul_rn(eta, 2.44140625e-4f));       // 2^-12
  C[6] = __fmul_rn(w, __fmul_rn(eta, 1.52587890625e-5f));    // 2^-16
  C[7] = __fmul_rn(w, __fmul_rn(eta, 2.3283064365386963e-10f));   // 2^-32
  int cur = 0;
  float curc = C[0], prev = __int_as_float(0x7F800000);
  const unsigned long long low = 0xFFFFFFFFull - u;
#pragma unroll 1
  for (int s = 0; s < kNS; ++s) {
    float be = 0.f;
    int bj = -1;
#pragma unroll
    for (int j = 1; j < kNB; ++j) {
      if (j > cur) {
        const float e = __fdiv_rn(__fsub_rn(curc, C[j]), (float)(c_bits[j] - c_bits[cur]));
        if (e > 0.f && e > be) {
          be = e;
          bj = j;
        }
      }
    }
    if (bj < 0) {
      for (int r = s; r < kNS; ++r) {
        keys[32 * r] = 0ull;
        reach[32 * r] = 0xFF;
      }
      return;
    }
    const float e = fminf(be, prev);
    keys[32 * s] = ((unsigned long long)__float_as_uint(e) << 32) | low;
    reach[32 * s] = (uint8_t)bj;
    curc = C[bj];
    cur = bj;
    prev = e;
  }
}

struct CostArgs {
  const float* p;
  const float* alpha;
  const float* beta;
  float gamma, k2, k3, k4;
  int64_t U;
  int d;
  AllocWs w;
  int lose;   // testing hook: the warps of block 0 take their second wait for a stage as run out
};

// floor(|x| 2^40) for |x| < 32 as A 2^22 + B with A = floor(y), B = floor(frac(y) 2^22),
// y = |x| 2^18 < 2^23: each is read off the bits of a round-toward-zero add of 2^23
// (2^23 + floor(v) for 0 <= v < 2^23).  The raw bit patterns are summed; the caller
// subtracts count * bits(2^23) (mod 2^32).  Also the running max |x|.
__device__ __forceinline__ void fix_add(float ax, float& mx, uint32_t& sa, uint32_t& sb) {
  mx = fmaxf(mx, ax);
  const float y = __fmul_rn(ax, 262144.f);                                          // 2^18
  const float ty = __fadd_rz(y, 8388608.f);                                         // 2^23 + floor(y)
  const float z = __fmul_rn(__fsub_rn(y, __fsub_rn(ty, 8388608.f)), 4194304.f);   // frac(y) 2^22
  sa += __float_as_uint(ty);
  sb += __float_as_uint(__fadd_rz(z, 8388608.f));
}

// Row k of the warp's 32: its max |p| and exact fixed-point sum over the lanes, kept by lane k (cnt: the
// elements a lane added).
__device__ __forceinline__ void row_sums(float mx, uint32_t sa, uint32_t sb, uint32_t cnt, int k, float& rho,
                                         long long& l1) {
  const uint32_t A = sa - cnt * 0x4B000000u, B = sb - cnt * 0x4B000000u;
  // 16-bit halves, so that the 32 lanes' sums fit; mx is never negative or NaN: its bits order as it does
  const unsigned a0 = __reduce_add_sync(0xFFFFFFFFu, A & 0xFFFFu), a1 = __reduce_add_sync(0xFFFFFFFFu, A >> 16);
  const unsigned b0 = __reduce_add_sync(0xFFFFFFFFu, B & 0xFFFFu), b1 = __reduce_add_sync(0xFFFFFFFFu, B >> 16);
  const unsigned m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx));
  if ((threadIdx.x & 31) == k) {
    rho = __uint_as_float(m);
    l1 = ((((long long)a1 << 16) + (long long)a0) << 22) + ((long long)b1 << 16) + (long long)b0;
  }
}

// Bits of the increments of a warp's lanes (take: the lane has one) added to their digits' counts: many share
// a digit (the leading digits hold the efficiency's exponent), so the lanes of a digit add up first.
__device__ __forceinline__ void count_digit(unsigned long long* hist, bool take, unsigned dgt, unsigned db, int lane) {
  const unsigned act = __ballot_sync(0xFFFFFFFFu, take);
  if (!take) return;
  const unsigned grp = __match_any_sync(act, dgt);
  const unsigned tot = __reduce_add_sync(grp, db);
  if (lane == __ffs(grp) - 1) atomicAdd(hist + dgt, (unsigned long long)tot);
}

// The hulls of a warp's 32 units (lane = unit), their rows of the workspace and the first digit's counts.
__device__ void warp_hulls(const CostArgs& a, int64_t base, int nu, float rho, long long l1, unsigned long long* sk,
                           uint8_t* sr) {
  const int lane = threadIdx.x & 31;
  if (lane < nu) {
    const int64_t u = base + lane;
    const float w = weight(__ldg(a.alpha + u), __ldg(a.beta + u), a.gamma);
    unit_hull(rho, l1, a.d, w, a.k2, a.k3, a.k4, (uint32_t)u, sk + lane, sr + lane);
  } else {
    for (int s = 0; s < kNS; ++s) {
      sk[32 * s + lane] = 0ull;
      sr[32 * s + lane] = 0xFF;
    }
  }
  __syncwarp();
  int pb = 0;
#pragma unroll 1
  for (int s = 0; s < kNS; ++s) {
    const unsigned long long key = sk[32 * s + lane];
    const uint8_t r = sr[32 * s + lane];
    if (lane < nu) {
      a.w.keys[(size_t)s * a.U + base + lane] = key;
      a.w.reach[(size_t)s * a.U + base + lane] = r;
    }
    const int b = key ? c_bits[r] : 0;
    count_digit(a.w.hist, key != 0ull, (unsigned)(key >> 48), (unsigned)(b - pb), lane);
    pb = b;
  }
  __syncwarp();
}

// One warp per 32 consecutive units; lane l keeps unit (base + l)'s rho and ||p||_1.  Rows of any length: the
// warp streams kUK units' rows side by side, so kUK 16-byte loads per lane are in flight at once.
constexpr int kUK = 8;
__global__ void __launch_bounds__(kAW * 32) k_alloc_cost(CostArgs a) {
  __shared__ unsigned long long sk[kAW][kNS * 32];
  __shared__ uint8_t sr[kAW][kNS * 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t nwarps = (int64_t)gridDim.x * kAW;
  const bool v4 = (a.d & 3) == 0;
  for (int64_t base = ((int64_t)blockIdx.x * kAW + (threadIdx.x >> 5)) * 32; base < a.U; base += nwarps * 32) {
    const int nu = a.U - base < 32 ? (int)(a.U - base) : 32;
    float my_rho = 0.f;
    long long my_l1 = 0;
    for (int k0 = 0; k0 < nu; k0 += kUK) {
      float mx[kUK];
      uint32_t sa[kUK], sb[kUK];
#pragma unroll
      for (int q = 0; q < kUK; ++q) {
        mx[q] = 0.f;
        sa[q] = sb[q] = 0u;
      }
      const float* rows[kUK];
#pragma unroll
      for (int q = 0; q < kUK; ++q) rows[q] = a.p + (size_t)(base + (k0 + q < nu ? k0 + q : 0)) * a.d;
      uint32_t cnt = 0;
      if (v4) {
        for (int i = lane; i < a.d / 4; i += 32) {
          float4 x[kUK];
#pragma unroll
          for (int q = 0; q < kUK; ++q) x[q] = __ldcs(reinterpret_cast<const float4*>(rows[q]) + i);
#pragma unroll
          for (int q = 0; q < kUK; ++q) {
            fix_add(fabsf(x[q].x), mx[q], sa[q], sb[q]);
            fix_add(fabsf(x[q].y), mx[q], sa[q], sb[q]);
            fix_add(fabsf(x[q].z), mx[q], sa[q], sb[q]);
            fix_add(fabsf(x[q].w), mx[q], sa[q], sb[q]);
          }
          cnt += 4;
        }
      } else {
        for (int i = lane; i < a.d; i += 32) {
          float x[kUK];
#pragma unroll
          for (int q = 0; q < kUK; ++q) x[q] = __ldcs(rows[q] + i);
#pragma unroll
          for (int q = 0; q < kUK; ++q) fix_add(fabsf(x[q]), mx[q], sa[q], sb[q]);
          cnt += 1;
        }
      }
#pragma unroll
      for (int q = 0; q < kUK; ++q) row_sums(mx[q], sa[q], sb[q], cnt, k0 + q, my_rho, my_l1);
    }
    warp_hulls(a, base, nu, my_rho, my_l1, sk[wid], sr[wid]);
  }
}

// The same for rows of whole 16-byte chunks up to kRowMax bytes: each warp takes a range of units, whose rows lie
// one after another, and streams them through its own two stages of `rows` rows by bulk copies, so that the
// next rows arrive while these are summed.  The warps' first hulls come after different numbers of units: with
// all of them at their hulls at once (several microseconds without a request) the stream stood still.
// HBM-bound: 262144 units of 768 floats, 805 MB: 196 us with the loads between the sums, 200 us by bulk copies
// with the hulls in step, 149 us so (5.4 TB/s, 0.81 of the copy bandwidth).
//
// A wait for a stage that runs out (its bound is about a second) costs speed, not results: the warp requests no more,
// reads the rows from that stage's on by ordinary loads, and before it leaves waits once more for the copies it
// still has in flight.
constexpr uint32_t kStageMax = 6144, kRowMax = kStageMax;

// Rows k0 .. k0 + r - 1 of a warp's units, the first at `rows` (rb bytes apart), two side by side.
__device__ __forceinline__ void rows_sums(const uint8_t* rows, uint32_t rb, int r, int d, int k0, float& rho, long long& l1) {
  const int lane = threadIdx.x & 31;
  for (int q0 = 0; q0 < r; q0 += 2) {
    float mx[2];
    uint32_t sa[2], sb[2], cnt = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      mx[q] = 0.f;
      sa[q] = sb[q] = 0u;
    }
#pragma unroll 2
    for (int i = lane; i < d / 4; i += 32) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float4 x = *reinterpret_cast<const float4*>(rows + (size_t)min(q0 + q, r - 1) * rb + 16 * i);
        fix_add(fabsf(x.x), mx[q], sa[q], sb[q]);
        fix_add(fabsf(x.y), mx[q], sa[q], sb[q]);
        fix_add(fabsf(x.z), mx[q], sa[q], sb[q]);
        fix_add(fabsf(x.w), mx[q], sa[q], sb[q]);
      }
      cnt += 4;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (q0 + q < r) row_sums(mx[q], sa[q], sb[q], cnt, k0 + q0 + q, rho, l1);
  }
}

__global__ void __launch_bounds__(kBW * 32) k_alloc_cost_bulk(CostArgs a, int rows) {
  extern __shared__ __align__(128) uint8_t ring_raw[];
  __shared__ unsigned long long sk[kBW][kNS * 32];
  __shared__ uint8_t sr[kBW][kNS * 32];
  __shared__ uint64_t bars[kBW][2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t rb = (uint32_t)a.d * 4u, sb_ = (uint32_t)rows * rb;
  uint8_t* ring = ring_raw + (size_t)wid * 2 * sb_;
  const int64_t nw = (int64_t)gridDim.x * kBW, gw = (int64_t)wid * gridDim.x + blockIdx.x;
  const int64_t u0 = a.U / nw * gw + min(gw, a.U % nw), u1 = u0 + a.U / nw + (gw < a.U % nw ? 1 : 0);
  if (u0 >= u1) return;
  // units of the group that starts at base
  auto group = [&](int64_t base) { return (int)min((int64_t)(base == u0 ? (wid + 1) * (32 / kBW) : 32), u1 - base); };
  if (lane == 0) {
    mbar_init(&bars[wid][0]);
    mbar_init(&bars[wid][1]);
  }
  __syncwarp();
  int64_t nb = u0;   // the stage to be requested next: rows nk .. of the group at nb
  int nk = 0;
  uint32_t asked = 0, had = 0;   // stages requested and consumed: the i-th is slot i & 1, parity (i >> 1) & 1
  auto request = [&]() {
    if (nb >= u1) return;
    const int nu = group(nb), r = min(rows, nu - nk), s = (int)(asked & 1u);
    if (lane == 0) {
      fence_proxy_async();   // the stage was last read by the generic proxy
      mbar_expect_tx(&bars[wid][s], (uint32_t)r * rb);
      bulk_g2s(ring + (size_t)s * sb_, a.p + (size_t)(nb + nk) * a.d, (uint32_t)r * rb, &bars[wid][s]);
    }
    ++asked;
    nk += r;
    if (nk == nu) {
      nk = 0;
      nb += nu;
    }
  };
  request();
  bool bulk = true;   // no wait has run out
  const bool lose = a.lose && blockIdx.x == 0;
  for (int64_t base = u0; base < u1;) {
    const int nu = group(base);
    float my_rho = 0.f;
    long long my_l1 = 0;
    for (int k0 = 0; k0 < nu; k0 += rows) {
      const int r = min(rows, nu - k0);
      if (bulk) {
        __syncwarp();   // the other stage has been read by every lane
        request();
        const bool here = mbar_wait(&bars[wid][had & 1u], (had >> 1) & 1u) && !(lose && had == 1u);
        bulk = __all_sync(0xFFFFFFFFu, here);
      }
      if (bulk) {
        rows_sums(ring + (size_t)(had & 1u) * sb_, rb, r, a.d, k0, my_rho, my_l1);
        ++had;
      } else {
        rows_sums(reinterpret_cast<const uint8_t*>(a.p + (size_t)(base + k0) * a.d), rb, r, a.d, k0, my_rho, my_l1);
      }
    }
    warp_hulls(a, base, nu, my_rho, my_l1, sk[wid], sr[wid]);
    base += nu;
  }
  for (; had != asked; ++had) mbar_wait(&bars[wid][had & 1u], (had >> 1) & 1u);   // (only after a wait that ran out)
}

// Bits of increment s of unit u (its key is not 0).
__device__ __forceinline__ int step_bits(const AllocWs& w, int s, int64_t u) {
  return c_bits[w.reach[(size_t)s * w.U + u]] - (s ? c_bits[w.reach[(size_t)(s - 1) * w.U + u]] : 0);
}

// The keys of the first digit's cut bucket into the list (as many as it holds), and their second digit's counts.
__global__ void k_alloc_compact(AllocWs w) {
  AllocState& st = *w.st;
  if (st.all_fit) return;
  const unsigned pre = (unsigned)(st.prefix >> 48);
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // whole warps walk the units together, so that every lane reaches the shuffles
  for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); u0 < w.U; u0 += stride) {
    const int64_t u = u0 + lane;
    unsigned long long key[kNS];
#pragma unroll
    for (int s = 0; s < kNS; ++s) key[s] = u < w.U ? w.keys[(size_t)s * w.U + u] : 0ull;
#pragma unroll
    for (int s = 0; s < kNS; ++s) {
      const bool take = key[s] != 0ull && (unsigned)(key[s] >> 48) == pre;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, take);
      if (!m) continue;
      const unsigned db = take ? (unsigned)step_bits(w, s, u) : 0u;
      unsigned at = 0;
      if (lane == __ffs(m) - 1) at = atomicAdd(&st.nlist, (unsigned)__popc(m));
      at = __shfl_sync(0xFFFFFFFFu, at, __ffs(m) - 1) + (unsigned)__popc(m & ((1u << lane) - 1u));
      if (take && at < (unsigned)kList) {
        w.lkey[at] = key[s];
        w.ldb[at] = (uint8_t)db;
      }
      count_digit(w.hist + kDigits, take, (unsigned)((key[s] >> 32) & 0xFFFFull), db, lane);
    }
  }
}

// A later radix pass: bits of the increments in the current bucket, by the digit at `shift`.
__global__ void k_alloc_hist(AllocWs w, int shift, int buf) {
  const AllocState& st = *w.st;
  if (st.all_fit) return;
  const int hs = shift + 16;
  const unsigned long long pre = st.prefix >> hs;
  unsigned long long* hist = w.hist + (size_t)buf * kDigits;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  if (st.nlist <= (unsigned)kList) {
    for (int64_t i = i0; i < (int64_t)st.nlist; i += stride) {
      const bool in = i + lane < (int64_t)st.nlist;
      const unsigned long long key = in ? w.lkey[i + lane] : 0ull;
      const bool take = in && (key >> hs) == pre;
      count_digit(hist, take, (unsigned)((key >> shift) & 0xFFFFull), take ? w.ldb[i + lane] : 0u, lane);
    }
    return;
  }
  for (int64_t u0 = i0; u0 < w.U; u0 += stride) {
    const int64_t u = u0 + lane;
#pragma unroll 1
    for (int s = 0; s < kNS; ++s) {
      const unsigned long long key = u < w.U ? w.keys[(size_t)s * w.U + u] : 0ull;
      const bool take = key != 0ull && (key >> hs) == pre;
      count_digit(hist, take, (unsigned)((key >> shift) & 0xFFFFull), take ? (unsigned)step_bits(w, s, u) : 0u, lane);
    }
  }
}

// Find the largest digit d with above + sum_{d' >= d} hist[d'] > budget: each block sums its 2048 digits; the
// last one to finish finds the block whose range holds the cut from the suffix sums of the totals, then scans
// that range's digits in pairs.  The other histogram is cleared for the next pass.
__global__ void __launch_bounds__(1024) k_alloc_scan(AllocWs w, long long budget, int shift, int buf, int last) {
  constexpr int kPerB = kDigits / kScanBlocks;
  __shared__ unsigned long long part[1024];
  __shared__ unsigned long long red[32];
  __shared__ unsigned long long wabove;
  __shared__ int cutb, found, final_block;
  AllocState& st = *w.st;
  const unsigned long long* hist = w.hist + (size_t)buf * kDigits;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const bool skip = st.all_fit != 0;
  {
    const int i = blockIdx.x * kPerB + 2 * t;
    unsigned long long sum = hist[i] + hist[i + 1];
    w.hist[(size_t)(buf ^ 1) * kDigits + i] = 0ull;
    w.hist[(size_t)(buf ^ 1) * kDigits + i + 1] = 0ull;
#pragma unroll
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if (lane == 0) red[wid] = sum;
  }
  __syncthreads();
  if (t == 0) {
    unsigned long long sum = 0;
    for (int i = 0; i < 32; ++i) sum += red[i];
    st.wtot[blockIdx.x] = sum;
    __threadfence();
    final_block = atomicAdd(&st.done, 1u) == kScanBlocks - 1;
    cutb = -1;
    found = 0;
  }
  __syncthreads();
  if (!final_block) return;
  __threadfence();
  const unsigned long long above = st.above;
  const unsigned long long bud = (unsigned long long)budget;
  if (wid == 0 && !skip) {
    const unsigned long long mine = __ldcg(&st.wtot[lane]);
    unsigned long long sfx = mine;   // sum of the blocks at or above this one
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long v = __shfl_down_sync(0xFFFFFFFFu, sfx, o);
      if (lane + o < 32) sfx += v;
    }
    if (above + sfx > bud && above + sfx - mine <= bud) {
      cutb = lane;
      wabove = sfx - mine;
    }
  }
  __syncthreads();
  const int cw = cutb;
  if (cw >= 0) {
    // the cut block's digits, two per thread (d0 = 2t, d1 = 2t + 1 of its range)
    const unsigned long long* hc = hist + (size_t)cw * kPerB;
    const unsigned long long h0 = hc[2 * t], h1 = hc[2 * t + 1];
    unsigned long long sfx = h0 + h1;   // inclusive suffix scan over the pairs: in the warp, then over the warps
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long v = __shfl_down_sync(0xFFFFFFFFu, sfx, o);
      if (lane + o < 32) sfx += v;
    }
    if (lane == 0) red[wid] = sfx;
    __syncthreads();
    for (int i = wid + 1; i < 32; ++i) sfx += red[i];
    part[t] = sfx;
    __syncthreads();
    const unsigned long long run = above + wabove + (t + 1 < 1024 ? part[t + 1] : 0ull);
    if (run + h0 + h1 > bud && run <= bud) {
      const int d1 = cw * kPerB + 2 * t + 1;
      if (run + h1 > bud) {
        st.prefix |= (unsigned long long)d1 << shift;
        st.above = run;
      } else {
        st.prefix |= (unsigned long long)(d1 - 1) << shift;
        st.above = run + h1;
      }
      found = 1;
    }
  }
  __syncthreads();
  if (t == 0) {
    st.done = 0;
    if (!skip) {
      if (!found) {   // only possible in the first pass: every increment fits
        st.all_fit = 1;
        st.kstar = 0ull;
      } else if (last) {
        st.kstar = st.prefix;
      }
    }
  }
}

// Units [u0, u1) of block b of the final pass.
__device__ __forceinline__ void final_range(int64_t U, int b, int64_t& u0, int64_t& u1) {
  const int64_t per = (U + kFinalBlocks - 1) / kFinalBlocks;
  u0 = min((int64_t)b * per, U);
  u1 = min(u0 + per, U);
}

// Step 3 for every unit, and its next increment for the fill.
__global__ void __launch_bounds__(256) k_alloc_final(AllocWs w, uint8_t* bits) {
  __shared__ unsigned long long best[kMaxDb + 1];
  const unsigned long long ks = w.st->kstar;
  unsigned long long used = 0;
  int64_t u0, u1;
  final_range(w.U, blockIdx.x, u0, u1);
  if (threadIdx.x <= kMaxDb) best[threadIdx.x] = 0ull;
  __syncthreads();
  for (int64_t u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
    unsigned long long key[kNS];
#pragma unroll
    for (int s = 0; s < kNS; ++s) key[s] = w.keys[(size_t)s * w.U + u];
    int t = 0;
    unsigned long long nk = key[0];   // the first key not taken
#pragma unroll
    for (int s = 0; s < kNS; ++s)
      if (t == s && key[s] > ks) {
        t = s + 1;
        nk = s + 1 < kNS ? key[s + 1] : 0ull;
      }
    const int b = t ? c_bits[w.reach[(size_t)(t - 1) * w.U + u]] : 0;
    bits[u] = (uint8_t)b;
    used += (unsigned long long)b;
    w.taken[u] = (uint8_t)t;
    const int db = nk ? c_bits[w.reach[(size_t)t * w.U + u]] - b : 0;
    w.nkey[u] = nk;
    w.ndb[u] = (uint8_t)db;
    if (nk && nk > best[db]) atomicMax(&best[db], nk);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) used += __shfl_xor_sync(0xFFFFFFFFu, used, o);
  if ((threadIdx.x & 31) == 0 && used) atomicAdd(&w.st->used, used);
  __syncthreads();
  if (threadIdx.x <= kMaxDb) w.best[(size_t)blockIdx.x * (kMaxDb + 1) + threadIdx.x] = best[threadIdx.x];
}

// The fill, one block: at most one increment per bit left.
__global__ void __launch_bounds__(1024) k_fill(AllocWs w, long long budget, uint8_t* bits) {
  __shared__ unsigned long long red[32];
  __shared__ unsigned long long row[kMaxDb + 1];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  long long left = budget - (long long)w.st->used;
  while (left > 0) {
    unsigned long long best = 0ull;   // the largest next key among those that fit
    for (int i = t; i < kFinalBlocks * (kMaxDb + 1); i += 1024) {
      const unsigned long long k = __ldcg(w.best + i);
      if (k > best && i % (kMaxDb + 1) <= left) best = k;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, best, o);
      best = v > best ? v : best;
    }
    if (lane == 0) red[wid] = best;
    if (t <= kMaxDb) row[t] = 0ull;
    __syncthreads();
    best = red[lane];
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, best, o);
      best = v > best ? v : best;
    }
    if (!best) break;   // (the same in every thread)
    const int64_t u = (int64_t)(0xFFFFFFFFull - (best & 0xFFFFFFFFull));
    if (u < 0 || u >= w.U) break;   // cannot happen: keys carry their unit
    const int db = w.ndb[u];
    left -= db;
    __syncthreads();   // every thread has read the unit's old state
    if (t == 0) {
      const int s = w.taken[u];
      const int b = c_bits[w.reach[(size_t)s * w.U + u]];
      bits[u] = (uint8_t)b;
      w.taken[u] = (uint8_t)(s + 1);
      const unsigned long long nk = s + 1 < kNS ? w.keys[(size_t)(s + 1) * w.U + u] : 0ull;
      w.nkey[u] = nk;
      w.ndb[u] = nk ? (uint8_t)(c_bits[w.reach[(size_t)(s + 1) * w.U + u]] - b) : (uint8_t)0;
    }
    __syncthreads();
    // the row of the unit's block again
    const int64_t per = (w.U + kFinalBlocks - 1) / kFinalBlocks;
    const int blk = (int)(u / per);
    int64_t u0, u1;
    final_range(w.U, blk, u0, u1);
    for (int64_t v = u0 + t; v < u1; v += 1024) {
      const unsigned long long nk = w.nkey[v];
      if (nk && nk > row[w.ndb[v]]) atomicMax(&row[w.ndb[v]], nk);
    }
    __syncthreads();
    if (t <= kMaxDb) w.best[(size_t)blk * (kMaxDb + 1) + t] = row[t];
    __threadfence_block();
    __syncthreads();
  }
}

int sms_of_current(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return e == cudaSuccess ? BITSMOE_OK : bmoe::record_cuda_error((int)e);
}

int allocate_impl(const float* p, const float* alpha, const float* beta, float gamma, int64_t U, int d,
                  const float* kappa, int64_t budget, uint8_t* bits, void* ws, size_t ws_bytes, cudaStream_t st,
                  float* phase_ms) {
  if (U < 0 || d < 1 || budget < 0 || !(gamma >= 0.f && gamma <= 1.f)) return BITSMOE_ERR_INVALID_ARG;
  if (U > 0xFFFFFFFEll || d > 16384) return BITSMOE_ERR_SHAPE;
  if (U == 0) return BITSMOE_OK;
  if (!p || !alpha || !beta || !kappa || !bits || !ws) return BITSMOE_ERR_INVALID_ARG;
  if ((uintptr_t)p % 16 || (uintptr_t)alpha % 4 || (uintptr_t)beta % 4 || (uintptr_t)ws % 256)
    return BITSMOE_ERR_ALIGNMENT;
  size_t off[kParts];
  if (ws_bytes < ws_layout(U, off)) return BITSMOE_ERR_WORKSPACE_TOO_SMALL;
  int sms = 0;
  int rc = sms_of_current(&sms);
  if (rc) return rc;
  uint8_t* wb = static_cast<uint8_t*>(ws);
  AllocWs w{reinterpret_cast<AllocState*>(wb + off[0]), reinterpret_cast<unsigned long long*>(wb + off[1]),
            reinterpret_cast<unsigned long long*>(wb + off[2]), wb + off[3], wb + off[4],
            reinterpret_cast<unsigned long long*>(wb + off[5]), wb + off[6],
            reinterpret_cast<unsigned long long*>(wb + off[7]), wb + off[8],
            reinterpret_cast<unsigned long long*>(wb + off[9]), U};
  cudaEvent_t ev[4] = {};
  if (phase_ms) {
    for (auto& e : ev)
      if (cudaEventCreate(&e) != cudaSuccess) return bmoe::record_cuda_error((int)cudaGetLastError());
  }
  auto fail = [&](cudaError_t e) {
    if (phase_ms)
      for (auto& x : ev) cudaEventDestroy(x);
    return bmoe::record_cuda_error((int)e);
  };
  cudaError_t e = cudaMemsetAsync(wb + off[0], 0, off[2], st);   // state and histograms
  if (e != cudaSuccess) return fail(e);
  if (phase_ms) cudaEventRecord(ev[0], st);
  CostArgs ca{p, alpha, beta, gamma, kappa[0], kappa[1], kappa[2], U, d, w, bmoe::debug_skip_arrival()};
  const int64_t groups = (U + 31) / 32;
  const uint32_t row = (uint32_t)d * 4u;
  if (d % 4 == 0 && row <= kRowMax) {
    const int rows = (int)std::min<uint32_t>(32u, kStageMax / row);
    const size_t smem = (size_t)kBW * 2 * rows * row;
    e = cudaFuncSetAttribute(k_alloc_cost_bulk, cudaFuncAttributeMaxDynamicSharedMemorySize, kBW * 2 * (int)kStageMax);
    if (e != cudaSuccess) return fail(e);
    const int64_t blocks = std::min<int64_t>((U + 4 * kBW - 1) / (4 * kBW), sms);   // four units a warp or more
    k_alloc_cost_bulk<<<(unsigned)blocks, kBW * 32, smem, st>>>(ca, rows);
  } else {
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_alloc_cost, kAW * 32, 0);
    if (e != cudaSuccess) return fail(e);
    const int64_t blocks = std::min<int64_t>((groups + kAW - 1) / kAW, (int64_t)sms * std::max(per_sm, 1));
    k_alloc_cost<<<(unsigned)blocks, kAW * 32, 0, st>>>(ca);
  }
  if (phase_ms) cudaEventRecord(ev[1], st);
  const unsigned ub = (unsigned)std::min<int64_t>((U + 255) / 256, (int64_t)sms * 8);
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 48 - 16 * pass, buf = pass & 1;
    if (pass == 1) k_alloc_compact<<<ub, 256, 0, st>>>(w);
    else if (pass > 1) k_alloc_hist<<<std::min(ub, (unsigned)kList / 256), 256, 0, st>>>(w, shift, buf);
    k_alloc_scan<<<kScanBlocks, 1024, 0, st>>>(w, (long long)budget, shift, buf, pass == 3);
  }
  k_alloc_final<<<kFinalBlocks, 256, 0, st>>>(w, bits);
  if (phase_ms) cudaEventRecord(ev[2], st);
  k_fill<<<1, 1024, 0, st>>>(w, (long long)budget, bits);
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(e);
  if (phase_ms) {
    cudaEventRecord(ev[3], st);
    e = cudaEventSynchronize(ev[3]);
    if (e != cudaSuccess) return fail(e);
    for (int i = 0; i < 3; ++i) cudaEventElapsedTime(&phase_ms[i], ev[i], ev[i + 1]);
    for (auto& x : ev) cudaEventDestroy(x);
  }
  return BITSMOE_OK;
}

}  // namespace

extern "C" int bitsmoe_projection_budget(int64_t E, int64_t n, int64_t m, int64_t beq_num, int64_t beq_den,
                                         int64_t* out) {
  // floor(E n b_eq - 16 n^2 / m), b_eq = num / den, in exact int64 arithmetic
  if (!out || E < 1 || n < 1 || m < 1 || beq_den < 1 || beq_num < 0) return BITSMOE_ERR_INVALID_ARG;
  if (E > (1 << 20) || n > (1 << 20) || m > (1 << 24) || beq_num > (1 << 16) || beq_den > (1 << 16))
    return BITSMOE_ERR_SHAPE;
  // a / den - b / m with a = E n num (< 2^56), b = 16 n^2 (< 2^45): whole parts q1 - q2, and
  // the fractional parts r1 / den - r2 / m in (-1, 1) take one more off when negative
  // (r1 m and r2 den stay below 2^40)
  const int64_t a = E * n * beq_num, b = 16 * n * n;
  const int64_t q1 = a / beq_den, r1 = a % beq_den, q2 = b / m, r2 = b % m;
  *out = q1 - q2 - (r1 * m < r2 * beq_den ? 1 : 0);
  return BITSMOE_OK;
}

extern "C" size_t bitsmoe_allocate_workspace_bytes(int64_t U) {
  if (U < 0 || U > 0xFFFFFFFEll) return 0;
  size_t off[kParts];
  return ws_layout(U, off);
}

extern "C" int bitsmoe_allocate_bits(const float* p, const float* alpha, const float* beta, float gamma, int64_t U,
                                     int d, const float* kappa, int64_t budget, uint8_t* bits, void* ws,
                                     size_t ws_bytes, void* stream) {
  return allocate_impl(p, alpha, beta, gamma, U, d, kappa, budget, bits, ws, ws_bytes,
                       static_cast<cudaStream_t>(stream), nullptr);
}

extern "C" int bitsmoe_profile_allocate_bits(const float* p, const float* alpha, const float* beta, float gamma,
                                             int64_t U, int d, const float* kappa, int64_t budget, uint8_t* bits,
                                             void* ws, size_t ws_bytes, void* stream, float phase_ms[3]) {
  if (!phase_ms) return BITSMOE_ERR_INVALID_ARG;
  return allocate_impl(p, alpha, beta, gamma, U, d, kappa, budget, bits, ws, ws_bytes,
                       static_cast<cudaStream_t>(stream), phase_ms);
}
