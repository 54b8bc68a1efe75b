// Importance beta of every spectral unit, from calibration tokens (the input of the bit
// allocation), on the GPU.
//
// The paper weighs the loss of quantising a unit by how strongly the calibration
// activations excite it (Sec. "Shared-basis Spectral Decomposition", the reconstruction
// loss; appendix Eqs. app_affinity_gram, app_beta_def, app_down_beta_approx,
// app_unified_beta_def):
//
//   H_e    = X Diag(g_e) X^T          activation metric of expert e (g_e: the tokens'
//                                     routing affinities to e, their gate weights)
//   beta   = phi_k^T H_e phi_k        gate, up   (phi_k: the shared input basis)
//          = sum_t g_{t,e} (phi_k^T x_t)^2 = sum_t g_{t,e} z_{k,t}^2
//   beta   = p_k^T H_e p_k            down       (p_k: the expert's spectral vector, H_e
//                                     over the expert's SwiGLU outputs h_t)
//          = sum_t g_{t,e} (p_k^T h_{t,e})^2
//
// all on the float factors of the decomposition, before anything is quantised.  Steps:
//
//   k_imp_route    one block per token: the k largest logits (ties to the lower index),
//                  softmax over them -> the dense affinity matrix G (T x E) and the tokens
//                  of each expert
//   k_imp_lists    each expert's tokens in token order with their gate weights, one block
//                  an expert
//   k_gemm<Z>      Z_h = Phi_h^T X for h = gate, up            (stored T x n)
//   k_gemm<BGU>    beta_h[e, k] = sum_t Z_h[k, t]^2 G[t, e]    (a contraction over tokens)
//   k_gemm<AG>     a_g = P_g,e (alpha_g,e * Z_g[:, tokens of e])          per expert
//   k_gemm<AUH>    h   = SiLU(a_g) * (P_u,e (alpha_u,e * Z_u[:, tokens]))  per expert
//   k_gemm<DN>     beta_dn[e, k] = sum_j g_j (P_dn,e^T h)[k, j]^2          per expert
//
// Every contraction is fp32 on the CUDA cores: the factors are fp32 and the result is
// compared with an fp64 oracle at a tight tolerance, which bf16 tensor-core operands would
// not meet.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"

namespace {

constexpr int kTM = 128, kTN = 64, kTK = 16;  // output tile and K step
constexpr int kGT = 256;                      // threads of a GEMM block (16 x 16, 8 x 4 outputs each)

enum GemmKind { kZ = 0, kBGU = 1, kAG = 2, kAUH = 3, kDN = 4 };

struct ImpArgs {
  const uint16_t* x;       // [T][D] bf16
  const float* logits;     // [T][E]
  const float* phi[2];     // gate, up: [D][n]
  const float* alpha[2];   // gate, up: [E][n]
  const float* P[3];       // gate, up, down: [E][I][n]
  float* beta;             // [3][E][n]
  int T, D, E, I, n, k;
  // workspace
  float* G;                // [T][E] affinities
  float* z;                // [2][T][n]
  int* cnt;                // [E] tokens per expert
  int* off;                // [E + 1] start of each expert's list (exclusive scan of cnt)
  int* toff;               // [E + 1] its first column tile (exclusive scan of the lists' tiles of kTN)
  int* tok;                // [T * k] token of each (expert, slot), grouped by expert
  float* tw;               // [T * k] its gate weight
  float* ag;               // [I][T * k] a_g, then h, by the expert's columns
  int* status;
};

__device__ __forceinline__ float bf16f(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }

// ---------------------------------------------------------------------------
// Routing of every token (one block each), the same rule as the forward.
// ---------------------------------------------------------------------------
__global__ void k_imp_route(ImpArgs a) {
  extern __shared__ uint32_t keys[];   // [E], then sel_e [k], sel_w [k]
  int* sel_e = reinterpret_cast<int*>(keys + a.E);
  float* sel_w = reinterpret_cast<float*>(sel_e + a.k);
  const int t = blockIdx.x, tid = threadIdx.x;
  for (int i = tid; i < a.E; i += blockDim.x) {
    keys[i] = order_key(a.logits[(size_t)t * a.E + i]);
    a.G[(size_t)t * a.E + i] = 0.f;
  }
  __syncthreads();
  for (int i = tid; i < a.E; i += blockDim.x) {
    const uint32_t key = keys[i];
    int rank = 0;
    for (int f = 0; f < a.E; ++f) {
      const uint32_t o = keys[f];
      rank += (o > key) | ((o == key) & (f < i));
    }
    if (rank < a.k) {
      sel_e[rank] = i;
      sel_w[rank] = key ? __uint_as_float((key & 0x80000000u) ? (key & 0x7FFFFFFFu) : ~key)
                        : __int_as_float(0x7FC00000);
    }
  }
  __syncthreads();
  if (tid < 32) {
    const float m = sel_w[0];
    const float ev = tid < a.k ? expf(sel_w[tid] - m) : 0.f;
    float sum = ev;
#pragma unroll
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if (tid < a.k) {
      const float w = ev * (1.f / sum);
      a.G[(size_t)t * a.E + sel_e[tid]] = w;
      if (w != 0.f) atomicAdd(a.cnt + sel_e[tid], 1);   // the lists keep the tokens with g > 0
    }
  }
}

// Token lists per expert, one block an expert: its start by a prefix over the counts, then
// its tokens in token order (each thread a contiguous part of the tokens).  One block for
// all experts, a thread an expert, read G one token after another.
constexpr int kLT = 256;
__global__ void __launch_bounds__(kLT) k_imp_lists(ImpArgs a) {
  __shared__ int red[3][kLT / 32];
  const int e = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int pre = 0, pret = 0;   // lists and tiles of the experts before
  for (int i = tid; i < e; i += kLT) {
    const int c = a.cnt[i];
    pre += c;
    pret += (c + kTN - 1) / kTN;
  }
  const int per = (a.T + kLT - 1) / kLT, t0 = min(a.T, tid * per), t1 = min(a.T, t0 + per);
  int c = 0;
  for (int t = t0; t < t1; ++t) c += a.G[(size_t)t * a.E + e] != 0.f;
  int ci = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, ci, o);
    if (lane >= o) ci += v;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    pre += __shfl_xor_sync(0xFFFFFFFFu, pre, o);
    pret += __shfl_xor_sync(0xFFFFFFFFu, pret, o);
  }
  if (lane == 31) red[0][wid] = ci;
  if (lane == 0) {
    red[1][wid] = pre;
    red[2][wid] = pret;
  }
  __syncthreads();
  int base = 0, tiles = 0, w = ci - c;
  for (int i = 0; i < kLT / 32; ++i) {
    base += red[1][i];
    tiles += red[2][i];
    if (i < wid) w += red[0][i];
  }
  if (tid == 0) {
    a.off[e] = base;
    a.toff[e] = tiles;
    if (e == a.E - 1) {
      const int n = a.cnt[e];
      a.off[a.E] = base + n;
      a.toff[a.E] = tiles + (n + kTN - 1) / kTN;
    }
  }
  w += base;
  for (int t = t0; t < t1; ++t) {
    const float g = a.G[(size_t)t * a.E + e];
    if (g != 0.f) {
      a.tok[w] = t;
      a.tw[w] = g;
      ++w;
    }
  }
}

// ---------------------------------------------------------------------------
// fp32 contractions C = A B (M x N over K) with the operands of each step read in place
// (transposed, gathered, squared or scaled on load) and the step's epilogue.
//
// Bound by the fp32 FMA pipe.  A 128 x 64 tile a block, 8 x 4 outputs a thread, multiplied
// in row pairs (fma.f32x2: two products an issue slot, so the shared-memory reads and the
// operand loads issue beside the FMAs); the next K step's operands are loaded while the
// current one is multiplied, into the other of two buffers.  64 columns: an expert's token
// list is cut into tiles of 64, its last tile computed 32 wide when no more are left.
// Qwen3-shaped layer, 2048 tokens: 64 x 64 tiles of 4 x 4 outputs, single-buffered with
// z gathered token by token, took 9.8 ms (19 TFLOP/s).
// ---------------------------------------------------------------------------
template <int KIND>
__host__ __device__ constexpr bool per_expert() { return KIND == kAG || KIND == kAUH || KIND == kDN; }
// whether consecutive kk are contiguous in memory (then a thread loads four kk of a row)
template <int KIND>
__host__ __device__ constexpr bool a_k_contig() { return KIND == kAG || KIND == kAUH; }
template <int KIND>
__host__ __device__ constexpr bool b_k_contig() { return KIND == kZ || KIND == kAG || KIND == kAUH; }

struct Op {
  int M, N, K, e, col0;   // e: expert (or projection); col0: first column of the expert's token list
};

__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// Four consecutive floats at p, of which `left` are inside (VEC: p 16-byte aligned when left >= 4)
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* p, int left) {
  if (VEC && left >= 4) return __ldg(reinterpret_cast<const float4*>(p));
  float4 v;
  v.x = left > 0 ? __ldg(p) : 0.f;
  v.y = left > 1 ? __ldg(p + 1) : 0.f;
  v.z = left > 2 ? __ldg(p + 2) : 0.f;
  v.w = left > 3 ? __ldg(p + 3) : 0.f;
  return v;
}

// Chunk q (of two) of this thread's part of the A tile at K step k0: four m of one kk, or four kk of one m.
template <int KIND, bool VEC>
__device__ __forceinline__ float4 a_load(const ImpArgs& a, const Op& o, int m0, int k0, int q) {
  const int lin = threadIdx.x + kGT * q;
  if (a_k_contig<KIND>()) {
    const int m = m0 + (lin >> 2), kk = k0 + (lin & 3) * 4;
    if (m >= o.M) return make_float4(0.f, 0.f, 0.f, 0.f);
    return load4<VEC>(a.P[KIND == kAG ? 0 : 1] + ((size_t)o.e * a.I + m) * a.n + kk, o.K - kk);
  }
  const int kk = k0 + (lin >> 5), m = m0 + (lin & 31) * 4;
  if (kk >= o.K) return make_float4(0.f, 0.f, 0.f, 0.f);
  if (KIND == kZ) return load4<VEC>(a.phi[o.e] + (size_t)kk * a.n + m, o.M - m);                     // Phi_h^T
  if (KIND == kDN) return load4<VEC>(a.P[2] + ((size_t)o.e * a.I + kk) * a.n + m, o.M - m);           // P_dn^T
  float4 v = load4<VEC>(a.z + ((size_t)o.e * a.T + kk) * a.n + m, o.M - m);                           // z^2
  v.x *= v.x;
  v.y *= v.y;
  v.z *= v.z;
  v.w *= v.w;
  return v;
}
template <int KIND>
__device__ __forceinline__ void a_store(float (*As)[kTM + 4], int q, const float4& v) {
  const int lin = threadIdx.x + kGT * q;
  if (a_k_contig<KIND>()) {
    const int m = lin >> 2, kk = (lin & 3) * 4;
    As[kk][m] = v.x;
    As[kk + 1][m] = v.y;
    As[kk + 2][m] = v.z;
    As[kk + 3][m] = v.w;
  } else {
    *reinterpret_cast<float4*>(&As[lin >> 5][(lin & 31) * 4]) = v;
  }
}

// This thread's four elements of the B tile: four kk of column j (row: this column's row of z or x), or four
// columns of one kk.
template <int KIND, bool VEC>
__device__ __forceinline__ float4 b_load(const ImpArgs& a, const Op& o, int j0, int k0, size_t row) {
  const size_t TK = (size_t)a.T * a.k;
  if (b_k_contig<KIND>()) {
    const int j = j0 + (threadIdx.x >> 2), kk = k0 + (threadIdx.x & 3) * 4, left = o.K - kk;
    if (j >= o.N || left <= 0) return make_float4(0.f, 0.f, 0.f, 0.f);
    if (KIND == kZ) {   // X^T
      const uint16_t* xp = a.x + row * a.D + kk;
      if (VEC && left >= 4) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(xp));
        return make_float4(bf16lo(w.x), bf16hi(w.x), bf16lo(w.y), bf16hi(w.y));
      }
      return make_float4(bf16f(xp[0]), left > 1 ? bf16f(xp[1]) : 0.f, left > 2 ? bf16f(xp[2]) : 0.f,
                         left > 3 ? bf16f(xp[3]) : 0.f);
    }
    const int h = KIND == kAG ? 0 : 1;
    const float4 z = load4<VEC>(a.z + ((size_t)h * a.T + row) * a.n + kk, left);
    const float4 al = load4<VEC>(a.alpha[h] + (size_t)o.e * a.n + kk, left);
    return make_float4(al.x * z.x, al.y * z.y, al.z * z.z, al.w * z.w);
  }
  const int kk = k0 + (threadIdx.x >> 4), j = j0 + (threadIdx.x & 15) * 4;
  if (kk >= o.K) return make_float4(0.f, 0.f, 0.f, 0.f);
  const float* p = KIND == kBGU ? a.G + (size_t)kk * a.E + j : a.ag + (size_t)kk * TK + o.col0 + j;   // G, h
  return load4<false>(p, o.N - j);   // (a list starts anywhere in its row)
}
template <int KIND>
__device__ __forceinline__ void b_store(float (*Bs)[kTN + 4], const float4& v) {
  if (b_k_contig<KIND>()) {
    const int j = threadIdx.x >> 2, kk = (threadIdx.x & 3) * 4;
    Bs[kk][j] = v.x;
    Bs[kk + 1][j] = v.y;
    Bs[kk + 2][j] = v.z;
    Bs[kk + 3][j] = v.w;
  } else {
    *reinterpret_cast<float4*>(&Bs[threadIdx.x >> 4][(threadIdx.x & 15) * 4]) = v;
  }
}

// One output tile, TN (4 or 2) columns a thread: 16 TN columns from j0.
template <int KIND, bool VEC, int TN>
__device__ __forceinline__ void tile(const ImpArgs& a, const Op& o, int m0, int j0, float (*As)[kTK][kTM + 4],
                                     float (*Bs)[kTK][kTN + 4]) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  size_t row = 0;   // the token of this thread's column of B
  if (b_k_contig<KIND>()) {
    const int j = min(j0 + (tid >> 2), o.N - 1);
    row = KIND == kZ ? (size_t)j : (size_t)a.tok[o.col0 + j];
  }
  unsigned long long acc[4][TN];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < TN; ++c) acc[r][c] = 0ull;
  float4 av[2], bv;
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) av[q] = a_load<KIND, VEC>(a, o, m0, k0, q);
    bv = b_load<KIND, VEC>(a, o, j0, k0, row);
  };
  auto put = [&](int s) {
#pragma unroll
    for (int q = 0; q < 2; ++q) a_store<KIND>(As[s], q, av[q]);
    b_store<KIND>(Bs[s], bv);
  };
  fetch(0);
  put(0);
  __syncthreads();
  for (int k0 = 0, s = 0; k0 < o.K; k0 += kTK, s ^= 1) {
    const bool more = k0 + kTK < o.K;
    if (more) fetch(k0 + kTK);
#pragma unroll
    for (int kk = 0; kk < kTK; ++kk) {
      const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(&As[s][kk][ty * 8]);
      const ulonglong2 p1 = *reinterpret_cast<const ulonglong2*>(&As[s][kk][ty * 8 + 4]);
      const unsigned long long ar[4] = {p0.x, p0.y, p1.x, p1.y};
      float br[TN];
      if (TN == 4) {
        const float4 w = *reinterpret_cast<const float4*>(&Bs[s][kk][tx * 4]);
        br[0] = w.x;
        br[1] = w.y;
        br[TN - 2] = w.z;
        br[TN - 1] = w.w;
      } else {
        const float2 w = *reinterpret_cast<const float2*>(&Bs[s][kk][tx * 2]);
        br[0] = w.x;
        br[1] = w.y;
      }
#pragma unroll
      for (int c = 0; c < TN; ++c) {
        const unsigned long long bb = pack2(br[c], br[c]);
#pragma unroll
        for (int r = 0; r < 4; ++r) fma2(acc[r][c], ar[r], bb);
      }
    }
    if (more) put(s ^ 1);
    __syncthreads();
  }
  // epilogues
  const size_t TK = (size_t)a.T * a.k;
  float v[8][TN];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < TN; ++c) {
      const float2 p = unpack2(acc[r][c]);
      v[2 * r][c] = p.x;
      v[2 * r + 1][c] = p.y;
    }
  const int gm0 = m0 + ty * 8, gj0 = j0 + tx * TN;
  if constexpr (KIND == kDN) {
    // beta_dn[e, m] += sum_j g_j acc(m, j)^2: the 16 threads of a row group add their columns
    float gw[TN];
#pragma unroll
    for (int c = 0; c < TN; ++c) gw[c] = gj0 + c < o.N ? a.tw[o.col0 + gj0 + c] : 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < TN; ++c)
        if (gj0 + c < o.N) s = fmaf(gw[c], v[r][c] * v[r][c], s);
#pragma unroll
      for (int sh = 8; sh; sh >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, sh);
      if (tx == 0 && gm0 + r < o.M && s != 0.f) atomicAdd(a.beta + ((size_t)2 * a.E + o.e) * a.n + gm0 + r, s);
    }
  } else {
#pragma unroll
  for (int c = 0; c < TN; ++c) {
    const int gj = gj0 + c;
    if (gj >= o.N) continue;
    if (KIND == kZ || KIND == kBGU) {   // rows contiguous
      float* p = KIND == kZ ? a.z + ((size_t)o.e * a.T + gj) * a.n + gm0 : a.beta + ((size_t)o.e * a.E + gj) * a.n + gm0;
#pragma unroll
      for (int r = 0; r < 8; r += 4) {
        if (VEC && gm0 + r + 4 <= o.M && KIND == kZ) {
          *reinterpret_cast<float4*>(p + r) = make_float4(v[r][c], v[r + 1][c], v[r + 2][c], v[r + 3][c]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (gm0 + r + q < o.M) p[r + q] = v[r + q][c];
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if (gm0 + r >= o.M) continue;
        float* hp = a.ag + (size_t)(gm0 + r) * TK + o.col0 + gj;
        if (KIND == kAG) {
          *hp = v[r][c];
        } else {   // h = SiLU(a_g) * a_u
          const float g = *hp;
          *hp = g / (1.f + expf(-g)) * v[r][c];
        }
      }
    }
  }
  }
}

// grid: x column tiles (of all experts' lists: the expert by its first tile), y row tiles, z projection
template <int KIND, bool VEC>
__global__ void __launch_bounds__(kGT, 2) k_gemm(ImpArgs a) {
  __shared__ __align__(16) float As[2][kTK][kTM + 4];
  __shared__ __align__(16) float Bs[2][kTK][kTN + 4];
  Op o;
  int jt = blockIdx.x;
  o.col0 = 0;
  if (per_expert<KIND>()) {
    if (jt >= a.toff[a.E]) return;
    int lo = 0, hi = a.E;   // the last expert whose first tile is at or before jt: one with tiles
    while (hi - lo > 1) {
      const int md = (lo + hi) >> 1;
      if (a.toff[md] <= jt) lo = md;
      else hi = md;
    }
    o.e = lo;
    jt -= a.toff[lo];
    o.col0 = a.off[lo];
    o.N = a.off[lo + 1] - o.col0;
    o.M = KIND == kDN ? a.n : a.I;
    o.K = KIND == kDN ? a.I : a.n;
  } else {
    o.e = blockIdx.z;
    o.M = a.n;
    o.N = KIND == kZ ? a.T : a.E;
    o.K = KIND == kZ ? a.D : a.T;
  }
  const int m0 = blockIdx.y * kTM, j0 = jt * kTN;
  if (o.N - j0 > kTN / 2) tile<KIND, VEC, 4>(a, o, m0, j0, As, Bs);
  else tile<KIND, VEC, 2>(a, o, m0, j0, As, Bs);
}

template <bool VEC>
void run_gemms(const ImpArgs& a, cudaStream_t st) {
  auto up = [](int64_t v, int d) { return (unsigned)((v + d - 1) / d); };
  // column tiles of all lists: at most one partial tile an expert
  const unsigned lists = (unsigned)((int64_t)a.T * a.k / kTN + a.E);
  k_gemm<kZ, VEC><<<dim3(up(a.T, kTN), up(a.n, kTM), 2), kGT, 0, st>>>(a);
  k_gemm<kBGU, VEC><<<dim3(up(a.E, kTN), up(a.n, kTM), 2), kGT, 0, st>>>(a);
  k_gemm<kAG, VEC><<<dim3(lists, up(a.I, kTM)), kGT, 0, st>>>(a);
  k_gemm<kAUH, VEC><<<dim3(lists, up(a.I, kTM)), kGT, 0, st>>>(a);
  k_gemm<kDN, VEC><<<dim3(lists, up(a.n, kTM)), kGT, 0, st>>>(a);
}

}  // namespace

namespace bmoe {

struct ImpLayout {
  size_t G, z, cnt, off, toff, tok, tw, ag, total;
};
static ImpLayout imp_layout(int64_t T, int E, int I, int n, int k) {
  ImpLayout l;
  size_t o = 0;
  auto put = [&](size_t bytes) {
    const size_t r = o;
    o = (o + bytes + 255) / 256 * 256;
    return r;
  };
  l.G = put((size_t)T * E * 4);
  l.z = put((size_t)2 * n * T * 4);
  l.cnt = put((size_t)E * 4);
  l.off = put(((size_t)E + 1) * 4);
  l.toff = put(((size_t)E + 1) * 4);
  l.tok = put((size_t)T * k * 4);
  l.tw = put((size_t)T * k * 4);
  l.ag = put((size_t)I * T * k * 4);
  l.total = o;
  return l;
}

}  // namespace bmoe

extern "C" {

size_t bitsmoe_importance_workspace_bytes(int64_t T, int E, int I, int n, int top_k) {
  if (T < 0 || E < 1 || I < 1 || n < 1 || top_k < 1 || top_k > std::min(E, 32)) return 0;
  return bmoe::imp_layout(T, E, I, n, top_k).total;
}

int bitsmoe_importance(const void* x, const float* logits, int64_t T, int D, int E, int I, int n, int top_k,
                       const float* const basis[2], const float* const alpha[2], const float* const factor[3],
                       float* beta, void* ws, size_t ws_bytes, void* stream) {
  if (T < 0 || D < 1 || E < 1 || E > 1024 || I < 1 || n < 1 || top_k < 1 || top_k > std::min(E, 32))
    return BITSMOE_ERR_INVALID_ARG;
  if (T > (1 << 24) || (int64_t)I * T * top_k > (1ll << 31)) return BITSMOE_ERR_SHAPE;
  if (!basis || !alpha || !factor || !beta || !ws) return BITSMOE_ERR_INVALID_ARG;
  if (!basis[0] || !basis[1] || !alpha[0] || !alpha[1] || !factor[0] || !factor[1] || !factor[2])
    return BITSMOE_ERR_INVALID_ARG;
  if (T > 0 && (!x || !logits)) return BITSMOE_ERR_INVALID_ARG;
  const bmoe::ImpLayout l = bmoe::imp_layout(T, E, I, n, top_k);
  if (ws_bytes < l.total) return BITSMOE_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  auto fail = [](cudaError_t e) { return bmoe::record_cuda_error((int)e); };
  cudaError_t e = cudaMemsetAsync(beta, 0, (size_t)3 * E * n * 4, st);
  if (e != cudaSuccess) return fail(e);
  if (T == 0) return BITSMOE_OK;
  uint8_t* w = static_cast<uint8_t*>(ws);
  ImpArgs a;
  a.x = static_cast<const uint16_t*>(x);
  a.logits = logits;
  for (int h = 0; h < 2; ++h) {
    a.phi[h] = basis[h];
    a.alpha[h] = alpha[h];
  }
  for (int h = 0; h < 3; ++h) a.P[h] = factor[h];
  a.beta = beta;
  a.T = (int)T; a.D = D; a.E = E; a.I = I; a.n = n; a.k = top_k;
  a.G = reinterpret_cast<float*>(w + l.G);
  a.z = reinterpret_cast<float*>(w + l.z);
  a.cnt = reinterpret_cast<int*>(w + l.cnt);
  a.off = reinterpret_cast<int*>(w + l.off);
  a.toff = reinterpret_cast<int*>(w + l.toff);
  a.tok = reinterpret_cast<int*>(w + l.tok);
  a.tw = reinterpret_cast<float*>(w + l.tw);
  a.ag = reinterpret_cast<float*>(w + l.ag);
  a.status = nullptr;
  if ((e = cudaMemsetAsync(a.cnt, 0, (size_t)E * 4, st)) != cudaSuccess) return fail(e);
  const size_t rsm = ((size_t)E + 2 * top_k) * 4;
  if (rsm > 48 * 1024) return BITSMOE_ERR_SHAPE;
  k_imp_route<<<(unsigned)T, 256, rsm, st>>>(a);
  k_imp_lists<<<(unsigned)E, kLT, 0, st>>>(a);
  // rows of the factors, bases, energies, z and x that a thread may read four elements at a time
  uintptr_t al = reinterpret_cast<uintptr_t>(a.z) | reinterpret_cast<uintptr_t>(x);
  for (int h = 0; h < 2; ++h) al |= reinterpret_cast<uintptr_t>(basis[h]) | reinterpret_cast<uintptr_t>(alpha[h]);
  for (int h = 0; h < 3; ++h) al |= reinterpret_cast<uintptr_t>(factor[h]);
  if (n % 4 == 0 && D % 4 == 0 && (al & 15) == 0) run_gemms<true>(a, st);
  else run_gemms<false>(a, st);
  e = cudaGetLastError();
  return e == cudaSuccess ? BITSMOE_OK : fail(e);
}

}  // extern "C"
